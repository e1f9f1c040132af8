// fgmres_res.cu -- the flexible GMRES solve of fgmres.cu on a resident team
// (resident.cuh): the FP32 matrix in registers, the Arnoldi basis of the
// CTA's own rows, its share of the level-0 transfer operators and the coarse
// operator in shared memory.  The method is the same -- FP64 residual and
// update around an FP32 Arnoldi process, classical Gram-Schmidt with one
// reorthogonalisation, one multigrid cycle per step -- with these changes of
// the step's schedule:
//
//   * z_{j+1} starts from u_{j+1} = w - V h, the vector after the first
//     orthogonalisation pass, scaled by 1 / h_{j+1,j}, instead of from
//     v_{j+1}: flexible GMRES takes any direction, and the two differ by the
//     second pass's corrections (FP32 rounding).  u_{j+1} is published by the
//     exchange that reduces the second pass, so v_{j+1} needs none.
//   * the level-0 smoother z_0 = 2 W b - W A (W b) uses the matrix in
//     registers instead of a second one (S_0 = 2 W - W A W).
//   * below level 1 the cycle is one dense matrix y_1 = B b_1 where level 1
//     is small (B = S_1 + sum_l Q_l Rh_l of the composed cycle, or the
//     coarsest inverse; RES_DENSE_N rows: 16 MB, 71 KB a CTA at 1 610 rows):
//     one phase and one exchange where the composed cycle has two.  Larger
//     level-1 problems run the composed cycle's two phases.
//
// Exchanges a step: b_1; y_1 (two without the dense operator); z_j; the two
// reductions -- five, against seven.
//
// Measured on GB300, a whole outer iteration (momentum included) with the
// streaming and with the resident p' solve: cavity 200^2 (q = 30, 140 steps)
// 8.4 -> 6.4 ms, cylinder 147 827 (q = 20, 110 steps) 11.6 -> 9.5 ms,
// Kovasznay 50^2 (one cluster, 115 steps) 4.9 -> 3.1 ms.
#include "fgmres.cuh"
#include "resident.cuh"

namespace rbffd {

namespace {

constexpr int LDH = FG_MAXM + 1;
constexpr int MAXV = FG_MAXM + 1;   // vectors V of a restart that are kept
constexpr int MAXR1 = 256;          // level-1 rows a CTA may own

struct FgResArgs {
  FgmresArgs f;
  ResPlan res;
  double omega;           // level 0's smoothing weight
  int n1;                 // level 1's rows
  AmgCsrT<float> R0, P0;  // level 0's R~ and P~
  AmgCsrT<float> S1;      // level 1's S, with the composed cycle's operators:
  AmgCompT<float> C;      //   used when B is null
  const float *B;         // dense coarse operator n1 x ldb, or null
  int ldb;
  float *b1, *y1;         // level-1 vectors
  float *u;               // n
  // shared-memory layout, in bytes from the dynamic base (host: fg_layout)
  int o_list, o_w, o_work, o_c1, o_v, o_b, o_r, o_p;
  int kv, ldv;            // basis vectors kept in shared memory, their stride
  int rcap, pcap;         // entries of the R~ and P~ slabs kept (0: read from L2)
  int bres;               // 1: B's rows kept
};

struct FgState {
  double bnorm, beta, scale, relres;
  float gtol;  // |g_{j+1}| at which the restart's residual estimate meets the tolerance
  int it, restarts, state, k, stop;
};

// Products of one step summed over the team: warp d < D holds its CTA's
// part; totals to tot[0..D).
__device__ __forceinline__ bool products(res::Team &t, float s, int D, float *tot, float *cpart,
                                         void *gpart) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned int ep = t.epoch;  // of this exchange, before its barrier
  auto at = [&](int v, int b) {
    return reinterpret_cast<float *>(static_cast<char *>(gpart) + res_slot(ep, v, b, 4));
  };
  if (w < D) {
    if (t.nb == 1) {
      if (lane == 0) tot[w] = s;
    } else if (t.cluster) {
      float *dst = cpart + res_cluster_slot(ep, 32, w, t.lb);
      if (lane < t.nb) *res::cg::this_cluster().map_shared_rank(dst, lane) = s;
    } else if (lane == 0) {
      *at(w, t.lb) = s;
    }
  }
  const bool ok = res::team_barrier(t);
  if (t.nb > 1) {
    if (w < D) {
      float r = 0.0f;
      if (t.cluster) {
        if (lane < t.nb) r = cpart[res_cluster_slot(ep, 32, w, lane)];
      } else {
        float p[RES_MAXB / 32];
#pragma unroll
        for (int u = 0; u < RES_MAXB / 32; ++u)
          p[u] = lane + 32 * u < t.nb ? __ldcg(at(w, lane + 32 * u)) : 0.0f;
#pragma unroll
        for (int u = 0; u < RES_MAXB / 32; ++u) r += p[u];
      }
      r = res::warp_total(r);
      if (lane == 0) tot[w] = r;
    }
    __syncthreads();
  }
  return ok;
}

template <int E>
__global__ void __launch_bounds__(RES_NT, 1) k_fgmres_res(const __grid_constant__ FgResArgs A) {
  __shared__ float H[LDH * FG_MAXM];
  __shared__ float cs[FG_MAXM], sn[FG_MAXM], g[FG_MAXM + 1], y[FG_MAXM];
  __shared__ float tot[32], cpart[2 * 32 * RES_CLUSTER];
  __shared__ double tot64[2], wsum64[2 * 32], cpart64[2 * 2 * RES_CLUSTER];
  __shared__ FgState st;
  __shared__ float rowpart[32];
  __shared__ int rptr[MAXR1 + 1];
  extern __shared__ __align__(16) unsigned char dyn[];
  const FgmresArgs &F = A.f;
  const int lb = blockIdx.x, nb = gridDim.x, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int n = F.n, q = F.q, ldn = F.ldn, m = F.m, T = A.res.T;
  const int r0 = min(n, lb * A.res.R), r1 = min(n, r0 + A.res.R), nr = r1 - r0;
  const int L = A.res.hinfo[2 * lb], own = A.res.hinfo[2 * lb + 1];
  const int n1 = A.n1, R1 = (n1 + nb - 1) / nb, k0 = min(n1, lb * R1), k1 = min(n1, k0 + R1);
  res::Team team{F.flags, &F.bar->err, lb, nb, A.res.cluster, 0u};
  int *list = reinterpret_cast<int *>(dyn + A.o_list);
  float *wj = reinterpret_cast<float *>(dyn + A.o_w);       // W on the halo
  float *hat = reinterpret_cast<float *>(dyn + A.o_work);   // staged operand of an SpMV
  double *xs = reinterpret_cast<double *>(dyn + A.o_work);  // FP64 x of the residual phase
  float *c1 = reinterpret_cast<float *>(dyn + A.o_c1);      // b_1, the coarse vector or y_1
  float *Vs = reinterpret_cast<float *>(dyn + A.o_v);
  float *Bs = reinterpret_cast<float *>(dyn + A.o_b);
  int2 *Rs = reinterpret_cast<int2 *>(dyn + A.o_r), *Ps = reinterpret_cast<int2 *>(dyn + A.o_p);
  float *ws = Vs + (size_t)A.kv * A.ldv;                    // w on the own rows (one more stride)
  const int kv = A.kv, ldv = A.ldv;

  for (int e = tid; e < L; e += RES_NT) {
    const int c = __ldg(A.res.hlist + (size_t)lb * A.res.hstride + e);
    list[e] = c;
    const double dg = __ldg(F.val + c);  // a row's first entry is its diagonal
    wj[e] = dg != 0.0 ? (float)(A.omega / dg) : 0.0f;
  }
  res::Rows<float, E, 4> row;
  row.place(r0, r1, T);
  row.indices(q, ldn, T, A.res.lidx);
#pragma unroll
  for (int u = 0; u < E; ++u) {
    const int j = row.lg + u * T;
    row.a[u] = (row.i >= 0 && j < q) ? __ldg(F.val32 + (size_t)j * ldn + row.i) : 0.0f;
  }
  // this CTA's rows of R~ and P~: contiguous entries of the CSR arrays
  const int rs0 = k1 > k0 ? __ldg(A.R0.ptr + k0) : 0, rs1 = k1 > k0 ? __ldg(A.R0.ptr + k1) : 0;
  const int ps0 = nr > 0 ? __ldg(A.P0.ptr + r0) : 0, ps1 = nr > 0 ? __ldg(A.P0.ptr + r1) : 0;
  for (int k = tid; k <= k1 - k0; k += RES_NT) rptr[k] = __ldg(A.R0.ptr + k0 + k) - rs0;
  const bool rres = rs1 - rs0 <= A.rcap, pres = ps1 - ps0 <= A.pcap;
  if (rres)
    for (int e = tid; e < rs1 - rs0; e += RES_NT)
      Rs[e] = make_int2(__ldg(A.R0.col + rs0 + e), __float_as_int(__ldg(A.R0.val + rs0 + e)));
  if (pres)
    for (int e = tid; e < ps1 - ps0; e += RES_NT)
      Ps[e] = make_int2(__ldg(A.P0.col + ps0 + e), __float_as_int(__ldg(A.P0.val + ps0 + e)));
  int pa = 0, pe = 0;  // this lane's row of P~ (its lanes take every T-th entry)
  if (row.i >= 0) {
    pa = __ldg(A.P0.ptr + row.i);
    pe = __ldg(A.P0.ptr + row.i + 1);
  }
  if (A.B && A.bres)
    for (int e = tid; e < (k1 - k0) * A.ldb; e += RES_NT)
      Bs[e] = __ldg(A.B + (size_t)k0 * A.ldb + e);
  if (tid == 0) {
    st.bnorm = st.beta = 0.0;
    st.relres = 1.0;
    st.it = st.restarts = 0;
    st.state = KRY_RUNNING;
    st.stop = 0;
  }
  bool ok = true;
  if (team.cluster) res::team_barrier(team);  // every CTA of the cluster has started
  else __syncthreads();

  auto row_sum = [&](float s) {
    float t = s;
    for (int u = 1; u < T; ++u) t += __shfl_sync(0xffffffffu, s, (lane + u) & 31);
    return t;
  };
  // (A hat) of this lane's row, complete on the row's first lane
  auto spmv = [&]() {
    const unsigned char *hb = reinterpret_cast<const unsigned char *>(hat);
    float s = 0.0f;
#pragma unroll
    for (int u = 0; u < E; ++u)
      s = fmaf(row.a[u], *reinterpret_cast<const float *>(hb + row.at(u)), s);
    return row_sum(s);
  };
  // the basis on the own rows: the first kv vectors in shared memory, the
  // rest in global memory (only this CTA touches its rows)
  auto v_get = [&](int i, int r) {
    return i < kv ? Vs[i * ldv + r] : __ldcg(F.V + (size_t)i * n + r0 + r);
  };
  auto v_put = [&](int i, int r, float v) {
    if (i < kv) Vs[i * ldv + r] = v;
    else F.V[(size_t)i * n + r0 + r] = v;
  };
  // sum_{i <= j} tot[i] V_i on this lane's row (first lane)
  auto combine = [&](int j) {
    float s = 0.0f;
    if (row.i >= 0) {
      const int js = min(j + 1, kv);
      int i = row.lg;
#pragma unroll 4
      for (; i < js; i += T) s = fmaf(tot[i], Vs[i * ldv + row.rl], s);
#pragma unroll 4
      for (; i <= j; i += T)
        s = fmaf(tot[i], __ldcg(F.V + (size_t)i * n + row.i), s);
    }
    return row_sum(s);
  };
  // warp d <= j + 1: (w, V_d) over the own rows, (w, w) for d = j + 1
  auto dots = [&](int j) {
    float s = 0.0f;
    if (warp <= j + 1) {
      if (warp == j + 1) {
        for (int r = lane; r < nr; r += 32) s = fmaf(ws[r], ws[r], s);
      } else if (warp < kv) {
        const float *v = Vs + warp * ldv;
#pragma unroll 4
        for (int r = lane; r < nr; r += 32) s = fmaf(ws[r], v[r], s);
      } else {
        const float *v = F.V + (size_t)warp * n + r0;
#pragma unroll 8
        for (int r = lane; r < nr; r += 32) s = fmaf(ws[r], __ldcg(v + r), s);
      }
      s = res::warp_total(s);
    }
    return s;
  };

  // ---- r = b - A x (FP64), (b, b) and (r, r)
  auto residual = [&](bool first) -> bool {
    for (int e = tid; e < L; e += RES_NT) xs[e] = __ldcg(F.x + list[e]);
    __syncthreads();
    double ax = 0.0;
    if (row.i >= 0) {
#pragma unroll 4
      for (int j = row.lg; j < q; j += T) {
        const size_t e = (size_t)j * ldn + row.i;
        ax += __ldg(F.val + e) * xs[__ldg(A.res.lidx + e)];
      }
    }
    const double s = ax;
    for (int u = 1; u < T; ++u) ax += __shfl_sync(0xffffffffu, s, (lane + u) & 31);
    double acc[2] = {0.0, 0.0};
    if (row.lead) {
      const double bi = __ldg(F.b + row.i), ri = bi - ax;
      F.r[row.i] = ri;
      acc[0] = bi * bi;
      acc[1] = ri * ri;
    }
    if (!res::team_totals<2, 2>(team, acc, tot64, wsum64, cpart64, A.res.part)) return false;
    if (tid == 0) {
      if (first) st.bnorm = sqrt(tot64[0]);
      st.beta = sqrt(tot64[1]);
      st.scale = st.beta > 0.0 ? 1.0 / st.beta : 0.0;
      st.relres = st.bnorm > 0.0 ? st.beta / st.bnorm : 0.0;
      if (st.bnorm == 0.0) st.state = KRY_OK;
      else if (!(st.relres == st.relres)) st.state = KRY_DIVERGED;
      else if (st.relres <= F.tol) st.state = KRY_OK;
      else if (st.it >= F.maxit) st.state = KRY_NOCONV;
    }
    __syncthreads();
    return true;
  };

  // sums over the entries of rows k0 .. k1 - 1: nparts warps a row, f(k)'s
  // parts meet in rowpart (at most 64 parts; more rows than warps take turns)
  const int nparts = R1 > 0 && R1 <= 32 ? 32 / R1 : 1;

  if (!residual(true)) ok = false;
  if (ok && st.bnorm == 0.0)
    for (int i = r0 + tid; i < r1; i += RES_NT) F.x[i] = 0.0;

  while (ok && st.state == KRY_RUNNING) {
    // ---- start of a restart: v_0 = r / beta, published
    {
      const double sc = st.scale;
      for (int r = tid; r < nr; r += RES_NT) {
        const float v = float(F.r[r0 + r] * sc);
        v_put(0, r, v);
        A.u[r0 + r] = v;
      }
      if (tid == 0) {
        st.gtol = (float)(F.tol * st.bnorm / st.beta);
        g[0] = 1.0f;
        for (int k = 1; k <= FG_MAXM; ++k) g[k] = 0.0f;
        st.k = 0;
      }
      if (!res::team_barrier(team)) { ok = false; break; }
    }
    float sigma = 1.0f;  // scale of u: z_j = M^-1 (sigma u)
    for (int j = 0; j < m; ++j) {
      // ---- A: z_0 = S_0 b and b_1 = R~_0 b with b = sigma u
      {
        float uv[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int e = tid + h * RES_NT;
          uv[h] = e < L ? __ldcg(A.u + list[e]) : 0.0f;
        }
        // R~'s gathers are in flight with the halo's
        for (int task = warp; task < (k1 - k0) * nparts; task += 32) {
          const int k = task / nparts, part = task - k * nparts;
          const int s = rptr[k], e1 = rptr[k + 1];
          float t = 0.0f;
          if (rres) {
#pragma unroll 4
            for (int e = s + lane + 32 * part; e < e1; e += 32 * nparts) {
              const int2 ce = Rs[e];
              t = fmaf(__int_as_float(ce.y), __ldcg(A.u + ce.x), t);
            }
          } else {
#pragma unroll 4
            for (int e = rs0 + s + lane + 32 * part; e < rs0 + e1; e += 32 * nparts)
              t = fmaf(__ldg(A.R0.val + e), __ldcg(A.u + __ldg(A.R0.col + e)), t);
          }
          t = res::warp_total(t);
          if (lane == 0) {
            if (nparts == 1) A.b1[k0 + k] = sigma * t;
            else rowpart[task] = t;
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int e = tid + h * RES_NT;
          if (e < L) hat[e] = wj[e] * (sigma * uv[h]);
        }
        for (int e = tid + 2 * RES_NT; e < L; e += RES_NT)
          hat[e] = wj[e] * (sigma * __ldcg(A.u + list[e]));
      }
      __syncthreads();
      if (nparts > 1 && tid < k1 - k0) {
        float t = rowpart[tid * nparts];
        for (int p = 1; p < nparts; ++p) t += rowpart[tid * nparts + p];
        A.b1[k0 + tid] = sigma * t;
      }
      float z0;
      {
        const float s = spmv();
        z0 = row.i >= 0 ? 2.0f * hat[own + row.rl] - wj[own + row.rl] * s : 0.0f;
      }
      if (!res::team_barrier(team)) { ok = false; break; }
      // ---- B: y_1
      if (A.B) {
        for (int e = tid; e < max(n1, A.ldb); e += RES_NT)
          c1[e] = e < n1 ? __ldcg(A.b1 + e) : 0.0f;
        __syncthreads();
        for (int task = warp; task < (k1 - k0) * nparts; task += 32) {
          const int k = task / nparts, part = task - k * nparts;
          const float *b = A.bres ? Bs + k * A.ldb : A.B + (size_t)(k0 + k) * A.ldb;
          float t = 0.0f;
          if ((A.ldb & 3) == 0) {  // rows and b_1 padded to whole quadruples
            const float4 *b4 = reinterpret_cast<const float4 *>(b);
            const float4 *c4 = reinterpret_cast<const float4 *>(c1);
#pragma unroll 4
            for (int e = lane + 32 * part; e < A.ldb / 4; e += 32 * nparts) {
              const float4 x = b4[e], y = c4[e];
              t = fmaf(x.x, y.x, t);
              t = fmaf(x.y, y.y, t);
              t = fmaf(x.z, y.z, t);
              t = fmaf(x.w, y.w, t);
            }
          } else {
            for (int e = lane + 32 * part; e < n1; e += 32 * nparts) t = fmaf(b[e], c1[e], t);
          }
          t = res::warp_total(t);
          if (lane == 0) {
            if (nparts == 1) A.y1[k0 + k] = t;
            else rowpart[task] = t;
          }
        }
        if (nparts > 1) {
          __syncthreads();
          if (tid < k1 - k0) {
            float t = rowpart[tid * nparts];
            for (int p = 1; p < nparts; ++p) t += rowpart[tid * nparts + p];
            A.y1[k0 + tid] = t;
          }
        }
      } else {
        // z_1 = S_1 b_1 on the own rows (kept), every deeper right-hand side
        // as chunk sums of the stacked restriction
        const AmgCompT<float> &C = A.C;
        float *z1 = c1 + C.nc;
        for (int k = warp; k < k1 - k0; k += 32) {
          const int s = __ldg(A.S1.ptr + k0 + k), e1 = __ldg(A.S1.ptr + k0 + k + 1);
          float t = 0.0f;
          for (int e = s + lane; e < e1; e += 32)
            t = fmaf(__ldg(A.S1.val + e), __ldcg(A.b1 + __ldg(A.S1.col + e)), t);
          t = res::warp_total(t);
          if (lane == 0) z1[k] = t;
        }
        for (int ch = (31 - warp) * nb + lb; ch < C.nchunk; ch += 32 * nb) {
          const int s = __ldg(C.cs + ch), e1 = __ldg(C.cs + ch + 1);
          float t = 0.0f;
#pragma unroll 8
          for (int e = s + lane; e < e1; e += 32)
            t = fmaf(__ldg(C.rval + e), __ldcg(A.b1 + __ldg(C.rcol + e)), t);
          t = res::warp_total(t);
          if (lane == 0) C.part[ch] = t;
        }
        if (!res::team_barrier(team)) { ok = false; break; }
        // the coarse vector in shared memory, y_1 = z_1 + Q c
        for (int k = tid; k < C.nc; k += RES_NT) {
          float t = 0.0f;
          for (int ch = __ldg(C.kc + k), e1 = __ldg(C.kc + k + 1); ch < e1; ++ch)
            t += __ldcg(C.part + ch);
          c1[k] = t;
        }
        __syncthreads();
        for (int k = warp; k < k1 - k0; k += 32) {
          const int s = __ldg(C.Q.ptr + k0 + k), e1 = __ldg(C.Q.ptr + k0 + k + 1);
          float t = 0.0f;
#pragma unroll 4
          for (int e = s + lane; e < e1; e += 32)
            t = fmaf(__ldg(C.Q.val + e), c1[__ldg(C.Q.col + e)], t);
          t = res::warp_total(t);
          if (lane == 0) A.y1[k0 + k] = z1[k] + t;
        }
      }
      if (!res::team_barrier(team)) { ok = false; break; }
      // ---- C: z = z_0 + P~_0 y_1 on the own rows
      float *zj = F.Z + (size_t)j * n;
      for (int e = tid; e < n1; e += RES_NT) c1[e] = __ldcg(A.y1 + e);
      __syncthreads();
      {
        float s = 0.0f;
        if (pres) {
#pragma unroll 4
          for (int e = pa + row.lg; e < pe; e += T) {
            const int2 ce = Ps[e - ps0];
            s = fmaf(__int_as_float(ce.y), c1[ce.x], s);
          }
        } else {
#pragma unroll 4
          for (int e = pa + row.lg; e < pe; e += T)
            s = fmaf(__ldg(A.P0.val + e), c1[__ldg(A.P0.col + e)], s);
        }
        s = row_sum(s);
        if (row.lead) zj[row.i] = z0 + s;
      }
      if (!res::team_barrier(team)) { ok = false; break; }
      // ---- w = A z, first pass
      for (int e = tid; e < L; e += RES_NT) hat[e] = __ldcg(zj + list[e]);
      __syncthreads();
      {
        const float s = spmv();
        if (row.lead) ws[row.rl] = s;
      }
      __syncthreads();
      if (!products(team, dots(j), j + 2, tot, cpart, A.res.part)) { ok = false; break; }
      {
        const float s = combine(j);
        if (tid <= j) H[tid + LDH * j] = tot[tid];
        __syncthreads();
        if (row.lead) {
          const float u = ws[row.rl] - s;
          ws[row.rl] = u;
          A.u[row.i] = u;
        }
      }
      __syncthreads();
      // ---- second pass; u is published by its exchange
      if (!products(team, dots(j), j + 2, tot, cpart, A.res.part)) { ok = false; break; }
      // h_{j+1,j} = sqrt((u, u) - sum c_i^2), by every warp in the same order
      float hn;
      {
        float c2 = lane <= j ? tot[lane] * tot[lane] : 0.0f;
        c2 = res::warp_total(c2);
        const float hn2 = tot[j + 1] - c2;
        hn = hn2 > 0.0f ? sqrtf(hn2) : 0.0f;
      }
      sigma = hn > 0.0f ? 1.0f / hn : 0.0f;
      if (j + 1 < m) {
        const float s = combine(j);
        if (row.lead) v_put(j + 1, row.rl, (ws[row.rl] - s) * sigma);
      }
      if (warp == 31) {
        // the second pass's coefficients join the column, then the previous
        // rotations and a new one (a lane's chain), the residual estimate
        if (lane <= j) H[lane + LDH * j] += tot[lane];
        __syncwarp();
        if (lane == 0) {
          float hc = H[LDH * j];
          for (int i = 0; i < j; ++i) {
            const float b = H[i + 1 + LDH * j];
            H[i + LDH * j] = cs[i] * hc + sn[i] * b;
            hc = -sn[i] * hc + cs[i] * b;
          }
          const float a = hc, b = hn;
          const float rr = sqrtf(a * a + b * b);
          const float ri = rr > 0.0f ? 1.0f / rr : 0.0f;
          cs[j] = rr > 0.0f ? a * ri : 1.0f;
          sn[j] = rr > 0.0f ? b * ri : 0.0f;
          H[j + LDH * j] = rr;
          g[j + 1] = -sn[j] * g[j];
          g[j] = cs[j] * g[j];
          st.it++;
          st.k = j + 1;
          const float ga = fabsf(g[j + 1]);
          st.stop = !(ga == ga) ? 2 : (ga <= st.gtol || hn == 0.0f || st.it >= F.maxit) ? 1 : 0;
          if (st.stop == 2) st.state = KRY_DIVERGED;
        }
      }
      __syncthreads();
      if (st.stop) break;
    }
    if (!ok || st.state != KRY_RUNNING) break;
    // ---- y = H^-1 g on the k columns, x += beta Z y in FP64
    if (tid == 0) {
      const int k = st.k;
      for (int i = k - 1; i >= 0; --i) {
        float t = g[i];
        for (int l = i + 1; l < k; ++l) t -= H[i + LDH * l] * y[l];
        y[i] = t / H[i + LDH * i];
      }
    }
    __syncthreads();
    {
      const int k = st.k;
      double s = 0.0;
      if (row.i >= 0) {
#pragma unroll 4
        for (int i = row.lg; i < k; i += T)
          s += (double)y[i] * (double)__ldcg(F.Z + (size_t)i * n + row.i);
      }
      const double s0 = s;
      for (int u = 1; u < T; ++u) s += __shfl_sync(0xffffffffu, s0, (lane + u) & 31);
      if (row.lead) F.x[row.i] = __ldcg(F.x + row.i) + st.beta * s;
    }
    if (tid == 0) st.restarts++;
    if (!res::team_barrier(team)) { ok = false; break; }
    // ---- true residual; stop or restart from it
    if (!residual(false)) { ok = false; break; }
  }

  if (team.cluster) res::team_barrier(team);  // no CTA leaves while others may write to it
  if (lb == 0 && tid == 0) {
    F.out->iters = st.it;
    F.out->restarts = st.restarts;
    F.out->status = ok ? st.state : KRY_TIMEOUT;
    F.out->relres = st.relres;
  }
}

// Row i of B = S_1 + sum_c Q(i, c) Rh(c, :): one CTA a row, the row's
// entries in shared memory; the rows of Rh are added one after another, so
// every entry is summed in a fixed order.  Once per build.
__global__ void __launch_bounds__(256) k_dense_coarse(int n1, int ldb, AmgCsrT<float> S,
                                                      AmgCompT<float> C, float *__restrict__ B) {
  extern __shared__ float acc[];
  const int i = blockIdx.x;
  for (int k = threadIdx.x; k < ldb; k += blockDim.x) acc[k] = 0.0f;
  __syncthreads();
  for (int e = S.ptr[i] + threadIdx.x; e < S.ptr[i + 1]; e += blockDim.x) acc[S.col[e]] = S.val[e];
  for (int e = C.Q.ptr[i]; e < C.Q.ptr[i + 1]; ++e) {
    const int c = C.Q.col[e];
    const float v = C.Q.val[e];
    const int s1 = C.cs[C.kc[c + 1]];
    __syncthreads();
    for (int s = C.cs[C.kc[c]] + threadIdx.x; s < s1; s += blockDim.x)
      acc[C.rcol[s]] = fmaf(v, C.rval[s], acc[C.rcol[s]]);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < ldb; k += blockDim.x) B[(size_t)i * ldb + k] = acc[k];
}

int round16(size_t v) { return (int)((v + 15) / 16 * 16); }

// The shared-memory layout: what every step needs first, then, as far as it
// fits, the dense operator's rows, the basis, R~'s and P~'s slabs.
bool fg_layout(FgResArgs &a, size_t *smem) {
  const int hm = a.res.hmax, R = a.res.R;
  const int n1 = a.n1, nb = a.res.nb, R1 = (n1 + nb - 1) / nb;
  size_t at = 0;
  auto take = [&](size_t bytes) {
    const size_t o = at;
    at += round16(bytes);
    return (int)o;
  };
  const size_t limit = RES_SMEM;
  a.o_list = take(4 * (size_t)hm);
  a.o_w = take(4 * (size_t)hm);
  a.o_work = take(8 * (size_t)hm);
  const size_t coarse = a.B ? 0 : (size_t)(a.C.nc + R1);
  a.o_c1 = take(4 * (coarse > (size_t)n1 ? coarse : (size_t)n1) + 16);
  a.ldv = R;
  while (a.ldv % 32 != (32 / a.res.T) % 32) ++a.ldv;
  const size_t vec = 4 * (size_t)a.ldv;
  if (at + vec > limit || R1 > MAXR1) return false;
  size_t left = limit - at - round16(vec);  // the vector w always has a place
  // basis vectors first, then B, then the transfer slabs: B and the slabs are
  // read once a step, a basis vector four times
  const size_t bb = a.B ? 4 * (size_t)R1 * a.ldb : 0;
  a.kv = (int)(left / vec < (size_t)MAXV ? left / vec : MAXV);
  left -= vec * a.kv;
  a.bres = a.B && (size_t)round16(bb) <= left;
  if (a.bres) left -= round16(bb);
  // a CTA's slab is about the mean; one that is longer reads L2
  a.rcap = (int)(left / 2 / 8);
  a.o_v = take(vec * (a.kv + 1));
  a.o_b = take(a.bres ? bb : 0);
  a.o_r = take(8 * (size_t)a.rcap);
  a.pcap = (int)((limit - at) / 8);
  if (a.pcap < 0) a.pcap = 0;
  a.o_p = take(8 * (size_t)a.pcap);
  *smem = at;
  return true;
}

const void *fg_res_fn(int E) {
  return E <= 6    ? (const void *)k_fgmres_res<6>
         : E <= 12 ? (const void *)k_fgmres_res<12>
         : E <= 24 ? (const void *)k_fgmres_res<24>
                   : nullptr;
}

}  // namespace

int fgmres_dense_ld(const AmgDevF &h) {
  const int n1 = h.nlev >= 2 ? h.lev[1].n : 0;
  if (h.nlev < 3 || h.comp.nc < 1 || n1 > RES_DENSE_N) return 0;
  return (n1 + 3) / 4 * 4;
}

int fgmres_dense_build(rbffd_ctx *ctx, const AmgDevF &h, float *B) {
  const int n1 = h.lev[1].n, ldb = fgmres_dense_ld(h);
  k_dense_coarse<<<n1, 256, 4 * (size_t)ldb, ctx->stream>>>(n1, ldb, h.lev[1].S, h.comp, B);
  return after_launch(ctx, "k_dense_coarse");
}

int fgmres_res_launch(rbffd_ctx *ctx, const FgmresArgs &args, const ResPlan &res,
                      const AmgDevF &h, double omega, const float *B, bool *ran) {
  *ran = false;
  // one level has no transfer operators; modes 0 and 2 of the
  // orthogonalisation and the level-by-level cycle keep the streaming kernel
  if (res.nb < 1 || res.hmax < 1 || res.hmax > res.hstride || args.reorth != 1 || h.nlev < 2 ||
      args.m > FG_MAXM || (h.nlev > 2 && h.comp.nc < 1))
    return RBFFD_OK;
  const int E = (args.q + res.T - 1) / res.T;
  const void *fn = fg_res_fn(E);
  if (!fn || 4 * res.hmax > 65535) return RBFFD_OK;
  FgResArgs a;
  memset(&a, 0, sizeof(a));
  a.f = args;
  a.res = res;
  a.omega = omega;
  a.n1 = h.lev[1].n;
  a.R0 = h.lev[0].R;
  a.P0 = h.lev[0].P;
  a.S1 = h.lev[1].S;
  a.C = h.comp;
  if (h.nlev == 2) {
    a.B = h.cinv;
    a.ldb = a.n1;
  } else if (B) {
    a.B = B;
    a.ldb = fgmres_dense_ld(h);
  }
  a.b1 = h.lev[1].b;
  a.y1 = h.lev[1].y;
  a.u = args.V + (size_t)args.m * args.n;  // the basis's last slot, unused by a restart's vectors
  size_t smem = 0;
  if (!fg_layout(a, &smem)) return RBFFD_OK;
  RBFFD_TRY(reset_barriers(ctx, args.bar, 1));
  if (!res.cluster)
    RBFFD_CK(cudaMemsetAsync(args.flags, 0, sizeof(unsigned int), ctx->stream));
  *ran = res_launch(ctx, res, fn, &a, smem);
  return RBFFD_OK;
}

}  // namespace rbffd
