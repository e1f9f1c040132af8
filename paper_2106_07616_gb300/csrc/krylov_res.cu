// krylov_res.cu -- the FP64 BiCGSTAB solves of krylov.cu on a resident team
// (resident.cuh): the CTA's rows of the matrix and the gathered vectors'
// halo in shared memory.
//
// With the Jacobi scaling, two exchanges an iteration instead of four: every
// CTA advances r, s, p and v of its whole halo with the same operations as
// their owners, so its neighbours need only t before the first product and v
// before the second.  The iteration's tests are those of krylov.cu, made
// after the exchange that follows (v = A p^ carries (r, r) and (r^, r)).
// With the multigrid cycle p and s are published for it; the cycle is three
// phases (level 0's smoother from the matrix itself; one dense matrix below
// level 1 where that is small, else the composed cycle's two phases; the
// prolongation), five exchanges a product instead of seven and more.
//
// What bounds it on GB300: an FP64 warp instruction occupies the pipe for 16
// cycles whatever its active lanes, so vector updates run on one thread a
// row, a row's products on T = 1, 2 or 4 lanes (a row sum costs log2 T more
// instructions), and the scalar recurrences' divisions (over 400 cycles
// each) side by side on different lanes.
//
// Measured on GB300, a whole FP64 outer iteration with the streaming and with
// this solve: cavity 99^2 (q = 20, multigrid) 7.0 -> 4.1 ms, Kovasznay 30^2
// (Jacobi, one cluster) 12.8 -> 4.8 ms; four requests of 5 184 to 8 836 rows
// served together, two time steps each, batched: 500 -> 372 ms.
#include "bicg_scalars.cuh"
#include "krylov.cuh"
#include "resident.cuh"

namespace rbffd {

namespace {

struct BicgResArgs {
  KrylovArgs k;
  int T;              // lanes a row
  double *pubt[1], *pubv[1];  // published vectors (Jacobi: t and v, NR side by side)
  // multigrid: level 0's smoothing weight, transfers, and what is below
  double omega;
  int n1, ldb;
  AmgCsrT<double> R0, P0, S1;
  AmgCompT<double> C;
  const double *B;    // dense coarse operator n1 x ldb, or null
  double *b1, *y1;
  // shared-memory layout, in bytes
  int o_val, o_idx, ld, o_list, o_w, o_vec, o_own, o_c1, o_b, o_rc, o_rv, o_pc, o_pv;
  int vres, bres, rcap, pcap;
  int o_tmp;          // scratch of a halo list made by the kernel (batched launches)
};

__device__ __forceinline__ void ld_l2v(const res::Vec<double, 1> *p, res::Vec<double, 1> &v) {
  v.x[0] = __ldcg(&p->x[0]);
}
__device__ __forceinline__ void ld_l2v(const res::Vec<double, 2> *p, res::Vec<double, 2> &v) {
  const double2 t = __ldcg(reinterpret_cast<const double2 *>(p));
  v.x[0] = t.x;
  v.x[1] = t.y;
}

// The solve of one system by the nb CTAs of a team; this CTA is number lb.
template <int NR, bool AMGP>
__device__ __forceinline__ void bicg_res_body(const BicgResArgs &A, const int lb, const int nb) {
  static_assert(!AMGP || NR == 1, "the multigrid preconditioner serves one right-hand side");
  using V = res::Vec<double, NR>;
  constexpr int VA = 3 * NR, VC = 5 * NR;
  __shared__ double wsum[VC * 32], cpart[2 * VC * RES_CLUSTER], tot[VC];
  __shared__ BicgScalars ks[NR];
  __shared__ int s_any;
  extern __shared__ __align__(16) unsigned char dyn[];
  const KrylovArgs &K = A.k;
  __shared__ int s_len, s_own;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = K.n, q = K.q, ldn = K.ldn, T = A.T;
  const int R = K.res.R, r0 = min(n, lb * R), r1 = min(n, r0 + R), nr = r1 - r0;
  const int hm = K.res.hmax;
  res::Team team{K.flags, &K.bar->err, lb, nb, K.res.cluster, 0u};
  double *val = reinterpret_cast<double *>(dyn + A.o_val);
  uint16_t *idx = reinterpret_cast<uint16_t *>(dyn + A.o_idx);
  int *list = reinterpret_cast<int *>(dyn + A.o_list);
  double *w = reinterpret_cast<double *>(dyn + A.o_w);  // 1 / d, or W = omega / d, on the halo
  // Jacobi: rs (r, then s), p, v and the product's operand on the halo, x own
  V *hat = reinterpret_cast<V *>(dyn + A.o_vec), *rs = hat + hm, *ph = rs + hm, *vh = ph + hm;
  // multigrid: own rows only, but for the operand
  double *own_v = reinterpret_cast<double *>(dyn + A.o_own);
  V *xo = reinterpret_cast<V *>(own_v);
  double *o_r = own_v + R, *o_p = o_r + R, *o_v = o_p + R, *o_t = o_v + R,
         *o_ph = o_t + R, *o_sh = o_ph + R;
  double *c1 = reinterpret_cast<double *>(dyn + A.o_c1);
  const int n1 = AMGP ? A.n1 : 0, R1 = AMGP ? (n1 + nb - 1) / nb : 0;
  const int k0 = min(n1, lb * R1), k1 = min(n1, k0 + R1);
  double *Bs = reinterpret_cast<double *>(dyn + A.o_b);
  int *Rc = reinterpret_cast<int *>(dyn + A.o_rc), *Pc = reinterpret_cast<int *>(dyn + A.o_pc);
  double *Rv = reinterpret_cast<double *>(dyn + A.o_rv),
         *Pv = reinterpret_cast<double *>(dyn + A.o_pv);
  V *pubt = reinterpret_cast<V *>(A.pubt[0]), *pubv = reinterpret_cast<V *>(A.pubv[0]);

  double rhat[NR];  // r^ of this row (first lane)
#pragma unroll
  for (int k = 0; k < NR; ++k) rhat[k] = 0.0;
  // ---- this thread's row
  const int gpw = 32 / T, g = lane / T, lg = lane - g * T, rl = warp * gpw + g;
  const bool mine = rl < nr, lead = mine && lg == 0, active = warp * gpw < nr;
  const int row = r0 + rl;

  // ---- load the CTA's share
  const bool listed = K.res.hlist != nullptr;
  if (listed) {
    if (tid == 0) {
      s_len = K.res.hinfo[2 * lb];
      s_own = K.res.hinfo[2 * lb + 1];
    }
    __syncthreads();
  } else {
    res::halo_local(n, q, ldn, K.col, r0, r1, reinterpret_cast<unsigned int *>(dyn + A.o_tmp),
                    list, idx, A.ld, &s_len, &s_own);
  }
  const int L = s_len, own = s_own;
  for (int e = tid; e < L; e += RES_NT) {
    const int c = listed ? __ldg(K.res.hlist + (size_t)lb * K.res.hstride + e) : list[e];
    list[e] = c;
    if (AMGP) {
      const double dg = __ldg(K.val + c);  // a row's first entry is its diagonal
      w[e] = dg != 0.0 ? A.omega / dg : 0.0;
    } else {
      w[e] = __ldg(K.dinv + c);
    }
  }
  for (int e = tid; e < nr * q; e += RES_NT) {
    const int j = e / nr, i = e - j * nr;
    const size_t s = (size_t)j * ldn + r0 + i;
    if (A.vres) val[j * A.ld + i] = __ldg(K.val + s);
    if (listed) idx[j * A.ld + i] = __ldg(K.res.lidx + s);
  }
  int rs0 = 0, rs1 = 0, ps0 = 0, ps1 = 0, pa = 0, pe = 0;
  bool rres = false, pres = false;
  if constexpr (AMGP) {
    if (k1 > k0) {
      rs0 = __ldg(A.R0.ptr + k0);
      rs1 = __ldg(A.R0.ptr + k1);
    }
    if (nr > 0) {
      ps0 = __ldg(A.P0.ptr + r0);
      ps1 = __ldg(A.P0.ptr + r1);
    }
    rres = rs1 - rs0 <= A.rcap;
    pres = ps1 - ps0 <= A.pcap;
    if (rres)
      for (int e = tid; e < rs1 - rs0; e += RES_NT) {
        Rc[e] = __ldg(A.R0.col + rs0 + e);
        Rv[e] = __ldg(A.R0.val + rs0 + e);
      }
    if (pres)
      for (int e = tid; e < ps1 - ps0; e += RES_NT) {
        Pc[e] = __ldg(A.P0.col + ps0 + e);
        Pv[e] = __ldg(A.P0.val + ps0 + e);
      }
    if (mine) {
      pa = __ldg(A.P0.ptr + row);
      pe = __ldg(A.P0.ptr + row + 1);
    }
    if (A.B && A.bres)
      for (int e = tid; e < (k1 - k0) * A.ldb; e += RES_NT)
        Bs[e] = __ldg(A.B + (size_t)k0 * A.ldb + e);
  }
  if (tid < NR) bicg_start(ks[tid]);
  for (int e = tid; e < nr; e += RES_NT)
#pragma unroll
    for (int k = 0; k < NR; ++k) xo[e].x[k] = K.x[k][r0 + e];
  bool ok = true;
  if (team.cluster) res::team_barrier(team);  // every CTA of the cluster has started
  else __syncthreads();

  auto row_sum = [&](double s) {
    for (int o = T >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  };
  // (A x) of this lane's row for the NR vectors staged at b (entry stride NR)
  auto product = [&](const V *b, double (&o)[NR]) {
    double s0[NR], s1[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) s0[k] = s1[k] = 0.0;
    if (mine) {
      int j = lg;
#pragma unroll 2
      for (; j + T < q; j += 2 * T) {
        const int e0 = j * A.ld + rl, e1 = e0 + T * A.ld;
        const double a0 = A.vres ? val[e0] : __ldg(K.val + (size_t)j * ldn + row);
        const double a1 = A.vres ? val[e1] : __ldg(K.val + (size_t)(j + T) * ldn + row);
        const V x0 = b[idx[e0]], x1 = b[idx[e1]];
#pragma unroll
        for (int k = 0; k < NR; ++k) {
          s0[k] = fma(a0, x0.x[k], s0[k]);
          s1[k] = fma(a1, x1.x[k], s1[k]);
        }
      }
      if (j < q) {
        const int e0 = j * A.ld + rl;
        const double a0 = A.vres ? val[e0] : __ldg(K.val + (size_t)j * ldn + row);
        const V x0 = b[idx[e0]];
#pragma unroll
        for (int k = 0; k < NR; ++k) s0[k] = fma(a0, x0.x[k], s0[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < NR; ++k) o[k] = active ? row_sum(s0[k] + s1[k]) : 0.0;
  };

  // ---- the multigrid cycle z = M^-1 u: u published (n), z to zp and to own
  // (the own rows); ends with z published
  auto cycle = [&](const double *u, double *zp, double *zown) -> bool {
    for (int e = tid; e < L; e += RES_NT) hat[e].x[0] = w[e] * __ldcg(u + list[e]);
    // b_1 = R~_0 u, 16 lanes a row
    for (int kb = 2 * warp; kb < k1 - k0; kb += 64) {
      const int k = kb + (lane >> 4), l = lane & 15;
      double t0 = 0.0, t1 = 0.0;
      if (k < k1 - k0) {
        const int s = __ldg(A.R0.ptr + k0 + k), e1 = __ldg(A.R0.ptr + k0 + k + 1);
#pragma unroll 4
        for (int e = s + l; e < e1; e += 32) {
          const bool two = e + 16 < e1;
          const int c0 = rres ? Rc[e - rs0] : __ldg(A.R0.col + e);
          const int c1i = two ? (rres ? Rc[e + 16 - rs0] : __ldg(A.R0.col + e + 16)) : c0;
          const double v0 = rres ? Rv[e - rs0] : __ldg(A.R0.val + e);
          const double v1 = two ? (rres ? Rv[e + 16 - rs0] : __ldg(A.R0.val + e + 16)) : 0.0;
          t0 = fma(v0, __ldcg(u + c0), t0);
          t1 = fma(v1, __ldcg(u + c1i), t1);
        }
      }
      t0 += t1;
      for (int o = 8; o > 0; o >>= 1) t0 += __shfl_xor_sync(0xffffffffu, t0, o);
      if (k < k1 - k0 && l == 0) A.b1[k0 + k] = t0;
    }
    __syncthreads();
    double ah[NR];
    product(hat, ah);
    const double z0 = lead ? 2.0 * hat[own + rl].x[0] - w[own + rl] * ah[0] : 0.0;
    if (!res::team_barrier(team)) return false;
    if (A.B) {
      for (int e = tid; e < n1; e += RES_NT) c1[e] = __ldcg(A.b1 + e);
      __syncthreads();
      for (int k = warp; k < k1 - k0; k += 32) {
        const double *b = A.bres ? Bs + k * A.ldb : A.B + (size_t)(k0 + k) * A.ldb;
        double t0 = 0.0, t1 = 0.0;
#pragma unroll 4
        for (int e = lane; e < n1; e += 64) {
          t0 = fma(b[e], c1[e], t0);
          if (e + 32 < n1) t1 = fma(b[e + 32], c1[e + 32], t1);
        }
        t0 = res::warp_total(t0 + t1);
        if (lane == 0) A.y1[k0 + k] = t0;
      }
    } else {
      const AmgCompT<double> &C = A.C;
      double *z1 = c1 + C.nc;
      for (int kb = 4 * warp; kb < k1 - k0; kb += 128) {  // 8 lanes a row
        const int k = kb + (lane >> 3);
        double t = 0.0;
        if (k < k1 - k0) {
          const int s = __ldg(A.S1.ptr + k0 + k), e1 = __ldg(A.S1.ptr + k0 + k + 1);
          for (int e = s + (lane & 7); e < e1; e += 8)
            t = fma(__ldg(A.S1.val + e), __ldcg(A.b1 + __ldg(A.S1.col + e)), t);
        }
        for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (k < k1 - k0 && (lane & 7) == 0) z1[k] = t;
      }
      for (int ch = (31 - warp) * nb + lb; ch < C.nchunk; ch += 32 * nb) {
        const int s = __ldg(C.cs + ch), e1 = __ldg(C.cs + ch + 1);
        double t = 0.0;
#pragma unroll 8
        for (int e = s + lane; e < e1; e += 32)
          t = fma(__ldg(C.rval + e), __ldcg(A.b1 + __ldg(C.rcol + e)), t);
        t = res::warp_total(t);
        if (lane == 0) C.part[ch] = t;
      }
      if (!res::team_barrier(team)) return false;
      for (int k = tid; k < C.nc; k += RES_NT) {
        double t = 0.0;
        for (int ch = __ldg(C.kc + k), e1 = __ldg(C.kc + k + 1); ch < e1; ++ch)
          t += __ldcg(C.part + ch);
        c1[k] = t;
      }
      __syncthreads();
      for (int k = warp; k < k1 - k0; k += 32) {
        const int s = __ldg(C.Q.ptr + k0 + k), e1 = __ldg(C.Q.ptr + k0 + k + 1);
        double t = 0.0;
#pragma unroll 4
        for (int e = s + lane; e < e1; e += 32)
          t = fma(__ldg(C.Q.val + e), c1[__ldg(C.Q.col + e)], t);
        t = res::warp_total(t);
        if (lane == 0) A.y1[k0 + k] = z1[k] + t;
      }
    }
    if (!res::team_barrier(team)) return false;
    for (int e = tid; e < n1; e += RES_NT) c1[e] = __ldcg(A.y1 + e);
    __syncthreads();
    double s = 0.0;
    if (pres) {
#pragma unroll 4
      for (int e = pa - ps0 + lg; e < pe - ps0; e += T) s = fma(Pv[e], c1[Pc[e]], s);
    } else {
#pragma unroll 4
      for (int e = pa + lg; e < pe; e += T)
        s = fma(__ldg(A.P0.val + e), c1[__ldg(A.P0.col + e)], s);
    }
    if (active) s = row_sum(s);
    if (lead) {
      zown[rl] = z0 + s;
      zp[row] = z0 + s;
    }
    return res::team_barrier(team);
  };

  for (;;) {
    // ---------------- (re)starts: r = b - A x, r^ = p = r
    bool ini[NR], any_ini = false;
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      ini[k] = ks[k].state == KRY_RUNNING && ks[k].need_init;
      any_ini |= ini[k];
    }
    if (any_ini) {
      for (int e = tid; e < nr; e += RES_NT)
#pragma unroll
        for (int k = 0; k < NR; ++k)
          if (ini[k]) {
            if (bicg_from_copy(ks[k])) xo[e].x[k] = K.w[k].xb[r0 + e];
            K.x[k][r0 + e] = xo[e].x[k];
          }
      if (!res::team_barrier(team)) { ok = false; break; }
      for (int e = tid; e < L; e += RES_NT)
#pragma unroll
        for (int k = 0; k < NR; ++k) hat[e].x[k] = __ldcg(K.x[k] + list[e]);
      __syncthreads();
      double ax[NR], acc[res::pow2_ge(2 * NR)];
      product(hat, ax);
#pragma unroll
      for (int k = 0; k < res::pow2_ge(2 * NR); ++k) acc[k] = 0.0;
      if (lead) {
#pragma unroll
        for (int k = 0; k < NR; ++k)
          if (ini[k]) {
            const double bi = __ldg(K.b[k] + row), ri = bi - ax[k];
            rhat[k] = ri;
            if constexpr (AMGP) {
              o_r[rl] = ri;
            } else {
              pubt[row].x[k] = ri;
            }
            acc[2 * k] = bi * bi;
            acc[2 * k + 1] = ri * ri;
          }
      }
      ok = res::team_totals<2 * NR, VC>(team, acc, tot, wsum, cpart, K.res.part, active);
      if (!ok) break;
      if (tid < NR && ks[tid].state == KRY_RUNNING && ks[tid].need_init)
        bicg_restarted(ks[tid], tot[2 * tid], tot[2 * tid + 1], K.tol);
      __syncthreads();
#pragma unroll
      for (int k = 0; k < NR; ++k)
        if (ks[k].half == 3)
          for (int e = tid; e < nr; e += RES_NT) xo[e].x[k] = 0.0;
    }
    if (tid == 0) {
      int any = 0;
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        ks[k].run = ks[k].state == KRY_RUNNING;
        any |= ks[k].run;
      }
      s_any = any;
    }
    __syncthreads();
    if (!s_any) break;
    bool run[NR];
    double alp[NR], omg[NR], bet[NR];
    bool first[NR], sav[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      run[k] = ks[k].run != 0;
      alp[k] = ks[k].alpha;
      omg[k] = ks[k].omega;
      bet[k] = ks[k].beta;
      first[k] = ks[k].first != 0;
      sav[k] = ks[k].save != 0;
    }

    // ---------------- A: x, r and the next direction; v = A p^
    if constexpr (AMGP) {
      for (int e = tid; e < nr; e += RES_NT) {
        if (sav[0]) K.w[0].xb[r0 + e] = xo[e].x[0];
        double r = o_r[e], p;
        if (first[0]) {
          p = r;
        } else {
          xo[e].x[0] = xo[e].x[0] + alp[0] * o_ph[e] + omg[0] * o_sh[e];
          r = fma(-omg[0], o_t[e], r);  // r holds s here
          p = fma(bet[0], fma(-omg[0], o_v[e], o_p[e]), r);
          o_r[e] = r;
        }
        o_p[e] = p;
        pubv[r0 + e].x[0] = p;
      }
      if (!res::team_barrier(team)) { ok = false; break; }
      if (!cycle(A.pubv[0], A.pubt[0], o_ph)) { ok = false; break; }
      for (int e = tid; e < L; e += RES_NT) hat[e].x[0] = __ldcg(A.pubt[0] + list[e]);
    } else {
      for (int e = tid; e < L; e += RES_NT) {
        V t;
        ld_l2v(pubt + list[e], t);
        V r = rs[e], p = ph[e], h;
        const V ve = vh[e];
        const double di = w[e];
        const bool own_e = e >= own && e < own + nr;
#pragma unroll
        for (int k = 0; k < NR; ++k) {
          if (!run[k]) {
            h.x[k] = 0.0;
            continue;
          }
          if (own_e && sav[k]) K.w[k].xb[r0 + e - own] = xo[e - own].x[k];
          if (first[k]) {
            r.x[k] = p.x[k] = t.x[k];
          } else {
            if (own_e)
              xo[e - own].x[k] = xo[e - own].x[k] + alp[k] * (p.x[k] * di) + omg[k] * (r.x[k] * di);
            r.x[k] = fma(-omg[k], t.x[k], r.x[k]);
            p.x[k] = fma(bet[k], fma(-omg[k], ve.x[k], p.x[k]), r.x[k]);
          }
          h.x[k] = p.x[k] * di;
        }
        rs[e] = r;
        ph[e] = p;
        hat[e] = h;
      }
    }
    __syncthreads();
    {
      double av[NR], acc[res::pow2_ge(VA)];
      product(hat, av);
#pragma unroll
      for (int k = 0; k < res::pow2_ge(VA); ++k) acc[k] = 0.0;
      if (lead) {
#pragma unroll
        for (int k = 0; k < NR; ++k) {
          if (!run[k]) continue;
          const double rh = rhat[k];
          const double r = AMGP ? o_r[rl] : rs[own + rl].x[k];
          if constexpr (AMGP) o_v[rl] = av[k];
          else pubv[row].x[k] = av[k];
          acc[3 * k] = rh * av[k];
          acc[3 * k + 1] = r * r;
          acc[3 * k + 2] = rh * r;
        }
      }
      ok = res::team_totals<VA, VC>(team, acc, tot, wsum, cpart, K.res.part, active);
    }
    if (!ok) break;
    if (tid < NR && ks[tid].run)
      bicg_after_v(ks[tid], tot[3 * tid], tot[3 * tid + 1], tot[3 * tid + 2], K.maxit);
    __syncthreads();
    bool anyc = false;
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      run[k] = ks[k].run != 0;
      alp[k] = ks[k].alpha;
      anyc |= run[k];
    }
    if (!anyc) continue;

    // ---------------- C: s = r - alpha v, t = A s^
    if constexpr (AMGP) {
      for (int e = tid; e < nr; e += RES_NT) {
        const double s = fma(-alp[0], o_v[e], o_r[e]);
        o_r[e] = s;
        pubv[r0 + e].x[0] = s;
      }
      if (!res::team_barrier(team)) { ok = false; break; }
      if (!cycle(A.pubv[0], A.pubt[0], o_sh)) { ok = false; break; }
      for (int e = tid; e < L; e += RES_NT) hat[e].x[0] = __ldcg(A.pubt[0] + list[e]);
    } else {
      for (int e = tid; e < L; e += RES_NT) {
        V ve, s = rs[e], h;
        ld_l2v(pubv + list[e], ve);
        const double di = w[e];
#pragma unroll
        for (int k = 0; k < NR; ++k) {
          h.x[k] = 0.0;
          if (!run[k]) continue;
          s.x[k] = fma(-alp[k], ve.x[k], s.x[k]);
          h.x[k] = s.x[k] * di;
        }
        rs[e] = s;
        vh[e] = ve;
        hat[e] = h;
      }
    }
    __syncthreads();
    {
      double at[NR], acc[res::pow2_ge(VC)];
      product(hat, at);
#pragma unroll
      for (int k = 0; k < res::pow2_ge(VC); ++k) acc[k] = 0.0;
      if (lead) {
#pragma unroll
        for (int k = 0; k < NR; ++k) {
          if (!run[k]) continue;
          const double rh = rhat[k];
          const double s = AMGP ? o_r[rl] : rs[own + rl].x[k];
          if constexpr (AMGP) o_t[rl] = at[k];
          else pubt[row].x[k] = at[k];
          acc[5 * k] = s * s;
          acc[5 * k + 1] = at[k] * at[k];
          acc[5 * k + 2] = at[k] * s;
          acc[5 * k + 3] = rh * s;
          acc[5 * k + 4] = rh * at[k];
        }
      }
      ok = res::team_totals<VC, VC>(team, acc, tot, wsum, cpart, K.res.part, active);
    }
    if (!ok) break;
    if (tid < 32) {
      // omega = ts / tt, rho' = (r^,s) - omega (r^,t), beta = rho' (alpha /
      // rho) / omega: the three divisions on lanes 4 k .. 4 k + 2
      const int k = lane >> 2, o = lane & 3;
      double tt = 1.0, ts = 1.0, num = 1.0, den = 1.0;
      if (k < NR) {
        tt = tot[5 * k + 1];
        ts = tot[5 * k + 2];
        num = o == 0 ? ts : o == 1 ? tt : ks[k].alpha;
        den = o == 0 ? tt : o == 1 ? ts : ks[k].rho;
      }
      const double quo = num / den;
      const double om0 = __shfl_sync(0xffffffffu, quo, lane & ~3);
      const double iom = __shfl_sync(0xffffffffu, quo, (lane & ~3) + 1);
      const double ar = __shfl_sync(0xffffffffu, quo, (lane & ~3) + 2);
      if (k < NR && o == 0)
        bicg_after_t(ks[k], tot[5 * k], tot[5 * k + 3], tot[5 * k + 4], tt == 0.0, om0, iom, ar,
                     K.maxit);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NR; ++k)
      if (run[k] && ks[k].half == 1) {  // x += alpha p^ and done
        for (int e = tid; e < nr; e += RES_NT) {
          const double pe = AMGP ? o_ph[e] : ph[own + e].x[k] * w[own + e];
          xo[e].x[k] = xo[e].x[k] + alp[k] * pe;
        }
      }
    __syncthreads();
  }
  // ---- the solution (also of a solve that stopped short)
  if (tid < NR && ok) ks[tid].half = bicg_end(ks[tid]) ? 4 : 0;
  __syncthreads();
  for (int e = tid; e < nr; e += RES_NT)
#pragma unroll
    for (int k = 0; k < NR; ++k)
      K.x[k][r0 + e] = ks[k].half == 4 ? K.w[k].xb[r0 + e] : xo[e].x[k];
  if (team.cluster) res::team_barrier(team);  // no CTA leaves while others may write to it
  if (lb == 0 && tid < NR) {
    const BicgScalars &c = ks[tid];
    K.out[tid].iters = c.it;
    K.out[tid].restarts = c.restarts + c.blowups;
    K.out[tid].status = ok ? c.state : KRY_TIMEOUT;
    K.out[tid].relres = c.bnorm > 0.0 ? sqrt(c.rr) / c.bnorm : 0.0;
  }
}

template <int NR, bool AMGP>
__global__ void __launch_bounds__(RES_NT, 1) k_bicg_res(const __grid_constant__ BicgResArgs A) {
  bicg_res_body<NR, AMGP>(A, blockIdx.x, gridDim.x);
}

// Batched: a persistent work list as in krylov.cu, teams of 1024-thread CTAs.
template <int NR, bool AMGP>
__global__ void __launch_bounds__(RES_NT, 1)
    k_bicg_res_batch(const BicgResArgs *__restrict__ sys, const int *__restrict__ cta_team,
                     const int *__restrict__ info) {
  __shared__ BicgResArgs A;
  const int t = cta_team[blockIdx.x];
  const int c0 = info[4 * t], nc = info[4 * t + 1], j0 = info[4 * t + 2], j1 = info[4 * t + 3];
  for (int j = j0; j < j1; ++j) {
    __syncthreads();
    const int *src = reinterpret_cast<const int *>(sys + info[j]);
    for (int k = threadIdx.x; k < (int)(sizeof(A) / 4); k += RES_NT)
      reinterpret_cast<int *>(&A)[k] = src[k];
    __syncthreads();
    bicg_res_body<NR, AMGP>(A, blockIdx.x - c0, nc);
  }
}

int round16(size_t v) { return (int)((v + 15) / 16 * 16); }

// Lanes a row: enough threads to hide the products' latency, no more (a
// row sum's FP64 instructions grow with them).
int lanes(int R) { return R <= 128 ? 4 : R <= 512 ? 2 : 1; }

bool layout(BicgResArgs &a, int nr, bool amg, size_t *smem) {
  const ResPlan &p = a.k.res;
  const int hm = p.hmax, R = p.R, q = a.k.q;
  size_t at = 0;
  auto take = [&](size_t bytes) {
    const size_t o = at;
    at += round16(bytes);
    return (int)o;
  };
  a.ld = R | 1;
  a.o_list = take(4 * (size_t)hm);
  a.o_w = take(8 * (size_t)hm);
  a.o_vec = take(8 * (size_t)nr * hm * (amg ? 1 : 4));
  a.o_own = take(8 * (size_t)R * (amg ? 7 : nr));
  a.o_idx = take(2 * (size_t)q * a.ld);
  const int R1 = amg ? (a.n1 + p.nb - 1) / p.nb : 0;
  if (amg) {
    const size_t coarse = a.B ? 0 : (size_t)(a.C.nc + R1);
    a.o_c1 = take(8 * (coarse > (size_t)a.n1 ? coarse : (size_t)a.n1));
  }
  // the list's scratch lies over what is loaded after it
  a.o_tmp = (int)at;
  const size_t tmp = p.hlist ? 0 : 8 * (size_t)((a.k.n + 31) / 32);
  if (at + tmp > RES_SMEM) return false;
  a.vres = at + 8 * (size_t)q * a.ld <= RES_SMEM;
  if (a.vres) a.o_val = take(8 * (size_t)q * a.ld);
  if (amg) {
    const size_t bb = a.B ? 8 * (size_t)R1 * a.ldb : 0;
    a.bres = a.B && at + bb <= RES_SMEM;
    if (a.bres) a.o_b = take(bb);
    const size_t left = at < RES_SMEM ? RES_SMEM - at : 0;
    a.rcap = a.pcap = (int)(left / 2 / 12) / 4 * 4;
    a.o_rv = take(8 * (size_t)a.rcap);
    a.o_rc = take(4 * (size_t)a.rcap);
    a.o_pv = take(8 * (size_t)a.pcap);
    a.o_pc = take(4 * (size_t)a.pcap);
  }
  *smem = at > (size_t)a.o_tmp + tmp ? at : (size_t)a.o_tmp + tmp;
  return true;
}

// The arguments and shared memory of a solve on the plan of args.res, or false.
bool res_args(int nr, const KrylovArgs &args, const AmgDev *h, double omega, const double *B,
              BicgResArgs *out, size_t *smem) {
  const ResPlan &p = args.res;
  const bool amg = args.amg != nullptr;
  if (amg && (!h || h->nlev < 2 || (h->nlev > 2 && h->comp.nc < 1))) return false;
  BicgResArgs &a = *out;
  memset(&a, 0, sizeof(a));
  a.k = args;
  a.T = lanes(p.R);
  // published vectors, up to two right-hand sides side by side: ph and s, sh
  // and t of the first system are adjacent in the allocation
  a.pubt[0] = args.w[0].ph;
  a.pubv[0] = args.w[0].sh;
  if (amg) {
    a.omega = omega;
    a.n1 = h->lev[1].n;
    a.R0 = h->lev[0].R;
    a.P0 = h->lev[0].P;
    a.S1 = h->lev[1].S;
    a.C = h->comp;
    a.b1 = h->lev[1].b;
    a.y1 = h->lev[1].y;
    if (h->nlev == 2) {
      a.B = h->cinv;
      a.ldb = a.n1;
    } else if (B) {
      a.B = B;
      a.ldb = a.n1;
    }
  }
  return layout(a, nr, amg, smem);
}

// Row i of B = S_1 + sum_c Q(i, c) Rh(c, :), as in fgmres_res.cu.
__global__ void __launch_bounds__(256) k_dense_coarse64(int n1, int ldb, AmgCsrT<double> S,
                                                        AmgCompT<double> C,
                                                        double *__restrict__ B) {
  extern __shared__ double acc64[];
  const int i = blockIdx.x;
  for (int k = threadIdx.x; k < ldb; k += blockDim.x) acc64[k] = 0.0;
  __syncthreads();
  for (int e = S.ptr[i] + threadIdx.x; e < S.ptr[i + 1]; e += blockDim.x)
    acc64[S.col[e]] = S.val[e];
  for (int e = C.Q.ptr[i]; e < C.Q.ptr[i + 1]; ++e) {
    const int c = C.Q.col[e];
    const double v = C.Q.val[e];
    const int s1 = C.cs[C.kc[c + 1]];
    __syncthreads();
    for (int s = C.cs[C.kc[c]] + threadIdx.x; s < s1; s += blockDim.x)
      acc64[C.rcol[s]] = fma(v, C.rval[s], acc64[C.rcol[s]]);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < ldb; k += blockDim.x) B[(size_t)i * ldb + k] = acc64[k];
}

}  // namespace

int krylov_dense_ld(const AmgDev &h) {
  const int n1 = h.nlev >= 2 ? h.lev[1].n : 0;
  return h.nlev < 3 || h.comp.nc < 1 || n1 > RES_DENSE64_N ? 0 : n1;
}

int krylov_dense_build(rbffd_ctx *ctx, const AmgDev &h, double *B) {
  const int n1 = h.lev[1].n;
  k_dense_coarse64<<<n1, 256, 8 * (size_t)n1, ctx->stream>>>(n1, n1, h.lev[1].S, h.comp, B);
  return after_launch(ctx, "k_dense_coarse64");
}

int krylov_res_launch(rbffd_ctx *ctx, int nr, const KrylovArgs &args, const AmgDev *h,
                      double omega, const double *B, bool *ran) {
  *ran = false;
  const ResPlan &p = args.res;
  if (p.nb < 1 || p.hmax < 1 || p.hmax > p.hstride) return RBFFD_OK;
  const bool amg = args.amg != nullptr;
  BicgResArgs a;
  size_t smem = 0;
  if (!res_args(nr, args, h, omega, B, &a, &smem)) return RBFFD_OK;
  RBFFD_TRY(reset_barriers(ctx, args.bar, 1));
  if (!p.cluster) RBFFD_CK(cudaMemsetAsync(args.flags, 0, sizeof(unsigned int), ctx->stream));
  const void *fn = amg       ? (const void *)k_bicg_res<1, true>
                   : nr == 1 ? (const void *)k_bicg_res<1, false>
                             : (const void *)k_bicg_res<2, false>;
  *ran = res_launch(ctx, p, fn, &a, smem);
  return RBFFD_OK;
}

size_t krylov_res_args_bytes() { return sizeof(BicgResArgs); }

bool krylov_res_args(int nr, const KrylovArgs &args, const AmgDev *h, double omega,
                     const double *B, void *out, size_t *smem) {
  static_assert(sizeof(BicgResArgs) % 8 == 0, "copied as words");
  BicgResArgs a;
  if (!res_args(nr, args, h, omega, B, &a, smem)) return false;
  if (out) memcpy(out, &a, sizeof(a));
  return true;
}

int krylov_res_batch_launch(rbffd_ctx *ctx, int nr, bool amg, int nctas, const void *d_sys,
                            const int *d_cta_team, const int *d_info, size_t smem, bool *ran) {
  const void *fn = amg       ? (const void *)k_bicg_res_batch<1, true>
                   : nr == 1 ? (const void *)k_bicg_res_batch<1, false>
                             : (const void *)k_bicg_res_batch<2, false>;
  void *kargs[] = {(void *)&d_sys, (void *)&d_cta_team, (void *)&d_info};
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, RES_SMEM);
  if (e == cudaSuccess)
    e = cudaLaunchCooperativeKernel(fn, dim3(nctas), dim3(RES_NT), kargs, smem, ctx->stream);
  *ran = e == cudaSuccess;  // refused: as res_launch
  if (*ran) ctx->launches++;
  else cudaGetLastError();
  return RBFFD_OK;
}

}  // namespace rbffd
