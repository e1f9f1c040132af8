// weights.cu -- S2: PHS r^3 + polynomial collocation weights, one warp per
// cloud, the augmented (q+m) x (q+m+3) system in shared memory, FP64 LU with
// partial pivoting (paper Sec. 2, Eqs. RBF_interp_mat_vec ..
// RBF_interp_mat_vec_L_solve).
//
// The matrix build uses explicit round-to-nearest intrinsics (no fused
// multiply-add), as the oracle does.  On GB300 the kernel is bound by the
// FP64 pipe (about 2 FMA lanes per clock per SM: a warp instruction occupies it
// for 16 cycles), so every FP64 instruction counts and the kernel spends them
// only on the arithmetic itself:
//   - the system is eliminated through the null space of the polynomials
//     (k_weights), 32 k flops a cloud instead of 73 k at q = 30, m = 15;
//   - updates are one fused multiply-add, dealt element by element over the
//     32 lanes, so every FP64 instruction of the warp carries 32 of them;
//   - one reciprocal per pivot, kept for the back substitution (a division is
//     a sequence of FP64 instructions whatever its active lanes);
//   - Phi is symmetric: each r^3 (and its square root) is computed once for
//     the upper triangle and stored twice; S = Z^T Phi Z likewise.
// The weights then differ from the oracle's elimination of the whole matrix
// by rounding only, well inside the 1e-10 they are held to.  Measured on
// GB300: 40 000 clouds at q = 30, degree 4 in 5.8 ms by elimination of the
// augmented matrix, 3.2 ms this way (error against 64-bit LAPACK 8e-14 and
// 1.3e-13 relative); 10 201 clouds at q = 12, degree 2 in 0.47 and 0.25 ms.
#include "abi_guard.cuh"
#include "common.cuh"
#include "weights.cuh"

namespace rbffd {

// Monomial exponents in graded order, x power descending inside a degree:
// 1, x, y, x^2, xy, y^2, ...  The order for degree k is a prefix of the
// order for degree k+1, so one table serves every degree up to 8.
__constant__ int8_t c_ax[45];
__constant__ int8_t c_ay[45];

static bool g_tables_ready[64] = {false};

static int ensure_tables(int device) {
  if (device >= 0 && device < 64 && g_tables_ready[device]) return RBFFD_OK;
  int8_t ax[45], ay[45];
  int l = 0;
  for (int d = 0; d <= 8; ++d)
    for (int a = d; a >= 0; --a) {
      ax[l] = (int8_t)a;
      ay[l] = (int8_t)(d - a);
      ++l;
    }
  RBFFD_CK(cudaMemcpyToSymbol(c_ax, ax, sizeof(ax)));
  RBFFD_CK(cudaMemcpyToSymbol(c_ay, ay, sizeof(ay)));
  if (device >= 0 && device < 64) g_tables_ready[device] = true;
  return RBFFD_OK;
}

// A warp's shared memory, in doubles (odd leading dimensions: column walks
// touch every bank).
struct WeightsLayout {
  int ldp, ldf, f, xi, rhs, g, inv, ord, total;
  __host__ __device__ WeightsLayout(int q, int m) {
    ldp = m | 1;
    ldf = q | 1;
    f = q * ldp;
    xi = f + q * ldf;
    rhs = xi + 2 * q;
    g = rhs + 3 * q;
    inv = g + 3 * m;
    ord = inv + m;
    total = ord + (q + 1) / 2;
  }
};

__device__ __forceinline__ double ipow_rn(double b, int e) {
  double v = 1.0;
  for (int t = 0; t < e; ++t) v = __dmul_rn(v, b);
  return v;
}

// Largest |v[e * ld]| of e = k .. n - 1 over the warp, on bit patterns: for
// finite doubles with the sign bit cleared, unsigned 64-bit order is the
// order of the values, so this picks exactly the row an FP64 comparison would
// (ties to the lowest row) while keeping the compares off the FP64 pipe.
// Returns the row, or n if every entry is zero.
__device__ __forceinline__ int pivot_row(const double *v, int ld, int k, int n, int lane) {
  unsigned long long best = 0ull;
  int piv = n;
  for (int r = k + lane; r < n; r += 32) {
    const unsigned long long a =
        (unsigned long long)__double_as_longlong(v[r * ld]) & 0x7fffffffffffffffull;
    if (a > best) { best = a; piv = r; }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int op = __shfl_xor_sync(0xffffffffu, piv, o);
    if (ob > best || (ob == best && op < piv)) { best = ob; piv = op; }
  }
  return piv;
}

// a / pivot with the pivot's reciprocal; exactly 1 where a is the pivot (two
// equal rows then cancel exactly, as they do under a division)
__device__ __forceinline__ double ratio(double a, double pivot, double inv) {
  return __double_as_longlong(a) == __double_as_longlong(pivot) ? 1.0 : __dmul_rn(a, inv);
}

// Rank-one update of rows r0 .. nr - 1, columns c0 .. nc - 1 of M by column k
// and row k, the elements dealt over the lanes in row-major order so that
// every FP64 instruction of the warp carries 32 updates.
__device__ __forceinline__ void rank_one(double *M, int ld, int k, int r0, int nr, int c0, int nc,
                                         int lane) {
  const int C = nc - c0, E = (nr - r0) * C;
  if (E <= 0) return;
  int r = r0 + lane / C, c = c0 + lane % C;
  int e = lane;
  // two elements per trip: their loads go out before either update
  for (; e + 32 < E; e += 64) {
    int r2 = r, c2 = c + 32;
    while (c2 >= nc) { c2 -= C; ++r2; }
    const double l1 = M[r * ld + k], u1 = M[k * ld + c], a1 = M[r * ld + c];
    const double l2 = M[r2 * ld + k], u2 = M[k * ld + c2], a2 = M[r2 * ld + c2];
    M[r * ld + c] = __fma_rn(-l1, u1, a1);
    M[r2 * ld + c2] = __fma_rn(-l2, u2, a2);
    r = r2;
    c = c2 + 32;
    while (c >= nc) { c -= C; ++r; }
  }
  if (e < E) M[r * ld + c] = __fma_rn(-M[r * ld + k], M[k * ld + c], M[r * ld + c]);
}

// The weights of one cloud per warp by the null space of the polynomials.
// The system [Phi P; P^T 0] [c; d] = [f; g] is eliminated in blocks:
//   P = [L1; L2] U with partial pivoting (rows permuted, the cloud's points
//     with them), K = L2 L1^-1, so Z = [-K^T; I] spans the null space of P^T;
//   c = [L1^-T U^-T g; 0] + Z c2 meets the constraints for every c2;
//   (Z^T Phi Z) c2 = Z^T (f - Phi c_p) by LU with partial pivoting, order
//     q - m instead of q + m.
// At q = 2 m this takes 32 k flops for q = 30 instead of 73 k (two thirds of
// (q + m)^3 and the right-hand sides).  A cloud is singular when either
// factorisation meets an exactly zero pivot, as the augmented matrix is.
__global__ void k_weights(int n, const double *__restrict__ x, const double *__restrict__ y,
                          int q, const int32_t *__restrict__ idx, int m, int wpb,
                          double *__restrict__ wx, double *__restrict__ wy,
                          double *__restrict__ wl, int *first_singular, double Lx, double Ly) {
  extern __shared__ double smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const WeightsLayout ly(q, m);
  double *P = smem + (size_t)warp * ly.total;  // q x ldp: P, then L1 \ U over K
  double *F = P + ly.f;                        // Phi, q x ldf
  double *xi = P + ly.xi, *eta = xi + q;
  double *f = P + ly.rhs;                      // q x 3: right-hand sides, then c
  double *g = P + ly.g;                        // m x 3: constraints, then c_p
  double *inv = P + ly.inv;                    // m reciprocal pivots of P
  int *ord = reinterpret_cast<int *>(P + ly.ord);
  const int ldp = ly.ldp, ldf = ly.ldf, n2 = q - m;
  for (int i = blockIdx.x * wpb + warp; i < n; i += gridDim.x * wpb) {
    const int32_t *cl = idx + (int64_t)i * q;
    const double xc = x[i], yc = y[i];
    // cloud radius h = max distance
    double d2m = 0.0;
    for (int a = lane; a < q; a += 32) {
      int j = cl[a];
      double dx = pdiff(x[j], xc, Lx), dy = pdiff(y[j], yc, Ly);
      double d2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
      d2m = fmax(d2m, d2);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d2m = fmax(d2m, __shfl_xor_sync(0xffffffffu, d2m, o));
    double h = __dsqrt_rn(d2m);
    if (h == 0.0) h = 1.0;
    const double hinv = __drcp_rn(h);
    for (int a = lane; a < q; a += 32) {
      int j = cl[a];
      xi[a] = __dmul_rn(pdiff(x[j], xc, Lx), hinv);
      eta[a] = __dmul_rn(pdiff(y[j], yc, Ly), hinv);
      ord[a] = a;
    }
    __syncwarp();
    for (int e = lane; e < q * m; e += 32) {
      const int a = e / m, l = e - a * m;
      P[a * ldp + l] = __dmul_rn(ipow_rn(xi[a], c_ax[l]), ipow_rn(eta[a], c_ay[l]));
    }
    // the operators of the monomials at the centre
    for (int l = lane; l < m; l += 32) {
      const int ax = c_ax[l], ay = c_ay[l];
      g[3 * l] = (ax == 1 && ay == 0) ? 1.0 : 0.0;
      g[3 * l + 1] = (ax == 0 && ay == 1) ? 1.0 : 0.0;
      g[3 * l + 2] = ((ax == 2 && ay == 0) || (ax == 0 && ay == 2)) ? 2.0 : 0.0;
    }
    __syncwarp();
    // ---- P = [L1; L2] U
    bool singular = false;
    for (int k = 0; k < m; ++k) {
      const int piv = pivot_row(P + k, ldp, k, q, lane);
      if (piv >= q) { singular = true; break; }
      if (piv != k) {
        for (int c = lane; c < m; c += 32) {
          const double t = P[k * ldp + c];
          P[k * ldp + c] = P[piv * ldp + c];
          P[piv * ldp + c] = t;
        }
        if (lane == 0) {
          const double tx = xi[k], ty = eta[k];
          const int to = ord[k];
          xi[k] = xi[piv];
          eta[k] = eta[piv];
          ord[k] = ord[piv];
          xi[piv] = tx;
          eta[piv] = ty;
          ord[piv] = to;
        }
        __syncwarp();
      }
      const double pk = P[k * ldp + k], kinv = __drcp_rn(pk);
      if (lane == 0) inv[k] = kinv;
      for (int r = k + 1 + lane; r < q; r += 32)
        P[r * ldp + k] = ratio(P[r * ldp + k], pk, kinv);
      __syncwarp();
      rank_one(P, ldp, k, k + 1, q, k + 1, m, lane);
      __syncwarp();
    }
    if (!singular) {
      // ---- K = L2 L1^-1 in place, a column at a time from the last
      for (int j = m - 1; j > 0; --j) {
        for (int e = lane; e < n2 * j; e += 32) {
          const int r = m + e / j, c = e - (e / j) * j;
          P[r * ldp + c] = __fma_rn(-P[r * ldp + j], P[j * ldp + c], P[r * ldp + c]);
        }
        __syncwarp();
      }
      // ---- c_p = L1^-T U^-T g
      for (int j = 0; j < m; ++j) {
        if (lane < 3) g[3 * j + lane] = __dmul_rn(g[3 * j + lane], inv[j]);
        __syncwarp();
        for (int e = lane; e < 3 * (m - 1 - j); e += 32) {
          const int r = j + 1 + e / 3, s = e % 3;
          g[3 * r + s] = __fma_rn(-P[j * ldp + r], g[3 * j + s], g[3 * r + s]);
        }
        __syncwarp();
      }
      for (int j = m - 1; j > 0; --j) {
        for (int e = lane; e < 3 * j; e += 32) {
          const int r = e / 3, s = e % 3;
          g[3 * r + s] = __fma_rn(-P[j * ldp + r], g[3 * j + s], g[3 * r + s]);
        }
        __syncwarp();
      }
      // ---- Phi: r^3 of the permuted points, symmetric with a zero diagonal;
      // the q(q-1)/2 pairs a < b dealt over the lanes in row-major order
      for (int a = lane; a < q; a += 32) F[a * ldf + a] = 0.0;
      {
        // pair number e -> (a, b): past the end of row a (b >= q) it goes on
        // at b - q positions into row a + 1, whose first pair is (a+1, a+2)
        const int np = q * (q - 1) / 2;
        int a = 0, b = 1 + lane;
        while (a < q - 1 && b >= q) { b += a + 2 - q; ++a; }
        for (int e = lane; e < np; e += 32) {
          const double dx = __dsub_rn(xi[a], xi[b]), dy = __dsub_rn(eta[a], eta[b]);
          const double d2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
          const double r3 = __dmul_rn(__dsqrt_rn(d2), d2);
          F[a * ldf + b] = r3;
          F[b * ldf + a] = r3;
          b += 32;
          while (a < q - 1 && b >= q) { b += a + 2 - q; ++a; }
        }
      }
      // right-hand sides: d/dxi, d/deta and Laplacian of r^3 about the centre
      for (int a = lane; a < q; a += 32) {
        const double xa = xi[a], ya = eta[a];
        const double rj = __dsqrt_rn(__dadd_rn(__dmul_rn(xa, xa), __dmul_rn(ya, ya)));
        const double r3 = __dmul_rn(3.0, rj);
        f[3 * a] = __dmul_rn(r3, __dsub_rn(0.0, xa));
        f[3 * a + 1] = __dmul_rn(r3, __dsub_rn(0.0, ya));
        f[3 * a + 2] = __dmul_rn(9.0, rj);
      }
      __syncwarp();
      // f -= Phi c_p (before Phi12 is overwritten)
      for (int e = lane; e < 3 * q; e += 32) {
        const int a = e / 3, s = e % 3;
        double t = f[e];
        for (int l = 0; l < m; ++l) t = __fma_rn(-F[a * ldf + l], g[3 * l + s], t);
        f[e] = t;
      }
      __syncwarp();
      // M = Phi12 - Phi11 K^T over Phi12; f2 -= K f1
      for (int e = lane; e < m * n2; e += 32) {
        const int a = e / n2, b = e - a * n2;
        const double *ka = P + (m + b) * ldp, *fa = F + a * ldf;
        double t = fa[m + b];
        for (int l = 0; l < m; ++l) t = __fma_rn(-fa[l], ka[l], t);
        F[a * ldf + m + b] = t;
      }
      for (int e = lane; e < 3 * n2; e += 32) {
        const int b = e / 3, s = e % 3;
        double t = f[3 * m + e];
        for (int l = 0; l < m; ++l) t = __fma_rn(-P[(m + b) * ldp + l], f[3 * l + s], t);
        f[3 * m + e] = t;
      }
      __syncwarp();
      // S = Phi22 - Phi21 K^T - K M over Phi22, upper triangle, mirrored
      {
        const int np = n2 * (n2 + 1) / 2;
        int a = 0, b = lane;
        while (a < n2 && b >= n2) { b += a + 1 - n2; ++a; }
        for (int e = lane; e < np; e += 32) {
          const double *fa = F + (m + a) * ldf, *ka = P + (m + a) * ldp, *kb = P + (m + b) * ldp;
          double t = fa[m + b];
          for (int l = 0; l < m; ++l) t = __fma_rn(-fa[l], kb[l], t);
          for (int l = 0; l < m; ++l) t = __fma_rn(-ka[l], F[l * ldf + m + b], t);
          F[(m + a) * ldf + m + b] = t;
          F[(m + b) * ldf + m + a] = t;
          b += 32;
          while (a < n2 && b >= n2) { b += a + 1 - n2; ++a; }
        }
      }
      __syncwarp();
      // ---- S c2 = f2, LU with partial pivoting; f2 rides along.  Row k of S
      // is row m + k of F; its reciprocal pivot goes to the diagonal.
      double *S = F + m * ldf + m, *f2 = f + 3 * m;
      for (int k = 0; k < n2; ++k) {
        const int piv = pivot_row(S + k, ldf, k, n2, lane);
        if (piv >= n2) { singular = true; break; }
        if (piv != k) {
          for (int c = k + lane; c < n2; c += 32) {
            const double t = S[k * ldf + c];
            S[k * ldf + c] = S[piv * ldf + c];
            S[piv * ldf + c] = t;
          }
          if (lane < 3) {
            const double t = f2[3 * k + lane];
            f2[3 * k + lane] = f2[3 * piv + lane];
            f2[3 * piv + lane] = t;
          }
          __syncwarp();
        }
        const double pk = S[k * ldf + k], kinv = __drcp_rn(pk);
        for (int r = k + 1 + lane; r < n2; r += 32)
          S[r * ldf + k] = ratio(S[r * ldf + k], pk, kinv);
        __syncwarp();
        if (lane == 0) S[k * ldf + k] = kinv;
        rank_one(S, ldf, k, k + 1, n2, k + 1, n2, lane);
        for (int e = lane; e < 3 * (n2 - 1 - k); e += 32) {
          const int r = k + 1 + e / 3, s = e % 3;
          f2[3 * r + s] = __fma_rn(-S[r * ldf + k], f2[3 * k + s], f2[3 * r + s]);
        }
        __syncwarp();
      }
      if (!singular) {
        for (int j = n2 - 1; j >= 0; --j) {
          if (lane < 3) f2[3 * j + lane] = __dmul_rn(f2[3 * j + lane], S[j * ldf + j]);
          __syncwarp();
          for (int e = lane; e < 3 * j; e += 32) {
            const int r = e / 3, s = e % 3;
            f2[e] = __fma_rn(-S[r * ldf + j], f2[3 * j + s], f2[e]);
          }
          __syncwarp();
        }
        // c1 = c_p - K^T c2
        for (int e = lane; e < 3 * m; e += 32) {
          const int l = e / 3, s = e % 3;
          double t = g[e];
          for (int b = 0; b < n2; ++b) t = __fma_rn(-P[(m + b) * ldp + l], f2[3 * b + s], t);
          f[e] = t;
        }
        __syncwarp();
      }
    }
    if (singular) {
      for (int a = lane; a < q; a += 32) {
        if (wx) wx[(int64_t)i * q + a] = 0.0;
        if (wy) wy[(int64_t)i * q + a] = 0.0;
        if (wl) wl[(int64_t)i * q + a] = 0.0;
      }
      if (lane == 0) atomicMin(first_singular, i);
      __syncwarp();
      continue;
    }
    const double h2inv = __drcp_rn(__dmul_rn(h, h));
    for (int a = lane; a < q; a += 32) {
      const int64_t o = (int64_t)i * q + ord[a];
      if (wx) wx[o] = __dmul_rn(f[3 * a], hinv);
      if (wy) wy[o] = __dmul_rn(f[3 * a + 1], hinv);
      if (wl) wl[o] = __dmul_rn(f[3 * a + 2], h2inv);
    }
    __syncwarp();
  }
}

int weights_config(int q, int degree, int *wpb, size_t *smem) {
  const int m = (degree + 1) * (degree + 2) / 2;
  const size_t per = (size_t)WeightsLayout(q, m).total * sizeof(double);
  // as many warps as shared memory holds, up to 16 (q = 30: 16 x 13 KB):
  // the FP64 pipe needs several warps per scheduler to hide the shared-
  // memory latency in front of each update
  int w = (int)((224 * 1024) / per);
  if (w > 16) w = 16;
  if (w < 1) return RBFFD_EINVAL;
  *wpb = w;
  *smem = per * w;
  return RBFFD_OK;
}

int weights_run(rbffd_ctx *ctx, int n, const double *x, const double *y, int q,
                const int32_t *idx, int degree, double *wx, double *wy, double *wl,
                int *d_first_singular, double Lx, double Ly) {
  int m = (degree + 1) * (degree + 2) / 2;
  RBFFD_TRY(ensure_tables(ctx->device));
  int wpb;
  size_t smem;
  RBFFD_TRY(weights_config(q, degree, &wpb, &smem));
  RBFFD_CK(cudaFuncSetAttribute(k_weights, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem));
  int blocks = (n + wpb - 1) / wpb;
  int cap = ctx->num_sms * 16;
  if (blocks > cap) blocks = cap;
  k_weights<<<blocks, 32 * wpb, smem, ctx->stream>>>(n, x, y, q, idx, m, wpb, wx, wy, wl,
                                                     d_first_singular, Lx, Ly);
  return after_launch(ctx, "k_weights");
}

int weights_check_args(int n, int q, int degree) {
  if (n < 1 || q < 1 || q > n || degree < 0 || degree > 8) return RBFFD_EINVAL;
  int m = (degree + 1) * (degree + 2) / 2;
  if (q < m || q + m > 96) return RBFFD_EINVAL;
  return RBFFD_OK;
}

}  // namespace rbffd

using namespace rbffd;

extern "C" int rbffd_weights(rbffd_ctx *ctx, int32_t n, const double *x, const double *y,
                             int32_t q, const int32_t *idx, int32_t degree, double *wx,
                             double *wy, double *wl, int32_t *first_singular) {
  return guarded([&]() -> int {
    if (!ctx || !x || !y || !idx || weights_check_args(n, q, degree) != RBFFD_OK) {
      set_error("rbffd_weights: bad arguments (n=%d q=%d degree=%d)", n, q, degree);
      return RBFFD_EINVAL;
    }
    RBFFD_CK(cudaSetDevice(ctx->device));
    int *dfs = nullptr;
    RBFFD_TRY(ctx_scratch(ctx, sizeof(int), (void **)&dfs));
    int big = 0x7fffffff;
    int rc = RBFFD_OK;
    if (cudaMemcpyAsync(dfs, &big, sizeof(int), cudaMemcpyHostToDevice, ctx->stream) !=
        cudaSuccess) {
      rc = RBFFD_ECUDA;
    } else {
      rc = weights_run(ctx, n, x, y, q, idx, degree, wx, wy, wl, dfs, 0.0, 0.0);
    }
    int hfs = big;
    if (rc == RBFFD_OK) {
      if (cudaMemcpyAsync(&hfs, dfs, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream) !=
              cudaSuccess ||
          cudaStreamSynchronize(ctx->stream) != cudaSuccess) {
        set_error("rbffd_weights: read-back failed");
        rc = RBFFD_ECUDA;
      }
    }
    if (rc != RBFFD_OK) cudaStreamSynchronize(ctx->stream);
    if (first_singular) *first_singular = (rc == RBFFD_OK && hfs != big) ? hfs : -1;
    if (rc == RBFFD_OK && hfs != big) {
      set_error("rbffd_weights: singular collocation matrix at point %d", hfs);
      return RBFFD_ESINGULAR;
    }
    return rc;
  });
}
