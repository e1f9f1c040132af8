// weights.cu -- S2: PHS r^3 + polynomial collocation weights (paper Sec. 2, Eqs.
// RBF_interp_mat_vec .. RBF_interp_mat_vec_L_solve), 4 to 32 lanes a cloud: the
// polynomials' factors and Phi with three right-hand sides in shared memory,
// FP64 LU with partial pivoting of the polynomials (q x m) and of Phi on their
// null space (q - m).
//
// The matrix build uses explicit round-to-nearest intrinsics (no fused
// multiply-add), as the oracle does.  On GB300 the kernel is bound by the
// FP64 pipe (about 2 FMA lanes per clock per SM: a warp instruction occupies it
// for 16 cycles), so every FP64 instruction counts and the kernel spends them
// only on the arithmetic itself:
//   - the system is eliminated through the null space of the polynomials
//     (k_weights), 32 k flops a cloud instead of 73 k at q = 30, m = 15;
//   - updates are one fused multiply-add, dealt element by element over the
//     cloud's lanes, so every FP64 instruction of the warp carries 32 of them;
//   - one reciprocal per pivot, kept for the back substitution (a division is
//     a sequence of FP64 instructions whatever its active lanes), and small
//     clouds several to a warp, which then share it;
//   - a monomial is one product of two powers that are there;
//   - Phi is symmetric: each r^3 (and its square root) is computed once for
//     the upper triangle and stored twice; S = Z^T Phi Z likewise.
// The weights then differ from the oracle's elimination of the whole matrix
// by rounding only, well inside the 1e-10 they are held to.  Measured on
// GB300: 40 000 clouds at q = 30, degree 4 in 5.8 ms by elimination of the
// augmented matrix, 3.2 ms by the null space with a warp a cloud and 16 warps a
// block, 2.5 ms now: some 1 200 FP64 instructions a cloud, 19 000 cycles, keep
// the pipe busy (89% of its cycles); 10 201 clouds at q = 12, degree 2 in 0.47,
// 0.25 and 0.11 ms.  Relative error against 80-bit elimination over 800 clouds
// each, this kernel, the augmented elimination before it and an unfused one (d/dx,
// d/dy, Laplacian): degree 2 7.5e-15 7.5e-15 5.1e-15, 8.5e-15 8.8e-15 6.2e-15,
// 8.7e-15 8.6e-15 6.2e-15; degree 3 4.7e-14 4.5e-14 2.5e-14, 3.9e-14 3.9e-14
// 2.4e-14, 4.1e-14 3.9e-14 2.4e-14; degree 4 0.96e-13 1.24e-13 5.7e-14, 0.96e-13
// 0.93e-13 4.8e-14, 1.17e-13 1.02e-13 4.8e-14 (graded cylinder 8.3e-14 7.8e-14
// 3.5e-14, 5.9e-14 5.9e-14 3.0e-14, 6.3e-14 6.9e-14 2.9e-14); degree 5 3.8e-13
// 4.1e-13 1.6e-13, 5.9e-13 5.7e-13 1.4e-13, 7.0e-13 7.9e-13 1.5e-13: up to 1.4
// times the augmented elimination's, and below it in some.  It comes from the
// rounding of Phi's entries and of the sums that form S: with both exact 3e-16.
#include "abi_guard.cuh"
#include "common.cuh"
#include "weights.cuh"

namespace rbffd {

// A cloud's shared memory, in doubles (odd leading dimensions: column walks
// touch every bank).
struct WeightsLayout {
  int ldp, ldf, f, xi, ord, total;
  __host__ __device__ WeightsLayout(int q, int m) {
    ldp = m | 1;
    ldf = (q + 3) | 1;
    f = (q + 3) * ldp;
    xi = f + q * ldf;
    ord = xi + 2 * q;
    total = ord + (q + 1) / 2;
  }
};

// Largest |v[e * ld]| of e = k .. n - 1 over the cloud's LW lanes, on bit patterns: for
// finite doubles with the sign bit cleared, unsigned 64-bit order is the
// order of the values, so this picks exactly the row an FP64 comparison would
// (ties to the lowest row) while keeping the compares off the FP64 pipe.
// Returns the row, or n if every entry is zero.
template <int LW>
__device__ __forceinline__ int pivot_row(const double *v, int ld, int k, int n, int lane) {
  unsigned long long best = 0ull;
  int piv = n;
  for (int r = k + lane; r < n; r += LW) {
    const unsigned long long a =
        (unsigned long long)__double_as_longlong(v[r * ld]) & 0x7fffffffffffffffull;
    if (a > best) { best = a; piv = r; }
  }
#pragma unroll
  for (int o = LW / 2; o > 0; o >>= 1) {
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
template <int LW>
__device__ __forceinline__ void rank_one(double *M, int ld, int k, int r0, int nr, int c0, int nc,
                                         int lane) {
  const int C = nc - c0, E = (nr - r0) * C;
  if (E <= 0) return;
  int r = r0 + lane / C, c = c0 + lane % C;
  int e = lane;
  // two elements per trip: their loads go out before either update
  for (; e + LW < E; e += 2 * LW) {
    int r2 = r, c2 = c + LW;
    while (c2 >= nc) { c2 -= C; ++r2; }
    const double l1 = M[r * ld + k], u1 = M[k * ld + c], a1 = M[r * ld + c];
    const double l2 = M[r2 * ld + k], u2 = M[k * ld + c2], a2 = M[r2 * ld + c2];
    M[r * ld + c] = __fma_rn(-l1, u1, a1);
    M[r2 * ld + c2] = __fma_rn(-l2, u2, a2);
    r = r2;
    c = c2 + LW;
    while (c >= nc) { c -= C; ++r; }
  }
  if (e < E) M[r * ld + c] = __fma_rn(-M[r * ld + k], M[k * ld + c], M[r * ld + c]);
}

// The weights of one cloud per LW lanes by the null space of the polynomials.
// The system [Phi P; P^T 0] [c; d] = [f; g] is eliminated in blocks:
//   P = [L1; L2] U with partial pivoting (rows permuted, the cloud's points
//     with them), K = L2 L1^-1, so Z = [-K^T; I] spans the null space of P^T;
//   c = [c_p; 0] + Z c2 with c_p = L1^-T U^-T g meets the constraints for
//     every c2;
//   (Z^T Phi Z) c2 = Z^T (f - Phi [c_p; 0]) by LU with partial pivoting,
//     order q - m instead of q + m.
// The right-hand sides ride along: g^T as three more rows of P (which become
// c_p^T by the steps that make K), f as three more columns of Phi.
// At q = 2 m this takes 32 k flops for q = 30 instead of 73 k (two thirds of
// (q + m)^3 and the right-hand sides).  A cloud is singular when either
// factorisation meets an exactly zero pivot, as the augmented matrix is; two
// cases that there cancel exactly and here only up to rounding are looked for:
// coinciding points (S is made by symmetry, which tells its two equal rows
// apart) and points on one line through the centre (x and y are one column).
// Lanes a cloud: a warp's clouds share the instructions that one lane would
// do for all (reciprocals) and the part-filled last ones of every loop.
template <int LW>
__global__ void __launch_bounds__(32)
    k_weights(int n, const double *__restrict__ x, const double *__restrict__ y, int q,
              const int32_t *__restrict__ idx, int m, int degree, double *__restrict__ wx,
              double *__restrict__ wy, double *__restrict__ wl, int *first_singular, double Lx,
              double Ly) {
  extern __shared__ double smem[];
  const int sub = threadIdx.x / LW, lane = threadIdx.x % LW;
  const WeightsLayout ly(q, m);
  double *P = smem + (size_t)sub * ly.total;  // (q + 3) x ldp: P, then L1 \ U over K, c_p^T
  double *F = P + ly.f;                       // q x ldf: Phi, then the right-hand sides
  double *xi = P + ly.xi, *eta = xi + q;
  int *ord = reinterpret_cast<int *>(P + ly.ord);
  const int ldp = ly.ldp, ldf = ly.ldf, n2 = q - m;
  // the warp's lanes stay together: past the last cloud they repeat it and
  // write nothing
  const int i0 = blockIdx.x * (32 / LW);
  const bool out = i0 + sub < n;
  const int i = out ? i0 + sub : n - 1;
  const int32_t *cl = idx + (int64_t)i * q;
  const double xc = x[i], yc = y[i];
  // cloud radius h = max distance
  double d2m = 0.0;
  for (int a = lane; a < q; a += LW) {
    int j = cl[a];
    double dx = pdiff(x[j], xc, Lx), dy = pdiff(y[j], yc, Ly);
    double d2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
    d2m = fmax(d2m, d2);
  }
#pragma unroll
  for (int o = LW / 2; o > 0; o >>= 1) d2m = fmax(d2m, __shfl_xor_sync(0xffffffffu, d2m, o));
  double h = __dsqrt_rn(d2m);
  if (h == 0.0) h = 1.0;
  const double hinv = __drcp_rn(h);
  for (int a = lane; a < q; a += LW) {
    int j = cl[a];
    const double xa = __dmul_rn(pdiff(x[j], xc, Lx), hinv),
                 ya = __dmul_rn(pdiff(y[j], yc, Ly), hinv);
    xi[a] = xa;
    eta[a] = ya;
    ord[a] = a;
    // monomials in graded order: degree d starts at d (d + 1) / 2 with x^d
    // and ends with y^d; those between from the powers
    double *p = P + a * ldp;
    double px = 1.0, py = 1.0;
    p[0] = 1.0;
    for (int d = 1; d <= degree; ++d) {
      px = __dmul_rn(px, xa);
      py = __dmul_rn(py, ya);
      double *pd = p + d * (d + 1) / 2;
      pd[0] = px;
      pd[d] = py;
      for (int b = 1; b < d; ++b)  // x^(d-b) y^b
        pd[b] = __dmul_rn(p[(d - b) * (d - b + 1) / 2], p[b * (b + 1) / 2 + b]);
    }
  }
  // the operators of the monomials at the centre: d/dx of x, d/dy of y, the
  // Laplacian of x^2 and y^2
  for (int e = lane; e < 3 * m; e += LW) {
    const int s = e / m, l = e - s * m;
    P[(q + s) * ldp + l] = s < 2 ? (l == s + 1 ? 1.0 : 0.0) : l == 3 || l == 5 ? 2.0 : 0.0;
  }
  __syncwarp();
  // all on the line through the centre and the last point?
  int off = degree < 1;
  {
    const double xl = xi[q - 1], yl = eta[q - 1];
    for (int a = lane; a < q; a += LW)
      off |= __double_as_longlong(__dsub_rn(__dmul_rn(xi[a], yl), __dmul_rn(xl, eta[a]))) << 1 != 0;
    off |= ((__double_as_longlong(xl) | __double_as_longlong(yl)) << 1) == 0;
  }
#pragma unroll
  for (int o = LW / 2; o > 0; o >>= 1) off |= __shfl_xor_sync(0xffffffffu, off, o);
  __syncwarp();
  // ---- P = [L1; L2] U
  bool singular = off == 0;
  for (int k = 0; k < m; ++k) {
    int piv = pivot_row<LW>(P + k, ldp, k, q, lane);
    if (piv >= q) { singular = true; piv = k; }
    if (piv != k) {
      for (int c = lane; c < m; c += LW) {
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
    }
    __syncwarp();
    const double pk = P[k * ldp + k], kinv = __drcp_rn(pk);
    for (int r = k + 1 + lane; r < q + 3; r += LW)
      P[r * ldp + k] = ratio(P[r * ldp + k], pk, kinv);
    __syncwarp();
    rank_one<LW>(P, ldp, k, k + 1, q + 3, k + 1, m, lane);
    __syncwarp();
  }
  // ---- K = L2 L1^-1 and c_p^T in place, a column at a time from the last
  for (int j = m - 1; j > 0; --j) {
    for (int e = lane; e < (n2 + 3) * j; e += LW) {
      const int r = m + e / j, c = e - (e / j) * j;
      P[r * ldp + c] = __fma_rn(-P[r * ldp + j], P[j * ldp + c], P[r * ldp + c]);
    }
    __syncwarp();
  }
  // ---- Phi: r^3 of the permuted points, symmetric with a zero diagonal;
  // the q(q-1)/2 pairs a < b dealt over the lanes in row-major order
  for (int a = lane; a < q; a += LW) F[a * ldf + a] = 0.0;
  int twice = 0;  // two points in one place: two equal rows
  {
    // pair number e -> (a, b): past the end of row a (b >= q) it goes on
    // at b - q positions into row a + 1, whose first pair is (a+1, a+2)
    const int np = q * (q - 1) / 2;
    int a = 0, b = 1 + lane;
    while (a < q - 1 && b >= q) { b += a + 2 - q; ++a; }
    for (int e = lane; e < np; e += LW) {
      const double dx = __dsub_rn(xi[a], xi[b]), dy = __dsub_rn(eta[a], eta[b]);
      twice |= ((__double_as_longlong(dx) | __double_as_longlong(dy)) << 1) == 0;
      const double d2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
      const double r3 = __dmul_rn(__dsqrt_rn(d2), d2);
      F[a * ldf + b] = r3;
      F[b * ldf + a] = r3;
      b += LW;
      while (a < q - 1 && b >= q) { b += a + 2 - q; ++a; }
    }
  }
#pragma unroll
  for (int o = LW / 2; o > 0; o >>= 1) twice |= __shfl_xor_sync(0xffffffffu, twice, o);
  singular |= twice != 0;
  // right-hand sides: d/dxi, d/deta and Laplacian of r^3 about the centre
  for (int a = lane; a < q; a += LW) {
    const double xa = xi[a], ya = eta[a];
    const double rj = __dsqrt_rn(__dadd_rn(__dmul_rn(xa, xa), __dmul_rn(ya, ya)));
    const double r3 = __dmul_rn(3.0, rj);
    double *f = F + a * ldf + q;
    f[0] = __dmul_rn(r3, __dsub_rn(0.0, xa));
    f[1] = __dmul_rn(r3, __dsub_rn(0.0, ya));
    f[2] = __dmul_rn(9.0, rj);
  }
  __syncwarp();
  // [M f1] = [Phi12 f1] - Phi11 [K^T c_p] over [Phi12 f1]
  for (int e = lane; e < m * (n2 + 3); e += LW) {
    const int a = e / (n2 + 3), b = e - a * (n2 + 3);
    const double *kb = P + (m + b) * ldp, *fa = F + a * ldf;
    double t = fa[m + b];
    for (int l = 0; l < m; ++l) t = __fma_rn(-fa[l], kb[l], t);
    F[a * ldf + m + b] = t;
  }
  __syncwarp();
  // [S f2] = [Phi22 f2] - Phi21 [K^T c_p] - K [M f1] over [Phi22 f2], the
  // upper triangle of S, mirrored
  {
    const int w = n2 + 3, np = n2 * (n2 + 1) / 2 + 3 * n2;
    int a = 0, b = lane;
    while (a < n2 && b >= w) { b += a + 1 - w; ++a; }
    for (int e = lane; e < np; e += LW) {
      const double *fa = F + (m + a) * ldf, *ka = P + (m + a) * ldp, *kb = P + (m + b) * ldp;
      double t = fa[m + b];
      for (int l = 0; l < m; ++l) t = __fma_rn(-fa[l], kb[l], t);
      for (int l = 0; l < m; ++l) t = __fma_rn(-ka[l], F[l * ldf + m + b], t);
      F[(m + a) * ldf + m + b] = t;
      if (b < n2) F[(m + b) * ldf + m + a] = t;
      b += LW;
      while (a < n2 && b >= w) { b += a + 1 - w; ++a; }
    }
  }
  __syncwarp();
  // ---- S c2 = f2, LU with partial pivoting; f2 (three more columns) rides
  // along.  Row k of S is row m + k of F; its reciprocal pivot goes to the
  // diagonal.
  double *S = F + m * ldf + m;
  for (int k = 0; k < n2; ++k) {
    int piv = pivot_row<LW>(S + k, ldf, k, n2, lane);
    if (piv >= n2) { singular = true; piv = k; }
    if (piv != k)
      for (int c = k + lane; c < n2 + 3; c += LW) {
        const double t = S[k * ldf + c];
        S[k * ldf + c] = S[piv * ldf + c];
        S[piv * ldf + c] = t;
      }
    __syncwarp();
    const double pk = S[k * ldf + k], kinv = __drcp_rn(pk);
    for (int r = k + 1 + lane; r < n2; r += LW)
      S[r * ldf + k] = ratio(S[r * ldf + k], pk, kinv);
    __syncwarp();
    if (lane == 0) S[k * ldf + k] = kinv;
    rank_one<LW>(S, ldf, k, k + 1, n2, k + 1, n2 + 3, lane);
    __syncwarp();
  }
  for (int j = n2 - 1; j >= 0; --j) {
    double *fj = S + j * ldf + n2;
    if (lane < 3) fj[lane] = __dmul_rn(fj[lane], S[j * ldf + j]);
    __syncwarp();
    for (int e = lane; e < 3 * j; e += LW) {
      const int r = e / 3, s = e % 3;
      double *fr = S + r * ldf + n2 + s;
      *fr = __fma_rn(-S[r * ldf + j], fj[s], *fr);
    }
    __syncwarp();
  }
  // c1 = c_p - K^T c2, over f1
  for (int e = lane; e < 3 * m; e += LW) {
    const int l = e / 3, s = e % 3;
    double t = P[(q + s) * ldp + l];
    for (int b = 0; b < n2; ++b) t = __fma_rn(-P[(m + b) * ldp + l], S[b * ldf + n2 + s], t);
    F[l * ldf + q + s] = t;
  }
  __syncwarp();
  if (out) {
    const double h2inv = __drcp_rn(__dmul_rn(h, h));
    for (int a = lane; a < q; a += LW) {
      const int64_t o = (int64_t)i * q + ord[a];
      const double *c = F + a * ldf + q;
      if (wx) wx[o] = singular ? 0.0 : __dmul_rn(c[0], hinv);
      if (wy) wy[o] = singular ? 0.0 : __dmul_rn(c[1], hinv);
      if (wl) wl[o] = singular ? 0.0 : __dmul_rn(c[2], h2inv);
    }
    if (singular && lane == 0) atomicMin(first_singular, i);
  }
}

// Shared memory an SM's clouds may take, and what every launch allows its
// kernel (resident.cuh: RES_SMEM says why not its own need).
constexpr int WEIGHTS_SMEM = 224 * 1024;

// Lanes a cloud of n (a block is one warp) and a block's shared memory.  The
// fewest lanes that leave each SM more than nine warps by shared memory and
// eight by n: with fewer the FP64 pipe waits for the steps' latencies.  Times
// in us with 32, 16, 8 and 4 lanes: 40 000 clouds, q = 12, m = 6: 658, 425,
// 347, 314 (11 warps with 4); q = 20, m = 10: 1188, 970, 922, 1386 (9.3 with
// 8, 4.6 with 4); q = 28, m = 10: 2051, 1876, 2518 (11 with 16); q = 30,
// m = 15: 2431, 2525 (9 with 16); q = 42, m = 21: 5691, 8368.  900 clouds,
// q = 12: 54, 55, 64, 81; 3 600, q = 20, m = 10: 137, 125, 127, 178.
// Blocks of 16 warps took 2 to 60% longer (2 500 clouds, q = 30: 327 us
// against 200): a new block needs only one warp's clouds to end.
int weights_config(int n, int q, int degree, int num_sms, int *lw, size_t *smem) {
  const int m = (degree + 1) * (degree + 2) / 2;
  const size_t per = (size_t)WeightsLayout(q, m).total * sizeof(double);
  const int fit = (int)(WEIGHTS_SMEM / per);  // clouds an SM
  if (fit < 1) return RBFFD_EINVAL;
  *lw = 4;
  while (*lw < 32 && (fit * *lw <= 9 * 32 || (long long)n * *lw < 8LL * 32 * num_sms)) *lw *= 2;
  *smem = per * (32 / *lw);
  return RBFFD_OK;
}

int weights_run(rbffd_ctx *ctx, int n, const double *x, const double *y, int q,
                const int32_t *idx, int degree, double *wx, double *wy, double *wl,
                int *d_first_singular, double Lx, double Ly) {
  const int m = (degree + 1) * (degree + 2) / 2;
  int lw;
  size_t smem;
  RBFFD_TRY(weights_config(n, q, degree, ctx->num_sms, &lw, &smem));
  const auto fn = lw == 4    ? k_weights<4>
                  : lw == 8  ? k_weights<8>
                  : lw == 16 ? k_weights<16>
                             : k_weights<32>;
  RBFFD_CK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, WEIGHTS_SMEM));
  const int cpb = 32 / lw;
  fn<<<(n + cpb - 1) / cpb, 32, smem, ctx->stream>>>(n, x, y, q, idx, m, degree, wx, wy, wl,
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
