// resident.cu -- teams and halo lists of the resident Krylov kernels
// (resident.cuh), made once per build of a problem.
#include "resident.cuh"

#include <algorithm>

#include "krylov.cuh"

namespace rbffd {

namespace {

// The halo list of CTA blockIdx.x's rows: the columns its ELL entries reach
// are marked in a bitmap of the n points in shared memory, a scan over the
// words' population counts gives every column its place, in ascending
// order.  One pass over the columns to mark, one to look the places up:
// 7 us for 40 000 x 30 entries, once per build.
__global__ void __launch_bounds__(RES_NT) k_halo_build(int n, int q, int ldn, int R, int hstride,
                                                       const int32_t *__restrict__ col,
                                                       int32_t *__restrict__ hlist,
                                                       int32_t *__restrict__ hinfo,
                                                       uint16_t *__restrict__ lidx, int *hmax) {
  extern __shared__ unsigned int bm[];
  const int W = (n + 31) / 32;
  unsigned int *pre = bm + W;
  __shared__ unsigned int wtot[RES_NT / 32];
  const int b = blockIdx.x, r0 = min(n, b * R), r1 = min(n, r0 + R), nr = r1 - r0;
  for (int k = threadIdx.x; k < W; k += RES_NT) bm[k] = 0;
  __syncthreads();
  for (int e = threadIdx.x; e < nr * q; e += RES_NT) {
    const int j = e / nr, i = r0 + e - j * nr;
    const int c = __ldg(col + (size_t)j * ldn + i);
    atomicOr(bm + (c >> 5), 1u << (c & 31));
  }
  __syncthreads();
  // exclusive scan of the words' counts: a run of words per thread, then
  // warps, then the block
  const int cw = (W + RES_NT - 1) / RES_NT, k0 = min(W, (int)threadIdx.x * cw),
            k1 = min(W, k0 + cw);
  unsigned int mine = 0;
  for (int k = k0; k < k1; ++k) mine += __popc(bm[k]);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned int inc = mine;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) wtot[w] = inc;
  __syncthreads();
  unsigned int base = 0, total = 0;
  for (int k = 0; k < RES_NT / 32; ++k) {
    if (k < w) base += wtot[k];
    total += wtot[k];
  }
  unsigned int at = base + inc - mine;
  for (int k = k0; k < k1; ++k) {
    pre[k] = at;
    unsigned int bits = bm[k];
    while (bits) {
      const int o = __ffs(bits) - 1;
      bits &= bits - 1;
      if (at < (unsigned int)hstride) hlist[(size_t)b * hstride + at] = 32 * k + o;
      ++at;
    }
  }
  __syncthreads();
  auto place = [&](int c) {
    return pre[c >> 5] + __popc(bm[c >> 5] & ((1u << (c & 31)) - 1u));
  };
  for (int e = threadIdx.x; e < nr * q; e += RES_NT) {
    const int j = e / nr, i = r0 + e - j * nr;
    lidx[(size_t)j * ldn + i] = (uint16_t)min(65535u, place(__ldg(col + (size_t)j * ldn + i)));
  }
  if (threadIdx.x == 0) {
    hinfo[2 * b] = (int)total;
    hinfo[2 * b + 1] = nr > 0 ? (int)place(r0) : 0;
    atomicMax(hmax, (int)total);
  }
}

// The longest list at each team size: CTA b is CTA b - first of size k's team.
struct SizeTable {
  int nb[RES_NSIZES], first[RES_NSIZES + 1];
};
__global__ void __launch_bounds__(RES_NT) k_halo_sizes(int n, int q, int ldn, SizeTable t,
                                                       const int32_t *__restrict__ col,
                                                       int *hm) {
  extern __shared__ unsigned int bm[];
  __shared__ int len, own;
  int k = 0;
  while (blockIdx.x >= t.first[k + 1]) ++k;
  const int R = (n + t.nb[k] - 1) / t.nb[k], b = blockIdx.x - t.first[k];
  const int r0 = min(n, b * R), r1 = min(n, r0 + R);
  res::halo_local(n, q, ldn, col, r0, r1, bm, nullptr, nullptr, 0, &len, &own);
  if (threadIdx.x == 0) atomicMax(hm + k, len);
}

}  // namespace

int res_halo_sizes(rbffd_ctx *ctx, int n, int q, int ldn, const int32_t *col, int *d_hm) {
  SizeTable t;
  int at = 0;
  for (int k = 0; k < RES_NSIZES; ++k) {
    t.first[k] = at;
    const int nb = t.nb[k] = RES_SIZES[k];
    if ((long long)nb * RES_NT >= n && nb <= ctx->num_sms) at += nb;
  }
  t.first[RES_NSIZES] = at;
  RBFFD_CK(cudaMemsetAsync(d_hm, 0, sizeof(int) * RES_NSIZES, ctx->stream));
  if (at == 0) return RBFFD_OK;
  const size_t smem = 2 * sizeof(unsigned int) * (size_t)((n + 31) / 32);
  RBFFD_CK(cudaFuncSetAttribute(k_halo_sizes, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(2 * sizeof(unsigned int) * ((RES_MAXN + 31) / 32))));
  k_halo_sizes<<<at, RES_NT, smem, ctx->stream>>>(n, q, ldn, t, col, d_hm);
  return after_launch(ctx, "k_halo_sizes");
}

ResPlan res_plan(rbffd_ctx *ctx, int n, int q) {
  ResPlan p;
  const int cap = ctx->num_sms < RES_MAXB ? ctx->num_sms : RES_MAXB;
  // eight lanes a row before the rows spread over fewer SMs
  long long want = ((long long)n * 8 + RES_NT - 1) / RES_NT;
  int nb = (int)(want < 1 ? 1 : want < cap ? want : cap);
  if ((long long)n > (long long)nb * RES_NT || n > RES_MAXN) return p;
  if (nb > 1 && n <= RES_CLUSTER_N) {
    p.cluster = 1;
    if (nb > RES_CLUSTER) nb = RES_CLUSTER;
  }
  p.nb = nb;
  p.R = (n + nb - 1) / nb;
  for (int t = 2; t <= 8; ++t)
    if ((32 / t) * (RES_NT / 32) >= p.R) p.T = t;
  // no list is longer than the cloud, or than its rows' entries
  p.hstride = (int)std::min({(long long)n, (long long)RES_HCAP, (long long)p.R * q});
  return p;
}

int res_halo_build(rbffd_ctx *ctx, const ResPlan &p, int n, int q, int ldn, const int32_t *col,
                   int32_t *hlist, int32_t *hinfo, uint16_t *lidx, int *d_hmax) {
  const size_t smem = 2 * sizeof(unsigned int) * (size_t)((n + 31) / 32);
  RBFFD_CK(cudaMemsetAsync(d_hmax, 0, sizeof(int), ctx->stream));
  RBFFD_CK(cudaFuncSetAttribute(k_halo_build, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(2 * sizeof(unsigned int) * ((RES_MAXN + 31) / 32))));
  k_halo_build<<<p.nb, RES_NT, smem, ctx->stream>>>(n, q, ldn, p.R, p.hstride, col, hlist, hinfo,
                                                    lidx, d_hmax);
  return after_launch(ctx, "k_halo_build");
}

bool res_launch(rbffd_ctx *ctx, const ResPlan &p, const void *fn, void *args, size_t smem) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.nb);
  cfg.blockDim = dim3(RES_NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = ctx->stream;
  cudaLaunchAttribute at[1];
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, RES_SMEM);
  if (p.cluster) {
    if (e == cudaSuccess && p.nb > 8)
      e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = p.nb;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = 1;
  void *kargs[] = {args};
  if (e == cudaSuccess) e = cudaLaunchKernelExC(&cfg, fn, kargs);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  ctx->launches++;
  return true;
}

}  // namespace rbffd
