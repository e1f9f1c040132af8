// resident.cuh -- building blocks of the Krylov kernels that keep a solve on
// chip: the matrix in registers, the gathered vectors in shared memory.
//
// A team of nb CTAs (the whole grid, or one thread-block cluster) shares one
// solve; CTA b owns the R = ceil(n / nb) consecutive rows from b R, T lanes a
// row.  Its rows' ELL entries reach a set of columns, the CTA's halo list
// (its own rows among them, consecutive, since a row's first entry is
// itself).  k_halo_build makes, once per build of a problem, the sorted list
// of every CTA and each entry's 16-bit place in it, so that a solve reads a
// vector's halo with one load an entry of the list and gathers from shared
// memory.
//
// Why: a solve of 10^3 .. 10^5 rows is bound by latency, not by bandwidth.
// Read from L2, a phase of the earlier kernels cost 2.5 - 8 us for loads
// whose bytes take 0.3 us (column and value, then the gather, each a round
// trip of 300 - 700 cycles, behind barriers that drain them); with the
// matrix in registers a phase is one round trip for the halo.
#pragma once
#include <cooperative_groups.h>

#include <cstring>

#include "common.cuh"
#include "inner_arith.cuh"

namespace rbffd {

constexpr int RES_NT = 1024;        // threads per CTA of a resident solve
constexpr int RES_MAXB = 160;       // CTAs of a team
constexpr int RES_CLUSTER = 16;     // most CTAs of a cluster team
// Most rows of a cluster team: where the FP64 solves stop gaining.  Outer
// iterations on Kovasznay lattices, cluster and grid, ms: 4 096 rows mixed 2.22
// and 2.80, FP64 multigrid 4.05 and 4.36, FP64 Jacobi 10.1 and 11.2 (900 rows: 1.8
// and 2.4, 2.8 and 3.3, 4.3 and 5.0); 5 184 rows mixed 2.67 and 2.93, FP64 5.20 and
// 4.58; 10 000 rows 3.40 and 2.97, 6.90 and 4.62.
constexpr int RES_CLUSTER_N = 4096;
constexpr int RES_HCAP = 8192;      // largest halo list (16-bit byte offsets of 8-byte entries)
constexpr int RES_MAXN = 150 * RES_NT;  // rows a team can own, one lane each
// Most dynamic shared memory of a resident launch.  Every launch allows its
// kernel this much, whatever it uses itself: the allowance belongs to the
// function on the device, and another context's thread that lowered it
// between this one's call and its launch would have the launch refused.
constexpr int RES_SMEM = 200 * 1024;

// The team's rows and halo lists of one problem (device arrays; plan on the host).
struct ResPlan {
  int nb = 0;                       // CTAs (0: no resident solves for this problem)
  int cluster = 0;                  // 1: the team is one cluster
  int R = 0, T = 1;                 // rows a CTA, lanes a row
  int hstride = 0;                  // entries between two CTAs' lists
  int hmax = 0;                     // longest list (0 until the build has read it back)
  const int32_t *hlist = nullptr;   // nb x hstride columns, ascending
  const int32_t *hinfo = nullptr;   // per CTA: length of its list, place of its first row
  const uint16_t *lidx = nullptr;   // ELL [q][ldn]: an entry's place in its CTA's list
  void *part = nullptr;             // RES_PART_BYTES of partial sums
};
// Partial sums of a grid team: two shares (a pair of single systems on one
// problem's memory takes one each) of two halves of up to 32 values of 8
// bytes.  Alternate exchanges of a solve use alternate halves, at offsets
// that no exchange's number of values or their type moves.
constexpr size_t RES_HALF_BYTES = 32 * RES_MAXB * 8;
constexpr size_t RES_SHARE_BYTES = 2 * RES_HALF_BYTES;
constexpr size_t RES_PART_BYTES = 2 * RES_SHARE_BYTES;
// Byte offset of value v of CTA b in the partial sums of exchange `epoch`
// whose values have `bytes` each.
__host__ __device__ constexpr size_t res_slot(unsigned int epoch, int v, int b, size_t bytes) {
  return (epoch & 1) * RES_HALF_BYTES + ((size_t)v * RES_MAXB + b) * bytes;
}
// The same for a cluster team's array in shared memory, halves of vmax values
// (the most of any exchange on that array), counted in values.
__host__ __device__ constexpr int res_cluster_slot(unsigned int epoch, int vmax, int v, int b) {
  return ((int)(epoch & 1) * vmax + v) * RES_CLUSTER + b;
}

// Team sizes a batched resident launch chooses from, and for a problem the
// longest halo list at each (0: the team would not fit its rows).
constexpr int RES_NSIZES = 15;
constexpr int RES_SIZES[RES_NSIZES] = {1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 152};
// Longest lists of the sizes that suit n rows to d_hm[RES_NSIZES] (device).
int res_halo_sizes(rbffd_ctx *ctx, int n, int q, int ldn, const int32_t *col, int *d_hm);

// Rows and lanes of a team for n rows (nb = 0 when a CTA would own more rows
// than it has threads).
ResPlan res_plan(rbffd_ctx *ctx, int n, int q);
// Lists of a packed matrix's columns; longest list to *d_hmax (device).
int res_halo_build(rbffd_ctx *ctx, const ResPlan &p, int n, int q, int ldn, const int32_t *col,
                   int32_t *hlist, int32_t *hinfo, uint16_t *lidx, int *d_hmax);
// Launch fn(args) on the plan's team: a cooperative grid, or one cluster.  False
// where the launch is refused -- a cluster of more than 8 CTAs or a CTA on every
// SM may not be there to have -- and the solve has to stream; an error that is
// no such refusal meets the streaming launch too, which reports it.  (Asking the
// occupancy before each launch instead cost 8 to 15 us a launch.)
bool res_launch(rbffd_ctx *ctx, const ResPlan &p, const void *fn, void *args, size_t smem);

namespace res {

namespace cg = cooperative_groups;

// ---- the team's exchange ------------------------------------------------

struct Team {
  unsigned int *cnt;   // grid team: the arrival counter (zeroed before the launch)
  int *err;            // error word of bounded waits
  int lb, nb, cluster;
  unsigned int epoch;  // exchanges made so far
};

template <typename P>
__device__ __forceinline__ P shfl_xor(P v, int o) {
  return __shfl_xor_sync(0xffffffffu, v, o);
}
__device__ __forceinline__ ff shfl_xor(ff v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
template <typename P>
__device__ __forceinline__ P shfl_at(P v, int src) {
  return __shfl_sync(0xffffffffu, v, src);
}
__device__ __forceinline__ ff shfl_at(ff v, int src) {
  return {__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src)};
}

template <typename P>
__device__ __forceinline__ P warp_total(P v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += shfl_xor(v, o);
  return v;
}

__host__ __device__ constexpr int pow2_ge(int v) { return v <= 1 ? 1 : 2 * pow2_ge((v + 1) / 2); }

// Warp totals of V values in log2 steps that halve the values a lane still
// holds: V + 5 - log2 V shuffles instead of 5 V.  Lane l ends with value
// l / (32 / pow2_ge(V)) in v[0].
template <int V, typename P>
__device__ __forceinline__ void warp_totals(P (&v)[pow2_ge(V)]) {
  const int lane = threadIdx.x & 31;
  int m = pow2_ge(V);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (m > 1) {
      m >>= 1;
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int i = 0; i < pow2_ge(V) / 2; ++i) {
        if (i < m) {
          const P send = up ? v[i] : v[i + m];
          const P keep = up ? v[i + m] : v[i];
          v[i] = keep + shfl_xor(send, o);
        }
      }
    } else {
      v[0] += shfl_xor(v[0], o);
    }
  }
}

__device__ __forceinline__ double ld_l2(const double *p) { return __ldcg(p); }
__device__ __forceinline__ float ld_l2(const float *p) { return __ldcg(p); }
__device__ __forceinline__ float2 ld_l2(const float2 *p) { return __ldcg(p); }
__device__ __forceinline__ float4 ld_l2(const float4 *p) { return __ldcg(p); }
__device__ __forceinline__ ff ld_l2(const ff *p) {
  const float2 t = __ldcg(reinterpret_cast<const float2 *>(p));
  return {t.x, t.y};
}

// All of the CTA's and, after it, the team's earlier writes are visible to
// the team's later L2 loads.  False: a wait gave up (grid teams only: a
// cluster's barrier is the hardware's, and every CTA takes the same branches
// up to it).
__device__ __forceinline__ bool team_barrier(Team &t) {
  __shared__ int s_ok;
  ++t.epoch;
  if (t.nb == 1) {
    __syncthreads();
    return true;
  }
  if (t.cluster) {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;"
                 ::: "memory");
    return true;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    cuda::atomic_ref<unsigned int, cuda::thread_scope_device> cnt(t.cnt[0]);
    cnt.fetch_add(1u, cuda::memory_order_release);
    const unsigned int target = t.epoch * (unsigned int)t.nb;
    bool ok = true;
    if (cnt.load(cuda::memory_order_acquire) < target) {
      const long long t0 = clock64(), lim = wait_cycles(t.err);
      for (unsigned int spin = 1; cnt.load(cuda::memory_order_acquire) < target; ++spin) {
        // another CTA gave up (it will not arrive): leave without the wait
        if ((spin & 1023u) == 0 && *(volatile int *)t.err != 0) {
          ok = false;
          break;
        }
        if (clock64() - t0 > lim) {
          ok = false;
          atomicExch(t.err, 1);
          break;
        }
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// active: false when the whole warp's values are zero (it then spends no
// arithmetic on them).
// Totals over the team of V values per thread, into tot[0..V) (shared; all
// threads may read it on return), with a team barrier on the way.  Sums run
// in a fixed order: every CTA gets bit-identical totals.  wsum: V x 32
// shared; cpart: 2 x VMAX x RES_CLUSTER shared (cluster teams), VMAX the most
// values of any exchange on that array; gpart: RES_SHARE_BYTES global (grid
// teams), for exchanges of any type and number of values.  A CTA that has
// left exchange e writes the partials of e + 1 while a slower one still reads
// those of e; it reaches e + 2 only after every CTA has arrived at e + 1, so
// after all reads of e.  Two halves are enough, then, as long as they are
// disjoint for every V and type of the exchanges that share the array.
template <int V, int VMAX, typename P>
__device__ __forceinline__ bool team_totals(Team &t, P (&val)[pow2_ge(V)], P *tot, P *wsum,
                                            P *cpart, void *gpart, bool active = true) {
  constexpr int VP = pow2_ge(V);
  static_assert(V <= VMAX, "a half of the cluster's array holds VMAX values");
  static_assert(res_slot(0, V, 0, sizeof(P)) <= RES_HALF_BYTES, "a half holds the values");
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (active) warp_totals<V>(val);
  else val[0] = P(0);
  if ((lane & (32 / VP - 1)) == 0 && lane / (32 / VP) < V)
    wsum[(lane / (32 / VP)) * 32 + w] = val[0];
  __syncthreads();
  const unsigned int ep = t.epoch;  // of this exchange, before its barrier
  auto slot = [&](int v, int b) {
    return reinterpret_cast<P *>(static_cast<char *>(gpart) + res_slot(ep, v, b, sizeof(P)));
  };
  if (w < V) {
    P s = lane < nw ? wsum[w * 32 + lane] : P(0);
    s = warp_total(s);
    if (t.nb == 1) {
      if (lane == 0) tot[w] = s;
    } else if (t.cluster) {
      P *dst = cpart + res_cluster_slot(ep, VMAX, w, t.lb);
      if (lane < t.nb) *cg::this_cluster().map_shared_rank(dst, lane) = s;
    } else if (lane == 0) {
      *slot(w, t.lb) = s;
    }
  }
  const bool ok = team_barrier(t);
  if (t.nb > 1) {
    if (w < V) {
      P s = P(0);
      if (t.cluster) {
        if (lane < t.nb) s = cpart[res_cluster_slot(ep, VMAX, w, lane)];
      } else {
        P p[RES_MAXB / 32];
#pragma unroll
        for (int u = 0; u < RES_MAXB / 32; ++u)
          p[u] = lane + 32 * u < t.nb ? ld_l2(slot(w, lane + 32 * u)) : P(0);
#pragma unroll
        for (int u = 0; u < RES_MAXB / 32; ++u) s += p[u];
      }
      s = warp_total(s);
      if (lane == 0) tot[w] = s;
    }
    __syncthreads();
  }
  return ok;
}

// The halo list of the CTA's rows [r0, r1) made by the CTA itself (a batched
// launch chooses its teams after the build): the sorted columns to list (n2
// at most), every entry's place to idx[j * ld + row].  bm: 2 ceil(n / 32)
// words of shared scratch.  The length and the place of the first row to
// *len and *own (shared).  Ends with a barrier.
__device__ __forceinline__ void halo_local(int n, int q, int ldn, const int32_t *__restrict__ col,
                                           int r0, int r1, unsigned int *bm, int *list,
                                           uint16_t *idx, int ld, int *len, int *own) {
  __shared__ unsigned int wtot[RES_NT / 32];
  const int W = (n + 31) / 32, nr = r1 - r0;
  unsigned int *pre = bm + W;
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
      if (list != nullptr) list[at] = 32 * k + o;
      ++at;
    }
  }
  __syncthreads();
  auto place = [&](int c) {
    return pre[c >> 5] + __popc(bm[c >> 5] & ((1u << (c & 31)) - 1u));
  };
  if (idx != nullptr)
    for (int e = threadIdx.x; e < nr * q; e += RES_NT) {
      const int j = e / nr, i = e - j * nr;
      idx[j * ld + i] = (uint16_t)place(__ldg(col + (size_t)j * ldn + r0 + i));
    }
  if (threadIdx.x == 0) {
    *len = (int)total;
    *own = nr > 0 ? (int)place(r0) : 0;
  }
  __syncthreads();
}

// ---- values of NR right-hand sides side by side -----------------------------

template <typename S, int NR>
struct __align__(sizeof(S) * NR) Vec {
  S x[NR];
};

template <typename S, int NR>
__device__ __forceinline__ Vec<S, NR> ldv(const Vec<S, NR> *p) {
  Vec<S, NR> r;
  if constexpr (sizeof(Vec<S, NR>) == 4) {
    const float t = __ldcg(reinterpret_cast<const float *>(p));
    memcpy(&r, &t, 4);
  } else if constexpr (sizeof(Vec<S, NR>) == 8) {
    const float2 t = __ldcg(reinterpret_cast<const float2 *>(p));
    memcpy(&r, &t, 8);
  } else {
    const float4 t = __ldcg(reinterpret_cast<const float4 *>(p));
    memcpy(&r, &t, 16);
  }
  return r;
}

// A thread's place in the team's row layout and its share of the matrix:
// entries lg, lg + T, ... of row i, at most E of them, in registers, each
// with its halo entry's byte offset (entry size ES) in 16 bits.
template <typename S, int E, int ES>
struct Rows {
  int i;          // the row, or -1
  int lg;         // lane of the row
  int rl;         // row within the CTA
  bool lead;      // first lane of a row
  S a[E];
  uint32_t off[(E + 1) / 2];

  __device__ __forceinline__ void place(int r0, int r1, int T) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int gpw = 32 / T, g = lane / T;
    lg = lane - g * T;
    rl = w * gpw + g;
    i = (g < gpw && r0 + rl < r1) ? r0 + rl : -1;
    lead = i >= 0 && lg == 0;
  }
  __device__ __forceinline__ void indices(int q, int ldn, int T,
                                          const uint16_t *__restrict__ lidx) {
#pragma unroll
    for (int u = 0; u < (E + 1) / 2; ++u) off[u] = 0;
#pragma unroll
    for (int u = 0; u < E; ++u) {
      const int j = lg + u * T;
      // entries past the row's end: value zero, at the row's own place
      uint32_t o = 0;
      if (i >= 0) o = (uint32_t)__ldg(lidx + (size_t)(j < q ? j : 0) * ldn + i) * (uint32_t)ES;
      off[u >> 1] |= o << (16 * (u & 1));
    }
  }
  __device__ __forceinline__ uint32_t at(int u) const {
    return (u & 1) ? off[u >> 1] >> 16 : off[u >> 1] & 0xffffu;
  }
};

}  // namespace res
}  // namespace rbffd
