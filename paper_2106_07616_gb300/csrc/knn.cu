// knn.cu -- S1: cloud selection (paper Sec. 2 clouds; one-sided clouds at
// boundaries, Sec. 3.1) with a uniform cell grid.
//
// Every point gets itself plus its q-1 nearest candidates under the total
// order (d^2, index).  d^2 is formed with explicit round-to-nearest
// intrinsics (no fused multiply-add), so the selected indices are exactly
// those of a brute-force search that evaluates dx*dx + dy*dy the same way.
// The ring search stops only when the current (q-1)-th distance is strictly
// below the clearance of the searched block of cells, so no unvisited point
// can enter or tie.  A periodic axis (period L > 0) measures differences to
// the nearest image and wraps the ring around the grid, each column (row)
// visited once at its smallest offset; a cell at wrapped offset r + 1 is
// still at least r cells away, so the clearance bound holds.
#include <mutex>
#include "abi_guard.cuh"
#include "common.cuh"
#include "knn.cuh"

namespace rbffd {

// The bounding box as four 64-bit keys: a key orders doubles as unsigned
// integers, and the minima are kept as maxima of the complement, so zeroed
// memory is the start of all four atomic maxima.
__device__ __forceinline__ unsigned long long order_key(double v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  return (u >> 63) ? ~u : u | 0x8000000000000000ull;
}
__device__ __forceinline__ double order_value(unsigned long long k) {
  return __longlong_as_double((long long)((k >> 63) ? k & 0x7fffffffffffffffull : ~k));
}

__global__ void __launch_bounds__(256) k_bbox(int n, const double *__restrict__ x,
                                              const double *__restrict__ y,
                                              unsigned long long *bbox) {
  unsigned long long k[4] = {0, 0, 0, 0};
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double a = x[i], b = y[i];
    if (a == a) {
      k[0] = max(k[0], ~order_key(a));
      k[1] = max(k[1], order_key(a));
    }
    if (b == b) {
      k[2] = max(k[2], ~order_key(b));
      k[3] = max(k[3], order_key(b));
    }
  }
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    for (int o = 16; o > 0; o >>= 1) k[v] = max(k[v], __shfl_xor_sync(0xffffffffu, k[v], o));
    if ((threadIdx.x & 31) == 0 && k[v]) atomicMax(bbox + v, k[v]);
  }
}

// A grid of at most m square cells over the bounding box: square so that a
// search block of cells has the same clearance on every side (in the graded
// cylinder cloud's 2:1 box, cells of the box's own shape doubled the
// candidates).
struct Grid {
  double x0, y0, ix, iy;  // origin, reciprocals of the cell sides
  // squares of the cells' sides, and of the smaller one, less what rounding may
  // move a point against the cells' edges: no point r cells away or more has a
  // smaller squared distance than r^2 times this
  double cx2, cy2, c2;
  int Gx, Gy;
};

__device__ __forceinline__ Grid make_grid(const unsigned long long *bbox, int m) {
  Grid g;
  double x1 = 0.0, y1 = 0.0;
  g.x0 = g.y0 = 0.0;
  if (bbox[1]) {
    g.x0 = order_value(~bbox[0]);
    x1 = order_value(bbox[1]);
  }
  if (bbox[3]) {
    g.y0 = order_value(~bbox[2]);
    y1 = order_value(bbox[3]);
  }
  const double w = x1 - g.x0, h = y1 - g.y0;
  // Gx = sqrt(m w / h) columns, within 1 .. m (also for a degenerate box)
  double gx = h > 0.0 ? floor(sqrt((double)m * (w / h))) : (w > 0.0 ? (double)m : 1.0);
  if (!(gx >= 1.0)) gx = 1.0;
  g.Gx = gx < (double)m ? (int)gx : m;
  g.Gy = max(1, m / g.Gx);
  double cx = w / g.Gx, cy = h / g.Gy;
  if (!(cx > 0.0)) cx = 1.0;
  if (!(cy > 0.0)) cy = 1.0;
  g.ix = 1.0 / cx;
  g.iy = 1.0 / cy;
  cx *= 1.0 - (1e-9 + 1e-15 * g.Gx);
  cy *= 1.0 - (1e-9 + 1e-15 * g.Gy);
  g.cx2 = cx * cx;
  g.cy2 = cy * cy;
  g.c2 = fmin(g.cx2, g.cy2);
  return g;
}

// Points outside the searched block, r cells around the point's own, have at
// least this squared distance: an axis along which the block holds every cell
// does not count.  (With the smaller of the two sides for both axes, a search in a
// box far longer than the grid could follow -- points on a line up to rounding
// -- walked every ring of the long axis.)
__device__ __forceinline__ double clearance2(const Grid &g, int r, bool all_x, bool all_y) {
  if (all_x && all_y) return __longlong_as_double(0x7ff0000000000000ll);
  return (double)r * (double)r * (all_x ? g.cy2 : all_y ? g.cx2 : g.c2);
}

// one thread's grid for the block (FP64 divisions take over 400 cycles); the
// search, in blocks of four points, reads the one that k_cell_count leaves
__device__ __forceinline__ const Grid &block_grid(const unsigned long long *bbox, int m) {
  __shared__ Grid g;
  if (threadIdx.x == 0) g = make_grid(bbox, m);
  __syncthreads();
  return g;
}

__device__ __forceinline__ int cell_coord(double v, double v0, double inv, int G) {
  const double t = floor((v - v0) * inv);
  return t >= 0.0 ? (t < (double)G ? (int)t : G - 1) : 0;
}

__global__ void k_cell_count(int n, const double *__restrict__ x, const double *__restrict__ y,
                             const unsigned long long *bbox, int m, int *__restrict__ cell,
                             int *__restrict__ cnt, Grid *grid) {
  const Grid &g = block_grid(bbox, m);
  if (blockIdx.x == 0 && threadIdx.x == 0) *grid = g;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int c = cell_coord(y[i], g.y0, g.iy, g.Gy) * g.Gx + cell_coord(x[i], g.x0, g.ix, g.Gx);
  cell[i] = c;
  atomicAdd(&cnt[c], 1);
}

// The sum of each tile of KNN_TILE counts.
constexpr int KNN_TILE = 1024;
__global__ void __launch_bounds__(KNN_TILE) k_tile_sums(const int *__restrict__ cnt,
                                                        int *__restrict__ sums, int m) {
  __shared__ int s[32];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, k = blockIdx.x * KNN_TILE + t;
  int v = k < m ? cnt[k] : 0;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) s[w] = v;
  __syncthreads();
  if (w == 0) {
    v = s[lane];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) sums[blockIdx.x] = v;
  }
}

// Exclusive scan of m counts, start[m] = total; a block a tile of 1024.  Each
// block sums what lies before its tile itself (a coalesced read, from L2)
// instead of waiting for the block before it: one block walking 75 000 counts
// took longer than the search of its points.  It reads the tiles' sums where
// they were made (sums not null), else the counts.
__global__ void __launch_bounds__(KNN_TILE) k_scan(const int *__restrict__ cnt,
                                                   const int *__restrict__ sums,
                                                   int *__restrict__ start, int m) {
  __shared__ int s[32], base_s;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, k0 = blockIdx.x * KNN_TILE;
  const int *lead = sums != nullptr ? sums : cnt;
  const int leads = sums != nullptr ? blockIdx.x : k0;
  int before = 0;
  for (int k = t; k < leads; k += KNN_TILE) before += lead[k];
  for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
  if (lane == 0) s[w] = before;
  __syncthreads();
  if (w == 0) {
    int v = s[lane];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) base_s = v;
  }
  __syncthreads();
  const int k = k0 + t, mine = k < m ? cnt[k] : 0;
  int inc = mine;
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) s[w] = inc;
  __syncthreads();
  int base = base_s;
  for (int v = 0; v < w; ++v) base += s[v];
  if (k < m) start[k] = base + inc - mine;
  if (k == m - 1) start[m] = base + inc;
}

// the counts run down to zero as the cells fill (the order within a cell does
// not matter: the search ranks by distance and index)
__global__ void k_cell_fill(int n, const int *__restrict__ cell, const int *__restrict__ start,
                            int *__restrict__ cnt, int *__restrict__ pts) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int c = cell[i];
  pts[start[c] + atomicSub(&cnt[c], 1) - 1] = i;
}

__device__ __forceinline__ bool key_less(double da, int ja, double db, int jb) {
  return da < db || (da == db && ja < jb);
}

// The search, one warp a point (bounded axes).  The candidates of the block
// of (2 r + 1)^2 cells around the point are contiguous runs of pts, one per
// row of cells, dealt over the lanes; those closer than the block's clearance
// are kept in shared memory.  With K of them or more no unvisited point can
// enter, and each one's place is the number of kept ones before it in the
// order (d^2, index), counted by every lane for its own: no sorting, no
// local memory.  A thread with an insertion-sorted list per point was bound
// by that list's local-memory traffic and by divergence: the whole search of
// 147 827 graded points at q = 20 took 1.20 ms with it, 0.55 ms this way, and
// 0.40 ms with the ranks counted by d^2 alone (the index decides only where a
// place stays empty), two candidates a lane at once, the grid's FP64 divisions
// made once instead of by every block of four points, and the block's limit
// one product.  It is bound
// by instruction issue and the FP64 distances (53% of the pipe before).
// Points whose block holds more than CAP candidates at every usable r go to
// the list `rest` (k_knn_query searches them).
constexpr int KNN_CAP = 256;

__global__ void __launch_bounds__(128) k_knn_warp(
    int n, const double *__restrict__ x, const double *__restrict__ y,
    const int8_t *__restrict__ tag, int q, const Grid *__restrict__ grid,
    const int *__restrict__ start, const int *__restrict__ pts, int32_t *__restrict__ idx,
    int *err, int *nrest, int *__restrict__ rest, int r_first) {
  __shared__ __align__(16) unsigned long long sd[4][KNN_CAP];
  __shared__ int sj[4][KNN_CAP], sp[4][32], sa[4][32];
  __shared__ uint16_t sr[4][KNN_CAP];
  const Grid g = *grid;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = blockIdx.x * 4 + w, K = q - 1;
  if (i >= n) return;
  const int64_t o = (int64_t)i * q;
  if (lane == 0) idx[o] = i;
  if (K == 0) return;
  const double xi = x[i], yi = y[i];
  const bool bnd = tag != nullptr && tag[i] != 0;
  const int ci = cell_coord(xi, g.x0, g.ix, g.Gx), cj = cell_coord(yi, g.y0, g.iy, g.Gy);
  unsigned long long *kd = sd[w];
  int *kj = sj[w];
  int kept = 0;
  int lo = 0, hi = 0x7fffffff;  // the largest r known to hold too few, the least too many
  bool fits = false;
  for (int r = r_first;;) {
    const int x0 = max(0, ci - r), x1 = min(g.Gx - 1, ci + r);
    const int y0 = max(0, cj - r), y1 = min(g.Gy - 1, cj + r), rows = y1 - y0 + 1;
    const bool all_x = x0 == 0 && x1 == g.Gx - 1, all_y = y0 == 0 && y1 == g.Gy - 1;
    const bool all = all_x && all_y;
    if (rows > 32) break;
    int s = 0, c = 0;
    if (lane < rows) {
      const int row = (y0 + lane) * g.Gx;
      s = __ldg(start + row + x0);
      c = __ldg(start + row + x1 + 1) - s;
    }
    int pre = c;  // inclusive scan of the rows' counts
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, pre, d);
      if (lane >= d) pre += v;
    }
    const int M = __shfl_sync(0xffffffffu, pre, 31);
    // run k ends before candidate sp[k]; candidate t of it is pts[sa[k] + t]
    __syncwarp();
    sp[w][lane] = lane < rows ? pre : 0x7fffffff;
    sa[w][lane] = s - (pre - c);
    __syncwarp();
    int row = 0;
    const double lim = clearance2(g, r, all_x, all_y);
    kept = 0;
    for (int t0 = 0; t0 < M; t0 += 32) {
      const int t = t0 + lane;
      bool keep = false;
      double d2 = 0.0;
      int j = 0;
      if (t < M) {
        while (t >= sp[w][row]) ++row;
        j = __ldg(pts + sa[w][row] + t);
        if (j != i && !(bnd && tag[j] != 0)) {
          const double dx = __dsub_rn(x[j], xi), dy = __dsub_rn(y[j], yi);
          d2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
          keep = d2 < lim || (all && !(d2 < lim));
        }
      }
      const unsigned int b = __ballot_sync(0xffffffffu, keep);
      const int p = kept + __popc(b & ((1u << lane) - 1u));
      if (keep && p < KNN_CAP) {
        kd[p] = (unsigned long long)__double_as_longlong(d2);
        kj[p] = j;
      }
      kept += __popc(b);
    }
    __syncwarp();
    if (kept <= KNN_CAP && (kept >= K || all)) {
      fits = true;
      break;
    }
    if (kept > KNN_CAP) hi = r;
    else lo = r;
    // the next block: between the two; a ring more while blocks are small (a
    // square one stays below 32 rows of cells), then twice the rings, so that
    // a long axis takes few steps
    if (hi - lo <= 1) break;
    const int up = lo < 16 ? lo + 1 : min(2 * lo, max(g.Gx, g.Gy));
    r = hi == 0x7fffffff ? up : lo == 0 ? hi - 1 : lo + (hi - lo) / 2;
  }
  if (!fits) {
    if (lane == 0) rest[atomicAdd(nrest, 1)] = i;
    return;
  }
  if (kept < K) {
    if (lane == 0) atomicExch(err, 1);
    for (int s = lane; s < K; s += 32) idx[o + 1 + s] = i;
    return;
  }
  // d^2 >= 0, so its bit pattern orders as its value.  Ranks by d^2 alone, two
  // candidates of a lane at once; where two are equal a place stays empty, and
  // the ranks are counted again with the index
  constexpr uint16_t EMPTY = 0xffff;
  uint16_t *kr = sr[w];
  for (int c = lane; c < kept; c += 32) kr[c] = EMPTY;
  __syncwarp();
  for (int c0 = 0; c0 < kept; c0 += 64) {
    const int ca = c0 + lane, cb = ca + 32;
    const unsigned long long da = ca < kept ? kd[ca] : 0ull, db = cb < kept ? kd[cb] : 0ull;
    int ra = 0, rb = 0, k = 0;
    for (; k + 2 <= kept; k += 2) {
      const ulonglong2 d = *reinterpret_cast<const ulonglong2 *>(kd + k);
      ra += d.x < da;
      rb += d.x < db;
      ra += d.y < da;
      rb += d.y < db;
    }
    if (k < kept) {
      ra += kd[k] < da;
      rb += kd[k] < db;
    }
    if (ca < kept) kr[ra] = (uint16_t)ca;
    if (cb < kept) kr[rb] = (uint16_t)cb;
  }
  __syncwarp();
  bool tie = false;
  for (int p = lane; p < kept; p += 32) {
    const int c = kr[p];
    tie |= c == EMPTY;
    if (p < K && c != EMPTY) idx[o + 1 + p] = kj[c];
  }
  if (!__any_sync(0xffffffffu, tie)) return;
  __syncwarp();
  for (int c = lane; c < kept; c += 32) {
    const unsigned long long dc = kd[c];
    const int jc = kj[c];
    int rank = 0;
    for (int k = 0; k < kept; ++k) {
      const unsigned long long dk = kd[k];
      rank += dk < dc || (dk == dc && kj[k] < jc);
    }
    if (rank < K) idx[o + 1 + rank] = jc;
  }
}

// Column (row) of the ring at offset d from c, or -1 to skip it: out of a
// bounded grid, or on a periodic axis not the smallest offset of its column.
__device__ __forceinline__ int ring_index(int c, int d, int G, bool periodic) {
  if (!periodic) {
    const int k = c + d;
    return (k < 0 || k >= G) ? -1 : k;
  }
  int canon = ((d % G) + G) % G;
  if (canon > G / 2) canon -= G;
  if (canon != d) return -1;
  return ((c + d) % G + G) % G;
}

// The general search, one thread a point with an insertion-sorted list: the
// points of `rest` (nrest of them), or all n (rest null): periodic axes.
template <int KMAX>
__global__ void __launch_bounds__(128) k_knn_query(
    int n, const double *__restrict__ x, const double *__restrict__ y,
    const int8_t *__restrict__ tag, int q, const Grid *__restrict__ grid,
    const int *__restrict__ start, const int *__restrict__ pts, int32_t *__restrict__ idx,
    int *err, const int *nrest, const int *rest, double Lx, double Ly) {
  if (rest != nullptr && blockIdx.x * blockDim.x >= *nrest) return;
  const Grid g = *grid;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (rest != nullptr ? *nrest : n)) return;
  if (rest != nullptr) i = rest[i];
  const int K = q - 1;
  int64_t o = (int64_t)i * q;
  idx[o] = i;
  if (K == 0) return;
  const double xi = x[i], yi = y[i];
  const bool bnd = tag != nullptr && tag[i] != 0;
  const int ci = cell_coord(xi, g.x0, g.ix, g.Gx), cj = cell_coord(yi, g.y0, g.iy, g.Gy);
  double bd[KMAX];
  int bj[KMAX];
  int cnt = 0;
  // offsets that exist along an axis: up to the grid's edges, or, periodic,
  // the smallest offset of every column (row)
  const int ymin = Ly > 0.0 ? -(g.Gy / 2) : -cj, ymax = Ly > 0.0 ? g.Gy / 2 : g.Gy - 1 - cj;
  const int xmin = Lx > 0.0 ? -(g.Gx / 2) : -ci, xmax = Lx > 0.0 ? g.Gx / 2 : g.Gx - 1 - ci;
  for (int r = 0;; ++r) {
    const bool ends = -r >= xmin || r <= xmax;
    for (int dy = max(-r, ymin); dy <= min(r, ymax); ++dy) {
      // the ring's first and last rows whole, of the others the two ends
      const bool edge = (dy == -r || dy == r);
      if (!edge && !ends) {
        dy = r - 1;
        continue;
      }
      const int yy = ring_index(cj, dy, g.Gy, Ly > 0.0);
      if (yy < 0) continue;
      const int stp = edge ? 1 : 2 * r;
      for (int dx = edge ? max(-r, xmin) : -r; dx <= (edge ? min(r, xmax) : r); dx += stp) {
        const int xx = ring_index(ci, dx, g.Gx, Lx > 0.0);
        if (xx < 0) continue;
        int c = yy * g.Gx + xx;
        for (int s = start[c], se = start[c + 1]; s < se; ++s) {
          int j = pts[s];
          if (j == i) continue;
          if (bnd && tag[j] != 0) continue;
          double ddx = pdiff(x[j], xi, Lx);
          double ddy = pdiff(y[j], yi, Ly);
          double d2 = __dadd_rn(__dmul_rn(ddx, ddx), __dmul_rn(ddy, ddy));
          int p;
          if (cnt < K) {
            p = cnt++;
          } else if (key_less(d2, j, bd[K - 1], bj[K - 1])) {
            p = K - 1;
          } else {
            continue;
          }
          while (p > 0 && key_less(d2, j, bd[p - 1], bj[p - 1])) {
            bd[p] = bd[p - 1];
            bj[p] = bj[p - 1];
            --p;
          }
          bd[p] = d2;
          bj[p] = j;
        }
      }
    }
    const bool all_x = -r <= xmin && r >= xmax, all_y = -r <= ymin && r >= ymax;
    if (all_x && all_y) break;  // every cell visited
    if (cnt == K && bd[K - 1] < clearance2(g, r, all_x, all_y)) break;
  }
  if (cnt < K) {
    atomicExch(err, 1);
    for (int s = 0; s < K; ++s) idx[o + 1 + s] = i;
    return;
  }
  for (int s = 0; s < K; ++s) idx[o + 1 + s] = bj[s];
}

// Tiles above which their sums are made first: below, every block's own sum is
// as fast as one launch more (150 000 points, 74 tiles: 273 us the whole call
// either way; 300 000, 147 tiles: 500 and 497 us), above, it grows with the
// square of the points (16 million: about 5 of 29 ms).
constexpr int KNN_SUM_TILES = 128;

int knn_workspace_bytes(int n, KnnLayout *lay) {
  int G = (int)ceil(sqrt((double)n / 2.0));
  if (G < 1) G = 1;
  const int m = G * G;
  lay->m = m;
  size_t off = 0;
  auto take = [&](size_t b) {
    size_t at = off;
    off += (b + 255) / 256 * 256;
    return at;
  };
  // bounding-box keys, error word, rest counter and cell counts: zeroed
  // together before every search
  lay->off_bbox = take(4 * sizeof(unsigned long long) + 2 * sizeof(int));
  lay->off_cnt = take((size_t)m * sizeof(int));
  lay->zero_bytes = off;
  lay->off_grid = take(sizeof(Grid));
  lay->off_cell = take((size_t)n * sizeof(int));
  lay->off_start = take((size_t)(m + 1) * sizeof(int));
  lay->off_sums = take((size_t)((m + KNN_TILE - 1) / KNN_TILE) * sizeof(int));
  lay->off_pts = take((size_t)n * sizeof(int));
  lay->bytes = off;
  return RBFFD_OK;
}

int knn_run(rbffd_ctx *ctx, void *ws, const KnnLayout &lay, int n, const double *x,
            const double *y, const int8_t *tag, int q, int32_t *idx, double Lx, double Ly) {
  char *b = (char *)ws;
  unsigned long long *bbox = (unsigned long long *)(b + lay.off_bbox);
  int *err = (int *)(bbox + 4), *nrest = err + 1;
  Grid *grid = (Grid *)(b + lay.off_grid);
  int *cell = (int *)(b + lay.off_cell);  // also, after the fill, the rest list
  int *cnt = (int *)(b + lay.off_cnt);
  int *start = (int *)(b + lay.off_start);
  int *pts = (int *)(b + lay.off_pts);
  const int m = lay.m;
  cudaStream_t st = ctx->stream;
  RBFFD_CK(cudaMemsetAsync(b, 0, lay.zero_bytes, st));
  const int nb = (n + 255) / 256;
  k_bbox<<<nb < 2 * ctx->num_sms ? nb : 2 * ctx->num_sms, 256, 0, st>>>(n, x, y, bbox);
  RBFFD_TRY(after_launch(ctx, "k_bbox"));
  k_cell_count<<<nb, 256, 0, st>>>(n, x, y, bbox, m, cell, cnt, grid);
  RBFFD_TRY(after_launch(ctx, "k_cell_count"));
  const int tiles = (m + KNN_TILE - 1) / KNN_TILE;
  int *sums = nullptr;
  if (tiles > KNN_SUM_TILES) {
    sums = (int *)(b + lay.off_sums);
    k_tile_sums<<<tiles, KNN_TILE, 0, st>>>(cnt, sums, m);
    RBFFD_TRY(after_launch(ctx, "k_tile_sums"));
  }
  k_scan<<<tiles, KNN_TILE, 0, st>>>(cnt, sums, start, m);
  RBFFD_TRY(after_launch(ctx, "k_scan"));
  k_cell_fill<<<nb, 256, 0, st>>>(n, cell, start, cnt, pts);
  RBFFD_TRY(after_launch(ctx, "k_cell_fill"));
  const int qb = (n + 127) / 128;
  int *rest = nullptr;
  if (!(Lx > 0.0) && !(Ly > 0.0)) {
    // about two points a cell: the circle of the q - 1 nearest has a radius of
    // sqrt((q - 1) / (2 pi)) cells
    int r_first = 1;
    while (6.2832 * r_first * r_first < q - 1) ++r_first;
    rest = cell;
    k_knn_warp<<<(n + 3) / 4, 128, 0, st>>>(n, x, y, tag, q, grid, start, pts, idx, err,
                                            nrest, rest, r_first);
    RBFFD_TRY(after_launch(ctx, "k_knn_warp"));
  }
  if (q - 1 <= 32) {
    k_knn_query<32><<<qb, 128, 0, st>>>(n, x, y, tag, q, grid, start, pts, idx, err, nrest,
                                        rest, Lx, Ly);
  } else if (q - 1 <= 64) {
    k_knn_query<64><<<qb, 128, 0, st>>>(n, x, y, tag, q, grid, start, pts, idx, err, nrest,
                                        rest, Lx, Ly);
  } else {
    k_knn_query<128><<<qb, 128, 0, st>>>(n, x, y, tag, q, grid, start, pts, idx, err, nrest,
                                         rest, Lx, Ly);
  }
  RBFFD_TRY(after_launch(ctx, "k_knn_query"));
  int herr = 0;
  RBFFD_CK(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st));
  RBFFD_CK(cudaStreamSynchronize(st));
  if (herr) {
    set_error("a boundary point has fewer than q-1 interior candidates");
    return RBFFD_EINVAL;
  }
  return RBFFD_OK;
}

}  // namespace rbffd

using namespace rbffd;

extern "C" int rbffd_build_stencils(rbffd_ctx *ctx, int32_t n, const double *x, const double *y,
                                    const int8_t *tag, int32_t q, int32_t *idx) {
  return guarded([&]() -> int {
    if (!ctx || !x || !y || !idx || n < 1 || q < 1 || q > n || q > 129) {
      set_error("rbffd_build_stencils: bad arguments (n=%d q=%d)", n, q);
      return RBFFD_EINVAL;
    }
    RBFFD_CK(cudaSetDevice(ctx->device));
    KnnLayout lay;
    knn_workspace_bytes(n, &lay);
    void *ws = nullptr;
    RBFFD_TRY(ctx_scratch(ctx, lay.bytes, &ws));
    return knn_run(ctx, ws, lay, n, x, y, tag, q, idx, 0.0, 0.0);
  });
}

// ---------------------------------------------------------------------------
// Cloud building without any device allocation.
//
// rbffd_build_stencils above takes its cell-grid workspace from the context,
// which allocates it at the first call and at larger ones.  Some callers
// cannot have that: a solver loop that must keep a fixed device-memory
// footprint once it has started, or an application whose other streams must
// not be stalled by the implicit device synchronisation of cudaMalloc.  For them,
// rbffd_build_stencils_static takes the same workspace from a fixed array in
// device global memory that is part of this library image.  Every GPU that
// loads the library holds the array (RBFFD_STATIC_SCRATCH_BYTES) until the
// process exits.

namespace rbffd {

static __device__ __align__(256) unsigned char g_knn_scratch[RBFFD_STATIC_SCRATCH_BYTES];

// Device address of g_knn_scratch per device.  In host code the symbol is
// only a host-side stand-in, so the address has to be asked of the runtime,
// once per device, with that device current.  The lookup runs under one
// std::once_flag per device, so host threads that make their first call on
// one device at the same time do not race on the cached pointer; the result
// (the address, or the CUDA error of the lookup) is published by call_once.
static void *g_knn_scratch_ptr[64] = {nullptr};
static cudaError_t g_knn_scratch_err[64];
static std::once_flag g_knn_scratch_once[64];

static int static_scratch(int device, void **out) {
  if (device < 0 || device >= 64) {
    set_error("rbffd_build_stencils_static: device %d not supported", device);
    return RBFFD_EINVAL;
  }
  std::call_once(g_knn_scratch_once[device], [device]() {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_knn_scratch);
    if (e == cudaSuccess && p == nullptr) e = cudaErrorInvalidSymbol;
    g_knn_scratch_err[device] = e;
    g_knn_scratch_ptr[device] = e == cudaSuccess ? p : nullptr;
  });
  if (g_knn_scratch_err[device] != cudaSuccess) {
    set_error("cudaGetSymbolAddress(static cloud scratch) failed: %s",
              cudaGetErrorString(g_knn_scratch_err[device]));
    return RBFFD_ECUDA;
  }
  *out = g_knn_scratch_ptr[device];
  return RBFFD_OK;
}

}  // namespace rbffd

extern "C" int rbffd_build_stencils_static(rbffd_ctx *ctx, int32_t n, const double *x,
                                           const double *y, const int8_t *tag, int32_t q,
                                           int32_t *idx) {
  return guarded([&]() -> int {
    if (!ctx || !x || !y || !idx || n < 1 || q < 1 || q > n || q > 129) {
      set_error("rbffd_build_stencils_static: bad arguments (n=%d q=%d)", n, q);
      return RBFFD_EINVAL;
    }
    if (n > RBFFD_STATIC_MAX_POINTS) {
      set_error("rbffd_build_stencils_static: n=%d exceeds the static limit of %d points", n,
                RBFFD_STATIC_MAX_POINTS);
      return RBFFD_EINVAL;
    }
    KnnLayout lay;
    knn_workspace_bytes(n, &lay);
    if (lay.bytes > sizeof(g_knn_scratch)) {
      set_error("rbffd_build_stencils_static: workspace of %zu bytes exceeds the %zu-byte array",
                lay.bytes, sizeof(g_knn_scratch));
      return RBFFD_EINVAL;
    }
    RBFFD_CK(cudaSetDevice(ctx->device));
    void *ws = nullptr;
    RBFFD_TRY(static_scratch(ctx->device, &ws));
    // knn_run clears the counters, cursors and error word it reads before
    // writing them, so the contents left by an earlier call do not matter.
    return knn_run(ctx, ws, lay, n, x, y, tag, q, idx, 0.0, 0.0);
  });
}
