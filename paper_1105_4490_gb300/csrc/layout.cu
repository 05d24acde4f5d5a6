// Geometry (Sec. 2): steepest descent on the energy of eq. graphenergysimple
// (Algorithm 4) inside the multilevel scheme of Algorithm 3.
//
// One step of a level, for every problem of a batch at once:
//   keys      cell of every point on a uniform grid over the bounding cube
//             (fp32, no FMA), row-major key of the finest cell
//   sort      counting sort by cell, the points of a cell by vertex; first
//             point of every finest cell recorded in a dense table, points
//             copied in that order
//   aggregate per cell weight and weighted mean: finest cells from their
//             points, coarser cells from their 2^d children (fixed order)
//   attract   y_n = sum_j c_j (x_n - z_j) (2-pin nets: c/2 (x_n - x_u))
//   repulse   near field exactly over the 3^d adjacent finest cells, far field
//             from the cells whose parent is adjacent to the target's parent
//             but which are not adjacent themselves; then the step
//             x_n <- x_n - s_t y_n / ||y_n|| and the next bounding box.
#include <algorithm>
#include <cmath>

#include <cooperative_groups.h>

#include "blocksort.cuh"
#include "layout.cuh"

namespace vmo {

namespace {

constexpr int kBlock = 256;

__host__ __device__ inline int64_t lvl_off(int d, int l) {
  // sum_{j<l} 2^(d j) = (2^(d l) - 1) / (2^d - 1)
  return ((int64_t(1) << (d * l)) - 1) / ((int64_t(1) << d) - 1);
}

__device__ inline int find_problem(const int64_t* __restrict__ base, int P, int64_t i) {
  int lo = 0, hi = P;  // base[lo] <= i < base[hi]
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (base[mid] <= i) lo = mid; else hi = mid;
  }
  return lo;
}

// Paired source tables.  The far field and the near field read their sources
// two at a time: sources 2j and 2j+1 share a pair of float4 (three for d = 4)
// holding each coordinate of both side by side, then both weights:
//   d <= 3: (x0, x1, y0, y1), (z0, z1, w0, w1)     (d = 2: z unused)
//   d = 4:  (x0, x1, y0, y1), (z0, z1, u0, u1), (w0, w1, -, -)
// so that one packed fp32x2 instruction (Blackwell f32x2 add / mul / fma)
// computes the same step for both sources.
template <int D>
struct Pair {
  static constexpr int N = D == 4 ? 3 : 2;  // float4 per pair
  static constexpr int WQ = D == 4 ? 2 : 1; // float4 holding the weights
  static constexpr int WO = D == 4 ? 0 : 2; // float offset of the weights in it
};

// Pair j of a table (read-only during the launch): one 32-byte load for
// d <= 3, where a pair starts on a 32-byte boundary.
template <int D>
__device__ __forceinline__ void pair_load(const float4* __restrict__ tab, int64_t j, float4* P) {
  const float4* p = tab + j * Pair<D>::N;
  if (Pair<D>::N == 2) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(P[0].x), "=f"(P[0].y), "=f"(P[0].z), "=f"(P[0].w), "=f"(P[1].x), "=f"(P[1].y), "=f"(P[1].z),
          "=f"(P[1].w)
        : "l"(p));
  } else {
#pragma unroll
    for (int i = 0; i < Pair<D>::N; ++i) P[i] = p[i];
  }
}
template <int D>
__device__ __forceinline__ void pair_zero(float4* P) {
#pragma unroll
  for (int i = 0; i < Pair<D>::N; ++i) P[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

template <int D>
__device__ __forceinline__ void pair_store(float4* __restrict__ tab, int64_t i, const float* c, float w) {
  float* f = reinterpret_cast<float*>(tab + (i >> 1) * Pair<D>::N);
  const int h = (int)(i & 1);
#pragma unroll
  for (int m = 0; m < D; ++m) f[4 * (m >> 1) + 2 * (m & 1) + h] = c[m];
  f[4 * Pair<D>::WQ + Pair<D>::WO + h] = w;
}

template <int D>
__device__ inline void cell_of(const float4& v, const float* lo, float s, int L, int32_t* c) {
  const int32_t cmax = (1 << L) - 1;
#pragma unroll
  for (int m = 0; m < D; ++m) {
    float t = __fmul_rn(__fsub_rn(comp(v, m), lo[m]), s);
    int32_t q = (int32_t)floorf(t);
    c[m] = q < cmax ? q : cmax;
  }
}

template <int D>
__device__ inline void grid_frame(const uint32_t* __restrict__ bb, int pb, int L, float* lo, float* s) {
  float E = 0.0f;
#pragma unroll
  for (int m = 0; m < D; ++m) {
    lo[m] = ord2f(bb[pb * 8 + m]);
    float hi = ord2f(bb[pb * 8 + 4 + m]);
    float e = __fsub_rn(hi, lo[m]);
    E = e > E ? e : E;
  }
  *s = (E > 0.0f) ? __fdiv_rn((float)(1 << L), E) : 0.0f;
}

template <int D>
__device__ inline int64_t rowmajor(const int32_t* c, int side) {
  int64_t r = 0;
#pragma unroll
  for (int m = D - 1; m >= 0; --m) r = r * side + c[m];
  return r;
}

__host__ __device__ constexpr int field_bits(int D) { return D == 4 ? 8 : 30 / D; }

// Coordinate m of a packed cell, kept inside the grid whatever the word holds
// (the ranges around a cell outside it would be empty or negative, and the
// loops over them would not end).
template <int D>
__device__ __forceinline__ int32_t cell_field(uint32_t packed, int m, int side) {
  return min((int32_t)((packed >> (m * field_bits(D))) & ((1u << field_bits(D)) - 1)), side - 1);
}

// Block-level bounding-box accumulation into ordered-uint min/max slots.
// uniform: every valid thread of the block belongs to problem pblock (the
// block result is then published once for pblock); otherwise each valid
// thread publishes its own point for its own problem pb.
template <int D>
__device__ void bbox_accumulate(const float4& v, bool valid, int pb, bool uniform, int pblock,
                                uint32_t* __restrict__ bb) {
  __shared__ uint32_t smn[kBlock / 32][4], smx[kBlock / 32][4];
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  if (!uniform) {
    if (valid)
#pragma unroll
      for (int m = 0; m < D; ++m) {
        uint32_t o = f2ord(comp(v, m));
        atomicMin(&bb[pb * 8 + m], o);
        atomicMax(&bb[pb * 8 + 4 + m], o);
      }
    return;
  }
#pragma unroll
  for (int m = 0; m < D; ++m) {
    uint32_t mn = valid ? f2ord(comp(v, m)) : 0xFFFFFFFFu;
    uint32_t mx = valid ? mn : 0u;
    mn = __reduce_min_sync(0xffffffffu, mn);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) { smn[warp][m] = mn; smx[warp][m] = mx; }
  }
  __syncthreads();
  if (threadIdx.x < D) {
    uint32_t mn = 0xFFFFFFFFu, mx = 0u;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      mn = min(mn, smn[w][threadIdx.x]);
      mx = max(mx, smx[w][threadIdx.x]);
    }
    if (mn != 0xFFFFFFFFu) atomicMin(&bb[pblock * 8 + threadIdx.x], mn);
    if (mx != 0u) atomicMax(&bb[pblock * 8 + 4 + threadIdx.x], mx);
  }
}

__global__ void k_bbox_reset(uint32_t* bb, int n) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) bb[i] = ((i & 7) < 4) ? 0xFFFFFFFFu : 0u;
}

template <int D>
__global__ void __launch_bounds__(kBlock) k_bbox(const float4* __restrict__ x, int64_t K,
                                                 const int32_t* __restrict__ vprob, uint32_t* __restrict__ bb) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int64_t first = (int64_t)blockIdx.x * blockDim.x;
  int64_t last = min(first + (int64_t)blockDim.x, K) - 1;
  const int pblock = vprob[first];
  bool uniform = pblock == vprob[last];
  bool valid = i < K;
  float4 v = valid ? x[i] : make_float4(0, 0, 0, 0);
  int pb = valid ? vprob[i] : 0;
  bbox_accumulate<D>(v, valid, pb, uniform, pblock, bb);
}

// Step length of a level: s0 = sigma * Lbox / k^(1/d), Lbox = d-th root of the
// box volume (largest extent if an extent is zero).
template <int D>
__global__ void k_step0(const uint32_t* __restrict__ bb, const ProbDev* __restrict__ prob, int P, float sigma,
                        float* __restrict__ s0) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  double vol = 1.0, emax = 0.0;
  bool degenerate = false;
  for (int m = 0; m < D; ++m) {
    double e = (double)ord2f(bb[p * 8 + 4 + m]) - (double)ord2f(bb[p * 8 + m]);
    if (!(e > 0.0)) degenerate = true;
    emax = e > emax ? e : emax;
    vol *= e;
  }
  int k = prob[p].k;
  double Lbox = degenerate ? emax : pow(vol, 1.0 / D);
  s0[p] = (k > 0) ? (float)(sigma * Lbox / pow((double)k, 1.0 / D)) : 0.0f;
}

// Binning of a level, device-wide: a counting sort by cell.  A step's cells
// are at most 8 points each on average, so instead of sorting (key, vertex)
// by digits (two passes of three kernels), every point takes a number in its
// cell, a scan of the cell counts gives the cell start table directly, and
// the points of a cell are then put into vertex order by counting the smaller
// ids among them:
//   k_keys      cell key of every point, its arrival number in the cell
//   k_cell_scan cell counts -> first sorted position of every cell
//   k_slots     vertex ids to their cells in arrival order
//   k_place     vertex order within the cell; sorted copies of the points
//   k_cells     cell sums and charges of every grid level
// The sorted order is that of a stable sort of (key, vertex), so nothing
// depends on the arrival order.  Five launches; the two-pass digit sort with
// its gather and per-level sums took eleven or more of about 4 us each, all
// bound by latency on the levels of a hierarchy.

// Cell keys of the points.  Each thread takes U points, strided by the block
// so that every load is coalesced, and issues all their loads before the
// arithmetic (U = 4 on large levels: more bytes in flight per SM; U = 1 on
// small ones: more blocks); thread 0 advances the level's step counter and
// the grid resets the next bounding boxes.
constexpr int64_t kKeyItemsMin = int64_t(1) << 20;  // points of a level that take 4 per thread

template <int D, int U>
__global__ void __launch_bounds__(kBlock) k_keys(const float4* __restrict__ x, int64_t K, const int32_t* __restrict__ vprob,
                                                 const ProbDev* __restrict__ prob, const uint32_t* __restrict__ bb,
                                                 uint32_t* __restrict__ keys, uint32_t* __restrict__ arrival,
                                                 int32_t* __restrict__ cnt, int P, uint32_t* __restrict__ bb_next,
                                                 int32_t* __restrict__ tctr) {
  pdl_enter();
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gt == 0) {
    ++tctr[0];    // the level's step (read by the step kernel of this step)
    tctr[1] = 0;  // set by the scan of the counts if a cell is crowded
  }
  const int64_t nreset = 8 * (int64_t)P;
  for (int64_t r = gt; r < nreset; r += (int64_t)gridDim.x * blockDim.x) bb_next[r] = ((r & 7) < 4) ? 0xFFFFFFFFu : 0u;
  const int64_t v0 = (int64_t)blockIdx.x * blockDim.x * U + threadIdx.x;
  float4 xv[U];
  int pb[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t v = v0 + (int64_t)u * blockDim.x;
    xv[u] = v < K ? x[v] : make_float4(0.f, 0.f, 0.f, 0.f);
    pb[u] = v < K ? vprob[v] : 0;
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t v = v0 + (int64_t)u * blockDim.x;
    const unsigned in = __ballot_sync(0xffffffffu, v < K);
    if (v >= K) continue;
    const int L = prob[pb[u]].L;
    float lo[D], s;
    grid_frame<D>(bb, pb[u], L, lo, &s);
    int32_t c[D];
    cell_of<D>(xv[u], lo, s, L, c);
    // the key indexes the count table: kept inside it whatever the coordinates are
    const uint32_t key = min((uint32_t)rowmajor<D>(c, 1 << L), (uint32_t)((int64_t(1) << (D * L)) - 1));
    keys[v] = key;
    // One atomic for the warp's points of the first cell that two neighbouring
    // lanes share: the points of a crowded cell would take their numbers one by
    // one (99,000 of 100,000 points in one cell, d = 2: 67 us, now 6.3 us).
    const int64_t slot = prob[pb[u]].fbase + pb[u] + key;
    const int64_t next = __shfl_down_sync(in, slot, 1);
    const unsigned shared = __ballot_sync(in, lane_id() < 31 && ((in >> (lane_id() + 1)) & 1u) && slot == next);
    unsigned same = 0;
    if (shared) same = __ballot_sync(in, slot == __shfl_sync(in, slot, __ffs(shared) - 1));
    const bool joined = (same >> lane_id()) & 1u;
    const unsigned below = same & ((1u << lane_id()) - 1u);
    uint32_t number = 0;
    if (!joined || !below) number = (uint32_t)atomicAdd(&cnt[slot], joined ? __popc(same) : 1);
    if (shared) {
      const uint32_t first = __shfl_sync(in, number, __ffs(same) - 1);
      if (joined) number = first + __popc(below);
    }
    arrival[v] = number;
  }
}

// Cell counts -> cell start table: the exclusive scan of cnt (every problem's
// finest cells and one empty end entry, problem after problem, as the
// problems' points are) is the first sorted position of every cell, of the
// end entry the problem's end.  With two targets per thread the scan of
// ceil(cnt / 2) next to it (cch) numbers the cells' chunks of two points.  One
// cluster scans a table of up to kCellScanTile entries; its blocks exchange
// their totals through distributed shared memory.
constexpr int kCellScanCtas = 8;
constexpr int kCellScanThreads = 1024;
constexpr int kCellScanItems = 16;
constexpr int64_t kCellScanTile = (int64_t)kCellScanCtas * kCellScanThreads * kCellScanItems;

__device__ __forceinline__ void load_items(const int32_t* __restrict__ a, int64_t i0, int64_t n, int32_t* v) {
  if (i0 + kCellScanItems <= n) {
#pragma unroll
    for (int j = 0; j < kCellScanItems / 4; ++j) {
      const int4 q = *reinterpret_cast<const int4*>(a + i0 + 4 * j);
      v[4 * j] = q.x;
      v[4 * j + 1] = q.y;
      v[4 * j + 2] = q.z;
      v[4 * j + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < kCellScanItems; ++j) v[j] = i0 + j < n ? a[i0 + j] : 0;
  }
}

__device__ __forceinline__ void store_items(int32_t* __restrict__ a, int64_t i0, int64_t n, const int32_t* e) {
  if (i0 + kCellScanItems <= n) {
#pragma unroll
    for (int j = 0; j < kCellScanItems / 4; ++j)
      *reinterpret_cast<int4*>(a + i0 + 4 * j) = make_int4(e[4 * j], e[4 * j + 1], e[4 * j + 2], e[4 * j + 3]);
  } else {
#pragma unroll
    for (int j = 0; j < kCellScanItems; ++j)
      if (i0 + j < n) a[i0 + j] = e[j];
  }
}

// Sum of a thread's items: points in the low, chunks in the high word (both
// below 2^31, so the words of a sum never mix).
__device__ __forceinline__ uint64_t items_sum(const int32_t* v) {
  uint64_t s = 0;
#pragma unroll
  for (int j = 0; j < kCellScanItems; ++j) s += ((uint64_t)(uint32_t)((v[j] + 1) >> 1) << 32) | (uint32_t)v[j];
  return s;
}

// The starts of a thread's items from the sums before it, and whether one of
// them is a crowded cell (see rank_large).
constexpr int kRankBlock = 1024;  // points of a cell from which a block places them together

__device__ __forceinline__ void store_starts(int32_t* __restrict__ cst, int32_t* __restrict__ cch,
                                             int32_t* __restrict__ crowded, int64_t i0, int64_t n, const int32_t* v,
                                             uint64_t before) {
  int32_t most = 0;
#pragma unroll
  for (int j = 0; j < kCellScanItems; ++j) most = max(most, v[j]);
  if (most > kRankBlock) *crowded = 1;
  int32_t e[kCellScanItems];
  int32_t run = (int32_t)(uint32_t)before;
#pragma unroll
  for (int j = 0; j < kCellScanItems; ++j) {
    e[j] = run;
    run += v[j];
  }
  store_items(cst, i0, n, e);
  if (!cch) return;
  run = (int32_t)(before >> 32);
#pragma unroll
  for (int j = 0; j < kCellScanItems; ++j) {
    e[j] = run;
    run += (v[j] + 1) >> 1;
  }
  store_items(cch, i0, n, e);
}

__global__ void __cluster_dims__(kCellScanCtas, 1, 1) __launch_bounds__(kCellScanThreads)
    k_cell_scan(const int32_t* __restrict__ cnt, int32_t* __restrict__ cst, int32_t* __restrict__ cch,
                int32_t* __restrict__ crowded, int64_t n) {
  pdl_enter();
  __shared__ uint64_t ws[33];
  __shared__ uint64_t tot;
  __shared__ uint64_t peer[kCellScanCtas];
  auto cluster = cooperative_groups::this_cluster();
  const unsigned r = cluster.block_rank();
  const int64_t i0 = ((int64_t)r * kCellScanThreads + threadIdx.x) * kCellScanItems;
  int32_t v[kCellScanItems];
  load_items(cnt, i0, n, v);
  uint64_t total;
  const uint64_t ex = block_exclusive<uint64_t>(items_sum(v), ws, &total);
  if (threadIdx.x == 0) tot = total;
  cluster.sync();
  if (threadIdx.x < kCellScanCtas) peer[threadIdx.x] = *cluster.map_shared_rank(&tot, threadIdx.x);
  cluster.sync();  // also: no block leaves while another may still read its total
  uint64_t before = ex;
#pragma unroll
  for (unsigned q = 0; q < kCellScanCtas; ++q) before += q < r ? peer[q] : 0;
  store_starts(cst, cch, crowded, i0, n, v, before);
}

// The same scan for larger tables in two launches: block totals, then every
// block adds up the totals before its own and scans its part (one cluster
// taking several tiles in turn needs 14 us for three, the two launches 9 us).
__global__ void __launch_bounds__(kCellScanThreads) k_cell_totals(const int32_t* __restrict__ cnt, int64_t n,
                                                                  uint64_t* __restrict__ tot) {
  pdl_enter();
  __shared__ uint64_t ws[33];
  int32_t v[kCellScanItems];
  load_items(cnt, ((int64_t)blockIdx.x * kCellScanThreads + threadIdx.x) * kCellScanItems, n, v);
  uint64_t total;
  block_exclusive<uint64_t>(items_sum(v), ws, &total);
  if (threadIdx.x == 0) tot[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kCellScanThreads) k_cell_starts(const int32_t* __restrict__ cnt, int64_t n,
                                                                  const uint64_t* __restrict__ tot,
                                                                  int32_t* __restrict__ cst, int32_t* __restrict__ cch,
                                                                  int32_t* __restrict__ crowded) {
  pdl_enter();
  __shared__ uint64_t ws[33];
  int32_t v[kCellScanItems];
  const int64_t i0 = ((int64_t)blockIdx.x * kCellScanThreads + threadIdx.x) * kCellScanItems;
  load_items(cnt, i0, n, v);
  uint64_t part = 0;
  for (unsigned b = threadIdx.x; b < blockIdx.x; b += kCellScanThreads) part += tot[b];
  uint64_t before;
  block_exclusive<uint64_t>(part, ws, &before);
  const uint64_t ex = block_exclusive<uint64_t>(items_sum(v), ws, nullptr);
  store_starts(cst, cch, crowded, i0, n, v, before + ex);
}

// Vertex ids to their cells, in arrival order.
__global__ void __launch_bounds__(kBlock) k_slots(const uint32_t* __restrict__ keys,
                                                  const uint32_t* __restrict__ arrival, int64_t K,
                                                  const int32_t* __restrict__ vprob, const ProbDev* __restrict__ prob,
                                                  const int32_t* __restrict__ cst, uint32_t* __restrict__ slot) {
  pdl_enter();
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= K) return;
  const int pb = vprob[v];
  slot[cst[prob[pb].fbase + pb + keys[v]] + arrival[v]] = (uint32_t)v;
}

// Places of a block's points in cells of more than kRankBlock points.  The block
// holds up to kBlock points of the cell (those of consecutive slots): it sorts
// their ids, then reads the cell's ids once, finds for each by binary search the
// first of its own that is larger, and counts there; the prefix sums of the
// counts are the places.  A thread that compared its point with the whole cell
// took kBlock / 8 times the operations (99,000 of 100,000 points in one cell, d = 2:
// 2,280 us, now 180 us; 50,000, d = 3: 1,140 and 83 us).  kRankBlock > kBlock, so only
// the cells of the block's first and last point can be large.  Every thread of the
// block calls it; `in` marks those with a point.
struct RankShared {
  uint32_t ids[kBlock], sorted[kBlock];
  int32_t count[kBlock], place[kBlock];
  int32_t seg[2][2];
  uint64_t scan[33];
};

__device__ __noinline__ void rank_large(const uint32_t* __restrict__ slot, bool in, bool last, uint32_t v, int32_t q0,
                                           int32_t q1, RankShared& sh) {
  const int tid = threadIdx.x;
  const int32_t b0 = (int32_t)(blockIdx.x * kBlock);
  const bool large = in && q1 - q0 > kRankBlock;
  if (tid == 0 || last) {
    const int e = last ? 1 : 0;
    sh.seg[e][0] = large ? q0 : 0;
    sh.seg[e][1] = large ? q1 : 0;
    if (tid == 0 && last) sh.seg[0][0] = sh.seg[0][1] = 0;  // one point: handled as the last
  }
  __syncthreads();
  for (int e = 0; e < 2; ++e) {
    const int32_t c0 = sh.seg[e][0], c1 = sh.seg[e][1];
    if (c0 == c1 || (e == 0 && c0 == sh.seg[1][0] && c1 == sh.seg[1][1])) continue;
    const bool mine = large && q0 == c0;
    const int a = max(c0 - b0, 0), m = min(c1 - b0, kBlock) - a;  // the block's points of the cell
    if (mine) sh.ids[tid - a] = v;
    sh.count[tid] = 0;
    __syncthreads();
    int r = 0;
    if (mine) {
      for (int i = 0; i < m; ++i) r += sh.ids[i] < v;
      sh.sorted[r] = v;
    }
    __syncthreads();
    const uint32_t lo = sh.sorted[0], hi = sh.sorted[m - 1];
    int below = 0;
    for (int64_t i = c0 + tid; i < c1; i += 8 * kBlock) {
      uint32_t u[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) u[j] = i + j * kBlock < c1 ? slot[i + j * kBlock] : 0xFFFFFFFFu;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        below += u[j] < lo;
        if (u[j] < lo || u[j] >= hi) continue;
        int x0 = 0, x1 = m - 1;  // sorted[x0] <= u < sorted[x1]
        while (x1 - x0 > 1) {
          const int mid = (x0 + x1) >> 1;
          if (sh.sorted[mid] <= u[j]) x0 = mid;
          else x1 = mid;
        }
        atomicAdd(&sh.count[x1], 1);
      }
    }
    below = __reduce_add_sync(0xffffffffu, below);
    if (lane_id() == 0 && below) atomicAdd(&sh.count[0], below);
    __syncthreads();
    const int own = sh.count[tid];
    const uint64_t before = block_exclusive<uint64_t>((uint64_t)(uint32_t)own, sh.scan, nullptr);
    sh.count[tid] = (int32_t)before + own;
    __syncthreads();
    if (mine) sh.place[tid] = sh.count[r];
    __syncthreads();
  }
}

// Sorted positions: the points of a cell by ascending vertex (a point's place
// is the number of smaller ids in its cell), coordinates and weights in
// sorted order (plain and in the paired table XP) and the packed cell of every
// point.  v is the vertex in the thread's slot (0 beyond the last).
template <int D, bool CROWDED>
__device__ __forceinline__ void place_points(const uint32_t* __restrict__ slot, const uint32_t* __restrict__ keys,
                                             uint32_t v, int64_t K, const float4* __restrict__ x, const float* __restrict__ w,
                                             const int32_t* __restrict__ vprob, const ProbDev* __restrict__ prob,
                                             const int32_t* __restrict__ cst, const int32_t* __restrict__ cch,
                                             int32_t* __restrict__ chunk, uint32_t* __restrict__ svals,
                                             float4* __restrict__ xs, float* __restrict__ ws,
                                             uint32_t* __restrict__ scell, float4* __restrict__ XP) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = t < K;
  if (!CROWDED && !in) return;
  const int pb = vprob[v];
  const uint32_t key = keys[v];
  const float4 xv = x[v];
  const int32_t* cs = cst + prob[pb].fbase + pb;
  const int32_t q0 = cs[key], q1 = cs[key + 1];
  const bool large = CROWDED && q1 - q0 > kRankBlock;
  __shared__ RankShared rank;
  if (CROWDED) {
    if (__syncthreads_or(large && in))
      rank_large(slot, in, in && (t == K - 1 || threadIdx.x == kBlock - 1), v, q0, q1, rank);
    if (!in) return;
  }
  const ProbDev pr = prob[pb];
  int32_t less = 0;
  if (large) {
    less = rank.place[threadIdx.x];
  } else {
    int32_t q = q0;
    for (; q < q1 && (q & 3); ++q) less += slot[q] < v;
    for (; q + 8 <= q1; q += 8) {  // 16-byte reads, two in flight
      const uint4 a = *reinterpret_cast<const uint4*>(slot + q), b = *reinterpret_cast<const uint4*>(slot + q + 4);
      less += (a.x < v) + (a.y < v) + (a.z < v) + (a.w < v) + (b.x < v) + (b.y < v) + (b.z < v) + (b.w < v);
    }
    for (; q < q1; ++q) less += slot[q] < v;
  }
  const int64_t p = (int64_t)q0 + less;
  if (cch && !(less & 1)) chunk[cch[pr.fbase + pb + key] + (less >> 1)] = (int32_t)p;
  svals[p] = v;
  xs[p] = xv;
  const float wv = w ? w[v] : 1.0f;
  if (ws) ws[p] = wv;
  // paired table: the problem's points start at an even slot, so the pairing
  // of its points does not depend on where the problem sits in the batch
  const int64_t e = (pr.vbase + pb + 1) & ~int64_t(1);
  const float xc[4] = {xv.x, xv.y, xv.z, xv.w};
  pair_store<D>(XP, e + (p - pr.vbase), xc, wv);
  if (p == pr.vbase + pr.k - 1 && (pr.k & 1)) {  // unused half of the last pair: finite, weight 0
    const float zero[4] = {0.f, 0.f, 0.f, 0.f};
    pair_store<D>(XP, e + pr.k, zero, 0.0f);
  }
  uint32_t packed = 0;
#pragma unroll
  for (int m = 0; m < D; ++m) packed |= ((key >> (m * pr.L)) & ((1u << pr.L) - 1u)) << (m * field_bits(D));
  scell[p] = packed;
}

// The launches of a level without a crowded cell (a flag of the scan) do without
// the barrier and the registers of the other path: with them in the same body the
// launch took 20.2 us at 500,000 points, without 16.5 us.
template <int D>
__device__ __noinline__ void place_crowded(const uint32_t* __restrict__ slot, const uint32_t* __restrict__ keys,
                                          uint32_t v, int64_t K, const float4* __restrict__ x, const float* __restrict__ w,
                                          const int32_t* __restrict__ vprob, const ProbDev* __restrict__ prob,
                                          const int32_t* __restrict__ cst, const int32_t* __restrict__ cch,
                                          int32_t* __restrict__ chunk, uint32_t* __restrict__ svals,
                                          float4* __restrict__ xs, float* __restrict__ ws,
                                          uint32_t* __restrict__ scell, float4* __restrict__ XP) {
  place_points<D, true>(slot, keys, v, K, x, w, vprob, prob, cst, cch, chunk, svals, xs, ws, scell, XP);
}

// Places of all points; the counts are cleared for the next step.
template <int D>
__global__ void __launch_bounds__(kBlock, 6) k_place(const uint32_t* __restrict__ slot,
                                                      const uint32_t* __restrict__ keys, int64_t K,
                                                      const float4* __restrict__ x, const float* __restrict__ w,
                                                      const int32_t* __restrict__ vprob,
                                                      const ProbDev* __restrict__ prob,
                                                      const int32_t* __restrict__ cst, int32_t* __restrict__ cnt,
                                                      int64_t ncnt, const int32_t* __restrict__ crowded,
                                                      const int32_t* __restrict__ cch, int32_t* __restrict__ chunk,
                                                      uint32_t* __restrict__ svals, float4* __restrict__ xs,
                                                      float* __restrict__ ws, uint32_t* __restrict__ scell,
                                                      float4* __restrict__ XP) {
  pdl_enter();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t v = t < K ? slot[t] : 0u;  // in flight together with the flag
  const int32_t any = *crowded;
  for (int64_t i = t; i < ncnt; i += (int64_t)gridDim.x * blockDim.x) cnt[i] = 0;
  if (any)
    place_crowded<D>(slot, keys, v, K, x, w, vprob, prob, cst, cch, chunk, svals, xs, ws, scell, XP);
  else
    place_points<D, false>(slot, keys, v, K, x, w, vprob, prob, cst, cch, chunk, svals, xs, ws, scell, XP);
}

// Cell sums (St, Wt) at cell index idx, and the cell's charge (weighted mean
// and weight) at index pidx of the paired cell table.
template <int D>
__device__ inline void store_cell(int64_t idx, int64_t pidx, const float* S, float W, float4* St, float* Wt,
                                  float4* CP) {
  St[idx] = make_float4(S[0], D > 1 ? S[1] : 0.f, D > 2 ? S[2] : 0.f, D > 3 ? S[3] : 0.f);
  Wt[idx] = W;
  float c[4] = {0.f, 0.f, 0.f, 0.f};
  if (W > 0.0f) {
    float iw = 1.0f / W;
#pragma unroll
    for (int m = 0; m < D; ++m) c[m] = S[m] * iw;
  }
  pair_store<D>(CP, pidx, c, W);
}

// A finest cell of at most kCellSerial points is summed by one thread in point
// order; a larger cell (dense clusters of the layout) by a whole warp:
// lane-strided partial sums from the cell's first point, then a fixed xor
// tree.  Either way the sums depend only on the cell.
constexpr int kCellSerial = 32;
constexpr int kCellHuge = 512;  // points of a cell from which a whole warp sums it

template <int D>
__device__ __forceinline__ void cell_add(const float4& p, float wq, float* S, float& W) {
  S[0] += wq * p.x;
  if (D > 1) S[1] += wq * p.y;
  if (D > 2) S[2] += wq * p.z;
  if (D > 3) S[3] += wq * p.w;
  W += wq;
}

// Points q0, q0 + stride, ... < q1 added in that order; U loads issued before
// their additions, those of the last, incomplete trip guarded.  The whole trips of a
// large cell go without guards, with which two loads' times passed per trip: the
// first step of 19,800 points in a cell, d = 2, 118 -> 88 us, the layout of the
// 64^3 grid 1.3% shorter (16 loads instead of 8: 53 us, but twice the registers,
// and a batch of 256 matrices 1% longer).
template <int D, int U>
__device__ __forceinline__ void cell_sum_long(const float4* xs, const float* ws, int64_t q0, int64_t q1, int64_t stride,
                                              float* S, float& W) {
  int64_t q = q0;
  for (; q + (U - 1) * stride < q1; q += U * stride) {
    float4 p[U];
    float wq[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      p[u] = xs[q + u * stride];
      wq[u] = ws ? ws[q + u * stride] : 1.0f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) cell_add<D>(p[u], wq[u], S, W);
  }
  if (q >= q1) return;
  float4 p[U];
  float wq[U];
#pragma unroll
  for (int u = 0; u + 1 < U; ++u) {
    const bool in = q + u * stride < q1;
    p[u] = in ? xs[q + u * stride] : make_float4(0.f, 0.f, 0.f, 0.f);
    wq[u] = in && ws ? ws[q + u * stride] : 1.0f;
  }
#pragma unroll
  for (int u = 0; u + 1 < U; ++u)
    if (q + u * stride < q1) cell_add<D>(p[u], wq[u], S, W);
}

// The same for cells of a few points, every load guarded.
template <int D, int U>
__device__ __forceinline__ void cell_sum(const float4* xs, const float* ws, int64_t q0, int64_t q1, int64_t stride,
                                         float* S, float& W) {
  for (int64_t q = q0; q < q1; q += U * stride) {
    float4 p[U];
    float wq[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool in = q + u * stride < q1;
      p[u] = in ? xs[q + u * stride] : make_float4(0.f, 0.f, 0.f, 0.f);
      wq[u] = in && ws ? ws[q + u * stride] : 1.0f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (q + u * stride < q1) cell_add<D>(p[u], wq[u], S, W);
  }
}

// Sum of the points [q0, q1) of a large cell (every lane gets it): 32 partial
// sums of every 32nd point, then the xor tree, by a whole warp ...
template <int D>
__device__ __forceinline__ void cell_sum_warp(const float4* xs, const float* ws, int64_t q0, int64_t q1, float* S,
                                              float& W) {
  cell_sum_long<D, 8>(xs, ws, q0 + lane_id(), q1, 32, S, W);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int m = 0; m < D; ++m) S[m] += __shfl_xor_sync(0xffffffffu, S[m], o);
    W += __shfl_xor_sync(0xffffffffu, W, o);
  }
}

// ... or by kCellLanes lanes that hold four of the partial sums each (the same
// sums; four cells per warp, so a brick of large cells takes a quarter of the
// turns).  Every lane of the warp calls it; an empty range gives zeros.
constexpr int kCellLanes = 8;

template <int D>
__device__ __forceinline__ void cell_sum_quarter(const float4* xs, const float* ws, int64_t q0, int64_t q1, float* S,
                                                 float& W) {
  float P[4][4], V[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    V[j] = 0.f;
#pragma unroll
    for (int m = 0; m < 4; ++m) P[j][m] = 0.f;
  }
  for (int64_t q = q0 + (lane_id() & (kCellLanes - 1)); q < q1; q += 64) {
    float4 p[8];
    float wq[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const bool in = q + 8 * u < q1;
      p[u] = in ? xs[q + 8 * u] : make_float4(0.f, 0.f, 0.f, 0.f);
      wq[u] = in && ws ? ws[q + 8 * u] : 1.0f;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (q + 8 * u < q1) cell_add<D>(p[u], wq[u], P[u & 3], V[u & 3]);
  }
  W = (V[0] + V[2]) + (V[1] + V[3]);
#pragma unroll
  for (int m = 0; m < D; ++m) S[m] = (P[0][m] + P[2][m]) + (P[1][m] + P[3][m]);
#pragma unroll
  for (int o = kCellLanes / 2; o > 0; o >>= 1) {
#pragma unroll
    for (int m = 0; m < D; ++m) S[m] += __shfl_xor_sync(0xffffffffu, S[m], o);
    W += __shfl_xor_sync(0xffffffffu, W, o);
  }
}

// Coarse cells: sums of the 2^d children (fixed order), charge at the mean.
template <int D>
__device__ inline void agg_cell(const ProbDev& pr, int pb, int l, int64_t c, float4* St, float* Wt, float4* CP) {
  const int side = 1 << l;
  int32_t cc[D];
  int64_t rem = c;
#pragma unroll
  for (int m = 0; m < D; ++m) {
    cc[m] = (int32_t)(rem % side);
    rem /= side;
  }
  const int64_t child_base = pr.cbase + lvl_off(D, l + 1);
  float S[4] = {0.f, 0.f, 0.f, 0.f};
  float W = 0.f;
#pragma unroll
  for (int ch = 0; ch < (1 << D); ++ch) {
    int32_t q[D];
#pragma unroll
    for (int m = 0; m < D; ++m) q[m] = 2 * cc[m] + ((ch >> m) & 1);
    const int64_t idx = child_base + rowmajor<D>(q, 2 * side);
    const float4 s4 = __ldcg(St + idx);  // written by other threads of this launch
    S[0] += s4.x;
    if (D > 1) S[1] += s4.y;
    if (D > 2) S[2] += s4.z;
    if (D > 3) S[3] += s4.w;
    W += __ldcg(Wt + idx);
  }
  const int64_t idx = pr.cbase + lvl_off(D, l) + c;
  store_cell<D>(idx, idx + pb + 1, S, W, St, Wt, CP);
}

// Cell sums and charges of every grid level (k_cells): one block per brick of
// 2^(d B) finest cells, B = kBrick(d) (the whole grid when L < B).  The block
// sums its finest cells from their points, then the B coarser levels from
// their children in shared memory; the problem's last block to arrive sums
// the levels above the bricks' roots from the roots' sums in global memory.
// Small bricks, so that the large cells of a dense cluster spread over many
// blocks (a warp took up to 32 of them in turn when a warp owned 32
// consecutive cells: 17 us on the 64^3 grid's finest level).  A problem of one
// grid level has no far field and so no bricks (the isolated vertices of a
// power-law pattern are thousands of such problems).
__host__ __device__ constexpr int brick_log2(int d) { return d == 2 ? 3 : 2; }
// A block's time is mostly its chain of dependent loads (9.5 us for 512 bricks, 36 us
// for 4,096 of clustered points); 64 threads are slower (large cells want
// threads), 256 equal. Finest cells first in a launch that spreads the cells
// of a cluster over all blocks was no faster (493 against 480 us a step).
constexpr int kCellsBlock = 128;

template <int D>
__global__ void __launch_bounds__(kCellsBlock) k_cells(const int32_t* __restrict__ bprob, const ProbDev* __restrict__ prob,
                                                  const float4* __restrict__ xs, const float* __restrict__ ws,
                                                  const int32_t* __restrict__ cst, float4* St, float* Wt, float4* CP,
                                                  int32_t* __restrict__ done) {
  pdl_enter();
  constexpr int B = brick_log2(D), NC = 1 << (D * B);
  constexpr int NT = ((1 << (D * (B + 1))) - 1) / ((1 << D) - 1);  // cells of a brick on its B + 1 levels
  __shared__ float sS[D][NT], sW[NT];  // finest level first
  __shared__ int32_t big[NC], bq0[NC], bq1[NC];
  __shared__ int nbig;
  __shared__ bool last;
  const int pb = bprob[blockIdx.x];
  const ProbDev pr = prob[pb];
  const int L = pr.L, lb = min(L, B), Lb = L - lb;
  const int64_t brick = (int64_t)blockIdx.x - pr.bbase;
  int32_t bc[D];
#pragma unroll
  for (int m = 0; m < D; ++m) bc[m] = (int32_t)((brick >> (m * Lb)) & ((1 << Lb) - 1));
  if (threadIdx.x == 0) nbig = 0;
  __syncthreads();
  // cell i of the brick on level l = L - j: row-major index in the level's grid
  auto cell_index = [&](int i, int j) {
    const int bits = lb - j;
    int32_t c[D];
#pragma unroll
    for (int m = 0; m < D; ++m) c[m] = (bc[m] << bits) | ((i >> (m * bits)) & ((1 << bits) - 1));
    return rowmajor<D>(c, 1 << (L - j));
  };
  auto store_charge = [&](int64_t c, int l, const float* S, float W) {
    float z[4] = {0.f, 0.f, 0.f, 0.f};
    if (W > 0.0f) {
      const float iw = 1.0f / W;
#pragma unroll
      for (int m = 0; m < D; ++m) z[m] = S[m] * iw;
    }
    pair_store<D>(CP, pr.cbase + lvl_off(D, l) + c + pb + 1, z, W);
  };
  const int nc = 1 << (D * lb);  // at most NC: 64, for d = 4 256
  const int32_t* cs = cst + pr.fbase + pb;
  for (int i = threadIdx.x; i < nc; i += kCellsBlock) {
    const int64_t c = cell_index(i, 0);
    const int32_t q0 = cs[c], q1 = cs[c + 1];
    if (q1 - q0 > kCellSerial) {
      const int b = atomicAdd(&nbig, 1);
      big[b] = i;
      bq0[b] = q0;
      bq1[b] = q1;
      continue;
    }
    float S[4] = {0.f, 0.f, 0.f, 0.f};
    float W = 0.f;
    cell_sum<D, 8>(xs, ws, q0, q1, 1, S, W);
#pragma unroll
    for (int m = 0; m < D; ++m) sS[m][i] = S[m];
    sW[i] = W;
    store_charge(c, L, S, W);
  }
  __syncthreads();
  auto keep = [&](int i, const float* S, float W) {
#pragma unroll
    for (int m = 0; m < D; ++m) sS[m][i] = S[m];
    sW[i] = W;
    store_charge(cell_index(i, 0), L, S, W);
  };
  for (int b0 = 0; b0 < nbig; b0 += kCellsBlock / kCellLanes) {  // large cells, four to a warp
    const int b = b0 + threadIdx.x / kCellLanes;
    const bool mine = b < nbig && bq1[b] - bq0[b] <= kCellHuge;
    float S[4] = {0.f, 0.f, 0.f, 0.f};
    float W = 0.f;
    cell_sum_quarter<D>(xs, ws, mine ? bq0[b] : 0, mine ? bq1[b] : 0, S, W);
    if (mine && (threadIdx.x & (kCellLanes - 1)) == 0) keep(big[b], S, W);
  }
  for (int b = threadIdx.x >> 5; b < nbig; b += kCellsBlock / 32) {  // the largest, a warp each
    if (bq1[b] - bq0[b] <= kCellHuge) continue;
    float S[4] = {0.f, 0.f, 0.f, 0.f};
    float W = 0.f;
    cell_sum_warp<D>(xs, ws, bq0[b], bq1[b], S, W);
    if (lane_id() == 0) keep(big[b], S, W);
  }
  int off = 0;  // first cell of level L - j + 1 in the shared sums
  for (int j = 1; j <= lb && L - j >= 2; ++j) {
    __syncthreads();
    const int bits = lb - j, n = 1 << (D * bits), next = off + (1 << (D * (bits + 1)));
    for (int i = threadIdx.x; i < n; i += kCellsBlock) {
      float S[4] = {0.f, 0.f, 0.f, 0.f};
      float W = 0.f;
#pragma unroll
      for (int ch = 0; ch < (1 << D); ++ch) {
        int q = 0;
#pragma unroll
        for (int m = 0; m < D; ++m)
          q |= (2 * ((i >> (m * bits)) & ((1 << bits) - 1)) + ((ch >> m) & 1)) << (m * (bits + 1));
#pragma unroll
        for (int m = 0; m < D; ++m) S[m] += sS[m][off + q];
        W += sW[off + q];
      }
#pragma unroll
      for (int m = 0; m < D; ++m) sS[m][next + i] = S[m];
      sW[next + i] = W;
      store_charge(cell_index(i, j), L - j, S, W);
    }
    off = next;
  }
  if (Lb <= 2) return;  // every level down to 2 lies inside the bricks
  __syncthreads();
  if (threadIdx.x == 0) {
    const int64_t idx = pr.cbase + lvl_off(D, Lb) + brick;  // the brick's root is cell `brick` of level Lb
    St[idx] = make_float4(sS[0][off], sS[1][off], D > 2 ? sS[D > 2 ? 2 : 0][off] : 0.f,
                          D > 3 ? sS[D > 3 ? 3 : 0][off] : 0.f);
    Wt[idx] = sW[off];
    __threadfence();
    last = atomicAdd(&done[pb], 1) == (1 << (D * Lb)) - 1;
    if (last) {
      done[pb] = 0;  // for the next step
      __threadfence();
    }
  }
  __syncthreads();
  if (!last) return;
  for (int l = Lb - 1; l >= 2; --l) {
    const int64_t n = int64_t(1) << (D * l);
    for (int64_t c = threadIdx.x; c < n; c += kCellsBlock) agg_cell<D>(pr, pb, l, c, St, Wt, CP);
    __syncthreads();
  }
}

// Rubber bands of 2-pin nets: y_v = sum_u c_vu (x_v - x_u) / 2.  Rows are
// split by degree: light rows (<= kLightMax) take one thread, medium rows a
// quarter warp and heavy rows a block; each class sums in a fixed order (sequential,
// lane-strided + xor tree, thread-strided + fixed tree), so the result of a
// vertex depends only on its own row.
constexpr int kLightMax = 32;
constexpr int kWarpMax = 4096;

__device__ inline void add_pull(float* a, const float4& xv, const float4& xu, float c) {
  a[0] += c * (xv.x - xu.x);
  a[1] += c * (xv.y - xu.y);
  a[2] += c * (xv.z - xu.z);
  a[3] += c * (xv.w - xu.w);
}

// a += sum over t = t0, t0 + stride, ... < t1 of c_t (xv - x[adj[t]]), in that
// order; U neighbours per trip with all their loads issued first.
template <int U>
__device__ __forceinline__ void pull_range(float* a, const float4& xv, const int32_t* __restrict__ adj,
                                           const float* __restrict__ acost, const float4* __restrict__ x, int32_t t,
                                           int32_t t1, int32_t stride) {
  for (; t < t1; t += U * stride) {
    int32_t u[U];
    float c[U];
    float4 q[U];
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const bool in = t + i * stride < t1;
      u[i] = in ? adj[t + i * stride] : -1;
      c[i] = in && acost ? acost[t + i * stride] : 1.0f;
    }
#pragma unroll
    for (int i = 0; i < U; ++i) q[i] = u[i] >= 0 ? x[u[i]] : xv;
#pragma unroll
    for (int i = 0; i < U; ++i)
      if (u[i] >= 0) add_pull(a, xv, q[i], c[i]);
  }
}

// All rows in one launch: first the blocks of the heavy rows (one each), then
// the blocks of medium rows, then the light rows' (a thread each, by vertex).
// A medium row's 32 partial sums (entries t0 + l, t0 + l + 32, ...; then the xor
// tree) are held four to a lane by kMidLanes = 8 lanes: four rows per warp, so
// that a row of 33 to 100 entries has all its gathers in flight at once and
// the tree's first two levels need no shuffle; rows longer than kMidMax take
// the whole warp with 16 entries of a lane in flight.  500,000-row power-law
// matrix, per step: 31 us, against 46 us of three launches (a thread, a warp
// and a block per row).
constexpr int kMidLanes = 8;
constexpr int kMidMax = 512;  // entries of a row from which the whole warp takes it

struct Attract {
  const int32_t *adj_ptr, *adj;
  const float* acost;
  const float4* x;
  int64_t K;
  const int32_t *heavy, *mid;
  int64_t n_heavy, n_mid, mid_blocks;  // mid_blocks: blocks of T threads for the medium rows
  float4* y;
  template <int T>
  int64_t blocks() const { return n_heavy + mid_blocks + (K + T - 1) / T; }
};

// The rows of blocks of T threads numbered b, medium and light rows.
template <int T>
__device__ __forceinline__ void attract_rows(const Attract& at, int64_t b) {
  const int32_t *adj_ptr = at.adj_ptr, *adj = at.adj, *mid = at.mid;
  const float* acost = at.acost;
  const float4* x = at.x;
  float4* y = at.y;
  const int64_t K = at.K, n_mid = at.n_mid, mid_blocks = at.mid_blocks;
  const int lane = lane_id();

  if (b < mid_blocks) {
    const int64_t i = (b * T + threadIdx.x) / kMidLanes;
    const int l = threadIdx.x & (kMidLanes - 1);
    const bool in = i < n_mid;
    const int32_t v = in ? mid[i] : 0;
    const int32_t t0 = in ? adj_ptr[v] : 0, t1 = in ? adj_ptr[v + 1] : 0;
    const bool quarter = in && t1 - t0 <= kMidMax;
    const float4 xv = x[v];
    float a[4][4];  // [partial sum l + 8 j][coordinate]
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int m = 0; m < 4; ++m) a[j][m] = 0.f;
    for (int32_t t = t0 + l; quarter && t < t1; t += 64) {  // two entries of every partial sum
      int32_t u[8];
      float c[8];
      float4 q[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const bool ok = t + 8 * j < t1;
        u[j] = ok ? adj[t + 8 * j] : v;
        c[j] = ok && acost ? acost[t + 8 * j] : 1.0f;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) q[j] = x[u[j]];
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (t + 8 * j < t1) add_pull(a[j & 3], xv, q[j], c[j]);
    }
    float s[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {  // the xor tree of 32 partial sums: distances 16, 8 here, 4, 2, 1 across lanes
      s[m] = (a[0][m] + a[2][m]) + (a[1][m] + a[3][m]);
#pragma unroll
      for (int o = kMidLanes / 2; o > 0; o >>= 1) s[m] += __shfl_xor_sync(0xffffffffu, s[m], o);
    }
    if (quarter && l == 0) y[v] = make_float4(0.5f * s[0], 0.5f * s[1], 0.5f * s[2], 0.5f * s[3]);
    unsigned todo = __ballot_sync(0xffffffffu, in && !quarter && l == 0);  // longer rows: the whole warp
    while (todo) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const int32_t w = __shfl_sync(0xffffffffu, v, src);
      const float4 xw = x[w];
      float g[4] = {0.f, 0.f, 0.f, 0.f};
      pull_range<16>(g, xw, adj, acost, x, adj_ptr[w] + lane, adj_ptr[w + 1], 32);
#pragma unroll
      for (int m = 0; m < 4; ++m)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) g[m] += __shfl_xor_sync(0xffffffffu, g[m], o);
      if (lane == 0) y[w] = make_float4(0.5f * g[0], 0.5f * g[1], 0.5f * g[2], 0.5f * g[3]);
    }
    return;
  }
  const int64_t v = (b - mid_blocks) * T + threadIdx.x;
  if (v >= K) return;
  const int32_t t0 = adj_ptr[v], t1 = adj_ptr[v + 1];
  if (t1 - t0 > kLightMax) return;  // a medium or heavy row
  const float4 xv = x[v];
  float a[4] = {0.f, 0.f, 0.f, 0.f};
  pull_range<4>(a, xv, adj, acost, x, t0, t1, 1);
  y[v] = make_float4(0.5f * a[0], 0.5f * a[1], 0.5f * a[2], 0.5f * a[3]);
}

__global__ void __launch_bounds__(kBlock) k_attract(Attract at) {
  pdl_enter();
  __shared__ float part[kBlock / 32][4];
  if (blockIdx.x >= at.n_heavy) {
    attract_rows<kBlock>(at, (int64_t)blockIdx.x - at.n_heavy);
    return;
  }
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  const float4* x = at.x;
  float4* y = at.y;
  const int32_t v = at.heavy[blockIdx.x];
  const float4 xv = x[v];
  float a[4] = {0.f, 0.f, 0.f, 0.f};
  pull_range<16>(a, xv, at.adj, at.acost, x, at.adj_ptr[v] + threadIdx.x, at.adj_ptr[v + 1], blockDim.x);
#pragma unroll
  for (int m = 0; m < 4; ++m)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a[m] += __shfl_xor_sync(0xffffffffu, a[m], o);
  if (lane == 0)
    for (int m = 0; m < 4; ++m) part[warp][m] = a[m];
  __syncthreads();
  if (threadIdx.x == 0) {
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w)
      for (int m = 0; m < 4; ++m) s[m] += part[w][m];
    y[v] = make_float4(0.5f * s[0], 0.5f * s[1], 0.5f * s[2], 0.5f * s[3]);
  }
}

// One-block binning of a step for levels whose problems all have at most
// kSortTile points and kBinCells finest cells: one block per problem does what
// the device-wide sequence does, with the counts, the sorted points and the
// sums of every grid level in shared memory: keys and arrival numbers, scan of
// the cell counts, vertex order within a cell, sorted copies, sums and charges.
// The arithmetic and the order of every sum are those kernels', so the results
// are bit-identical, from one launch instead of five.  The blocks after the
// problems' do the attraction (no row of such a level is heavy), so that a step
// of few problems is two launches in a row without a second stream.  As a sort of
// 8-bit digits with the coarse sums read back through L2, and the attraction on
// a second stream, a whole step took 12.2 / 17.4 us of 256 / 1,024 points (d =
// 2) and 15.4 / 24.5 us of 512 / 1,728 (d = 3); now 8.2 / 12.3 and 11.3 / 19.5.
// With four points per thread a problem may have 2 kSortTile points where the
// level has few problems and d = 2 (a whole layout of 4,096 points 16.3 -> 15.7
// ms); for d = 3 the block's one pass over the cells made that slower (24 us
// for the launch, 17 for the device-wide sequence with its launches overlapped).
constexpr int kBinCells = 4096;
constexpr int kFusedProblems = 64;  // most problems of a level whose binning launch does the attraction
constexpr int kBinWide = 2 * kSortTile;  // most points of a problem of a level of at most kFusedProblems
constexpr int kBinSorted = 64;  // points of a cell from which its ids are sorted (blocks of kSortTile points or more)
constexpr int kBinBig = kBinWide / (kCellSerial + 1) + 1;  // most large cells of a problem

// Shared memory of a block: sorted points and weights, slots, cell starts, sums.
struct BinShape {
  int points, cells, sums;  // capacities: points, finest cells, cells of all levels >= 2
  constexpr size_t bytes(int d) const {
    return (size_t)points * (sizeof(float4) + sizeof(float) + sizeof(uint32_t)) + (size_t)(cells + 1) * sizeof(int32_t) +
           (size_t)sums * (d + 1) * sizeof(float);
  }
};

// Shared-memory limit of the kernel for blocks of T threads with ITEMS points
// each: its largest shape.  The limit belongs to the function, for all host
// threads, and a smaller one set by one of them would have another's larger
// launch refused, so it is this constant whatever shape a level has.
template <int D, int T, int ITEMS>
constexpr size_t bin_limit() {
  constexpr int L = 12 / D;  // finest level of at most kBinCells cells
  static_assert((1 << (D * L)) <= kBinCells, "cells of the finest level");
  return BinShape{T * ITEMS, 1 << (D * L), ((1 << (D * (L + 1))) - 1) / ((1 << D) - 1)}.bytes(D);
}
static_assert(bin_limit<2, 1024, 4>() <= 220 * 1024 && bin_limit<3, 1024, 2>() <= 220 * 1024 &&
                  bin_limit<4, 1024, 2>() <= 220 * 1024,
              "a block's shared memory, with room for the static arrays");

template <int D, int T, int ITEMS>  // up to ITEMS points per thread
__global__ void __launch_bounds__(T) k_bin_small(
    const float4* __restrict__ x, const float* __restrict__ w, const ProbDev* __restrict__ prob, int P,
    const uint32_t* __restrict__ bb, uint32_t* __restrict__ bb_next, int32_t* __restrict__ tctr,
    uint32_t* __restrict__ keys, uint32_t* __restrict__ svals, float4* __restrict__ xs, float* __restrict__ ws,
    uint32_t* __restrict__ scell, int32_t* __restrict__ cst, float4* __restrict__ XP, float4* __restrict__ CP,
    int32_t* __restrict__ cch, int32_t* __restrict__ chunk, BinShape shape, Attract at) {
  pdl_enter();
  if ((int)blockIdx.x >= P) {
    attract_rows<T>(at, (int64_t)blockIdx.x - P);
    return;
  }
  constexpr bool SORT = ITEMS * T >= kSortTile;
  extern __shared__ __align__(16) unsigned char bin_raw[];
  float4* sx = reinterpret_cast<float4*>(bin_raw);
  float* sw = reinterpret_cast<float*>(sx + shape.points);
  uint32_t* slot = reinterpret_cast<uint32_t*>(sw + shape.points);
  int32_t* cs = reinterpret_cast<int32_t*>(slot + shape.points);
  float* sS = reinterpret_cast<float*>(cs + shape.cells + 1);  // [D + 1][sums]
  __shared__ uint64_t scan[33];
  __shared__ int32_t big[kBinBig];
  __shared__ int nbig;
  const int pb = blockIdx.x;
  const ProbDev pr = prob[pb];
  const int k = pr.k, L = pr.L;
  const int64_t vb = pr.vbase;
  if (pb == 0 && threadIdx.x == 0) ++*tctr;  // the level's step
  if (threadIdx.x < 8) bb_next[pb * 8 + threadIdx.x] = threadIdx.x < 4 ? 0xFFFFFFFFu : 0u;
  const int ncell = 1 << (D * L);
  for (int c = threadIdx.x; c <= ncell; c += T) cs[c] = 0;
  if (threadIdx.x == 0) nbig = 0;
  // the thread's points and weights
  float4 xv[ITEMS];
  float wv[ITEMS];
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const int i = threadIdx.x + j * T;
    xv[j] = i < k ? x[vb + i] : make_float4(0.f, 0.f, 0.f, 0.f);
    wv[j] = (i < k && w) ? w[vb + i] : 1.0f;
  }
  float lo[D], s;
  grid_frame<D>(bb, pb, L, lo, &s);
  __syncthreads();
  uint32_t key[ITEMS], arr[ITEMS];
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const int i = threadIdx.x + j * T;
    key[j] = arr[j] = 0;
    if (i < k) {
      int32_t c[D];
      cell_of<D>(xv[j], lo, s, L, c);
      key[j] = min((uint32_t)rowmajor<D>(c, 1 << L), (uint32_t)(ncell - 1));
      arr[j] = (uint32_t)atomicAdd(&cs[key[j]], 1);
      if (keys) keys[vb + i] = key[j];
    }
  }
  __syncthreads();
  {  // cell counts -> starts, and the chunks of two points (see k_cell_scan)
    const int per = (ncell + T - 1) / T, c0 = min((int)threadIdx.x * per, ncell), c1 = min(c0 + per, ncell);
    uint64_t sum = 0;
    for (int c = c0; c < c1; ++c) sum += ((uint64_t)(uint32_t)((cs[c] + 1) >> 1) << 32) | (uint32_t)cs[c];
    uint64_t total;
    const uint64_t ex = block_exclusive<uint64_t>(sum, scan, &total);
    int32_t run = (int32_t)(uint32_t)ex, chk = (int32_t)(ex >> 32);
    for (int c = c0; c < c1; ++c) {
      const int32_t n = cs[c];
      cs[c] = run;
      if (SORT && n > kBinSorted) big[atomicAdd(&nbig, 1)] = c;
      cst[pr.fbase + pb + c] = (int32_t)vb + run;
      if (cch) cch[pr.fbase + pb + c] = (int32_t)vb + chk;  // a problem's chunks are listed from its first point on
      run += n;
      chk += (n + 1) >> 1;
    }
    if (threadIdx.x == 0) {
      cs[ncell] = k;
      cst[pr.fbase + pb + ncell] = (int32_t)vb + k;
      if (cch) cch[pr.fbase + pb + ncell] = (int32_t)vb + (int32_t)(total >> 32);
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const int i = threadIdx.x + j * T;
    if (i < k) slot[cs[key[j]] + arr[j]] = (uint32_t)i;
  }
  __syncthreads();
  if (SORT && nbig > 0) {
    // the ids of a crowded cell in order, a warp per cell: a bit per point of the
    // problem, set for the cell's, the prefix sums of the set bits, and the bits
    // read off (4,000 / 2,000 points, 99 % of them in one cell: 32 / 20 us of the launch, 311 / 86 us
    // when every two points of a cell were compared)
    uint32_t* bits = reinterpret_cast<uint32_t*>(sx) + (threadIdx.x >> 5) * ((k + 31) / 32);
    const int lane = lane_id(), words = (k + 31) / 32, per = (words + 31) / 32;
    for (int b = threadIdx.x >> 5; b < nbig; b += T / 32) {
      const int q0 = cs[big[b]], q1 = cs[big[b] + 1];
      for (int i = lane; i < words; i += 32) bits[i] = 0;
      __syncwarp();
      for (int q = q0 + lane; q < q1; q += 32) atomicOr(&bits[slot[q] >> 5], 1u << (slot[q] & 31));
      __syncwarp();
      const int i0 = min(lane * per, words), i1 = min(i0 + per, words);
      int own = 0;
      for (int i = i0; i < i1; ++i) own += __popc(bits[i]);
      int q = q0 + warp_inclusive(own) - own;
      for (int i = i0; i < i1; ++i)
        for (uint32_t m = bits[i]; m; m &= m - 1) slot[q++] = (uint32_t)(32 * i + __ffs(m) - 1);
      __syncwarp();
    }
    __syncthreads();
    if (threadIdx.x == 0) nbig = 0;
  }
  const int64_t e = (vb + pb + 1) & ~int64_t(1);
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const int i = threadIdx.x + j * T;
    if (i >= k) continue;
    const int q0 = cs[key[j]], q1 = cs[key[j] + 1];
    int less = 0;
    if (!SORT || q1 - q0 <= kBinSorted) {
      for (int q = q0; q < q1; ++q) less += slot[q] < (uint32_t)i;
    } else {  // the first of the sorted ids that is not smaller
      for (int n = q1 - q0; n > 0;) {
        const int half = n >> 1;
        const bool up = slot[q0 + less + half] < (uint32_t)i;
        less += up ? half + 1 : 0;
        n = up ? n - half - 1 : half;
      }
    }
    const int q = q0 + less;
    const int64_t p = vb + q;
    sx[q] = xv[j];
    sw[q] = wv[j];
    svals[p] = (uint32_t)(vb + i);
    xs[p] = xv[j];
    if (ws) ws[p] = wv[j];
    const float xc[4] = {xv[j].x, xv[j].y, xv[j].z, xv[j].w};
    pair_store<D>(XP, e + q, xc, wv[j]);
    if (q == k - 1 && (k & 1)) {
      const float zero[4] = {0.f, 0.f, 0.f, 0.f};
      pair_store<D>(XP, e + k, zero, 0.0f);
    }
    uint32_t packed = 0;
#pragma unroll
    for (int m = 0; m < D; ++m) packed |= ((key[j] >> (m * L)) & ((1u << L) - 1u)) << (m * field_bits(D));
    scell[p] = packed;
    if (cch && !(less & 1)) chunk[cch[pr.fbase + pb + key[j]] + (less >> 1)] = (int32_t)p;
  }
  if (L < 2) return;  // no far field
  __syncthreads();
  // sums of the finest cells, then of every coarser level from its children
  auto keep = [&](int l, int at_, int c, const float* S, float W) {
    float z[4] = {0.f, 0.f, 0.f, 0.f};
    if (W > 0.0f) {
      const float iw = 1.0f / W;
#pragma unroll
      for (int m = 0; m < D; ++m) z[m] = S[m] * iw;
    }
#pragma unroll
    for (int m = 0; m < D; ++m) sS[m * shape.sums + at_ + c] = S[m];
    sS[D * shape.sums + at_ + c] = W;
    pair_store<D>(CP, pr.cbase + lvl_off(D, l) + c + pb + 1, z, W);
  };
  for (int c = threadIdx.x; c < ncell; c += T) {
    const int q0 = cs[c], q1 = cs[c + 1];
    if (q1 - q0 > kCellSerial) {
      big[atomicAdd(&nbig, 1)] = c;
      continue;
    }
    float S[4] = {0.f, 0.f, 0.f, 0.f};
    float W = 0.f;
    for (int q = q0; q < q1; ++q) cell_add<D>(sx[q], sw[q], S, W);
    keep(L, 0, c, S, W);
  }
  __syncthreads();
  for (int b0 = 0; b0 < nbig; b0 += T / kCellLanes) {
    const int b = b0 + threadIdx.x / kCellLanes;
    const bool mine = b < nbig;
    float S[4] = {0.f, 0.f, 0.f, 0.f};
    float W = 0.f;
    cell_sum_quarter<D>(sx, sw, mine ? cs[big[b]] : 0, mine ? cs[big[b] + 1] : 0, S, W);
    if (mine && (threadIdx.x & (kCellLanes - 1)) == 0) keep(L, 0, big[b], S, W);
  }
  int from = 0, to = ncell;
  for (int l = L - 1; l >= 2; --l) {
    __syncthreads();
    const int n = 1 << (D * l), side = 1 << l;
    for (int c = threadIdx.x; c < n; c += T) {
      float S[4] = {0.f, 0.f, 0.f, 0.f};
      float W = 0.f;
#pragma unroll
      for (int ch = 0; ch < (1 << D); ++ch) {
        int q = 0;
#pragma unroll
        for (int m = 0; m < D; ++m)
          q |= (2 * ((c >> (m * l)) & (side - 1)) + ((ch >> m) & 1)) << (m * (l + 1));
#pragma unroll
        for (int m = 0; m < D; ++m) S[m] += sS[m * shape.sums + from + q];
        W += sS[D * shape.sums + from + q];
      }
      keep(l, to, c, S, W);
    }
    from = to;
    to += n;
  }
}

// Degree class of every row, counted by one scan: 1 medium, 2^32 heavy.
__global__ void k_degree_class(const int32_t* __restrict__ adj_ptr, int64_t K, uint64_t* __restrict__ cls) {
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= K) return;
  const int32_t deg = adj_ptr[v + 1] - adj_ptr[v];
  cls[v] = deg <= kLightMax ? 0ull : (deg <= kWarpMax ? 1ull : 1ull << 32);
}

__global__ void k_class_lists(const uint64_t* __restrict__ cls, const uint64_t* __restrict__ pos, int64_t K,
                              int32_t* __restrict__ mid, int32_t* __restrict__ heavy) {
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= K) return;
  const uint64_t c = cls[v];
  if (c == 1) mid[(uint32_t)pos[v]] = (int32_t)v;
  else if (c) heavy[pos[v] >> 32] = (int32_t)v;
}

// Net centres z_j of general nets (Algorithm 4).
__global__ void k_net_center(const int32_t* __restrict__ net_ptr, const int32_t* __restrict__ pins, int64_t l,
                             const float4* __restrict__ x, float4* __restrict__ z) {
  pdl_enter();
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= l) return;
  int32_t a = net_ptr[j], b = net_ptr[j + 1];
  float4 s = make_float4(0, 0, 0, 0);
  for (int32_t t = a; t < b; ++t) {
    float4 q = x[pins[t]];
    s.x += q.x; s.y += q.y; s.z += q.z; s.w += q.w;
  }
  float inv = (b > a) ? 1.0f / (float)(b - a) : 0.f;
  z[j] = make_float4(s.x * inv, s.y * inv, s.z * inv, s.w * inv);
}

__global__ void k_attract_hyper(const int32_t* __restrict__ vtx_ptr, const int32_t* __restrict__ vnets,
                                const float4* __restrict__ x, const float4* __restrict__ z, int64_t K,
                                float4* __restrict__ y) {
  pdl_enter();
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= K) return;
  float4 xv = x[v];
  float4 a = make_float4(0, 0, 0, 0);
  for (int32_t t = vtx_ptr[v]; t < vtx_ptr[v + 1]; ++t) {
    float4 q = z[vnets[t]];
    a.x += xv.x - q.x; a.y += xv.y - q.y; a.z += xv.z - q.z; a.w += xv.w - q.w;
  }
  y[v] = a;
}

// Approximate reciprocal and reciprocal square root (PTX rcp/rsqrt.approx,
// flush-to-zero) for the force terms; the decisions elsewhere use exactly
// rounded intrinsics.
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Added to every squared distance fed to the kernels.  A source at the
// target's own position (the target itself, a coincident point) has dx = 0
// and so contributes exactly 0 * g = 0; the offset keeps g finite for it.
// Masked sources (weight 0) contribute 0 the same way.  For real pairs the
// relative change of r^2 is 1e-15 / r^2, negligible at the spacings of a
// layout (mean point spacing ~1).
constexpr float kR2Floor = 1e-15f;

// w r^-d of the two sources of a pair at the differences dx.
template <int D, bool UNIT>
__device__ __forceinline__ float2 pair_factor(const float2* dx, float2 w) {
  float2 r2 = make_float2(kR2Floor, kR2Floor);  // offset: a source at the target's position gives 0 * finite
#pragma unroll
  for (int m = 0; m < D; ++m) r2 = __ffma2_rn(dx[m], dx[m], r2);
  float2 g;
  if (D == 2) {
    const float2 i2 = make_float2(rcp_approx(r2.x), rcp_approx(r2.y));
    g = UNIT ? i2 : __fmul2_rn(w, i2);
  } else if (D == 3) {
    const float2 ir = make_float2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
    g = UNIT ? __fmul2_rn(ir, __fmul2_rn(ir, ir)) : __fmul2_rn(__fmul2_rn(w, ir), __fmul2_rn(ir, ir));
  } else {
    const float2 i2 = make_float2(rcp_approx(r2.x), rcp_approx(r2.y));
    g = UNIT ? __fmul2_rn(i2, i2) : __fmul2_rn(__fmul2_rn(w, i2), i2);
  }
  return g;
}

// F += w r^-d (src - xn) for the two sources of a pair; nx holds -xn twice
// per coordinate, w the (masked) weights.  UNIT: both weights are 1 (the
// multiply by w is left out; a half is masked by giving it the target's own
// coordinates instead, so that its dx = 0 contributes 0).
template <int D, bool UNIT = false>
__device__ __forceinline__ void pair_charge(float2* F, const float4* P, const float2* nx, float2 w) {
  float2 dx[D];
  dx[0] = __fadd2_rn(make_float2(P[0].x, P[0].y), nx[0]);
  if (D > 1) dx[1] = __fadd2_rn(make_float2(P[0].z, P[0].w), nx[1]);
  if (D > 2) dx[2] = __fadd2_rn(make_float2(P[1].x, P[1].y), nx[2]);
  if (D > 3) dx[3] = __fadd2_rn(make_float2(P[1].z, P[1].w), nx[3]);
  const float2 g = pair_factor<D, UNIT>(dx, w);
#pragma unroll
  for (int m = 0; m < D; ++m) F[m] = __ffma2_rn(g, dx[m], F[m]);
}

// Gives half h of a pair the target's coordinates (-nx), so it contributes 0.
template <int D>
__device__ __forceinline__ void pair_mask_half(float4* P, int h, bool mask, const float2* nx) {
  float* f = reinterpret_cast<float*>(P);
#pragma unroll
  for (int m = 0; m < D; ++m) {
    const int i = 4 * (m >> 1) + 2 * (m & 1);
    if (h == 0) f[i] = mask ? -nx[m].x : f[i];
    else f[i + 1] = mask ? -nx[m].x : f[i + 1];
  }
}

template <int D>
__device__ __forceinline__ float2 pair_weight(const float4* P) {
  const float4& q = P[Pair<D>::WQ];
  return Pair<D>::WO == 0 ? make_float2(q.x, q.y) : make_float2(q.z, q.w);
}

// The targets of one thread: T points of one finest cell, so that every
// loaded source pair serves all of them (T = 2 halves the L1 bandwidth per
// interaction).  nx holds -x twice per coordinate, F the force sums of the
// even and the odd sources.  A target's sums take the same sources in the same
// order whatever T is.
template <int D, int T>
struct Targets {
  float2 nx[T][D], F[T][D];
};

template <int D, bool UNIT, int T>
__device__ __forceinline__ void charge_all(Targets<D, T>& g, const float4* P, float2 w) {
#pragma unroll
  for (int t = 0; t < T; ++t) pair_charge<D, UNIT>(g.F[t], P, g.nx[t], w);
}

// Far field.  Of level l the cells of the 6^d box spanned by the children of
// the cells around the target's parent cell act as charges, minus the 3^d
// cells adjacent to the target's cell.  One row of the box along coordinate 0
// starts at an even cell and holds 4 or 6 cells, i.e. 2 or 3 pairs.  The rows
// (row-major, coordinate 1 fastest) go round-robin to the G lanes of the
// target's group: FarRows steps through one lane's rows of every level
// l = 2..L in that order.
template <int D>
struct FarRows {
  int64_t cell0;  // table index of the problem's level-0 cell (lvl_off(0) = 0), odd
  int l, L, G, lane_g;
  int32_t c[D];   // the target's finest cell
  int32_t me[D], lo[D], hi[D];
  int q[D];       // current row: q[1..D-1]
  int half;       // pairs per row of the level's grid
  int64_t base;   // first pair of the level plus lo[0] / 2

  __device__ __forceinline__ void init(int64_t cell, const int32_t* cc, int LL, int GG, int lg) {
    cell0 = cell;
    L = LL;
    G = GG;
    lane_g = lg;
#pragma unroll
    for (int m = 0; m < D; ++m) c[m] = cc[m];
    l = 1;
    next_level();
  }
  __device__ __forceinline__ bool done() const { return l > L; }
  __device__ __forceinline__ void next_level() {
    do {
      ++l;
      if (l > L) return;
      const int sl = 1 << l;
#pragma unroll
      for (int m = 0; m < D; ++m) {
        me[m] = c[m] >> (L - l);
        const int par = me[m] >> 1;
        lo[m] = max(2 * par - 2, 0);
        hi[m] = min(2 * par + 3, sl - 1);
        q[m] = lo[m];
      }
      half = sl >> 1;
      base = ((cell0 + lvl_off(D, l)) >> 1) + (lo[0] >> 1);
      q[1] += lane_g;
      carry();
    } while (q[D - 1] > hi[D - 1]);  // fewer rows than lanes
  }
  __device__ __forceinline__ void carry() {
#pragma unroll
    for (int m = 1; m + 1 < D; ++m) {
      const int e = hi[m] - lo[m] + 1;
      while (q[m] > hi[m]) {
        q[m] -= e;
        ++q[m + 1];
      }
    }
  }
  __device__ __forceinline__ void advance() {
    q[1] += G;
    carry();
    if (q[D - 1] > hi[D - 1]) next_level();
  }
  // first pair of the row, whether it has a third pair, and the mask of its
  // cells (bit i: cell lo[0] + i) that are adjacent to the target's cell
  __device__ __forceinline__ int64_t row(bool& third, unsigned& mask) const {
    int64_t idx = 0;
    bool in = true;
#pragma unroll
    for (int m = D - 1; m >= 1; --m) {
      idx = (idx << l) + q[m];
      in = in && q[m] >= me[m] - 1 && q[m] <= me[m] + 1;
    }
    third = hi[0] - lo[0] > 4;
    const int o = me[0] - lo[0];  // 0, 1, 2 or 3
    mask = in ? (o > 0 ? 7u << (o - 1) : 3u) : 0u;
    return base + idx * half;
  }
};

// Loads of a row: all issued together; a pair beyond the row reads as zeros
// and weighs 0.
template <int D>
__device__ __forceinline__ void row_load(const float4* __restrict__ CP, int64_t row, bool third,
                                         float4 (*P)[Pair<D>::N]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (i < 2 || third) pair_load<D>(CP, row + i, P[i]);
    else pair_zero<D>(P[i]);
  }
}

template <int D, bool COUNT, int T>
__device__ __forceinline__ void row_apply(float4 (*P)[Pair<D>::N], unsigned mask, Targets<D, T>& g,
                                          unsigned long long& nint) {
  float2 w[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) w[i] = pair_weight<D>(P[i]);
  if (mask) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      w[i].x = (mask >> (2 * i)) & 1u ? 0.0f : w[i].x;
      w[i].y = (mask >> (2 * i + 1)) & 1u ? 0.0f : w[i].y;
    }
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    charge_all<D, false, T>(g, P[i], w[i]);
    if (COUNT) nint += (w[i].x > 0.0f) + (w[i].y > 0.0f);
  }
}

// PIPE: the next two rows are loaded before the current two are accumulated
// (launches with too few warps to hide a load behind other warps); else one
// row at a time.
template <int D, bool COUNT, int T, bool PIPE>
__device__ __forceinline__ void far_field(const float4* CP, int64_t cell0, const int32_t* c, int L, int G, int lane_g,
                                          Targets<D, T>& g, unsigned long long& nint) {
  constexpr int N = Pair<D>::N;
  FarRows<D> it;
  it.init(cell0, c, L, G, lane_g);
  if (!PIPE) {
    while (!it.done()) {
      float4 P[3][N];
      bool third;
      unsigned mask;
      const int64_t r = it.row(third, mask);
      row_load<D>(CP, r, third, P);
      it.advance();
      row_apply<D, COUNT, T>(P, mask, g, nint);
    }
    return;
  }
  float4 A[2][3][N], B[2][3][N];
  unsigned ma[2] = {0u, 0u}, mb[2] = {0u, 0u};
  int na = 0, nb = 0;
  auto fetch = [&](float4 (*P)[3][N], unsigned* m, int& n) {
    n = 0;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (it.done()) break;
      bool third;
      const int64_t r = it.row(third, m[u]);
      row_load<D>(CP, r, third, P[u]);
      it.advance();
      ++n;
    }
  };
  auto apply = [&](float4 (*P)[3][N], unsigned* m, int n) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (u < n) row_apply<D, COUNT, T>(P[u], m[u], g, nint);
  };
  fetch(A, ma, na);
  while (na > 0) {
    fetch(B, mb, nb);
    apply(A, ma, na);
    if (nb == 0) break;
    fetch(A, ma, na);
    apply(B, mb, nb);
  }
}

// Next bounding box, folded in by the step kernel: lane 0 of every warp (a
// warp never straddles two problems) applies atomic min / max of the
// order-preserving integer images of its lanes' new coordinates to the
// problem's box, which k_keys reset earlier in the step.  Min and max are
// exact, so the order of the atomics does not matter.
template <int D, int T>
__device__ inline void bbox_warp_fold(const float4* v, const bool* valid, uint32_t* __restrict__ box) {
  uint32_t mn[4], mx[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    uint32_t a = 0xFFFFFFFFu, b = 0u;
#pragma unroll
    for (int t = 0; t < T; ++t)
      if (valid[t] && m < D) {
        const uint32_t o = f2ord(comp(v[t], m));
        a = min(a, o);
        b = max(b, o);
      }
    mn[m] = __reduce_min_sync(0xffffffffu, a);
    mx[m] = __reduce_max_sync(0xffffffffu, b);
  }
  if (lane_id() == 0 && mn[0] != 0xFFFFFFFFu) {
#pragma unroll
    for (int m = 0; m < D; ++m) {
      atomicMin(box + m, mn[m]);
      atomicMax(box + 4 + m, mx[m]);
    }
  }
}

// Near field of one row range [qa, qb) of problem-local sorted positions for
// one lane of the targets' group: source pairs j = qa/2 + lane_g, + G, ...,
// U pairs per trip (all loads issued before the arithmetic).  Only the first
// pair can start before qa and only the last can end at or after qb; those
// halves are masked (weight 0, or the target's own coordinates when UNIT).
template <int D, bool COUNT, bool UNIT, int T, int U, bool GUARD>
__device__ __forceinline__ void near_trip(const float4* __restrict__ xp, int j, int qa, int qb, int G, int64_t tgt,
                                          Targets<D, T>& g, unsigned long long& nint) {
  constexpr int N = Pair<D>::N;
  float4 Q[U][N];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (!GUARD || u == 0 || 2 * (j + u * G) < qb) {
      // the coordinates alone, half the bytes through the load unit (99,000 of 100,000
      // points in one cell: 4.86 -> 3.70 ms a step)
      if (D == 2 && UNIT) {
        Q[u][0] = xp[(int64_t)(j + u * G) * N];
        Q[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
      } else {
        pair_load<D>(xp, j + u * G, Q[u]);
      }
    } else {
      pair_zero<D>(Q[u]);
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int h0 = 2 * (j + u * G);
    if (GUARD && u > 0 && h0 >= qb) break;
    const bool m0 = u == 0 && h0 < qa, m1 = (GUARD || u == U - 1) && h0 + 1 >= qb;
    if (UNIT) {
#pragma unroll
      for (int t = 0; t < T; ++t) {
        float4 R[N];
#pragma unroll
        for (int i = 0; i < N; ++i) R[i] = Q[u][i];
        if (u == 0) pair_mask_half<D>(R, 0, m0, g.nx[t]);
        if (GUARD || u == U - 1) pair_mask_half<D>(R, 1, m1, g.nx[t]);
        pair_charge<D, true>(g.F[t], R, g.nx[t], make_float2(1.0f, 1.0f));
      }
    } else {
      float2 w = pair_weight<D>(Q[u]);
      w.x = m0 ? 0.0f : w.x;
      w.y = m1 ? 0.0f : w.y;
      charge_all<D, false, T>(g, Q[u], w);
    }
    if (COUNT) nint += (h0 >= qa && h0 != tgt) + (h0 + 1 < qb && h0 + 1 != tgt);
  }
}

template <int D, bool COUNT, bool UNIT, int T, int BIG>
__device__ __forceinline__ void near_range(const float4* __restrict__ xp, int qa, int qb, int G, int lane_g,
                                           int64_t tgt, Targets<D, T>& g, unsigned long long& nint) {
  int j = (qa >> 1) + lane_g;
  if (BIG > 4)
    for (; 2 * (j + (BIG - 1) * G) < qb; j += BIG * G)
      near_trip<D, COUNT, UNIT, T, BIG, false>(xp, j, qa, qb, G, tgt, g, nint);
  for (; 2 * (j + 3 * G) < qb; j += 4 * G)
    near_trip<D, COUNT, UNIT, T, 4, false>(xp, j, qa, qb, G, tgt, g, nint);
  if (2 * j < qb) near_trip<D, COUNT, UNIT, T, 3, true>(xp, j, qa, qb, G, tgt, g, nint);
}

// Gradient and step of the point at sorted position p from its repulsion sums.
template <int D>
__device__ __forceinline__ float4 step_target(int64_t p, const float4& xn, const float* Fs, const float* __restrict__ ws,
                                              const uint32_t* __restrict__ svals, const float4* __restrict__ yatt,
                                              float kappa, float step_override, const float* __restrict__ s0, int pb,
                                              const float* __restrict__ scale_tab, const int32_t* __restrict__ tctr,
                                              float4* __restrict__ x, float4* __restrict__ y_out) {
  const float wn = ws ? ws[p] : 1.0f;
  const uint32_t v = svals[p];
  float4 ya = yatt[v];
  float y0 = kappa * wn * Fs[0] + ya.x;
  float y1 = D > 1 ? kappa * wn * Fs[1] + ya.y : 0.f;
  float y2 = D > 2 ? kappa * wn * Fs[2] + ya.z : 0.f;
  float y3 = D > 3 ? kappa * wn * Fs[3] + ya.w : 0.f;
  if (y_out) y_out[v] = make_float4(y0, y1, y2, y3);
  float ny = sqrtf(y0 * y0 + y1 * y1 + y2 * y2 + y3 * y3);
  float step = step_override > 0.0f ? step_override : s0[pb] * scale_tab[*tctr];
  float a = ny > 0.0f ? step / ny : 0.0f;
  const float4 xnew = make_float4(xn.x - a * y0, D > 1 ? xn.y - a * y1 : 0.f, D > 2 ? xn.z - a * y2 : 0.f,
                                  D > 3 ? xn.w - a * y3 : 0.f);
  x[v] = xnew;
  return xnew;
}

// Gradient (eq. graphenergygradientsimple with the grid pyramid) and step of
// every target.  Each problem gives its targets G lanes (G from the problem's
// own size), padded to whole warps; the lanes of a group split the near field
// (strided source pairs) and the far field (rows of every level's box) and
// combine with a fixed xor tree, so a target's result depends only on its own
// problem.  Lane 0 of the group applies the step.  Near field: points are
// sorted by row-major cell index, so the 3 cells of a row along coordinate 0
// form one contiguous range of the sorted points, read in pairs from the
// paired point table XP (a problem's points start at the even slot
// (vbase + pb + 1) & ~1; the halves outside the range weigh 0).  Far field:
// the paired cell table CP, whose index of (problem pb, level l, cell c) is
// cbase + pb + lvl_off(l) + 1 + c (even for even c).
//
// T = 1: a group handles the point at its own sorted position.  T = 2: a
// group handles a chunk of one or two consecutive points of one finest cell;
// the binning lists the chunks' first positions in cell order (cch[c]: first
// chunk of cell c, as cst[c] is its first point), and the problem's threads are
// numbered from tbase2.
// One target per thread is bound by the 32 bytes a pair costs every lane of
// L1 bandwidth (65% busy, FMA pipe 59%, 500,000 clustered points, d = 3, 587
// us); two per thread halve that (36%) and leave the FMA pipe (66%): 568 us,
// 400 against 461 us in that level's later steps.  Measured and not kept:
// leaving out the middle pair of a row where every lane of the warp has it
// masked (8% of the far field's work, 1% slower), other block sizes and
// register limits (within 2%).
constexpr int kStepBlock = 128;

// Which step kernel a level takes, by d and by the threads of one target lane
// each (per step, one level, GB300):
//  - d >= 3, at most 5/8 of g_tuning.small_step_threads (12,160): the split
//    kernel; 3-D grids of 1,728 / 8,000 / 13,824 points 25.2 / 34.9 / 50.2 us
//    against 29.7 / 45.0 / 48.5 us with one thread per lane.
//  - d = 2, at most g_tuning.small_step_threads (4 warps per SM): two far-field
//    rows in flight; 2-D grids of 1,024 / 4,096 points 16.4 / 20.5 us against
//    17.4 / 21.5 us (a target's sums are too short there for the split: 17.6 /
//    22.3 us).
//  - at least kPairThreadsMin: two targets per thread; 110,592 / 262,144 grid
//    points and 500,000 clustered ones 104 / 176 / 480 us against 95 / 196 /
//    538 us with one.
//  - else one target per thread.
constexpr int64_t kPairThreadsMin = 196608;

enum StepMode { kStepPlain = 0, kStepPipe = 1, kStepPair = 2 };
__host__ __device__ constexpr int step_min_blocks(int mode) { return mode == kStepPlain ? 6 : (mode == kStepPipe ? 3 : 4); }

template <int D, bool COUNT, int MODE>
__global__ void __launch_bounds__(kStepBlock, step_min_blocks(MODE)) k_repulse_update(
    const float4* __restrict__ xs, const float* __restrict__ ws, const float4* __restrict__ XP,
    const uint32_t* __restrict__ svals, const uint32_t* __restrict__ scell, const int32_t* __restrict__ cst,
    const float4* __restrict__ CP, const float4* __restrict__ yatt, const int32_t* __restrict__ wprob,
    const ProbDev* __restrict__ prob, int64_t nthreads, const int32_t* __restrict__ chunk,
    const int32_t* __restrict__ cch, float kappa, const float* __restrict__ s0,
    const float* __restrict__ scale_tab, const int32_t* __restrict__ tctr,
    float step_override, float4* __restrict__ x, float4* __restrict__ y_out, uint32_t* __restrict__ bb_next,
    unsigned long long* __restrict__ icount) {
  pdl_enter();
  constexpr int N = Pair<D>::N;
  constexpr int T = MODE == kStepPair ? 2 : 1;
  constexpr bool PIPE = MODE == kStepPipe;
  constexpr int BIG = MODE == kStepPair ? 4 : 8;
  const int64_t th = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int pb = wprob[(th < nthreads ? th : nthreads - 1) >> 5];  // a warp never straddles two problems
  const ProbDev pr = prob[pb];
  const int G = pr.group;
  const int64_t rel = th - (T == 2 ? pr.tbase2 : pr.tbase);
  const int lane_g = (int)(rel & (G - 1));
  int64_t tgt = rel / G;  // problem-local sorted position of the first target
  int first = 0, ntgt = pr.k;  // chunks of the problem, or points
  if (T == 2) {
    first = cch[pr.fbase + pb];
    ntgt = cch[pr.fbase + pb + (int64_t(1) << (D * pr.L))] - first;
  }
  const bool valid = th < nthreads && tgt < ntgt;
  int64_t p = pr.vbase + tgt;
  if (T == 2 && valid) {
    p = chunk[first + tgt];
    tgt = p - pr.vbase;
  }
  unsigned long long nint = 0;
  Targets<D, T> g;
  float4 xn[T];
  bool ok[T];
#pragma unroll
  for (int t = 0; t < T; ++t) {
    ok[t] = valid && t == 0;
    xn[t] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int m = 0; m < D; ++m) g.F[t][m] = make_float2(0.f, 0.f);
  }
  if (valid) {
    const int L = pr.L, side = 1 << L;
    const uint32_t packed = scell[p];
    xn[0] = xs[p];
    if (T == 2) {  // the second target (the first again when the chunk has one)
      ok[T - 1] = tgt + 1 < pr.k && scell[p + (tgt + 1 < pr.k)] == packed;
      xn[T - 1] = xs[p + ok[T - 1]];
    }
#pragma unroll
    for (int t = 0; t < T; ++t)
#pragma unroll
      for (int m = 0; m < D; ++m) g.nx[t][m] = make_float2(-comp(xn[t], m), -comp(xn[t], m));
    int32_t c[D];
#pragma unroll
    for (int m = 0; m < D; ++m) c[m] = cell_field<D>(packed, m, side);
    // near field: rows of 3 cells along coordinate 0 around the target's cell
    const int32_t* cs = cst + pr.fbase + pb;
    const float4* xp = XP + ((pr.vbase + pb + 1) >> 1) * N;  // the problem's first pair
    const int xa = max(c[0] - 1, 0), xb = min(c[0] + 1, side - 1);
    constexpr int NR = D == 2 ? 3 : (D == 3 ? 9 : 27);
    // the row ranges [qa, qb) of the problem's sorted points (empty: outside the grid)
    auto row_range = [&](int o, int& qa, int& qb) {
      int32_t cc[D];
      int oo = o;
      bool inside = true;
      cc[0] = xa;
#pragma unroll
      for (int m = 1; m < D; ++m) {
        cc[m] = c[m] + (oo % 3) - 1;
        oo /= 3;
        inside = inside && cc[m] >= 0 && cc[m] < side;
      }
      qa = qb = 0;
      if (!inside) return;
      const int64_t r0 = rowmajor<D>(cc, side);
      qa = cs[r0] - (int)pr.vbase;  // problem-local
      qb = cs[r0 + (xb - xa) + 1] - (int)pr.vbase;
    };
    auto near_row = [&](int qa, int qb) {
      if (qa >= qb) return;
      if (ws)
        near_range<D, COUNT, false, T, BIG>(xp, qa, qb, G, lane_g, tgt, g, nint);
      else
        near_range<D, COUNT, true, T, BIG>(xp, qa, qb, G, lane_g, tgt, g, nint);
    };
    if (PIPE) {
      // small launches: all rows' ranges loaded before the first row is used
      int qa[NR], qb[NR];
#pragma unroll
      for (int o = 0; o < NR; ++o) row_range(o, qa[o], qb[o]);
#pragma unroll
      for (int o = 0; o < NR; ++o) near_row(qa[o], qb[o]);
    } else {
      for (int o = 0; o < NR; ++o) {
        int qa, qb;
        row_range(o, qa, qb);
        near_row(qa, qb);
      }
    }
    far_field<D, COUNT, T, PIPE>(CP, pr.cbase + pb + 1, c, L, G, lane_g, g, nint);
  }
  float4 xnew[T];
  bool leader[T];
#pragma unroll
  for (int t = 0; t < T; ++t) {
    float Fs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int m = 0; m < D; ++m) Fs[m] = g.F[t][m].x + g.F[t][m].y;
    // combine the lanes of the group (groups never straddle a warp)
    for (int o = G >> 1; o > 0; o >>= 1)
#pragma unroll
      for (int m = 0; m < D; ++m) Fs[m] += __shfl_xor_sync(0xffffffffu, Fs[m], o);
    leader[t] = ok[t] && lane_g == 0;
    xnew[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (leader[t])
      xnew[t] = step_target<D>(p + t, xn[t], Fs, ws, svals, yatt, kappa, step_override, s0, pb, scale_tab, tctr, x, y_out);
  }
  if (COUNT) {
    unsigned long long tot = nint;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    if (lane_id() == 0 && tot) atomicAdd(icount, tot);
  }
  bbox_warp_fold<D, T>(xnew, leader, bb_next + (int64_t)pb * 8);
}

// The same step for launches that leave most of the GPU idle at one thread
// per target lane.  The force sums of a lane are chains of additions whose
// order is part of the result, so they cannot be split; but only the
// additions are serial.  kSplitR threads of the producer warps work for each
// target lane: each evaluates the terms (factor g and difference dx of each
// half) of its own source pairs of the lane's sequence, a round of up to
// kSplitS pairs at a time, and leaves them in shared memory; meanwhile the
// block's last warp, one thread per target lane and half, adds the round
// before in sequence order with the same fused operations.  The sums are those
// of k_repulse_update bit for bit.
constexpr int kSplitR = 8;                          // threads per target lane
constexpr int kSplitS = 4 * kSplitR;                // pairs of a round
constexpr int kSplitWarps = 4;                      // producer warps
constexpr int kSplitLanes = kSplitWarps * 32 / kSplitR;  // target lanes of a block: 16, two threads each of the last warp
constexpr int kSplitBlock = 32 * (kSplitWarps + 1);
static_assert(32 % kSplitLanes == 0 && kSplitLanes % kGroupMax == 0, "a block's lanes: whole targets of one problem");
// Pair indices fit 32 bits: two targets per thread take over at kPairThreadsMin, so a
// level has fewer points than that, and its grids at most 17 cells a point (d = 4).
static_assert(kPairThreadsMin * 16 * 2 < INT32_MAX, "pairs of a level's cell tables");
constexpr int kSplitPitch = kSplitS + 1;            // terms between two halves: 16-byte reads of 8 threads miss no bank twice

// Far-field rows of a target lane as one sequence over the levels (the rows
// and the order of FarRows), visited by one of R threads: rows first, first + R, ...
template <int D, int R>
struct FarSeq {
  int l, L, G, lane_g;
  int32_t c[D], me[D], lo[D], hi[D];
  int i, n;      // the lane's row of the level and how many it has there
  int64_t base;  // first pair of the level plus lo[0] / 2
  int64_t cell0;

  __device__ __forceinline__ void level() {
    if (l > L) return;
    const int sl = 1 << l;
    int rows = 1;
#pragma unroll
    for (int m = 0; m < D; ++m) {
      me[m] = c[m] >> (L - l);
      const int par = me[m] >> 1;
      lo[m] = max(2 * par - 2, 0);
      hi[m] = min(2 * par + 3, sl - 1);
      if (m > 0) rows *= hi[m] - lo[m] + 1;
    }
    n = rows > lane_g ? (rows - lane_g + G - 1) / G : 0;
    base = ((cell0 + lvl_off(D, l)) >> 1) + (lo[0] >> 1);
  }
  __device__ __forceinline__ void init(int64_t cell, const int32_t* cc, int LL, int GG, int lg, int first) {
    cell0 = cell;
    L = LL;
    G = GG;
    lane_g = lg;
#pragma unroll
    for (int m = 0; m < D; ++m) c[m] = cc[m];
    l = 2;
    n = 0;
    level();
    i = first;
    settle();
  }
  __device__ __forceinline__ void settle() {
    while (l <= L && i >= n) {
      i -= n;
      ++l;
      level();
    }
  }
  __device__ __forceinline__ bool done() const { return l > L; }
  // rows of the lane on all levels
  __device__ __forceinline__ int count(int64_t cell, const int32_t* cc, int LL, int GG, int lg) const {
    FarSeq<D, R> s;
    s.init(cell, cc, LL, GG, lg, 0);
    int sum = 0;
    for (s.l = 2; s.l <= LL; ++s.l) {
      s.level();
      sum += s.n;
    }
    return sum;
  }
  __device__ __forceinline__ void advance() {
    i += R;
    settle();
  }
  __device__ __forceinline__ int64_t row(bool& third, unsigned& mask) const {
    int rr = lane_g + G * i;
    int q[D];
    bool in = true;
#pragma unroll
    for (int m = 1; m < D; ++m) {
      const int e = hi[m] - lo[m] + 1;  // 4 or 6 cells
      const int t = m + 1 < D ? (e == 4 ? rr >> 2 : (rr * 10923) >> 16) : 0;
      q[m] = lo[m] + rr - t * e;
      rr = t;
      in = in && q[m] >= me[m] - 1 && q[m] <= me[m] + 1;
    }
    int64_t idx = 0;
#pragma unroll
    for (int m = D - 1; m >= 1; --m) idx = (idx << l) + q[m];
    third = hi[0] - lo[0] > 4;
    const int o = me[0] - lo[0];
    mask = in ? (o > 0 ? 7u << (o - 1) : 3u) : 0u;
    return base + idx * (int64_t(1) << (l - 1));
  }
};

// Terms of one pair, with pair_charge's operations: (g, dx0, dx1, dx2) of the
// even and the odd source to slot `at` of their halves (dx3 beside them).
template <int D, bool UNIT>
__device__ __forceinline__ void pair_terms(const float4* P, const float2* nx, float2 w, float4* terms, float* dx3,
                                           int at) {
  float2 dx[4];
  dx[0] = __fadd2_rn(make_float2(P[0].x, P[0].y), nx[0]);
  dx[1] = __fadd2_rn(make_float2(P[0].z, P[0].w), nx[1]);
  dx[2] = __fadd2_rn(make_float2(P[1].x, P[1].y), nx[2]);
  dx[3] = make_float2(0.f, 0.f);
  if (D > 3) dx[3] = __fadd2_rn(make_float2(P[1].z, P[1].w), nx[D > 3 ? 3 : 0]);
  const float2 g = pair_factor<D, UNIT>(dx, w);
  terms[at] = make_float4(g.x, dx[0].x, dx[1].x, dx[2].x);
  terms[kSplitPitch + at] = make_float4(g.y, dx[0].y, dx[1].y, dx[2].y);
  if (D > 3) {
    dx3[at] = dx[3].x;
    dx3[kSplitPitch + at] = dx[3].y;
  }
}

// The end of a round, where the producer warps and the adding warp arrive from
// different code: a barrier of its own number, which counts the block's
// threads wherever they come from (__syncthreads() wants one place for all).
__device__ __forceinline__ void split_round_barrier() {
  asm volatile("bar.sync 1, %0;" ::"n"(kSplitBlock) : "memory");
}

template <int D>
__global__ void __launch_bounds__(kSplitBlock, 4) k_repulse_split(
    const float4* __restrict__ xs, const float* __restrict__ ws, const float4* __restrict__ XP,
    const uint32_t* __restrict__ svals, const uint32_t* __restrict__ scell, const int32_t* __restrict__ cst,
    const float4* __restrict__ CP, const float4* __restrict__ yatt, const int32_t* __restrict__ wprob,
    const ProbDev* __restrict__ prob, float kappa, const float* __restrict__ s0,
    const float* __restrict__ scale_tab, const int32_t* __restrict__ tctr, float step_override,
    float4* __restrict__ x, float4* __restrict__ y_out, uint32_t* __restrict__ bb_next) {
  pdl_enter();
  constexpr int N = Pair<D>::N, R = kSplitR, S = kSplitS, PITCH = kSplitPitch, LN = kSplitLanes;
  static_assert(D > 2, "the sums of d = 2 are too short");
  constexpr int NR = D == 3 ? 9 : 27;  // near-field rows
  __shared__ float4 terms[2][LN * 2 * PITCH];
  __shared__ float terms3[2][D > 3 ? LN * 2 * PITCH : 1];
  __shared__ int32_t rq[LN][NR][2];     // near rows: [qa, qb)
  __shared__ int32_t rpre[LN][NR + 1];  // pairs of the lane before each row
  __shared__ int rounds[2];             // near, far
  const bool producer = threadIdx.x < 32 * kSplitWarps;
  const int grp = producer ? threadIdx.x / R : (threadIdx.x & 31) >> 1;  // target lane of the block
  const int r = threadIdx.x & (R - 1);
  const int64_t vl = (int64_t)blockIdx.x * LN + grp;  // a block's target lanes lie in one problem
  const int pb = wprob[((int64_t)blockIdx.x * LN) >> 5];
  const ProbDev pr = prob[pb];
  const int G = pr.group;
  const int64_t rel = vl - pr.tbase;
  const int lane_g = (int)(rel & (G - 1));
  const int64_t tgt = rel / G;
  const bool valid = tgt < pr.k;
  const int64_t p = valid ? pr.vbase + tgt : pr.vbase;
  const int L = pr.L, side = 1 << L;
  float4 xn = make_float4(0.f, 0.f, 0.f, 0.f);
  uint32_t packed = 0;
  if (valid) {
    xn = xs[p];
    packed = scell[p];
  }
  int32_t c[D];
#pragma unroll
  for (int m = 0; m < D; ++m) c[m] = cell_field<D>(packed, m, side);
  if (threadIdx.x < 2) rounds[threadIdx.x] = 0;
  if (producer) {  // near field: the lane's pairs of the 3^(d-1) rows as one sequence
    for (int o = r; o < NR; o += R) {
      int32_t cc[D];
      int oo = o;
      bool inside = valid;
      cc[0] = max(c[0] - 1, 0);
#pragma unroll
      for (int m = 1; m < D; ++m) {
        cc[m] = c[m] + (oo % 3) - 1;
        oo /= 3;
        inside = inside && cc[m] >= 0 && cc[m] < side;
      }
      int qa = 0, qb = 0, np = 0;
      if (inside) {
        const int32_t* cs = cst + pr.fbase + pb;
        const int64_t r0 = rowmajor<D>(cc, side);
        qa = cs[r0] - (int)pr.vbase;  // problem-local
        qb = cs[r0 + min(c[0] + 1, side - 1) - cc[0] + 1] - (int)pr.vbase;
        if (qb > qa) np = max(((qb + 1) >> 1) - (qa >> 1) - lane_g, 0);
      }
      rq[grp][o][0] = qa;
      rq[grp][o][1] = qb;
      rpre[grp][o + 1] = (np + G - 1) / G;
    }
  }
  __syncthreads();
  FarSeq<D, R> it;
  it.init(pr.cbase + pb + 1, c, valid ? L : 1, G, lane_g, r);
  if (producer && r == 0) {
    int run = 0;
    rpre[grp][0] = 0;
    for (int o = 1; o <= NR; ++o) rpre[grp][o] = run += rpre[grp][o];
    atomicMax(&rounds[0], (run + S - 1) / S);
    atomicMax(&rounds[1], valid ? (it.count(pr.cbase + pb + 1, c, L, G, lane_g) + R - 1) / R : 0);
  }
  __syncthreads();
  const int near = rounds[0], all = near + rounds[1];
  if (producer) {
    float2 nx[D];
#pragma unroll
    for (int m = 0; m < D; ++m) nx[m] = make_float2(-comp(xn, m), -comp(xn, m));
    const int total = rpre[grp][NR];
    const float4* xp = XP + ((pr.vbase + pb + 1) >> 1) * N;  // the problem's first pair
    float4* out = nullptr;
    float* out3 = nullptr;
    int o = 0, h0[4], qa[4], qb[4];
    float4 Q[4][N];
    // the thread's pairs of a near round: r, r + R, ... of the round's part of
    // the sequence, so that the R threads read consecutive pairs
    auto load_near = [&](int rd) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int f = rd * S + u * R + r;
        h0[u] = -1;
        if (f < total) {
          while (f >= rpre[grp][o + 1]) ++o;
          qa[u] = rq[grp][o][0];
          qb[u] = rq[grp][o][1];
          const int j = (qa[u] >> 1) + lane_g + G * (f - rpre[grp][o]);
          h0[u] = 2 * j;
          pair_load<D>(xp, j, Q[u]);
        }
      }
    };
    // its pairs of a far round: thread r steps through row r of the round's R
    // rows, and the R threads share out the rows' 3 R pairs in order (three
    // neighbours read one row; a row each would scatter every load over R lines)
    unsigned mask[3] = {0u, 0u, 0u};
    bool have[3] = {false, false, false};
    auto load_far = [&]() {
      bool third = false;
      unsigned m = 0u;
      const bool live = !it.done();
      const int row = live ? (int)it.row(third, m) : -1;
      m |= third ? 64u : 0u;
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        const int f = u * R + r, q = (f * 11) >> 5, i = f - 3 * q;  // f / 3 for f < 24
        const int rq_ = __shfl_sync(0xffffffffu, row, (threadIdx.x & 31 & ~(R - 1)) + q);
        const unsigned mq = __shfl_sync(0xffffffffu, m, (threadIdx.x & 31 & ~(R - 1)) + q);
        have[u] = rq_ >= 0 && (i < 2 || (mq & 64u));
        mask[u] = mq >> (2 * i);
        if (have[u]) pair_load<D>(CP, (int64_t)rq_ + i, Q[u]);
      }
      it.advance();
    };
    auto put_zero = [&](int at) {
      out[at] = out[PITCH + at] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (D > 3) out3[at] = out3[PITCH + at] = 0.f;
    };
    if (near > 0) load_near(0);
    else if (all > 0) load_far();
    for (int t = 0; t < all; ++t) {
      out = &terms[t & 1][grp * 2 * PITCH];
      out3 = &terms3[t & 1][D > 3 ? grp * 2 * PITCH : 0];
      if (t < near) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int at = u * R + r;  // 16-byte writes of the R threads side by side
          if (h0[u] < 0) {
            put_zero(at);
            continue;
          }
          const bool m0 = h0[u] < qa[u], m1 = h0[u] + 1 >= qb[u];
          if (ws) {
            float2 w = pair_weight<D>(Q[u]);
            w.x = m0 ? 0.0f : w.x;
            w.y = m1 ? 0.0f : w.y;
            pair_terms<D, false>(Q[u], nx, w, out, out3, at);
          } else {
            pair_mask_half<D>(Q[u], 0, m0, nx);
            pair_mask_half<D>(Q[u], 1, m1, nx);
            pair_terms<D, true>(Q[u], nx, make_float2(1.0f, 1.0f), out, out3, at);
          }
        }
        if (t + 1 < near) load_near(t + 1);
        else if (t + 1 < all) load_far();
      } else {
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          if (!have[u]) {
            put_zero(u * R + r);
            continue;
          }
          float2 w = pair_weight<D>(Q[u]);
          w.x = mask[u] & 1u ? 0.0f : w.x;
          w.y = mask[u] & 2u ? 0.0f : w.y;
          pair_terms<D, false>(Q[u], nx, w, out, out3, u * R + r);
        }
        if (t + 1 < all) load_far();
      }
      split_round_barrier();
    }
    return;
  }
  // the adding warp: thread = target lane and half
  float F[D];
#pragma unroll
  for (int m = 0; m < D; ++m) F[m] = 0.f;
  const int half = (threadIdx.x & 31) * PITCH;
  auto add = [&](const float4* in, const float* in3, auto U) {
#pragma unroll
    for (int f = 0; f < R * decltype(U)::value; ++f) {
      const float4 v = in[half + f];
      F[0] = __fmaf_rn(v.x, v.y, F[0]);
      F[1] = __fmaf_rn(v.x, v.z, F[1]);
      F[2] = __fmaf_rn(v.x, v.w, F[2]);
      if (D > 3) F[D > 3 ? 3 : 0] = __fmaf_rn(v.x, in3[half + f], F[D > 3 ? 3 : 0]);
    }
  };
  auto add_round = [&](int t) {
    if (t < near) add(terms[t & 1], terms3[t & 1], std::integral_constant<int, 4>());
    else add(terms[t & 1], terms3[t & 1], std::integral_constant<int, 3>());
  };
  for (int t = 0; t < all; ++t) {
    if (t > 0) add_round(t - 1);
    split_round_barrier();
  }
  if (all > 0) add_round(all - 1);
  // even + odd sources, then the G lanes of the target with the same xor tree
  float Fs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int m = 0; m < D; ++m) Fs[m] = F[m] + __shfl_xor_sync(0xffffffffu, F[m], 1);
  for (int o = G >> 1; o > 0; o >>= 1)
#pragma unroll
    for (int m = 0; m < D; ++m) Fs[m] += __shfl_xor_sync(0xffffffffu, Fs[m], 2 * o);
  const bool leader = valid && lane_g == 0 && (threadIdx.x & 1) == 0;
  float4 xnew = make_float4(0.f, 0.f, 0.f, 0.f);
  if (leader)
    xnew = step_target<D>(p, xn, Fs, ws, svals, yatt, kappa, step_override, s0, pb, scale_tab, tctr, x, y_out);
  bbox_warp_fold<D, 1>(&xnew, &leader, bb_next + (int64_t)pb * 8);
}

// Step-length factors decay^t, t < iters: the running double product, each
// rounded to fp32 (one thread, the same operations in the same order on every
// call), so that no host table has to be uploaded per level.
__global__ void k_scale_tab(int iters, double decay, float* __restrict__ tab) {
  double scale = 1.0;
  for (int t = 0; t < iters; ++t) {
    tab[t] = (float)scale;
    scale *= decay;
  }
}

// ------------------------------ initial layout -----------------------------
__global__ void k_init_coords(int64_t K, const int32_t* __restrict__ vprob, const ProbDev* __restrict__ prob,
                              const uint64_t* __restrict__ seeds, const int32_t* __restrict__ start, int D,
                              float4* __restrict__ x) {
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= K) return;
  int pb = vprob[v];
  if (start && !start[pb]) return;
  ProbDev pr = prob[pb];
  uint64_t lv = (uint64_t)(v - pr.vbase);
  float side = (float)pr.side;
  float c[4] = {0.f, 0.f, 0.f, 0.f};
  for (int m = 0; m < D; ++m) {
    uint64_t r = rand64(seeds[pb] ^ kTagCoord, lv, (uint64_t)m);
    float u = __fmul_rn((float)(r >> 40), 0x1p-24f);
    c[m] = __fmul_rn(u, side);
  }
  x[v] = make_float4(c[0], c[1], c[2], c[3]);
}

// Prolongation (Algorithm 3): x(v) = f * x_coarse(pi(v)) + jitter.
__global__ void k_prolong(const float4* __restrict__ xc, const int32_t* __restrict__ pi, int64_t K,
                          const int32_t* __restrict__ vprob, const ProbDev* __restrict__ prob,
                          const float* __restrict__ fac, const uint64_t* __restrict__ seeds, int level, int D,
                          float4* __restrict__ x) {
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= K) return;
  int pb = vprob[v];
  float f = fac[pb];
  if (!(f > 0.0f)) return;
  uint64_t lv = (uint64_t)(v - prob[pb].vbase);
  float4 q = xc[pi[v]];
  float c[4] = {q.x, q.y, q.z, q.w};
  float o[4] = {0.f, 0.f, 0.f, 0.f};
  for (int m = 0; m < D; ++m) {
    uint64_t r = rand64(seeds[pb] ^ kTagJitter, lv, (uint64_t)(4 * level + m));
    float u = (float)(r >> 40) * 0x1p-24f;
    o[m] = f * c[m] + 0.1f * (u - 0.5f);
  }
  x[v] = make_float4(o[0], o[1], o[2], o[3]);
}

// ------------------------------- coarsening --------------------------------
// Handshake heavy-edge matching round: every unmatched vertex of an active
// problem proposes to its unmatched neighbour with the largest cost, ties by
// the smaller hash of the (local) pair and then the smaller id.  The choice is
// an arg-max under a total order, so light (thread), medium (warp) and heavy
// (block) rows all give the same answer.
struct Proposal {
  float c;
  uint64_t h;
  int32_t u;
};

__device__ inline bool better(const Proposal& a, const Proposal& b) {
  if (a.u < 0) return false;
  if (b.u < 0) return true;
  return a.c > b.c || (a.c == b.c && (a.h < b.h || (a.h == b.h && a.u < b.u)));
}

__device__ inline Proposal scan_row(const int32_t* __restrict__ adj_ptr, const int32_t* __restrict__ adj,
                                    const float* __restrict__ acost, const int32_t* __restrict__ mate, int64_t v,
                                    int64_t vb, uint64_t seed, uint64_t b, int32_t start, int32_t stride) {
  // `better` is a total order on the candidates (a row's neighbours are
  // distinct), so the best does not depend on the order they are seen in:
  // four neighbours per trip, their loads issued together
  Proposal best{0.f, 0ull, -1};
  auto consider = [&](int32_t u, int32_t mu, float c) {
    if (u == v || mu >= 0) return;
    uint64_t lu = (uint64_t)(u - vb), lv = (uint64_t)(v - vb);
    uint64_t lo = lu < lv ? lu : lv, hi = lu < lv ? lv : lu;
    Proposal cand{c, rand64(seed, (lo << 32) | hi, b), u};
    if (better(cand, best)) best = cand;
  };
  const int32_t t1 = adj_ptr[v + 1];
  int32_t t = adj_ptr[v] + start;
  for (; t + 3 * stride < t1; t += 4 * stride) {
    int32_t u[4], mu[4];
    float c[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) u[q] = adj[t + q * stride];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      mu[q] = mate[u[q]];
      c[q] = acost ? acost[t + q * stride] : 1.0f;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) consider(u[q], mu[q], c[q]);
  }
  for (; t < t1; t += stride) {
    const int32_t u = adj[t];
    consider(u, mate[u], acost ? acost[t] : 1.0f);
  }
  return best;
}

__device__ inline Proposal warp_best(Proposal p) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Proposal q;
    q.c = __shfl_xor_sync(0xffffffffu, p.c, o);
    q.h = __shfl_xor_sync(0xffffffffu, p.h, o);
    q.u = __shfl_xor_sync(0xffffffffu, p.u, o);
    if (better(q, p)) p = q;
  }
  return p;
}

__global__ void k_propose(const int32_t* __restrict__ adj_ptr, const int32_t* __restrict__ adj,
                          const float* __restrict__ acost, int64_t K, const int32_t* __restrict__ vprob,
                          const ProbDev* __restrict__ prob, const int32_t* __restrict__ active,
                          const uint64_t* __restrict__ seeds, int level, int round, const int32_t* __restrict__ mate,
                          int32_t* __restrict__ prop) {
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= K) return;
  if (adj_ptr[v + 1] - adj_ptr[v] > kLightMax) return;  // k_propose_wide
  int pb = vprob[v];
  int32_t best = -1;
  if (active[pb] && mate[v] < 0)
    best = scan_row(adj_ptr, adj, acost, mate, v, prob[pb].vbase, seeds[pb] ^ kTagMatch,
                    (uint64_t)level * 256 + (uint64_t)round, 0, 1).u;
  prop[v] = best;
}

// Medium rows (list, warp each) or heavy rows (list, block each).
__global__ void __launch_bounds__(kBlock) k_propose_wide(const int32_t* __restrict__ list, int64_t n, int per_block,
                                                         const int32_t* __restrict__ adj_ptr,
                                                         const int32_t* __restrict__ adj,
                                                         const float* __restrict__ acost,
                                                         const int32_t* __restrict__ vprob,
                                                         const ProbDev* __restrict__ prob,
                                                         const int32_t* __restrict__ active,
                                                         const uint64_t* __restrict__ seeds, int level, int round,
                                                         const int32_t* __restrict__ mate,
                                                         int32_t* __restrict__ prop) {
  __shared__ Proposal part[kBlock / 32];
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  int64_t item = per_block ? (int64_t)blockIdx.x : (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  bool ok = item < n;
  int32_t v = ok ? list[item] : 0;
  int pb = ok ? vprob[v] : 0;
  bool act = ok && active[pb] && mate[v] < 0;
  Proposal best{0.f, 0ull, -1};
  if (act) {
    int32_t start = per_block ? (int32_t)threadIdx.x : lane;
    int32_t stride = per_block ? (int32_t)blockDim.x : 32;
    best = scan_row(adj_ptr, adj, acost, mate, v, prob[pb].vbase, seeds[pb] ^ kTagMatch,
                    (uint64_t)level * 256 + (uint64_t)round, start, stride);
  }
  best = warp_best(best);
  if (!per_block) {
    if (ok && lane == 0) prop[v] = best.u;
    return;
  }
  if (lane == 0) part[warp] = best;
  __syncthreads();
  if (threadIdx.x == 0 && ok) {
    Proposal b = part[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
      if (better(part[w], b)) b = part[w];
    prop[v] = b.u;
  }
}

__global__ void k_resolve(const int32_t* __restrict__ prop, int64_t K, int32_t* __restrict__ mate) {
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= K) return;
  int32_t u = prop[v];
  if (u >= 0 && prop[u] == v) mate[v] = u;
}

__global__ void k_anchor(const int32_t* __restrict__ adj_ptr, const int32_t* __restrict__ adj, int64_t K,
                         const int32_t* __restrict__ mate, int32_t* __restrict__ anchor, int32_t* __restrict__ isanc) {
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= K) return;
  int32_t mv = mate[v];
  int32_t a = mv >= 0 ? min((int32_t)v, mv) : (int32_t)v;
  if (mv < 0 && adj_ptr[v + 1] - adj_ptr[v] == 1) {
    int32_t u = adj[adj_ptr[v]];
    if (u != v) {
      int32_t mu = mate[u];
      a = mu >= 0 ? min(u, mu) : u;
    }
  }
  anchor[v] = a;
  isanc[a] = 1;
}

__global__ void k_kc(const int32_t* __restrict__ rank, const int32_t* __restrict__ total, const int64_t* __restrict__ vb,
                     int P, int64_t K, int64_t* __restrict__ kc) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  int64_t a = vb[p], b = vb[p + 1];
  int64_t ra = a < K ? rank[a] : *total;
  int64_t rb = b < K ? rank[b] : *total;
  kc[p] = rb - ra;
}

__global__ void k_pi(const int32_t* __restrict__ anchor, const int32_t* __restrict__ rank, int64_t K,
                     const int32_t* __restrict__ vprob, const ProbDev* __restrict__ prob,
                     const int64_t* __restrict__ newbase, int32_t* __restrict__ pi) {
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= K) return;
  int pb = vprob[v];
  int64_t nb = newbase[pb];
  pi[v] = nb >= 0 ? (int32_t)(nb + rank[anchor[v]] - rank[prob[pb].vbase]) : -1;
}

// Coarse-edge key and cost of the adjacency entries t, t + stride, ... < t1 of
// a row whose vertex has group a: key (a, pi[adj[t]]) in row-major order of
// the coarse pair, the sentinel for an edge inside a group or of a dropped
// vertex.  Every entry's output depends only on the entry, so rows are split
// by degree as for the attraction: a thread per light row (k_contract_keys),
// a warp per medium row, a block per heavy row (the power-law hubs).
__device__ __forceinline__ void contract_row(const int32_t* __restrict__ adj, const float* __restrict__ acost,
                                             const int32_t* __restrict__ pi, int32_t a, int32_t t, int32_t t1,
                                             int32_t stride, uint64_t Kc, uint64_t* __restrict__ keys,
                                             uint32_t* __restrict__ vals) {
  const uint64_t sentinel = Kc * Kc;
  for (; t < t1; t += stride) {
    const int32_t b = a >= 0 ? pi[adj[t]] : -1;
    keys[t] = (a >= 0 && b >= 0 && a != b) ? (uint64_t)a * Kc + (uint64_t)b : sentinel;
    vals[t] = __float_as_uint(acost ? acost[t] : 1.0f);
  }
}

__global__ void k_contract_keys(const int32_t* __restrict__ adj_ptr, const int32_t* __restrict__ adj,
                                const float* __restrict__ acost, int64_t K, const int32_t* __restrict__ pi,
                                uint64_t Kc, uint64_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= K) return;
  const int32_t t0 = adj_ptr[v], t1 = adj_ptr[v + 1];
  if (t1 - t0 > kLightMax) return;  // medium and heavy rows: k_contract_keys_warp / _block
  contract_row(adj, acost, pi, pi[v], t0, t1, 1, Kc, keys, vals);
}

__global__ void k_contract_keys_warp(const int32_t* __restrict__ list, int64_t n, const int32_t* __restrict__ adj_ptr,
                                     const int32_t* __restrict__ adj, const float* __restrict__ acost,
                                     const int32_t* __restrict__ pi, uint64_t Kc, uint64_t* __restrict__ keys,
                                     uint32_t* __restrict__ vals) {
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= n) return;
  const int32_t v = list[w];
  contract_row(adj, acost, pi, pi[v], adj_ptr[v] + (int32_t)lane_id(), adj_ptr[v + 1], 32, Kc, keys, vals);
}

__global__ void k_contract_keys_block(const int32_t* __restrict__ list, const int32_t* __restrict__ adj_ptr,
                                      const int32_t* __restrict__ adj, const float* __restrict__ acost,
                                      const int32_t* __restrict__ pi, uint64_t Kc, uint64_t* __restrict__ keys,
                                      uint32_t* __restrict__ vals) {
  const int32_t v = list[blockIdx.x];
  contract_row(adj, acost, pi, pi[v], adj_ptr[v] + (int32_t)threadIdx.x, adj_ptr[v + 1], (int32_t)blockDim.x, Kc,
               keys, vals);
}

__global__ void k_run_flags(const uint64_t* __restrict__ keys, int64_t n, uint64_t sentinel, int32_t* __restrict__ flag) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  uint64_t k = keys[t];
  flag[t] = (k != sentinel && (t == 0 || keys[t - 1] != k)) ? 1 : 0;
}

__global__ void k_emit_coarse(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ vals, int64_t n,
                              const int32_t* __restrict__ flag, const int32_t* __restrict__ pos, uint64_t Kc,
                              int32_t* __restrict__ adj, float* __restrict__ acost, int32_t* __restrict__ rowcount) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n || !flag[t]) return;
  uint64_t k = keys[t];
  float c = 0.f;
  for (int64_t u = t; u < n && keys[u] == k; ++u) c += __uint_as_float(vals[u]);
  adj[pos[t]] = (int32_t)(k % Kc);
  acost[pos[t]] = c;
  atomicAdd(&rowcount[k / Kc], 1);
}

// Coarse vertex weights (Algorithm 3: a group weighs what its members weigh).
// The fp32 weights are added in FP64, where the sum of a group of fp32 values
// is exact (their exponents lie within the 29 spare bits), so the order of the
// atomics does not change the rounded fp32 result.
__global__ void k_coarse_w(const float* __restrict__ w, const int32_t* __restrict__ pi, int64_t K,
                           double* __restrict__ wc) {
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= K) return;
  int32_t a = pi[v];
  if (a >= 0) atomicAdd(&wc[a], (double)(w ? w[v] : 1.0f));
}

__global__ void k_round_w(const double* __restrict__ wd, int64_t n, float* __restrict__ w) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) w[i] = (float)wd[i];
}

// Problem of every item of four tables whose problems start at base[t][0..P].
struct ProbMaps {
  int32_t* out[4];
  int64_t n[4];
};

__global__ void k_fill_prob(const int64_t* __restrict__ base, int P, ProbMaps maps) {
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    if (v < maps.n[t]) maps.out[t][v] = find_problem(base + (int64_t)t * (P + 1), P, v);
  }
}

__global__ void k_set_last(int32_t* ptr, int64_t n, const int32_t* total) { ptr[n] = *total; }

template <class F>
void dispatch_d(int d, F&& f) {
  if (d == 2) f(std::integral_constant<int, 2>());
  else if (d == 3) f(std::integral_constant<int, 3>());
  else f(std::integral_constant<int, 4>());
}

int lmax(int d) { return d == 2 ? 15 : (d == 3 ? 10 : 7); }

}  // namespace

int grid_levels(int64_t k, int d, int occ) {
  int L = 1;
  while (L < lmax(d) && (int64_t)occ * (int64_t(1) << (d * L)) < k) ++L;
  return L;
}

// Lanes per target of the step kernel: enough threads to fill the GPU for a
// small problem; a function of the problem's own size only.
int group_size(int64_t k) {
  // G lanes per target give a small problem (a latency-bound level) G-fold
  // shorter per-target chains, at the cost of the lanes' combining and of the
  // work each lane repeats; in a batch, where many problems already fill the
  // GPU, that cost is all that remains (measured: 4 / 2 lanes for <= 512 /
  // 4,096 vertices order the 4,096-matrix batch 17% faster than 16 / 4, a
  // single small matrix 3% slower).
  if (k <= 512) return kGroupMax;
  if (k <= 4096) return 2;
  return 1;
}

static vmo_status classify_degrees(LevelBatch& lb, cudaStream_t s) {
  lb.n_mid = lb.n_heavy = 0;
  if (!lb.adj_ptr || lb.K == 0) return VMO_OK;
  Scratch sc(s);
  uint64_t *cls, *pos, *tot;
  VMO_TRY(sc.alloc(&cls, lb.K));
  VMO_TRY(sc.alloc(&pos, lb.K));
  VMO_TRY(sc.alloc(&tot, 1));
  launch(k_degree_class, grid_for(lb.K, kBlock), kBlock, 0, s, lb.adj_ptr, lb.K, cls);
  VMO_LAUNCHED("degree_class");
  VMO_TRY(scan_exclusive<uint64_t>(cls, pos, lb.K, tot, s, sc));
  uint64_t h = 0;
  VMO_CUDA(cudaMemcpyAsync(&h, tot, 8, cudaMemcpyDeviceToHost, s));
  VMO_CUDA(cudaStreamSynchronize(s));  // also: the host tables of level_setup have been copied
  lb.n_mid = (int64_t)(h & 0xffffffffu);
  lb.n_heavy = (int64_t)(h >> 32);
  VMO_TRY(lb.mid_list.resize(std::max<int64_t>(lb.n_mid, 1)));
  VMO_TRY(lb.heavy_list.resize(std::max<int64_t>(lb.n_heavy, 1)));
  if (h) {
    launch(k_class_lists, grid_for(lb.K, kBlock), kBlock, 0, s, cls, pos, lb.K, lb.mid_list.ptr, lb.heavy_list.ptr);
    VMO_LAUNCHED("class_lists");
  }
  return VMO_OK;
}

int init_side(int64_t k, int d) {
  int64_t s = 1;
  for (;;) {
    int64_t p = 1;
    for (int i = 0; i < d; ++i) p *= s;
    if (p >= k) return (int)s;
    ++s;
  }
}

vmo_status level_setup(LevelBatch& lb, int d, int occ, cudaStream_t s) {
  const int P = lb.P;
  lb.L.assign(P, 1);
  lb.cbase.assign(P + 1, 0);
  lb.fbase.assign(P + 1, 0);
  std::vector<ProbDev> pd(P);
  // per problem: vertices, warps of the step kernel (one and two targets per
  // thread), bricks; each with the map from the item to its problem
  std::vector<int64_t> base((size_t)4 * (P + 1), 0);
  int64_t *vb = base.data(), *wb = vb + P + 1, *wb2 = wb + P + 1, *bk = wb2 + P + 1;
  int64_t chunks = 0;
  lb.maxL = 1;
  for (int p = 0; p < P; ++p) {
    int64_t k = lb.vbase[p + 1] - lb.vbase[p];
    int L = grid_levels(k, d, occ);
    lb.L[p] = L;
    lb.maxL = std::max(lb.maxL, L);
    lb.cbase[p + 1] = lb.cbase[p] + lvl_off(d, L + 1);
    lb.fbase[p + 1] = lb.fbase[p] + (int64_t(1) << (d * L));
    pd[p].vbase = lb.vbase[p];
    pd[p].cbase = lb.cbase[p];
    pd[p].fbase = lb.fbase[p];
    pd[p].k = (int32_t)k;
    pd[p].L = L;
    pd[p].side = init_side(std::max<int64_t>(k, 1), d);
    pd[p].group = group_size(k);
    pd[p].tbase = 32 * wb[p];
    pd[p].tbase2 = 32 * wb2[p];
    pd[p].bbase = bk[p];
    // at most one chunk of a single point per cell
    const int64_t ch = (k + std::min<int64_t>(k, int64_t(1) << (d * L))) / 2;
    chunks += ch;
    vb[p + 1] = lb.vbase[p + 1];
    wb[p + 1] = wb[p] + (k * pd[p].group + 31) / 32;
    wb2[p + 1] = wb2[p] + (ch * pd[p].group + 31) / 32;
    bk[p + 1] = bk[p] + (L > 1 ? int64_t(1) << (d * std::max(L - brick_log2(d), 0)) : 0);
  }
  lb.threads = 32 * wb[P];
  lb.threads2 = 32 * wb2[P];
  lb.bricks = bk[P];
  lb.chunks = chunks;
  VMO_TRY(lb.prob.resize(std::max(P, 1)));
  VMO_TRY(lb.vprob.resize((size_t)std::max<int64_t>(lb.K, 1)));
  VMO_CUDA(cudaMemcpyAsync(lb.prob.ptr, pd.data(), P * sizeof(ProbDev), cudaMemcpyHostToDevice, s));
  VMO_TRY(lb.wprob.resize((size_t)std::max<int64_t>(wb[P], 1)));
  VMO_TRY(lb.wprob2.resize((size_t)std::max<int64_t>(wb2[P], 1)));
  VMO_TRY(lb.bprob.resize((size_t)std::max<int64_t>(bk[P], 1)));
  int64_t* db;
  VMO_CUDA(cudaMallocAsync((void**)&db, base.size() * sizeof(int64_t), s));
  g_device_allocs.fetch_add(1, std::memory_order_relaxed);
  VMO_CUDA(cudaMemcpyAsync(db, base.data(), base.size() * sizeof(int64_t), cudaMemcpyHostToDevice, s));
  ProbMaps maps{{lb.vprob.ptr, lb.wprob.ptr, lb.wprob2.ptr, lb.bprob.ptr}, {lb.K, wb[P], wb2[P], bk[P]}};
  const int64_t items = std::max(std::max(lb.K, wb[P]), std::max(wb2[P], bk[P]));
  if (items > 0) launch(k_fill_prob, grid_for(items, kBlock), kBlock, 0, s, db, P, maps);
  VMO_LAUNCHED("fill_prob");
  VMO_CUDA(cudaFreeAsync(db, s));

  VMO_TRY(classify_degrees(lb, s));
  if (!lb.adj_ptr || lb.K == 0) VMO_CUDA(cudaStreamSynchronize(s));  // host tables must outlive the copies
  return VMO_OK;
}

vmo_status init_coords_level(LevelBatch& lb, int d, const uint64_t* seeds_dev, float4* x, const int32_t* start_dev,
                             cudaStream_t s) {
  if (lb.K == 0) return VMO_OK;
  launch(k_init_coords, grid_for(lb.K, kBlock), kBlock, 0, s, lb.K, lb.vprob.ptr, lb.prob.ptr, seeds_dev, start_dev, d, x);
  VMO_LAUNCHED("init_coords");
  return VMO_OK;
}

constexpr int kGraphMinIters = 8;

// Streams of one layout call, shared by its levels (made for each of 22 levels
// they cost 2 ms of the 64^3 grid's layout): `side` for the attraction (fork /
// join events per step) and `main` for the steps when they are replayed from a
// graph (capture needs a stream of its own: the caller's may be the legacy
// stream).
struct SideStream {
  cudaStream_t stream = nullptr, main = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr, start = nullptr, done = nullptr;
  SideStream() {
    if (cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&main, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&join, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&start, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&done, cudaEventDisableTiming) != cudaSuccess) {
      (void)cudaGetLastError();
      release();
    }
  }
  void release() {
    for (cudaEvent_t* e : {&fork, &join, &start, &done}) {
      if (*e) cudaEventDestroy(*e);
      *e = nullptr;
    }
    if (stream) cudaStreamDestroy(stream);
    if (main) cudaStreamDestroy(main);
    stream = main = nullptr;
  }
  ~SideStream() { release(); }
};

// Streams, step-length factors and graphs of one layout call.  A graph is
// destroyed and the streams are closed only when nothing of them is queued any
// more: destroyed behind their last launch, as the levels are queued far ahead
// of the device, they left the request server's slots (four host threads)
// standing after some 100,000 steps, kernels not started and hosts inside the
// driver.  The graphs go level by level while the last level runs; the rest is
// held by the call's Scratch to its end, so that the host does not wait for the
// last level here (1% of a 64 x 64 ordering).
struct LayoutContext {
  struct Replay {
    cudaGraphExec_t graph;
    cudaEvent_t done;  // behind its last launch (null if it could not be made)
  };
  SideStream streams;
  float* scale_tab = nullptr;  // decay^t of the layout's steps
  std::vector<Replay> replays;
  void keep(cudaGraphExec_t graph) {
    Replay r{graph, nullptr};
    if (cudaEventCreateWithFlags(&r.done, cudaEventDisableTiming) != cudaSuccess) {
      (void)cudaGetLastError();
      r.done = nullptr;
    } else {
      cudaEventRecord(r.done, streams.main);
    }
    replays.push_back(r);
  }
  void destroy_all_but(size_t last) {
    size_t n = 0;
    for (; n + last < replays.size(); ++n) {
      const Replay& r = replays[n];
      if (r.done) cudaEventSynchronize(r.done);
      else cudaStreamSynchronize(streams.main);
      cudaGraphExecDestroy(r.graph);
      if (r.done) cudaEventDestroy(r.done);
    }
    replays.erase(replays.begin(), replays.begin() + n);
  }
  ~LayoutContext() {
    destroy_all_but(0);
    for (cudaStream_t st : {streams.main, streams.stream})
      if (st) cudaStreamSynchronize(st);
  }
};

// Step lengths s0 * decay^t: decay^t as the running double product, rounded to
// fp32 (a table read by the step kernel at the level's step counter, which
// k_keys advances).
static vmo_status make_scale_tab(const LayoutOptions& o, int iters, float** tab, cudaStream_t s, Scratch& sc) {
  VMO_TRY(sc.alloc(tab, std::max(iters, 1)));
  launch(k_scale_tab, 1, 1, 0, s, iters, (double)o.decay, *tab);
  VMO_LAUNCHED("scale_tab");
  return VMO_OK;
}

// Points a Scratch at another stream for a scope (its allocations and frees
// then follow that stream's order).
struct ScratchOnStream {
  Scratch& sc;
  cudaStream_t prev;
  ScratchOnStream(Scratch& s, cudaStream_t st) : sc(s), prev(s.stream) { sc.stream = st; }
  ~ScratchOnStream() { sc.stream = prev; }
};

vmo_status layout_level(LevelBatch& lb, const LayoutOptions& o, float4* x, int iters, float step_override,
                        float4* y_out, uint32_t* keys_out, LayoutContext* ctx, cudaStream_t s, Scratch& sc) {
  const int64_t K = lb.K;
  const int P = lb.P;
  const int d = o.d;
  if (K == 0 || iters <= 0) return VMO_OK;
  ScratchFrame frame(sc);
  uint32_t *keys, *arrival = nullptr, *slot = nullptr, *svals, *scell, *bb;
  float4 *xs, *XP, *yatt, *St = nullptr, *CP, *z = nullptr;
  float *ws = nullptr, *Wt = nullptr, *s0;
  int32_t *cst, *cnt = nullptr, *done = nullptr, *chunk = nullptr, *cch = nullptr;
  uint64_t* tot = nullptr;
  const int64_t ncell = lb.cbase[P], nfine = lb.fbase[P];
  VMO_TRY(sc.alloc(&keys, K));
  VMO_TRY(sc.alloc(&svals, K));
  VMO_TRY(sc.alloc(&scell, K));
  VMO_TRY(sc.alloc(&xs, K));
  VMO_TRY(sc.alloc(&yatt, K));
  if (lb.w) VMO_TRY(sc.alloc(&ws, K));
  VMO_TRY(sc.alloc(&CP, (size_t)((ncell + P) / 2 + 1) * (d == 4 ? 3 : 2)));
  VMO_TRY(sc.alloc(&XP, (size_t)((K + P + 1) / 2 + 1) * (d == 4 ? 3 : 2)));
  VMO_TRY(sc.alloc(&cst, nfine + P));
  VMO_TRY(sc.alloc(&bb, (size_t)2 * 8 * P));
  VMO_TRY(sc.alloc(&s0, P));
  if (lb.net_ptr) VMO_TRY(sc.alloc(&z, std::max<int64_t>(lb.nnets, 1)));
  // levels whose problems all fit one sort tile are binned by one block per
  // problem (k_bin_small) when the tuning allows it
  int64_t kmax = 0;
  for (int p = 0; p < P; ++p) kmax = std::max(kmax, lb.vbase[p + 1] - lb.vbase[p]);
  const int64_t bin_points = g_tuning.small_bin_points.load(std::memory_order_relaxed);
  bool bin1 = kmax <= (bin_points >= kSortTile && P <= kFusedProblems && d == 2 ? kBinWide : bin_points);
  for (int p = 0; p < P && bin1; ++p) bin1 = (int64_t(1) << (d * lb.L[p])) <= kBinCells;
  BinShape shape{(int)std::max<int64_t>((kmax + 3) / 4 * 4, 4), 1 << (d * std::min(lb.maxL, 12 / d)),
                 (int)(lvl_off(d, std::min(lb.maxL, 12 / d) + 1))};
  // (512 threads up to 1,024 points: 13.4 -> 12.3 us a step of one problem for d = 2, the launch of
  // 168 problems 10.9 -> 9.0 us; one problem of d = 3 9.2 -> 9.8 us, so that keeps 1,024)
  const int64_t mid = d == 2 || P > kFusedProblems ? 1024 : 512;
  const auto bin_size = [&](auto DC, auto&& f) {  // threads of a problem's block and points of a thread
    using std::integral_constant;
    if (kmax > kSortTile) {
      if constexpr (decltype(DC)::value == 2) f(integral_constant<int, 1024>(), integral_constant<int, 4>());
    } else if (kmax > mid) f(integral_constant<int, 1024>(), integral_constant<int, 2>());
    else if (kmax > 512) f(integral_constant<int, 512>(), integral_constant<int, 1024 / 512>());
    else f(integral_constant<int, 256>(), integral_constant<int, 2>());
  };
  if (bin1 && shape.bytes(d) > 40 * 1024)  // with the static arrays above the default limit of 48 KB
    dispatch_d(d, [&](auto DC) {
      constexpr int D = decltype(DC)::value;
      cudaError_t err = cudaSuccess;
      bin_size(DC, [&](auto TC, auto IC) {
        constexpr int T = decltype(TC)::value, ITEMS = decltype(IC)::value;
        err = cudaFuncSetAttribute(k_bin_small<D, T, ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)bin_limit<D, T, ITEMS>());
      });
      if (err != cudaSuccess) {
        (void)cudaGetLastError();
        bin1 = false;  // the device-wide sequence then
      }
    });
  const bool pair = lb.threads >= kPairThreadsMin;
  const int64_t ncnt = nfine + P;  // entries of the cell start table
  if (pair) {
    VMO_TRY(sc.alloc(&chunk, K));
    VMO_TRY(sc.alloc(&cch, ncnt));
  }
  const bool one_cluster = ncnt <= kCellScanTile;
  const unsigned scan_blocks = grid_for(ncnt, kCellScanThreads * kCellScanItems);
  if (!bin1) {
    VMO_TRY(sc.alloc(&St, ncell));
    VMO_TRY(sc.alloc(&Wt, ncell));
    VMO_TRY(sc.alloc(&arrival, K));
    VMO_TRY(sc.alloc(&slot, K));
    VMO_TRY(sc.alloc(&cnt, ncnt));
    VMO_TRY(sc.alloc(&done, P));
    if (!one_cluster) VMO_TRY(sc.alloc(&tot, scan_blocks));
    VMO_CUDA(cudaMemsetAsync(cnt, 0, ncnt * sizeof(int32_t), s));
    VMO_CUDA(cudaMemsetAsync(done, 0, P * sizeof(int32_t), s));
  }
  launch(k_bbox_reset, grid_for(16 * P, kBlock), kBlock, 0, s, bb, 16 * P);
  VMO_LAUNCHED("bbox_reset");
  const float kappa = d == 2 ? 1.0f : (float)(d - 2);
  float* scale_tab = ctx ? ctx->scale_tab : nullptr;
  int32_t* tctr;
  const bool own_step = step_override <= 0.0f;  // the step length comes from the box, not from the caller
  if (!scale_tab && own_step) VMO_TRY(make_scale_tab(o, iters, &scale_tab, s, sc));
  VMO_TRY(sc.alloc(&tctr, 2));
  int32_t* crowded = tctr + 1;
  VMO_CUDA(cudaMemsetAsync(tctr, 0xFF, sizeof(int32_t), s));  // -1: k_keys advances it at every step
  vmo_status st = VMO_OK;
  // streams: the layout's, the level's own, or none for a few steps (making them
  // costs more than the overlap of so few gives) or if they cannot be made
  if (!ctx && iters >= kGraphMinIters) {
    auto own = std::make_shared<LayoutContext>();
    ctx = own.get();
    sc.held.push_back(own);
  }
  SideStream* ss = ctx ? &ctx->streams : nullptr;
  const cudaStream_t side = ss ? ss->stream : nullptr;
  dispatch_d(d, [&](auto DC) {
    constexpr int D = decltype(DC)::value;
    launch(k_bbox<D>, grid_for(K, kBlock), kBlock, 0, s, x, K, lb.vprob.ptr, bb);
    if (own_step) launch(k_step0<D>, grid_for(P, kBlock), kBlock, 0, s, bb, lb.prob.ptr, P, o.sigma, s0);
    cudaStream_t ms = s;  // stream of the steps
    // one step t of Algorithm 4 for every problem (only the parity of t and
    // whether it is the first step matter to the launches)
    auto step = [&](int t) -> vmo_status {
      ScratchFrame f2(sc);
      PdlScope pdl;  // every kernel of a step starts with pdl_wait()
      uint32_t* cur = bb + (t & 1) * 8 * P;
      uint32_t* nxt = bb + ((t + 1) & 1) * 8 * P;
      // attraction depends only on x: in the one-block binning's launch, or on
      // the side stream, overlapped with the binning, joined before the step kernel
      Attract at{lb.adj_ptr, lb.adj, lb.acost, x, K, lb.heavy_list.ptr, lb.mid_list.ptr, lb.n_heavy, lb.n_mid, 0, yatt};
      // (with many problems the wide blocks of the binning fill the SMs and the
      // attraction would wait for them)
      const bool fused = bin1 && lb.adj_ptr && lb.n_heavy == 0 && P <= kFusedProblems;
      const bool fork = side && !fused;
      cudaStream_t as = fork ? side : ms;
      if (fork) {
        cudaEventRecord(ss->fork, ms);
        cudaStreamWaitEvent(side, ss->fork, 0);
      }
      if (fused) {
      } else if (lb.adj_ptr) {
        at.mid_blocks = (lb.n_mid * kMidLanes + kBlock - 1) / kBlock;
        launch(k_attract, (unsigned)at.blocks<kBlock>(), kBlock, 0, as, at);
      } else if (lb.net_ptr) {
        if (lb.nnets > 0) launch(k_net_center, grid_for(lb.nnets, kBlock), kBlock, 0, as, lb.net_ptr, lb.pins, lb.nnets, x, z);
        launch(k_attract_hyper, grid_for(K, kBlock), kBlock, 0, as, lb.vtx_ptr, lb.vnets, x, z, K, yatt);
      } else {
        cudaMemsetAsync(yatt, 0, K * sizeof(float4), as);
      }
      if (fork) cudaEventRecord(ss->join, side);
      if (bin1) {
        bin_size(DC, [&](auto TC, auto IC) {
          constexpr int T = decltype(TC)::value;
          at.mid_blocks = (lb.n_mid * kMidLanes + T - 1) / T;
          const unsigned blocks = (unsigned)(P + (fused ? at.blocks<T>() : 0));
          launch(k_bin_small<D, T, decltype(IC)::value>, blocks, T, shape.bytes(D), ms, x, lb.w, lb.prob.ptr, P, cur, nxt,
                 tctr, keys_out && t == 0 ? keys : nullptr, svals, xs, ws, scell, cst, XP, CP, cch, chunk, shape, at);
        });
        if (keys_out && t == 0) cudaMemcpyAsync(keys_out, keys, K * 4, cudaMemcpyDeviceToDevice, ms);
      } else {
        auto keys_kernel = K >= kKeyItemsMin ? k_keys<D, 4> : k_keys<D, 1>;
        launch(keys_kernel, grid_for(K >= kKeyItemsMin ? (K + 3) / 4 : K, kBlock), kBlock, 0, ms, x, K, lb.vprob.ptr,
               lb.prob.ptr, cur, keys, arrival, cnt, P, nxt, tctr);
        if (keys_out && t == 0) cudaMemcpyAsync(keys_out, keys, K * 4, cudaMemcpyDeviceToDevice, ms);
        if (one_cluster) {
          launch(k_cell_scan, kCellScanCtas, kCellScanThreads, 0, ms, cnt, cst, cch, crowded, ncnt);
        } else {
          launch(k_cell_totals, scan_blocks, kCellScanThreads, 0, ms, cnt, ncnt, tot);
          launch(k_cell_starts, scan_blocks, kCellScanThreads, 0, ms, cnt, ncnt, tot, cst, cch,
                 crowded);
        }
        launch(k_slots, grid_for(K, kBlock), kBlock, 0, ms, keys, arrival, K, lb.vprob.ptr, lb.prob.ptr, cst, slot);
        launch(k_place<D>, grid_for(K, kBlock), kBlock, 0, ms, slot, keys, K, x, lb.w, lb.vprob.ptr, lb.prob.ptr, cst,
               cnt, ncnt, crowded, cch, chunk, svals, xs, ws, scell, XP);
        if (lb.bricks > 0)
          launch(k_cells<D>, (unsigned)lb.bricks, kCellsBlock, 0, ms, lb.bprob.ptr, lb.prob.ptr, xs, ws, cst, St, Wt,
                 CP, done);
      }
      if (fork) cudaStreamWaitEvent(ms, ss->join, 0);
      if (g_refused == cudaSuccess) begin_launches();  // also of the events and copies so far
      const bool timed = stats_timing();
      if (timed) stats_time_begin(ms);
      unsigned long long* icount = stats_interaction_counter();
      const int64_t small = g_tuning.small_step_threads.load(std::memory_order_relaxed);
      auto step_launch = [&](auto kernel, int64_t nth, const int32_t* wprob) {
        launch(kernel, grid_for(nth, kStepBlock), kStepBlock, 0, ms, xs, ws, XP, svals, scell, cst, CP, yatt, wprob,
               lb.prob.ptr, nth, chunk, cch, kappa, s0, scale_tab, tctr, step_override, x, y_out, nxt, icount);
      };
      if (icount) {
        step_launch(k_repulse_update<D, true, kStepPlain>, lb.threads, lb.wprob.ptr);
      } else if (pair) {
        step_launch(k_repulse_update<D, false, kStepPair>, lb.threads2, lb.wprob2.ptr);
      } else if (lb.threads <= (D > 2 ? small / 8 * 5 : small)) {
        if constexpr (D > 2)
          launch(k_repulse_split<D>, (unsigned)(lb.threads / kSplitLanes), kSplitBlock, 0, ms, xs, ws, XP, svals, scell,
                 cst, CP, yatt, lb.wprob.ptr, lb.prob.ptr, kappa, s0, scale_tab, tctr, step_override, x, y_out, nxt);
        else
          step_launch(k_repulse_update<D, false, kStepPipe>, lb.threads, lb.wprob.ptr);
      } else {
        step_launch(k_repulse_update<D, false, kStepPlain>, lb.threads, lb.wprob.ptr);
      }
      if (timed) stats_time_end(ms, (uint64_t)K);
      const cudaError_t e = launch_status();
      if (e != cudaSuccess) return cuda_fail(e, "layout step", __FILE__, __LINE__);
      return VMO_OK;
    };
    // Steps are replayed from a CUDA graph of two steps (even and odd parity)
    // when the level runs plain steps; the host then issues one graph launch
    // per two steps instead of ~20 kernel launches per step.
    const bool graphs = ss && ss->main && iters >= kGraphMinIters && !y_out && !keys_out && step_override <= 0.0f &&
                        !stats_timing() && !stats_interaction_counter();
    int t = 0;
    if (graphs) {
      // the steps run on the call's own stream, joined back to s at the end
      cudaEventRecord(ss->start, s);
      cudaStreamWaitEvent(ss->main, ss->start, 0);
      ms = ss->main;
    }
    ScratchOnStream on(sc, ms);  // scratch of a step follows the stream of the step
    if (graphs) {
      cudaGraph_t g = nullptr;
      cudaGraphExec_t ge = nullptr;
      const uint64_t before = g_launches.load();
      bool ok = cudaStreamBeginCapture(ms, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
      vmo_status cst0 = VMO_OK;
      if (ok) {
        cst0 = step(0);
        if (cst0 == VMO_OK) cst0 = step(1);
        // a capture that another thread has ended (by a device-wide wait) says
        // nothing about the steps: they are launched directly then
        const cudaError_t ended = cudaStreamEndCapture(ms, &g);
        if (ended == cudaErrorStreamCaptureInvalidated) cst0 = VMO_OK;
        ok = ended == cudaSuccess && cst0 == VMO_OK;
      }
      if (ok) ok = cudaGraphInstantiate(&ge, g, 0) == cudaSuccess;
      const uint64_t per_graph = g_launches.load() - before;
      g_launches.fetch_sub(per_graph);  // captured, not launched: counted per replay below
      if (ok) {
        for (; t + 2 <= iters; t += 2) {
          cudaError_t e = cudaGraphLaunch(ge, ms);
          if (e != cudaSuccess) {
            st = cuda_fail(e, "cudaGraphLaunch (layout steps)", __FILE__, __LINE__);
            break;
          }
          g_launches.fetch_add(per_graph);
        }
      } else {
        (void)cudaGetLastError();  // fall back to direct launches
        if (cst0 != VMO_OK) st = cst0;
      }
      if (ge) ctx->keep(ge);
      if (g) cudaGraphDestroy(g);
    }
    for (; t < iters && st == VMO_OK; ++t) st = step(t);
    if (ms != s) {
      cudaEventRecord(ss->done, ms);
      cudaStreamWaitEvent(s, ss->done, 0);
    }
  });
  return st;
}

vmo_status coarsen_level(LevelBatch& lb, const uint64_t* seeds_dev, int j, int rounds, const int32_t* active_dev,
                         int32_t* mate, int32_t* anchor, int32_t* rank, std::vector<int64_t>& kc, cudaStream_t s,
                         Scratch& sc) {
  const int64_t K = lb.K;
  const int P = lb.P;
  ScratchFrame frame(sc);
  int32_t *prop, *isanc, *total;
  int64_t *kcd, *vb;
  VMO_TRY(sc.alloc(&prop, K));
  VMO_TRY(sc.alloc(&isanc, K));
  VMO_TRY(sc.alloc(&total, 1));
  VMO_TRY(sc.alloc(&kcd, P));
  VMO_TRY(sc.alloc(&vb, P + 1));
  VMO_CUDA(cudaMemcpyAsync(vb, lb.vbase.data(), (P + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, s));
  VMO_CUDA(cudaMemsetAsync(mate, 0xFF, K * sizeof(int32_t), s));
  VMO_CUDA(cudaMemsetAsync(isanc, 0, K * sizeof(int32_t), s));
  for (int r = 0; r < rounds; ++r) {
    launch(k_propose, grid_for(K, kBlock), kBlock, 0, s, lb.adj_ptr, lb.adj, lb.acost, K, lb.vprob.ptr, lb.prob.ptr,
           active_dev, seeds_dev, j, r, mate, prop);
    if (lb.n_mid)
      launch(k_propose_wide, grid_for(lb.n_mid * 32, kBlock), kBlock, 0, s, lb.mid_list.ptr, lb.n_mid, 0, lb.adj_ptr,
             lb.adj, lb.acost, lb.vprob.ptr, lb.prob.ptr, active_dev, seeds_dev, j, r, mate, prop);
    if (lb.n_heavy)
      launch(k_propose_wide, (unsigned)lb.n_heavy, kBlock, 0, s, lb.heavy_list.ptr, lb.n_heavy, 1, lb.adj_ptr, lb.adj,
             lb.acost, lb.vprob.ptr, lb.prob.ptr, active_dev, seeds_dev, j, r, mate, prop);
    launch(k_resolve, grid_for(K, kBlock), kBlock, 0, s, prop, K, mate);
  }
  launch(k_anchor, grid_for(K, kBlock), kBlock, 0, s, lb.adj_ptr, lb.adj, K, mate, anchor, isanc);
  VMO_LAUNCHED("matching");
  VMO_TRY(scan_exclusive<int32_t>(isanc, rank, K, total, s, sc));
  launch(k_kc, grid_for(P, kBlock), kBlock, 0, s, rank, total, vb, P, K, kcd);
  VMO_LAUNCHED("kc");
  kc.resize(P);
  VMO_CUDA(cudaMemcpyAsync(kc.data(), kcd, P * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  VMO_CUDA(cudaStreamSynchronize(s));
  return VMO_OK;
}

// Builds the next (coarser) level from level `lb` for the problems with
// newbase[p] >= 0 (host), using the grouping (anchor, rank).
static vmo_status contract_level(LevelBatch& lb, const std::vector<int64_t>& newbase, int64_t Kc, const int32_t* anchor,
                                 const int32_t* rank, int32_t* pi, LevelBatch& out, cudaStream_t s, Scratch& sc) {
  const int64_t K = lb.K;
  const int P = lb.P;
  ScratchFrame frame(sc);
  int64_t* nb;
  VMO_TRY(sc.alloc(&nb, P));
  VMO_CUDA(cudaMemcpyAsync(nb, newbase.data(), P * sizeof(int64_t), cudaMemcpyHostToDevice, s));
  launch(k_pi, grid_for(K, kBlock), kBlock, 0, s, anchor, rank, K, lb.vprob.ptr, lb.prob.ptr, nb, pi);
  VMO_LAUNCHED("pi");
  const int64_t n = lb.nadj;
  uint64_t *keys, *skeys;
  uint32_t *vals, *svals;
  int32_t *flag, *pos, *total;
  VMO_TRY(sc.alloc(&keys, std::max<int64_t>(n, 1)));
  VMO_TRY(sc.alloc(&skeys, std::max<int64_t>(n, 1)));
  VMO_TRY(sc.alloc(&vals, std::max<int64_t>(n, 1)));
  VMO_TRY(sc.alloc(&svals, std::max<int64_t>(n, 1)));
  VMO_TRY(sc.alloc(&flag, std::max<int64_t>(n, 1)));
  VMO_TRY(sc.alloc(&pos, std::max<int64_t>(n, 1)));
  VMO_TRY(sc.alloc(&total, 1));
  const uint64_t sentinel = (uint64_t)Kc * (uint64_t)Kc;
  launch(k_contract_keys, grid_for(K, kBlock), kBlock, 0, s, lb.adj_ptr, lb.adj, lb.acost, K, pi, (uint64_t)Kc, keys, vals);
  if (lb.n_mid)
    launch(k_contract_keys_warp, grid_for(lb.n_mid * 32, kBlock), kBlock, 0, s, lb.mid_list.ptr, lb.n_mid, lb.adj_ptr,
           lb.adj, lb.acost, pi, (uint64_t)Kc, keys, vals);
  if (lb.n_heavy)
    launch(k_contract_keys_block, (unsigned)lb.n_heavy, kBlock, 0, s, lb.heavy_list.ptr, lb.adj_ptr, lb.adj, lb.acost,
           pi, (uint64_t)Kc, keys, vals);
  VMO_LAUNCHED("contract_keys");
  VMO_TRY(radix_sort_u64(keys, vals, skeys, svals, n, bits_for(sentinel), s, sc));
  if (n > 0) {
    launch(k_run_flags, grid_for(n, kBlock), kBlock, 0, s, skeys, n, sentinel, flag);
    VMO_LAUNCHED("run_flags");
  }
  VMO_TRY(scan_exclusive<int32_t>(flag, pos, n, total, s, sc));
  int32_t nadj_c = 0;
  VMO_CUDA(cudaMemcpyAsync(&nadj_c, total, 4, cudaMemcpyDeviceToHost, s));
  VMO_CUDA(cudaStreamSynchronize(s));
  VMO_TRY(out.own_adj_ptr.resize((size_t)Kc + 1));
  VMO_TRY(out.own_adj.resize(std::max<int32_t>(nadj_c, 1)));
  VMO_TRY(out.own_acost.resize(std::max<int32_t>(nadj_c, 1)));
  VMO_TRY(out.own_w.resize((size_t)std::max<int64_t>(Kc, 1)));
  double* wsum;
  VMO_TRY(sc.alloc(&wsum, std::max<int64_t>(Kc, 1)));
  VMO_CUDA(cudaMemsetAsync(out.own_adj_ptr.ptr, 0, (Kc + 1) * sizeof(int32_t), s));
  VMO_CUDA(cudaMemsetAsync(wsum, 0, std::max<int64_t>(Kc, 1) * sizeof(double), s));
  if (n > 0) {
    launch(k_emit_coarse, grid_for(n, kBlock), kBlock, 0, s, skeys, svals, n, flag, pos, (uint64_t)Kc, out.own_adj.ptr,
                                                         out.own_acost.ptr, out.own_adj_ptr.ptr);
    VMO_LAUNCHED("emit_coarse");
  }
  VMO_TRY(scan_exclusive<int32_t>(out.own_adj_ptr.ptr, out.own_adj_ptr.ptr, Kc, total, s, sc));
  launch(k_set_last, 1, 1, 0, s, out.own_adj_ptr.ptr, Kc, total);
  launch(k_coarse_w, grid_for(K, kBlock), kBlock, 0, s, lb.w, pi, K, wsum);
  if (Kc > 0) launch(k_round_w, grid_for(Kc, kBlock), kBlock, 0, s, wsum, Kc, out.own_w.ptr);
  VMO_LAUNCHED("coarse_w");
  out.K = Kc;
  out.adj_ptr = out.own_adj_ptr.ptr;
  out.adj = out.own_adj.ptr;
  out.acost = out.own_acost.ptr;
  out.w = out.own_w.ptr;
  out.nadj = nadj_c;
  return VMO_OK;
}

vmo_status build_hierarchy(LevelBatch& fine, const LayoutOptions& o, const std::vector<uint64_t>& seeds,
                           int match_rounds, int coarse_min, bool multilevel, Hierarchy& H, cudaStream_t s,
                           Scratch& sc) {
  std::vector<LevelBatch*>& levels = H.levels;
  std::vector<std::unique_ptr<LevelBatch>>& owned = H.owned;
  std::vector<int32_t*>& pis = H.pis;
  std::vector<std::vector<uint64_t>>& lseeds = H.seeds;
  levels.push_back(&fine);
  lseeds.push_back(seeds);
  const bool graph = fine.adj_ptr != nullptr;
  while (multilevel && graph && levels.size() < 41) {
    LevelBatch& cur = *levels.back();
    const int P = cur.P;
    std::vector<int32_t> active(P);
    bool any = false;
    for (int p = 0; p < P; ++p) {
      active[p] = (cur.vbase[p + 1] - cur.vbase[p]) > coarse_min ? 1 : 0;
      any = any || active[p];
    }
    if (!any) break;
    int32_t *act, *mate, *anchor, *rank, *pi;
    uint64_t* sd;
    VMO_TRY(sc.alloc(&act, P));
    VMO_TRY(sc.alloc(&sd, P));
    VMO_TRY(sc.alloc(&mate, cur.K));
    VMO_TRY(sc.alloc(&anchor, cur.K));
    VMO_TRY(sc.alloc(&rank, cur.K));
    VMO_TRY(sc.alloc(&pi, cur.K));
    VMO_CUDA(cudaMemcpyAsync(act, active.data(), P * 4, cudaMemcpyHostToDevice, s));
    VMO_CUDA(cudaMemcpyAsync(sd, lseeds.back().data(), P * 8, cudaMemcpyHostToDevice, s));
    std::vector<int64_t> kc;
    VMO_TRY(coarsen_level(cur, sd, (int)levels.size() - 1, match_rounds, act, mate, anchor, rank, kc, s, sc));
    std::vector<int64_t> newbase(P, -1);
    auto nxt = std::make_unique<LevelBatch>();
    nxt->vbase.push_back(0);
    std::vector<uint64_t> nseeds;
    for (int p = 0; p < P; ++p) {
      int64_t k = cur.vbase[p + 1] - cur.vbase[p];
      if (!active[p] || (double)kc[p] > 0.95 * (double)k) continue;
      newbase[p] = nxt->vbase.back();
      nxt->vbase.push_back(nxt->vbase.back() + kc[p]);
      nxt->src.push_back(cur.src[p]);
      nseeds.push_back(lseeds.back()[p]);
    }
    nxt->P = (int32_t)nxt->src.size();
    if (nxt->P == 0) break;
    int64_t Kc = nxt->vbase.back();
    VMO_TRY(contract_level(cur, newbase, Kc, anchor, rank, pi, *nxt, s, sc));
    VMO_TRY(level_setup(*nxt, o.d, o.occupancy, s));
    pis.push_back(pi);
    levels.push_back(nxt.get());
    lseeds.push_back(nseeds);
    owned.push_back(std::move(nxt));
  }
  return VMO_OK;
}

// Host tables of level j's start: which problems start here (not present one
// level up) and, for the others, the scale (k_f / k_c)^(1/d) of the
// prolongation.
static void prolong_tables(const Hierarchy& H, int j, int d, std::vector<int32_t>& start, std::vector<float>& fac) {
  const std::vector<LevelBatch*>& levels = H.levels;
  const int nl = (int)levels.size();
  const LevelBatch& cur = *levels[j];
  const int P = cur.P;
  start.assign(P, 1);
  fac.assign(P, -1.0f);
  if (j + 1 < nl) {
    const LevelBatch& up = *levels[j + 1];
    size_t q = 0;
    for (int p = 0; p < P && q < up.src.size(); ++p) {
      if (cur.src[p] == up.src[q]) {
        start[p] = 0;
        double kf = (double)(cur.vbase[p + 1] - cur.vbase[p]);
        double kcq = (double)(up.vbase[q + 1] - up.vbase[q]);
        fac[p] = (float)std::pow(kf / kcq, 1.0 / d);
        ++q;
      }
    }
  }
}

// Level j's start from device tables (start flags, scales, seeds of its
// problems): initial coordinates for the problems that start here, the
// prolongation of xc for the others.
static vmo_status prolong_level_dev(const Hierarchy& H, int j, int d, const float4* xc, float4* xj,
                                    const int32_t* st, const float* fc, const uint64_t* sd, cudaStream_t s) {
  LevelBatch& cur = *H.levels[j];
  VMO_TRY(init_coords_level(cur, d, sd, xj, st, s));
  if (xc && cur.K > 0) {
    launch(k_prolong, grid_for(cur.K, kBlock), kBlock, 0, s, xc, H.pis[j], cur.K, cur.vprob.ptr, cur.prob.ptr, fc, sd,
           j, d, xj);
    VMO_LAUNCHED("prolong");
  }
  return VMO_OK;
}

vmo_status prolong_level(const Hierarchy& H, int j, int d, const float4* xc, float4* xj, cudaStream_t s,
                         Scratch& sc) {
  const int P = H.levels[j]->P;
  std::vector<int32_t> start;
  std::vector<float> fac;
  prolong_tables(H, j, d, start, fac);
  int32_t* st;
  float* fc;
  uint64_t* sd;
  VMO_TRY(sc.alloc(&st, P));
  VMO_TRY(sc.alloc(&fc, P));
  VMO_TRY(sc.alloc(&sd, P));
  VMO_CUDA(cudaMemcpyAsync(st, start.data(), P * 4, cudaMemcpyHostToDevice, s));
  VMO_CUDA(cudaMemcpyAsync(fc, fac.data(), P * 4, cudaMemcpyHostToDevice, s));
  VMO_CUDA(cudaMemcpyAsync(sd, H.seeds[j].data(), P * 8, cudaMemcpyHostToDevice, s));
  VMO_TRY(prolong_level_dev(H, j, d, xc, xj, st, fc, sd, s));
  VMO_CUDA(cudaStreamSynchronize(s));  // host vectors above must outlive the copies
  return VMO_OK;
}

vmo_status layout_multilevel(LevelBatch& fine, const LayoutOptions& o, const std::vector<uint64_t>& seeds,
                             int match_rounds, int coarse_min, bool multilevel, float4* x, cudaStream_t s,
                             Scratch& sc) {
  Hierarchy H;
  VMO_TRY(build_hierarchy(fine, o, seeds, match_rounds, coarse_min, multilevel, H, s, sc));
  // the start tables of every level uploaded at once, so that the levels are
  // then queued without waiting for the device
  const int nl = (int)H.levels.size();
  std::vector<int64_t> tb(nl + 1, 0);
  for (int j = 0; j < nl; ++j) tb[j + 1] = tb[j] + H.levels[j]->P;
  std::vector<int32_t> start_all((size_t)tb[nl]);
  std::vector<float> fac_all((size_t)tb[nl]);
  std::vector<uint64_t> seed_all((size_t)tb[nl]);
  for (int j = 0; j < nl; ++j) {
    std::vector<int32_t> st;
    std::vector<float> fc;
    prolong_tables(H, j, o.d, st, fc);
    std::copy(st.begin(), st.end(), start_all.begin() + tb[j]);
    std::copy(fc.begin(), fc.end(), fac_all.begin() + tb[j]);
    std::copy(H.seeds[j].begin(), H.seeds[j].end(), seed_all.begin() + tb[j]);
  }
  int32_t* st_d;
  float* fc_d;
  uint64_t* sd_d;
  VMO_TRY(sc.alloc(&st_d, std::max<int64_t>(tb[nl], 1)));
  VMO_TRY(sc.alloc(&fc_d, std::max<int64_t>(tb[nl], 1)));
  VMO_TRY(sc.alloc(&sd_d, std::max<int64_t>(tb[nl], 1)));
  VMO_CUDA(cudaMemcpyAsync(st_d, start_all.data(), tb[nl] * 4, cudaMemcpyHostToDevice, s));
  VMO_CUDA(cudaMemcpyAsync(fc_d, fac_all.data(), tb[nl] * 4, cudaMemcpyHostToDevice, s));
  VMO_CUDA(cudaMemcpyAsync(sd_d, seed_all.data(), tb[nl] * 8, cudaMemcpyHostToDevice, s));
  VMO_CUDA(cudaStreamSynchronize(s));  // the host tables must outlive the copies
  // layout from the coarsest level down
  auto ctx = std::make_shared<LayoutContext>();
  sc.held.push_back(ctx);
  if (o.iters > 0) VMO_TRY(make_scale_tab(o, o.iters, &ctx->scale_tab, s, sc));
  float4* xc = nullptr;
  for (int j = nl - 1; j >= 0; --j) {
    LevelBatch& cur = *H.levels[j];
    float4* xj = (j == 0) ? x : nullptr;
    if (!xj) VMO_TRY(sc.alloc(&xj, std::max<int64_t>(cur.K, 1)));
    VMO_TRY(prolong_level_dev(H, j, o.d, xc, xj, st_d + tb[j], fc_d + tb[j], sd_d + tb[j], s));
    VMO_TRY(layout_level(cur, o, xj, o.iters, -1.0f, nullptr, nullptr, ctx.get(), s, sc));
    xc = xj;
  }
  ctx->destroy_all_but(1);
  return VMO_OK;
}

}  // namespace vmo
