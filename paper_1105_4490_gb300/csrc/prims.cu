// Device-wide primitives: scans and a stable LSD radix sort.
//
// Scan: reduce tiles -> scan each tile with its offset (tiles of 2048 elements
// staged through shared memory so global loads and stores are coalesced).  A
// tile adds up the sums of the tiles before it itself, up to kScanSelfTiles of
// them (a launch less, 2.5 us of the 12 of a small scan); above, one block scans the
// sums in a launch between the two.
//
// Radix sort: 8-bit digits, one histogram kernel and one scatter kernel per
// pass plus a scan of the (digit, tile)-ordered histogram.  The scatter ranks
// keys stably inside a warp with __match_any_sync, so equal keys keep their
// input order.
#include <algorithm>

#include <type_traits>

#include "blocksort.cuh"

namespace vmo {

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

template <class T>
__global__ void scan_reduce_kernel(const T* __restrict__ in, int64_t n, T* __restrict__ partial) {
  __shared__ T ws[33];
  pdl_enter();
  int64_t base = (int64_t)blockIdx.x * kScanTile;
  T acc = 0;
  for (int i = threadIdx.x; i < kScanTile; i += kScanThreads) {
    int64_t g = base + i;
    if (g < n) acc += in[g];
  }
  T tot;
  block_exclusive<T>(acc, ws, &tot);
  if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

template <class T>
__global__ void scan_partials_kernel(T* partial, int64_t ntiles, T* total) {
  __shared__ T ws[33];
  pdl_enter();
  T carry = 0;
  for (int64_t b = 0; b < ntiles; b += blockDim.x) {
    int64_t i = b + threadIdx.x;
    T v = (i < ntiles) ? partial[i] : T(0);
    T tot;
    T ex = block_exclusive<T>(v, ws, &tot);
    if (i < ntiles) partial[i] = ex + carry;
    carry += tot;
  }
  if (threadIdx.x == 0 && total) *total = carry;
}

constexpr int64_t kScanSelfTiles = 4096;

// SELF: partial holds the tiles' sums (the last tile writes the total), else
// their exclusive prefixes.
template <class T, bool Inclusive, bool SELF>
__global__ void scan_tile_kernel(const T* __restrict__ in, T* __restrict__ out, int64_t n,
                                 const T* __restrict__ partial, T* __restrict__ total) {
  __shared__ T tile[kScanTile];
  __shared__ T ws[33];
  pdl_enter();
  int64_t base = (int64_t)blockIdx.x * kScanTile;
  for (int i = threadIdx.x; i < kScanTile; i += kScanThreads) {
    int64_t g = base + i;
    tile[i] = (g < n) ? in[g] : T(0);
  }
  __syncthreads();
  T loc[kScanItems];
  T acc = 0;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    loc[j] = tile[threadIdx.x * kScanItems + j];
    acc += loc[j];
  }
  T before = SELF ? T(0) : partial[blockIdx.x];
  if (SELF) {
    T part = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += kScanThreads) part += partial[b];
    block_exclusive<T>(part, ws, &before);
  }
  T sum;
  T ex = block_exclusive<T>(acc, ws, &sum) + before;
  if (SELF && total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total = before + sum;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    T v = loc[j];
    tile[threadIdx.x * kScanItems + j] = Inclusive ? ex + v : ex;
    ex += v;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kScanTile; i += kScanThreads) {
    int64_t g = base + i;
    if (g < n) out[g] = tile[i];
  }
}

template <class T, bool Inclusive>
void scan_launch(const T* in, T* out, int64_t n, int64_t ntiles, T* partial, T* total, cudaStream_t s) {
  launch(scan_reduce_kernel<T>, (unsigned)ntiles, kScanThreads, 0, s, in, n, partial);
  if (ntiles <= kScanSelfTiles) {
    launch(scan_tile_kernel<T, Inclusive, true>, (unsigned)ntiles, kScanThreads, 0, s, in, out, n, partial, total);
  } else {
    launch(scan_partials_kernel<T>, 1, 1024, 0, s, partial, ntiles, total);
    launch(scan_tile_kernel<T, Inclusive, false>, (unsigned)ntiles, kScanThreads, 0, s, in, out, n, partial,
           (T*)nullptr);
  }
}

template <class T, bool Inclusive>
vmo_status scan_impl(const T* in, T* out, int64_t n, T* total, cudaStream_t s, Scratch& sc) {
  if (n <= 0) {
    if (total) VMO_CUDA(cudaMemsetAsync(total, 0, sizeof(T), s));
    return VMO_OK;
  }
  int64_t ntiles = (n + kScanTile - 1) / kScanTile;
  T* partial;
  VMO_TRY(sc.alloc(&partial, (size_t)ntiles));
  scan_launch<T, Inclusive>(in, out, n, ntiles, partial, total, s);
  VMO_LAUNCHED("scan");
  return VMO_OK;
}

// ------------------------------- radix sort --------------------------------
// LSD passes of B-bit digits, B in {6, 8, 9, 10} chosen per sort: the fewest
// passes of at most 10 bits (or the tuned cap, 8 or 9), then the smallest
// listed width covering the key bits in that many passes (18-bit cell keys:
// 2 passes of 9 bits).
constexpr int kMaxRadixBits = 10;

template <class K, int BITS>
__global__ void radix_hist_kernel(const K* __restrict__ keys, int64_t n, int shift, uint32_t* __restrict__ hist) {
  constexpr int R = 1 << BITS;
  __shared__ uint32_t h[R];
  for (int i = threadIdx.x; i < R; i += blockDim.x) h[i] = 0;
  __syncthreads();
  const int64_t start = (int64_t)blockIdx.x * kSortTile;
  const int count = (int)min((int64_t)kSortTile, n - start);
  for (int i = threadIdx.x; i < count; i += blockDim.x) {
    uint32_t dg = (uint32_t)(keys[start + i] >> shift) & (R - 1);
    atomicAdd(&h[dg], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < R; i += blockDim.x) hist[(int64_t)i * gridDim.x + blockIdx.x] = h[i];
}

// Row prefix of the tile histograms: one warp per digit (its counts in the nt
// tiles, contiguous): exclusive prefix in place, row total to rowtot.
__global__ void radix_rowscan(uint32_t* __restrict__ hist, int64_t nt, int R, uint32_t* __restrict__ rowtot) {
  const int64_t d = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (d >= R) return;
  const int lane = lane_id();
  uint32_t* row = hist + d * nt;
  uint32_t carry = 0;
  for (int64_t b = 0; b < nt; b += 32) {
    const int64_t t = b + lane;
    const uint32_t c = t < nt ? row[t] : 0u;
    const uint32_t inc = warp_inclusive(c);
    if (t < nt) row[t] = carry + inc - c;
    carry += __shfl_sync(0xffffffffu, inc, 31);
  }
  if (lane == 0) rowtot[d] = carry;
}

template <class K, bool HasVal, int BITS>
__global__ void __launch_bounds__(kSortThreads) radix_scatter_kernel(
    const K* __restrict__ keys, const uint32_t* __restrict__ vals, K* __restrict__ keys_out,
    uint32_t* __restrict__ vals_out, int64_t n, int shift, const uint32_t* __restrict__ offs,
    const uint32_t* __restrict__ rowtot) {
  constexpr int R = 1 << BITS;
  constexpr int PER = (R + kSortThreads - 1) / kSortThreads;
  // the per-warp digit counts, then (once every element knows its place) the
  // tile's keys and values in digit order, so that the writes of a digit's
  // run go out as consecutive addresses
  constexpr int kCountBytes = kSortWarps * R * 4;
  constexpr int kStageBytes = kSortTile * ((int)sizeof(K) + (HasVal ? 4 : 0));
  __shared__ __align__(16) unsigned char raw[kCountBytes > kStageBytes ? kCountBytes : kStageBytes];
  uint32_t(*wcnt)[R] = reinterpret_cast<uint32_t(*)[R]>(raw);
  K* skey = reinterpret_cast<K*>(raw);
  uint32_t* sval = reinterpret_cast<uint32_t*>(raw + kSortTile * sizeof(K));
  __shared__ uint32_t tbase[R];
  __shared__ uint32_t lbase[R];  // the tile's exclusive digit offsets
  __shared__ uint32_t ws[33];
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kSortWarps * R; i += blockDim.x) (&wcnt[0][0])[i] = 0;
  const int64_t start = (int64_t)blockIdx.x * kSortTile;
  const int count = (int)min((int64_t)kSortTile, n - start);
  const bool single = gridDim.x == 1;  // one tile: bases from its own counts
  // destination of digit d in this tile: keys with a smaller digit (scan of
  // the row totals) + keys of digit d in the earlier tiles (row prefix)
  if (!single) {
    uint32_t v[PER];
    uint32_t sum = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int d = threadIdx.x * PER + j;
      v[j] = d < R ? rowtot[d] : 0u;
      sum += v[j];
    }
    uint32_t ex = block_exclusive<uint32_t>(sum, ws, nullptr);
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int d = threadIdx.x * PER + j;
      if (d < R) tbase[d] = ex + offs[(int64_t)d * gridDim.x + blockIdx.x];
      ex += v[j];
    }
  }
  __syncthreads();
  K key[kSortItems];
  uint32_t val[kSortItems];
  uint32_t rank[kSortItems];
  uint32_t dig[kSortItems];
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int j = 0; j < kSortItems; ++j) {
    int idx = warp * (32 * kSortItems) + j * 32 + lane;
    bool valid = idx < count;
    key[j] = valid ? keys[start + idx] : K(0);
    if (HasVal) val[j] = valid ? vals[start + idx] : 0u;
    uint32_t dg = valid ? ((uint32_t)(key[j] >> shift) & (R - 1)) : (uint32_t)R;
    dig[j] = dg;
    unsigned peers = __match_any_sync(0xffffffffu, dg);
    uint32_t before = __popc(peers & lt);
    uint32_t base = valid ? wcnt[warp][dg] : 0u;
    rank[j] = base + before;
    __syncwarp();
    if (valid && lane == __ffs(peers) - 1) wcnt[warp][dg] = base + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  for (int dg = threadIdx.x; dg < R; dg += blockDim.x) {
    uint32_t run = 0;
    for (int w = 0; w < kSortWarps; ++w) {
      uint32_t c = wcnt[w][dg];
      wcnt[w][dg] = run;
      run += c;
    }
    lbase[dg] = run;  // the tile's count of digit dg
  }
  __syncthreads();
  {  // exclusive scan of the tile's digit counts
    uint32_t v[PER];
    uint32_t sum = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int d = threadIdx.x * PER + j;
      v[j] = d < R ? lbase[d] : 0u;
      sum += v[j];
    }
    uint32_t ex = block_exclusive<uint32_t>(sum, ws, nullptr);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int d = threadIdx.x * PER + j;
      if (d < R) {
        lbase[d] = ex;
        if (single) tbase[d] = ex;
      }
      ex += v[j];
    }
  }
  __syncthreads();
  // place of every element in the tile's digit order (stable: within a digit,
  // by warp, then item, then lane, i.e. input order)
  uint32_t lpos[kSortItems];
#pragma unroll
  for (int j = 0; j < kSortItems; ++j)
    lpos[j] = dig[j] < (uint32_t)R ? lbase[dig[j]] + wcnt[warp][dig[j]] + rank[j] : 0u;
  __syncthreads();  // wcnt is overwritten by the staged tile from here on
#pragma unroll
  for (int j = 0; j < kSortItems; ++j) {
    if (dig[j] >= (uint32_t)R) continue;
    skey[lpos[j]] = key[j];
    if (HasVal) sval[lpos[j]] = val[j];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < count; e += blockDim.x) {
    const K k = skey[e];
    const uint32_t d = (uint32_t)(k >> shift) & (R - 1);
    const uint32_t dst = tbase[d] + ((uint32_t)e - lbase[d]);
    keys_out[dst] = k;
    if (HasVal) vals_out[dst] = sval[e];
  }
}

// Whole sort of at most one tile (2,048 keys), all passes of 8-bit digits in
// shared memory, by one block (one launch instead of three per pass).  Ranks
// within a digit follow the input order exactly as in radix_scatter_kernel.
__global__ void __launch_bounds__(kSortThreads) radix_tile_sort_kernel(const uint32_t* __restrict__ keys,
                                                                       const uint32_t* __restrict__ vals,
                                                                       uint32_t* __restrict__ keys_out,
                                                                       uint32_t* __restrict__ vals_out, int n,
                                                                       int bits) {
  __shared__ TileSortSmem sm;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    sm.key[0][i] = keys[i];
    sm.val[0][i] = vals[i];
  }
  const int cur = tile_sort_smem(sm, n, bits);
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    keys_out[i] = sm.key[cur][i];
    vals_out[i] = sm.val[cur][i];
  }
}

inline int digit_bits(int bits, int* passes) {
  const int maxb = std::min(kMaxRadixBits, std::max(8, g_tuning.radix_max_bits.load(std::memory_order_relaxed)));
  const int p = (bits + maxb - 1) / maxb;
  const int need = (bits + p - 1) / p;
  *passes = p;
  return need <= 6 ? 6 : need <= 8 ? 8 : need <= 9 ? 9 : 10;
}

template <class K, int BITS>
void radix_pass(const K* ka, const uint32_t* va, K* kb, uint32_t* vb, int64_t n, int shift, int64_t ntiles,
                uint32_t* hist, uint32_t* rowtot, cudaStream_t s) {
  constexpr int R = 1 << BITS;
  launch(radix_hist_kernel<K, BITS>, (unsigned)ntiles, 256, 0, s, ka, n, shift, hist);
  if (ntiles > 1) launch(radix_rowscan, (unsigned)((R * 32 + 255) / 256), 256, 0, s, hist, ntiles, R, rowtot);
  if (va)
    launch(radix_scatter_kernel<K, true, BITS>, (unsigned)ntiles, kSortThreads, 0, s, ka, va, kb, vb, n, shift, hist,
           rowtot);
  else
    launch(radix_scatter_kernel<K, false, BITS>, (unsigned)ntiles, kSortThreads, 0, s, ka, nullptr, kb, nullptr, n,
           shift, hist, rowtot);
}

template <class K>
vmo_status radix_sort_impl(K* keys_in, uint32_t* vals_in, K* keys_out, uint32_t* vals_out, int64_t n, int bits,
                           cudaStream_t s, Scratch& sc) {
  if (n <= 0) return VMO_OK;
  const int64_t ntiles = (n + kSortTile - 1) / kSortTile;
  int passes = 0;
  const int B = bits > 0 ? digit_bits(bits, &passes) : 8;
  if (passes == 0) {
    VMO_CUDA(cudaMemcpyAsync(keys_out, keys_in, n * sizeof(K), cudaMemcpyDeviceToDevice, s));
    if (vals_in) VMO_CUDA(cudaMemcpyAsync(vals_out, vals_in, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
    return VMO_OK;
  }
  if constexpr (std::is_same<K, uint32_t>::value) {
    if (ntiles == 1 && vals_in && bits <= 32) {
      launch(radix_tile_sort_kernel, 1, kSortThreads, 0, s, keys_in, vals_in, keys_out, vals_out, (int)n, bits);
      VMO_LAUNCHED("radix_tile_sort");
      return VMO_OK;
    }
  }
  uint32_t *hist, *rowtot;
  VMO_TRY(sc.alloc(&hist, (size_t)(ntiles << B)));
  VMO_TRY(sc.alloc(&rowtot, (size_t)1 << B));
  K* ka = keys_in;
  K* kb = keys_out;
  uint32_t* va = vals_in;
  uint32_t* vb = vals_out;
  for (int p = 0; p < passes; ++p) {
    const int shift = p * B;
    switch (B) {
      case 6: radix_pass<K, 6>(ka, va, kb, vb, n, shift, ntiles, hist, rowtot, s); break;
      case 8: radix_pass<K, 8>(ka, va, kb, vb, n, shift, ntiles, hist, rowtot, s); break;
      case 9: radix_pass<K, 9>(ka, va, kb, vb, n, shift, ntiles, hist, rowtot, s); break;
      default: radix_pass<K, 10>(ka, va, kb, vb, n, shift, ntiles, hist, rowtot, s); break;
    }
    VMO_LAUNCHED("radix_sort");
    K* tk = ka; ka = kb; kb = tk;
    uint32_t* tv = va; va = vb; vb = tv;
  }
  if (ka != keys_out) {
    VMO_CUDA(cudaMemcpyAsync(keys_out, ka, n * sizeof(K), cudaMemcpyDeviceToDevice, s));
    if (vals_in) VMO_CUDA(cudaMemcpyAsync(vals_out, va, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
  }
  return VMO_OK;
}

}  // namespace

template <class T>
vmo_status scan_exclusive(const T* in, T* out, int64_t n, T* total, cudaStream_t s, Scratch& sc) {
  return scan_impl<T, false>(in, out, n, total, s, sc);
}
template <class T>
vmo_status scan_inclusive(const T* in, T* out, int64_t n, cudaStream_t s, Scratch& sc) {
  return scan_impl<T, true>(in, out, n, nullptr, s, sc);
}

template vmo_status scan_exclusive<int32_t>(const int32_t*, int32_t*, int64_t, int32_t*, cudaStream_t, Scratch&);
template vmo_status scan_exclusive<int64_t>(const int64_t*, int64_t*, int64_t, int64_t*, cudaStream_t, Scratch&);
template vmo_status scan_exclusive<uint32_t>(const uint32_t*, uint32_t*, int64_t, uint32_t*, cudaStream_t,
                                             Scratch&);
template vmo_status scan_exclusive<uint64_t>(const uint64_t*, uint64_t*, int64_t, uint64_t*, cudaStream_t,
                                             Scratch&);
template vmo_status scan_inclusive<uint64_t>(const uint64_t*, uint64_t*, int64_t, cudaStream_t, Scratch&);
template vmo_status scan_inclusive<int32_t>(const int32_t*, int32_t*, int64_t, cudaStream_t, Scratch&);
template vmo_status scan_inclusive<int64_t>(const int64_t*, int64_t*, int64_t, cudaStream_t, Scratch&);

vmo_status scan_inclusive_u64_into(const uint64_t* in, uint64_t* out, int64_t n, uint64_t* partial, cudaStream_t s) {
  if (n <= 0) return VMO_OK;
  int64_t ntiles = (n + kScanTile - 1) / kScanTile;
  scan_launch<uint64_t, true>(in, out, n, ntiles, partial, (uint64_t*)nullptr, s);
  VMO_LAUNCHED("scan");
  return VMO_OK;
}

int64_t scan_partials_needed(int64_t n) { return (n + kScanTile - 1) / kScanTile; }

vmo_status radix_sort_u32(uint32_t* keys_in, uint32_t* vals_in, uint32_t* keys_out, uint32_t* vals_out, int64_t n,
                          int bits, cudaStream_t s, Scratch& sc) {
  return radix_sort_impl<uint32_t>(keys_in, vals_in, keys_out, vals_out, n, bits, s, sc);
}

vmo_status radix_sort_u64(uint64_t* keys_in, uint32_t* vals_in, uint64_t* keys_out, uint32_t* vals_out, int64_t n,
                          int bits, cudaStream_t s, Scratch& sc) {
  return radix_sort_impl<uint64_t>(keys_in, vals_in, keys_out, vals_out, n, bits, s, sc);
}

}  // namespace vmo
