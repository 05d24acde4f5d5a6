// m-way k-means++ (Algorithm 5 with m centres): a one-shot m-way partition of
// a point set, in the readings of the recursion's 2-means (integer D^2
// weights on the grid 2^-(34-2e), draws keyed by (seed, key, centre index),
// fp32 distances without FMA, ties to the smaller centre, exact fixed-point
// means on the grid 2^-(30-e)); for m = 2 it is vmo_bisect.
//
// Seeding takes m - 1 rounds of (running minimum distance and block sums of
// the weights, pick); a Lloyd round is one assignment kernel (centres in shared
// memory, per-block fixed-point sums in shared memory folded into global int64
// sums with atomics, exact and order-free) and one update kernel.
#include <algorithm>

#include "blocksort.cuh"
#include "vmo_internal.cuh"

namespace vmo {

vmo_status ensure_device_public();

namespace {

constexpr int kKmBlock = 256;
constexpr int kKmMaxCentres = 256;
constexpr int kKmPickBlock = 1024;

struct KmState {
  int e;             // max |x| < 2^e
  int chosen;        // centres picked by the seeding
  int stopped;       // seeding stopped: every point on a chosen centre
  int converged;     // no label changed in a Lloyd round
  int changed;       // a label changed in the current round
  uint32_t maxabs;   // float bits of max |x|
};

template <int D>
__global__ void k_km_gather(const float4* __restrict__ x, const int32_t* __restrict__ verts, int64_t n,
                            float4* __restrict__ xo, KmState* __restrict__ st) {
  pdl_enter();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t mx = 0;
  if (i < n) {
    const float4 p = x[verts[i]];
    xo[i] = p;
#pragma unroll
    for (int m = 0; m < D; ++m) mx = max(mx, __float_as_uint(fabsf(comp(p, m))));
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane_id() == 0 && mx) atomicMax(&st->maxabs, mx);
}

// First centre: point floor(n * r0 / 2^64).
__global__ void k_km_seed0(const float4* __restrict__ xo, int64_t n, uint64_t seed, uint64_t key,
                           float4* __restrict__ z, KmState* __restrict__ st) {
  pdl_enter();
  st->e = exponent_of(st->maxabs);
  st->chosen = 1;
  st->stopped = 0;
  st->converged = 0;
  st->changed = 0;
  z[0] = xo[scale_draw((uint64_t)n, rand64(seed ^ kTagKmeans, key, 0))];
}

// Seeding of centre c, two launches.  First the running minimum squared
// distance to the chosen centres (centre c - 1 just picked) and the block's
// sum of the integer D^2 weights floor(dmin * 2^(34 - 2e)); then the first
// point whose inclusive prefix of the weights exceeds floor(total * r_c /
// 2^64) is found from the block sums and, in the one block that holds it, from the
// weights computed again (a zero total stops the seeding).  The weights and their
// prefixes are never stored: as five launches with 40 bytes a point a centre
// took 25 us of a million points, bound by launches and traffic alike.
constexpr int kKmItems = 8;                        // points per thread
constexpr int kKmTile = kKmBlock * kKmItems;       // points per block
static_assert(kKmBlock == 256, "eight warps");

__device__ __forceinline__ unsigned long long km_weight(float dm, int e) {
  return (unsigned long long)floorf(__fmul_rn(dm, exp2i_f(34 - 2 * e)));
}

template <int D>
__global__ void __launch_bounds__(kKmBlock) k_km_weights(const float4* __restrict__ xo, int64_t n,
                                                         const float4* __restrict__ z, int c, float* __restrict__ dmin,
                                                         unsigned long long* __restrict__ bsum,
                                                         const KmState* __restrict__ st) {
  __shared__ unsigned long long red[kKmBlock / 32];
  pdl_enter();
  if (st->stopped) return;  // grid-uniform
  const int e = st->e;
  const float4 zc = z[c - 1];
  const int64_t i0 = (int64_t)blockIdx.x * kKmTile + threadIdx.x;
  float4 p[kKmItems];
  float old[kKmItems];
#pragma unroll
  for (int u = 0; u < kKmItems; ++u) {  // every load in flight together
    const int64_t i = i0 + u * kKmBlock;
    p[u] = i < n ? xo[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    old[u] = i < n && c > 1 ? dmin[i] : 0.f;
  }
  unsigned long long w = 0;
#pragma unroll
  for (int u = 0; u < kKmItems; ++u) {
    const int64_t i = i0 + u * kKmBlock;
    if (i >= n) break;
    const float dd = sqdist32<D>(p[u], zc);
    const float dm = c == 1 ? dd : fminf(old[u], dd);
    dmin[i] = dm;
    w += km_weight(dm, e);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
  if (lane_id() == 0) red[threadIdx.x >> 5] = w;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long sum = 0;
    for (int q = 0; q < kKmBlock / 32; ++q) sum += red[q];
    bsum[blockIdx.x] = sum;
  }
}

// One block: the block of points that holds the draw, then the point in it.
__global__ void __launch_bounds__(kKmPickBlock) k_km_pick(const float4* __restrict__ xo, int64_t n,
                                                          const float* __restrict__ dmin,
                                                          const unsigned long long* __restrict__ bsum, int nb,
                                                          uint64_t seed, uint64_t key, int c, float4* __restrict__ z,
                                                          KmState* __restrict__ st) {
  __shared__ unsigned long long ws[33];
  __shared__ unsigned long long s_before;
  __shared__ int s_block;
  pdl_enter();
  if (st->stopped) return;
  // block sums: contiguous parts of the threads, prefixes by a block scan
  const int per = (nb + kKmPickBlock - 1) / kKmPickBlock;
  const int a = min((int)threadIdx.x * per, nb), b = min(a + per, nb);
  unsigned long long sum = 0;
  for (int q = a; q < b; ++q) sum += bsum[q];
  unsigned long long total;
  const unsigned long long ex = block_exclusive<unsigned long long>(sum, ws, &total);
  if (total == 0) {
    if (threadIdx.x == 0) st->stopped = 1;
    return;
  }
  const unsigned long long thr = scale_draw(total, rand64(seed ^ kTagKmeans, key, (uint64_t)c));
  if (threadIdx.x == 0) s_block = -1;
  __syncthreads();
  if (thr >= ex && thr - ex < sum) {
    unsigned long long run = ex;
    for (int q = a; q < b; ++q) {
      const unsigned long long w = bsum[q];
      if (thr - run < w) {
        s_block = q;
        s_before = run;
        break;
      }
      run += w;
    }
  }
  __syncthreads();
  if (s_block < 0) return;
  const int e = st->e;
  const int64_t base = (int64_t)s_block * kKmTile;
  constexpr int kPer = kKmTile / kKmPickBlock;
  unsigned long long w[kPer], own = 0;
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    const int64_t i = base + threadIdx.x * kPer + u;
    w[u] = i < n ? km_weight(dmin[i], e) : 0ull;
    own += w[u];
  }
  unsigned long long run = s_before + block_exclusive<unsigned long long>(own, ws, nullptr);
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    if (run <= thr && thr < run + w[u]) {
      z[c] = xo[base + threadIdx.x * kPer + u];
      st->chosen = c + 1;
    }
    run += w[u];
  }
}

// Centres the seeding did not reach are copies of the first (they never win).
__global__ void k_km_fill(float4* __restrict__ z, int m, const KmState* __restrict__ st) {
  pdl_enter();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < m && c >= st->chosen) z[c] = z[0];
}

// One Lloyd assignment (it >= 0) or the final labelling (it < 0).  Each thread
// takes kKmAssign points at a time, so that a centre read from shared memory serves
// all of them, and a block walks over tiles of the points and keeps the
// clusters' sums in shared memory until its end.  The fixed-point values are
// added as two 32-bit words (their low 16 bits and the rest): shared memory has
// native 32-bit additions but adds 64 bits by a compare-and-swap loop, which took most
// of the 150 us a round of a million points and 64 centres (now 35); a flush into
// 64-bit sums after kKmFlush points keeps the words from overflowing.
constexpr int kKmAssign = 4;
constexpr int kKmFlush = 8192;  // points of a block between flushes: 8192 (2^16 + 2^14) < 2^31

template <int D>
__global__ void __launch_bounds__(kKmBlock) k_km_assign(const float4* __restrict__ xo, int64_t n, int m, int it,
                                                        const float4* __restrict__ z, int32_t* __restrict__ lab,
                                                        unsigned long long* __restrict__ S,
                                                        unsigned long long* __restrict__ cnt,
                                                        KmState* __restrict__ st) {
  __shared__ float4 zs[kKmMaxCentres];
  __shared__ unsigned lo[kKmMaxCentres * D];
  __shared__ int hi[kKmMaxCentres * D];
  __shared__ int sc[kKmMaxCentres];
  const bool final_pass = it < 0;
  pdl_enter();
  if (!final_pass && st->converged) return;  // block-uniform
  for (int j = threadIdx.x; j < m; j += blockDim.x) {
    zs[j] = z[j];
    sc[j] = 0;
#pragma unroll
    for (int q = 0; q < D; ++q) {
      lo[j * D + q] = 0u;
      hi[j * D + q] = 0;
    }
  }
  __syncthreads();
  const float fx = exp2i_f(30 - st->e);
  bool changed = false;
  auto flush = [&]() {
    __syncthreads();
    for (int j = threadIdx.x; j < m; j += blockDim.x) {
      if (sc[j] == 0) continue;
      atomicAdd(&cnt[j], (unsigned long long)sc[j]);
      sc[j] = 0;
      if (final_pass) continue;
#pragma unroll
      for (int q = 0; q < D; ++q) {
        atomicAdd(&S[j * 4 + q], (unsigned long long)(((long long)hi[j * D + q] << 16) + (long long)lo[j * D + q]));
        lo[j * D + q] = 0u;
        hi[j * D + q] = 0;
      }
    }
    __syncthreads();
  };
  int held = 0;  // points since the last flush
  constexpr int kTile = kKmBlock * kKmAssign;
  for (int64_t base = (int64_t)blockIdx.x * kTile; base < n; base += (int64_t)gridDim.x * kTile) {
    if (held + kTile > kKmFlush) {
      flush();
      held = 0;
    }
    held += kTile;
    float4 p[kKmAssign];
    float bd[kKmAssign];
    int best[kKmAssign];
    const int64_t i0 = base + threadIdx.x;
#pragma unroll
    for (int u = 0; u < kKmAssign; ++u) {
      const int64_t i = i0 + u * kKmBlock;
      p[u] = i < n ? xo[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      bd[u] = sqdist32<D>(p[u], zs[0]);
      best[u] = 0;
    }
    for (int j = 1; j < m; ++j) {
      const float4 c = zs[j];
#pragma unroll
      for (int u = 0; u < kKmAssign; ++u) {
        const float dj = sqdist32<D>(p[u], c);
        if (dj < bd[u]) {
          bd[u] = dj;
          best[u] = j;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kKmAssign; ++u) {
      const int64_t i = i0 + u * kKmBlock;
      if (i >= n) continue;
      const int l = best[u];
      if (!final_pass && it > 0 && lab[i] != l) changed = true;
      lab[i] = l;
      atomicAdd(&sc[l], 1);
      if (final_pass) continue;
#pragma unroll
      for (int q = 0; q < D; ++q) {  // |value| < 2^30
        const int v = __float2int_rn(__fmul_rn(comp(p[u], q), fx));
        atomicAdd(&lo[l * D + q], (unsigned)v & 0xffffu);
        atomicAdd(&hi[l * D + q], v >> 16);
      }
    }
  }
  flush();
  if (changed) st->changed = 1;
}

// Centre update: z = fp32((double(sum) / count) * 2^-(30 - e)) for non-empty
// clusters; a round without a change ends the iteration.
template <int D>
__global__ void k_km_update(float4* __restrict__ z, int m, int it, unsigned long long* __restrict__ S,
                            unsigned long long* __restrict__ cnt, KmState* __restrict__ st) {
  const int j = threadIdx.x;  // one block of at least m threads
  pdl_enter();
  const bool done = st->converged || (it > 0 && !st->changed);
  __syncthreads();
  if (j < m) {
    if (!done && cnt[j] > 0) {
      const double inv = __longlong_as_double((long long)(1023 - (30 - st->e)) << 52);  // 2^-P
      float c[4] = {z[j].x, z[j].y, z[j].z, z[j].w};
#pragma unroll
      for (int q = 0; q < D; ++q)
        c[q] = __double2float_rn(__dmul_rn(__ddiv_rn(__ll2double_rn((long long)S[j * 4 + q]), (double)cnt[j]), inv));
      z[j] = make_float4(c[0], c[1], c[2], c[3]);
    }
    cnt[j] = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) S[j * 4 + q] = 0;
  }
  __syncthreads();
  if (j == 0) {
    if (done) st->converged = 1;
    st->changed = 0;
  }
}

__global__ void k_km_nonempty(const unsigned long long* __restrict__ cnt, int m, int32_t* __restrict__ out) {
  pdl_enter();
  int c = 0;
  for (int j = 0; j < m; ++j) c += cnt[j] > 0;
  *out = c;
}

template <class F>
void km_dispatch(int d, F&& f) {
  if (d == 2) f(std::integral_constant<int, 2>());
  else if (d == 3) f(std::integral_constant<int, 3>());
  else f(std::integral_constant<int, 4>());
}

}  // namespace

vmo_status kmeans_m(int32_t d, const float* coords, const int32_t* verts, int32_t nverts, int32_t m, uint64_t seed,
                    uint64_t key, int32_t km_iters, int32_t* labels, float* centres, int32_t* nonempty,
                    cudaStream_t s) {
  if (d < 2 || d > 4) return unsupported("d must be 2, 3 or 4");
  if (m < 1 || m > kKmMaxCentres) return invalid("m must be in [1, 256]");
  if (nverts < 0 || km_iters < 0) return invalid("negative size");
  if (!centres || ((uintptr_t)centres & 15u)) return invalid("centres null or not 16-byte aligned");
  if (nverts > 0 && (!coords || !verts || !labels || ((uintptr_t)coords & 15u)))
    return invalid("null or unaligned argument");
  VMO_CUDA(cudaMemsetAsync(centres, 0, (size_t)m * sizeof(float4), s));
  if (nverts == 0) {
    if (nonempty) *nonempty = 0;
    return VMO_OK;
  }
  Scratch sc(s);
  const int64_t n = nverts;
  float4 *xo, *z = reinterpret_cast<float4*>(centres);
  float* dmin;
  unsigned long long *bsum, *S, *cnt;
  KmState* st;
  int32_t* ne;
  VMO_TRY(sc.alloc(&xo, n));
  VMO_TRY(sc.alloc(&dmin, n));
  const int nt = (int)((n + kKmTile - 1) / kKmTile);  // tiles of the seeding
  VMO_TRY(sc.alloc(&bsum, nt));
  VMO_TRY(sc.alloc(&S, (size_t)m * 4));
  VMO_TRY(sc.alloc(&cnt, (size_t)m));
  VMO_TRY(sc.alloc(&st, 1));
  VMO_TRY(sc.alloc(&ne, 1));
  VMO_CUDA(cudaMemsetAsync(st, 0, sizeof(KmState), s));
  VMO_CUDA(cudaMemsetAsync(S, 0, (size_t)m * 4 * sizeof(unsigned long long), s));
  VMO_CUDA(cudaMemsetAsync(cnt, 0, (size_t)m * sizeof(unsigned long long), s));
  const unsigned nb = (unsigned)((n + kKmBlock - 1) / kKmBlock);
  // assignment blocks: one wave, so that the clusters' sums leave a block once
  const unsigned na = (unsigned)std::min<int64_t>((n + kKmBlock * kKmAssign - 1) / (kKmBlock * kKmAssign), 152 * 6);
  vmo_status stt = VMO_OK;
  PdlScope pdl;  // every kernel below starts with pdl_enter()
  km_dispatch(d, [&](auto DC) {
    constexpr int D = decltype(DC)::value;
    launch(k_km_gather<D>, nb, kKmBlock, 0, s, reinterpret_cast<const float4*>(coords), verts, n, xo, st);
    launch(k_km_seed0, 1, 1, 0, s, xo, n, seed, key, z, st);
    for (int c = 1; c < m; ++c) {
      launch(k_km_weights<D>, (unsigned)nt, kKmBlock, 0, s, xo, n, z, c, dmin, bsum, st);
      launch(k_km_pick, 1, kKmPickBlock, 0, s, xo, n, dmin, bsum, nt, seed, key, c, z, st);
    }
    launch(k_km_fill, 1, kKmMaxCentres, 0, s, z, m, st);
    for (int it = 0; it < km_iters; ++it) {
      launch(k_km_assign<D>, na, kKmBlock, 0, s, xo, n, m, it, z, labels, S, cnt, st);
      launch(k_km_update<D>, 1, kKmMaxCentres, 0, s, z, m, it, S, cnt, st);
      if (it % 4 == 3 && it + 1 < km_iters) {  // stop early once converged
        KmState h;
        cudaError_t e = cudaMemcpyAsync(&h, st, sizeof(h), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) {
          stt = cuda_fail(e, "kmeans convergence check", __FILE__, __LINE__);
          break;
        }
        if (h.converged) break;
      }
    }
    if (stt != VMO_OK) return;
    launch(k_km_assign<D>, na, kKmBlock, 0, s, xo, n, m, -1, z, labels, S, cnt, st);
    launch(k_km_nonempty, 1, 1, 0, s, cnt, m, ne);
  });
  VMO_TRY(stt);
  VMO_LAUNCHED("kmeans");
  int32_t h = 0;
  VMO_CUDA(cudaMemcpyAsync(&h, ne, 4, cudaMemcpyDeviceToHost, s));
  VMO_CUDA(cudaStreamSynchronize(s));
  if (nonempty) *nonempty = h;
  return VMO_OK;
}

}  // namespace vmo

extern "C" vmo_status vmo_kmeans(int32_t d, const float* coords, const int32_t* verts, int32_t nverts, int32_t m,
                                 uint64_t seed, uint64_t key, int32_t km_iters, int32_t* labels, float* centres,
                                 int32_t* nonempty, void* stream) {
  VMO_TRY(vmo::ensure_device_public());
  return vmo::kmeans_m(d, coords, verts, nverts, m, seed, key, km_iters, labels, centres, nonempty,
                       (cudaStream_t)stream);
}
