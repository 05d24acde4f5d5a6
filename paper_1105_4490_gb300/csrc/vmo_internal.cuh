// Internal declarations of the VMO CUDA library (not part of the C-ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <memory>
#include <string>
#include <utility>
#include <vector>

#include "../../include/vmo.h"

namespace vmo {

// ---------------------------------------------------------------------------
// Errors: a failing call records a message for vmo_last_error() and returns a
// status; nothing throws across the C-ABI.
// ---------------------------------------------------------------------------
void set_error(const std::string& msg);

struct Status {
  vmo_status code = VMO_OK;
  bool ok() const { return code == VMO_OK; }
};

#define VMO_TRY(expr)                          \
  do {                                         \
    vmo_status _s = (expr);                    \
    if (_s != VMO_OK) return _s;               \
  } while (0)

vmo_status cuda_fail(cudaError_t e, const char* what, const char* file, int line);

#define VMO_CUDA(call)                                                   \
  do {                                                                   \
    cudaError_t _e = (call);                                             \
    if (_e != cudaSuccess) return ::vmo::cuda_fail(_e, #call, __FILE__, __LINE__); \
  } while (0)

// The thread's first error that has not been collected: of a refused launch, or
// one that a call found pending when it began.  A kernel of a sequence reads
// what the ones before it wrote, so launch() leaves out every launch behind it
// until launch_status() or cuda_fail() has collected it: kernels on unwritten
// tables would read out of range or loop on what they find there.  (A look at
// the runtime's own last error at every launch cost a step of 4,096 points 6 of
// its 203 us.)
extern thread_local cudaError_t g_refused;
inline void begin_launches() { g_refused = cudaPeekAtLastError(); }
inline cudaError_t launch_status() {
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = g_refused;
  g_refused = cudaSuccess;
  return e;
}

#define VMO_LAUNCHED(name)                                                     \
  do {                                                                         \
    cudaError_t _e = ::vmo::launch_status();                                   \
    if (_e != cudaSuccess) return ::vmo::cuda_fail(_e, name, __FILE__, __LINE__); \
  } while (0)

vmo_status invalid(const std::string& msg);
vmo_status unsupported(const std::string& msg);

// ---------------------------------------------------------------------------
// Device memory.  Scratch of one call is taken from the stream-ordered pool
// (cudaMallocAsync) and released on the same stream when the call ends.
// ---------------------------------------------------------------------------
struct Scratch {
  cudaStream_t stream = nullptr;
  std::vector<void*> ptrs;
  std::vector<std::shared_ptr<void>> held;  // what must outlive the call's queued work, destroyed first
  explicit Scratch(cudaStream_t s) : stream(s) {}
  ~Scratch();
  template <class T>
  vmo_status alloc(T** p, size_t count) {
    return alloc_bytes(reinterpret_cast<void**>(p), count * sizeof(T));
  }
  vmo_status alloc_bytes(void** p, size_t bytes);
  size_t mark() const { return ptrs.size(); }
  void release_to(size_t m);  // frees (stream-ordered) everything allocated after mark m
};

// Returns the scratch taken inside a scope to the pool when the scope ends.
struct ScratchFrame {
  Scratch& sc;
  size_t m;
  explicit ScratchFrame(Scratch& s) : sc(s), m(s.mark()) {}
  ~ScratchFrame() { sc.release_to(m); }
};

// Stream for the allocations of DevArray in the calling thread.  By default a
// DevArray uses cudaMalloc / cudaFree; inside a DevArrayStreamScope it takes
// its memory from the stream-ordered pool on the scope's stream and returns it
// on that stream, so threads working on different streams (the request
// server's slots) never wait for each other in an allocation or a free, and a
// layout's levels cost no device-wide wait each (a dozen arrays a level). A
// scope may name a pool: the arrays of handles and the large ones of a layout's
// levels come from one of their own each, which keeps at most kPoolKeep bytes of
// what was freed and returns the rest at the next synchronisation (a call's own
// end).  A level's small arrays stay in the default pool: with a second pool for
// them too a step of 4,096 points took 191 us instead of 182.
extern std::atomic<uint64_t> g_device_allocs;
enum PoolKind { kDefaultPool, kHandlePool, kLevelPool };
extern thread_local cudaStream_t g_devarray_stream;
extern thread_local bool g_devarray_async;
extern thread_local PoolKind g_devarray_pool;
constexpr uint64_t kPoolKeep = uint64_t(1) << 30;
constexpr size_t kLevelPoolMin = size_t(16) << 20;  // bytes of an array from which a level takes it there
cudaMemPool_t library_pool(PoolKind kind);  // of the current device; null if it cannot be made
uint64_t level_pool_peak(int device);       // most bytes of its level pool in use at once (0: none made)

struct DevArrayStreamScope {
  cudaStream_t prev_s;
  bool prev_a;
  PoolKind prev_p;
  explicit DevArrayStreamScope(cudaStream_t s, PoolKind pool = kDefaultPool)
      : prev_s(g_devarray_stream), prev_a(g_devarray_async), prev_p(g_devarray_pool) {
    g_devarray_stream = s;
    g_devarray_async = true;
    g_devarray_pool = pool;
  }
  ~DevArrayStreamScope() {
    g_devarray_stream = prev_s;
    g_devarray_async = prev_a;
    g_devarray_pool = prev_p;
  }
};

// Persistent device buffer owned by a handle.
template <class T>
struct DevArray {
  T* ptr = nullptr;
  size_t count = 0;
  bool async = false;            // allocated from the stream-ordered pool
  cudaStream_t astream = nullptr;
  vmo_status resize(size_t n);  // contents not preserved
  void release();
  ~DevArray() { release(); }
  DevArray() = default;
  DevArray(const DevArray&) = delete;
  DevArray& operator=(const DevArray&) = delete;
};

template <class T>
vmo_status DevArray<T>::resize(size_t n) {
  if (n <= count && ptr) return VMO_OK;
  release();
  if (n == 0) n = 1;
  const bool as = g_devarray_async;
  void** pp = reinterpret_cast<void**>(&ptr);
  const PoolKind kind = g_devarray_pool;
  const bool own = as && (kind == kHandlePool || (kind == kLevelPool && n * sizeof(T) >= kLevelPoolMin));
  cudaMemPool_t pool = own ? library_pool(kind) : nullptr;
  cudaError_t e = !as ? cudaMalloc(pp, n * sizeof(T))
                  : pool ? cudaMallocFromPoolAsync(pp, n * sizeof(T), pool, g_devarray_stream)
                         : cudaMallocAsync(pp, n * sizeof(T), g_devarray_stream);
  if (e != cudaSuccess) {
    ptr = nullptr;
    (void)cudaGetLastError();
    set_error("device allocation of " + std::to_string(n * sizeof(T)) + " bytes failed");
    return VMO_ERR_OOM;
  }
  count = n;
  async = as;
  astream = g_devarray_stream;
  g_device_allocs.fetch_add(1, std::memory_order_relaxed);
  return VMO_OK;
}

template <class T>
void DevArray<T>::release() {
  if (ptr) {
    if (async) cudaFreeAsync(ptr, astream);
    else cudaFree(ptr);
  }
  ptr = nullptr;
  count = 0;
}

// ---------------------------------------------------------------------------
// Hypergraph handle.
// ---------------------------------------------------------------------------
struct Graph {
  // Adjacency CSR over global vertex ids, with optional per-entry edge costs
  // and per-vertex weights (null = 1).
  int64_t k = 0;
  int64_t nadj = 0;
  const int32_t* adj_ptr = nullptr;  // k+1 (int32 offsets)
  const int32_t* adj = nullptr;
  const float* acost = nullptr;      // nadj or null
  const float* w = nullptr;          // k or null
};

}  // namespace vmo

struct vmo_hg_s {
  vmo_model model;
  int32_t m = 0, n = 0;
  int32_t k = 0;        // vertices
  int64_t l = 0;        // nets
  vmo::DevArray<int32_t> adj_ptr, adj;      // graph models
  vmo::DevArray<int32_t> net_ptr, pins;     // all models
  vmo::DevArray<int32_t> vtx_ptr, vnets;    // all models
  vmo::DevArray<float> weight;              // optional vertex weights
  int64_t nadj = 0, npins = 0, nvnets = 0;
  bool has_weight = false;
  int device = 0;
  void* fence = nullptr;  // of a user's handle: freeing it waits for the device (vmo_destroy)
};

namespace vmo {

// ---------------------------------------------------------------------------
// Primitives (prims.cu).
// ---------------------------------------------------------------------------
// Exclusive scan of n values; if total != nullptr the sum is written there
// (device).  In-place (in == out) is allowed.
template <class T>
vmo_status scan_exclusive(const T* in, T* out, int64_t n, T* total, cudaStream_t s, Scratch& sc);
template <class T>
vmo_status scan_inclusive(const T* in, T* out, int64_t n, cudaStream_t s, Scratch& sc);

// Inclusive scan that allocates nothing: `partial` must hold
// scan_partials_needed(n) values.
vmo_status scan_inclusive_u64_into(const uint64_t* in, uint64_t* out, int64_t n, uint64_t* partial, cudaStream_t s);
int64_t scan_partials_needed(int64_t n);

constexpr int kSortTile = 2048;  // 256 threads x 8 keys

// Stable LSD radix sort of (key, value) pairs on bits [0, bits).  Buffers are
// ping-ponged; the sorted result ends in (keys_out, vals_out).  vals may be
// null (keys only).
vmo_status radix_sort_u32(uint32_t* keys_in, uint32_t* vals_in, uint32_t* keys_out, uint32_t* vals_out,
                          int64_t n, int bits, cudaStream_t s, Scratch& sc);
vmo_status radix_sort_u64(uint64_t* keys_in, uint32_t* vals_in, uint64_t* keys_out, uint32_t* vals_out,
                          int64_t n, int bits, cudaStream_t s, Scratch& sc);

// ---------------------------------------------------------------------------
// Instrumentation: every kernel launch of the library goes through launch(),
// which counts it; the layout step kernel can also be timed with CUDA events
// and can count the interactions it evaluates (vmo_stats_* in the C-ABI).
// ---------------------------------------------------------------------------
extern std::atomic<uint64_t> g_launches;
bool stats_timing();
unsigned long long* stats_interaction_counter();  // null unless counting is on
void stats_time_begin(cudaStream_t s);
void stats_time_end(cudaStream_t s, uint64_t points);

// Programmatic dependent launch: inside a PdlScope the calling thread's
// launches carry the programmatic-serialization attribute, so a kernel's launch
// is processed while its predecessor in the stream still runs.  Every kernel
// launched that way starts with pdl_wait(), which returns once the preceding
// kernel has completed and its writes are visible (and at once when the kernel
// was launched without the attribute).
extern thread_local bool g_pdl;

// Launch-shape choices that never change a result (tune.cu): the largest step
// launch that takes the step kernel of small levels (two far-field rows in
// flight for d = 2, split terms up to five eighths of it for d = 3 and 4), the
// widest radix digit, the positions per thread of the Lloyd assignment of nodes
// beyond a cluster, and the largest problem binned by one block.
// Process-wide; set by vmo_set_tuning / vmo_autotune.
struct Tuning {
  std::atomic<int64_t> small_step_threads{152 * 4 * 32};
  std::atomic<int> radix_max_bits{10};
  std::atomic<int> assign_items{4};  // 4 measured best for a million-point Lloyd round (8 and 2 slower)
  std::atomic<int> small_bin_points{kSortTile};
};
extern Tuning g_tuning;
struct PdlScope {
  bool prev;
  PdlScope() : prev(g_pdl) { g_pdl = true; }
  ~PdlScope() { g_pdl = prev; }
};

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// pdl_wait(), then lets the next kernel of the stream be placed as soon as
// every block of this one has started (it waits in its own pdl_wait until this
// kernel has completed, so its launch overlaps this kernel's last wave).
__device__ __forceinline__ void pdl_enter() {
  pdl_wait();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... KArgs, class... Args>
inline void launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
  if (g_refused != cudaSuccess) return;
  g_launches.fetch_add(1, std::memory_order_relaxed);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  if (g_pdl) {
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
  g_refused = cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

inline int bits_for(uint64_t maxval) {
  int b = 0;
  while (b < 64 && (maxval >> b) != 0) ++b;
  return b;
}

inline unsigned grid_for(int64_t n, int block) {
  int64_t g = (n + block - 1) / block;
  if (g < 1) g = 1;
  return (unsigned)g;
}

// ---------------------------------------------------------------------------
// Device helpers.  Floating point that decides an integer uses explicitly
// rounded intrinsics so the compiler cannot contract or reorder it.
// ---------------------------------------------------------------------------
constexpr uint64_t kGolden = 0x9E3779B97F4A7C15ull;
constexpr uint64_t kTagCoord = 0x636f6f7264000000ull;   // initial layout
constexpr uint64_t kTagKmeans = 0x6b6d65616e730000ull;  // k-means++ draws
constexpr uint64_t kTagMatch = 0x6d61746368000000ull;   // matching tie-breaks
constexpr uint64_t kTagJitter = 0x6a69747465720000ull;  // prolongation jitter

__host__ __device__ inline uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__host__ __device__ inline uint64_t rand64(uint64_t seed, uint64_t a, uint64_t b) {
  return mix64(mix64(seed + kGolden * (a + 1)) + kGolden * (b + 1));
}

// floor(n * r / 2^64)
__device__ inline uint64_t scale_draw(uint64_t n, uint64_t r) { return __umul64hi(n, r); }

// Exponent e with max |x| < 2^e (0 for max = 0) from the float bits of the max
// (the fixed-point grid of the k-means sums is 2^-(30 - e)).
__device__ inline int exponent_of(uint32_t maxbits) {
  float mx = __uint_as_float(maxbits);
  if (mx == 0.0f) return 0;
  int e;
  frexpf(mx, &e);
  return e;
}

// Order-preserving map float -> uint32 (for atomicMin/Max on floats).
__device__ inline uint32_t f2ord(float f) {
  uint32_t b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__host__ __device__ inline float ord2f(uint32_t u) {
  uint32_t b = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float f;
  memcpy(&f, &b, 4);
  return f;
#endif
}

// Exact 2^e as float for -126 <= e <= 127.
__device__ inline float exp2i_f(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }

// Squared distance of two points in fp32, coordinates 0..d-1 in order, no FMA.
template <int D>
__device__ inline float sqdist32(const float4& a, const float4& b) {
  float q = __fsub_rn(a.x, b.x);
  float s = __fmul_rn(q, q);
  if (D > 1) { q = __fsub_rn(a.y, b.y); s = __fadd_rn(s, __fmul_rn(q, q)); }
  if (D > 2) { q = __fsub_rn(a.z, b.z); s = __fadd_rn(s, __fmul_rn(q, q)); }
  if (D > 3) { q = __fsub_rn(a.w, b.w); s = __fadd_rn(s, __fmul_rn(q, q)); }
  return s;
}

__device__ inline float comp(const float4& v, int m) {
  return m == 0 ? v.x : (m == 1 ? v.y : (m == 2 ? v.z : v.w));
}

__device__ inline unsigned lane_id() { return threadIdx.x & 31u; }

}  // namespace vmo
