// Hypergraph models of a sparse pattern (Table 1, Sec. 1.1), connected
// components (Algorithm 1) and cut metrics (Sec. 4.1 footnote, Sec. 5).
//
// Any pattern can be built the general way: each nonzero emits 64-bit pair
// keys (row * ncols + col), a radix sort orders them, a flag/scan pass drops
// duplicates and the surviving keys become CSR rows whose pointers come from
// per-row counts and a scan.  Graph models emit both orientations of {u, v} so
// the result is the symmetric adjacency with ascending neighbours.
//
// A pattern whose rows ascend strictly, as matrices are usually stored, needs
// no such sort (the validation pass finds out): its rows are already the rows of
// the model, its columns come from one stable sort of 32-bit column keys with the
// entry numbers (two passes instead of four of 64-bit keys), and a symmetric
// pattern is its own adjacency, with every entry's mirror found by a binary
// search in its row.  27-point mesh of 10^6 rows in random numbering, symmetric
// model with copies of its arrays: 7.6 -> 1.05 ms; 400k x 300k bipartite model: 2.1 -> 0.61 ms.
#include <algorithm>

#include "vmo_internal.cuh"

namespace vmo {

namespace {

__device__ inline int32_t row_of(const int32_t* __restrict__ rowptr, int32_t m, int64_t t) {
  int32_t lo = 0, hi = m;  // rowptr[lo] <= t < rowptr[hi]
  while (hi - lo > 1) {
    int32_t mid = (lo + hi) >> 1;
    if (rowptr[mid] <= t) lo = mid; else hi = mid;
  }
  return lo;
}

// Error bits: 1 rowptr not monotone, 2 its ends, 4 a column out of range.
// steps (optional): [0] entries that do not ascend from the entry before them,
// [1] how many of these start a row; every row ascends strictly iff the two
// agree (a search of the row at each step took five times the pass).
__global__ void __launch_bounds__(256) validate_csr_kernel(const int32_t* __restrict__ rowptr,
                                                           const int32_t* __restrict__ colidx, int32_t m, int32_t n,
                                                           int64_t nnz, int32_t* __restrict__ bad,
                                                           int32_t* __restrict__ steps) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x, first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int err = 0, down = 0, starts = 0;
  if (first == 0 && (rowptr[0] != 0 || (int64_t)rowptr[m] != nnz)) err |= 2;
  for (int64_t r = first; r < m; r += stride) {
    const int32_t a = rowptr[r], b = rowptr[r + 1];
    if (b < a) err |= 1;
    if (steps && a > 0 && a < b && b <= nnz) starts += colidx[a] <= colidx[a - 1];
  }
  for (int64_t t = first; t < nnz; t += 4 * stride) {
    int32_t c[4], p[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t i = t + u * stride;
      c[u] = i < nnz ? colidx[i] : 0;
      p[u] = steps && i < nnz && i > 0 ? colidx[i - 1] : INT32_MIN;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (t + u * stride >= nnz) break;
      if (c[u] < 0 || c[u] >= n) err |= 4;
      down += c[u] <= p[u];
    }
  }
  err = __reduce_or_sync(0xffffffffu, err);
  if (lane_id() == 0 && err) atomicOr(bad, err);
  if (!steps) return;
  down = __reduce_add_sync(0xffffffffu, down);
  starts = __reduce_add_sync(0xffffffffu, starts);
  if (lane_id() == 0) {
    if (down) atomicAdd(&steps[0], down);
    if (starts) atomicAdd(&steps[1], starts);
  }
}

// ----- models of patterns with strictly ascending rows -----
constexpr int kRowTile = 2048;  // entries per block

// Row of the entries [t0, t0 + count) of a tile, count <= kRowTile, from the row starts of
// the tile's rows in shared memory (in global memory when empty rows make them
// more than fit).
struct TileRows {
  int32_t ptr[kRowTile + 2];
  int32_t r0, r1;  // rows of the tile's first and last entry
};

__device__ inline void tile_rows_load(TileRows& s, const int32_t* __restrict__ rowptr, int32_t m, int64_t t0,
                                      int64_t count) {
  if (threadIdx.x == 0) s.r0 = row_of(rowptr, m, t0);
  if (threadIdx.x == 32) s.r1 = row_of(rowptr, m, t0 + count - 1);
  __syncthreads();
  const int32_t rows = s.r1 - s.r0 + 1;
  if (rows <= kRowTile + 1)
    for (int32_t i = threadIdx.x; i < rows; i += blockDim.x) s.ptr[i] = rowptr[s.r0 + i];
  __syncthreads();
}

__device__ inline int32_t tile_row(const TileRows& s, const int32_t* __restrict__ rowptr, int64_t t) {
  const int32_t rows = s.r1 - s.r0 + 1;
  const int32_t* p = rows <= kRowTile + 1 ? s.ptr : rowptr + s.r0;
  return s.r0 + row_of(p, rows, t);
}

// Column keys, entry numbers and rows of the entries (for the column sort).
__global__ void __launch_bounds__(256) entry_rows_kernel(const int32_t* __restrict__ rowptr,
                                                         const int32_t* __restrict__ colidx, int32_t m, int64_t nnz,
                                                         uint32_t* __restrict__ key, uint32_t* __restrict__ val,
                                                         int32_t* __restrict__ row) {
  __shared__ TileRows s;
  const int64_t t0 = (int64_t)blockIdx.x * kRowTile;
  const int64_t count = min((int64_t)kRowTile, nnz - t0);
  tile_rows_load(s, rowptr, m, t0, count);
  for (int64_t t = t0 + threadIdx.x; t < t0 + count; t += blockDim.x) {
    key[t] = (uint32_t)colidx[t];
    val[t] = (uint32_t)t;
    row[t] = tile_row(s, rowptr, t);
  }
}

// First sorted entry of every column, and the end.
__global__ void column_starts_kernel(const uint32_t* __restrict__ key, int64_t nnz, int32_t n, int32_t add,
                                     int32_t* __restrict__ ptr) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c > n) return;
  int64_t lo = 0, hi = nnz;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((int64_t)key[mid] < c) lo = mid + 1; else hi = mid;
  }
  ptr[c] = add + (int32_t)lo;
}

// The column side of a model: idx[s] (vertex or net of the s-th entry in
// column order) is its row, or its entry number when row is null.
__global__ void column_entries_kernel(const uint32_t* __restrict__ val, const int32_t* __restrict__ row, int64_t nnz,
                                      int32_t* __restrict__ idx, int32_t* __restrict__ entry) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nnz) return;
  const uint32_t t = val[s];
  if (idx) idx[s] = row[t];
  if (entry) entry[s] = (int32_t)t;
}

// The row side of the bipartite model: entry t is net t, of row i and column
// vertex m + j.
__global__ void bipartite_rows_kernel(const int32_t* __restrict__ colidx, const int32_t* __restrict__ row, int32_t m,
                                      int64_t nnz, int32_t* __restrict__ adj, int32_t* __restrict__ vnets,
                                      int32_t* __restrict__ net_ptr, int2* __restrict__ pins) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t > nnz) return;
  net_ptr[t] = (int32_t)(2 * t);
  if (t == nnz) return;
  const int32_t v = m + colidx[t];
  adj[t] = v;
  vnets[t] = (int32_t)t;
  pins[t] = make_int2(row[t], v);
}

// Rows of a square pattern: entry on the diagonal (0 or 1) and entries right of it.
__global__ void row_parts_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx, int32_t m,
                                 int32_t* __restrict__ diag, int32_t* __restrict__ right) {
  const int32_t u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= m) return;
  int32_t lo = rowptr[u];
  const int32_t end = rowptr[u + 1];
  int32_t hi = end;
  while (lo < hi) {
    const int32_t mid = (lo + hi) >> 1;
    if (colidx[mid] < u) lo = mid + 1; else hi = mid;
  }
  const int32_t d = lo < end && colidx[lo] == u ? 1 : 0;
  diag[u] = d;
  right[u] = end - lo - d;
}

// First entry of every row and the diagonal entries before it, side by side (a
// mirror's row is looked up once per net).
__global__ void row_heads_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ dpre, int32_t m,
                                 int2* __restrict__ head) {
  const int32_t u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u <= m) head[u] = make_int2(rowptr[u], dpre[u]);
}

// Adjacency of a symmetric pattern: the entries off the diagonal.  Every entry
// (u, v) right of the diagonal is net number e, and sets the incidence of its
// mirror (v, u) too; *missing is set when an entry has no mirror.  dpre and rpre:
// diagonal entries and entries right of the diagonal in the rows before.
// Bound by the mirrors' scattered sectors (six per net).
__global__ void __launch_bounds__(256) symmetric_kernel(const int32_t* __restrict__ rowptr,
                                                        const int32_t* __restrict__ colidx, int32_t m, int64_t nnz,
                                                        const int2* __restrict__ head,
                                                        const int32_t* __restrict__ rpre, int32_t* __restrict__ adj,
                                                        int32_t* __restrict__ vnets, int32_t* __restrict__ net_ptr,
                                                        int2* __restrict__ pins, int32_t* __restrict__ missing) {
  __shared__ TileRows s;
  const int64_t t0 = (int64_t)blockIdx.x * kRowTile;
  const int64_t count = min((int64_t)kRowTile, nnz - t0);
  tile_rows_load(s, rowptr, m, t0, count);
  for (int64_t t = t0 + threadIdx.x; t < t0 + count; t += blockDim.x) {
    const int32_t v = colidx[t], u = tile_row(s, rowptr, t);
    if (v == u) continue;
    if (v < u) {
      adj[t - head[u].y] = v;
      continue;
    }
    const int2 next = head[u + 1];
    const int32_t e = rpre[u + 1] - (next.x - (int32_t)t);  // entries right of the diagonal end the row
    const int32_t place = (int32_t)t - next.y;
    adj[place] = v;
    vnets[place] = e;
    net_ptr[e] = 2 * e;
    pins[e] = make_int2(u, v);
    const int2 hv = head[v];
    const int32_t b1 = head[v + 1].x;
    int32_t lo = hv.x, hi = b1;
    while (lo < hi) {
      const int32_t mid = (lo + hi) >> 1;
      if (colidx[mid] < u) lo = mid + 1; else hi = mid;
    }
    if (lo < b1 && colidx[lo] == u) vnets[lo - hv.y] = e;  // left of the diagonal of row v
    else *missing = 1;
  }
}

__global__ void symmetric_ptr_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ dpre, int32_t m,
                                     int32_t nets, int32_t* __restrict__ adj_ptr, int32_t* __restrict__ vtx_ptr,
                                     int32_t* __restrict__ net_ptr) {
  const int32_t u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u > m) return;
  adj_ptr[u] = vtx_ptr[u] = rowptr[u] - dpre[u];
  if (u == 0) net_ptr[nets] = 2 * nets;
}

// Pair keys of the graph models: both orientations of every off-diagonal
// pattern entry (symmetric: {i, j}; bipartite: {r_i, c_j} = {i, m + j}).
__global__ void graph_keys_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx, int32_t m,
                                  int64_t nnz, int bipartite, uint64_t K, uint64_t sentinel,
                                  uint64_t* __restrict__ keys) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nnz) return;
  uint64_t u = (uint64_t)row_of(rowptr, m, t);
  uint64_t v = bipartite ? (uint64_t)m + (uint64_t)colidx[t] : (uint64_t)colidx[t];
  if (u == v) {
    keys[2 * t] = sentinel;
    keys[2 * t + 1] = sentinel;
  } else {
    keys[2 * t] = u * K + v;
    keys[2 * t + 1] = v * K + u;
  }
}

// Pair keys (row, col) or transposed (col, row) of the pattern itself.
__global__ void pattern_keys_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx, int32_t m,
                                    int32_t n, int64_t nnz, int transpose, uint64_t* __restrict__ keys) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nnz) return;
  uint64_t i = (uint64_t)row_of(rowptr, m, t), j = (uint64_t)colidx[t];
  keys[t] = transpose ? j * (uint64_t)m + i : i * (uint64_t)n + j;
}

__global__ void unique_flags_kernel(const uint64_t* __restrict__ keys, int64_t n, uint64_t sentinel,
                                    int32_t* __restrict__ flag) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  uint64_t k = keys[t];
  flag[t] = (k != sentinel && (t == 0 || keys[t - 1] != k)) ? 1 : 0;
}

__global__ void emit_csr_kernel(const uint64_t* __restrict__ keys, int64_t n, const int32_t* __restrict__ flag,
                                const int32_t* __restrict__ pos, uint64_t ncols, int32_t* __restrict__ idx,
                                int32_t* __restrict__ rowcount) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n || !flag[t]) return;
  uint64_t k = keys[t];
  idx[pos[t]] = (int32_t)(k % ncols);
  atomicAdd(&rowcount[k / ncols], 1);
}

__global__ void set_last_kernel(int32_t* ptr, int64_t n, const int32_t* total) { ptr[n] = *total; }

// Edge list (nets) of a graph model: the adjacency entries u -> v with u < v,
// in adjacency order (lexicographic).  pins[2e], pins[2e+1] = u, v.
__global__ void forward_flags_kernel(const int32_t* __restrict__ adj_ptr, const int32_t* __restrict__ adj, int32_t k,
                                     int64_t nadj, int32_t* __restrict__ flag) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nadj) return;
  int32_t u = row_of(adj_ptr, k, t);
  flag[t] = adj[t] > u ? 1 : 0;
}

__global__ void emit_edges_kernel(const int32_t* __restrict__ adj_ptr, const int32_t* __restrict__ adj, int32_t k,
                                  int64_t nadj, const int32_t* __restrict__ flag, const int32_t* __restrict__ pos,
                                  int32_t* __restrict__ net_ptr, int32_t* __restrict__ pins,
                                  int32_t* __restrict__ vnets) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nadj || !flag[t]) return;
  int32_t u = row_of(adj_ptr, k, t), v = adj[t];
  int32_t e = pos[t];
  net_ptr[e] = 2 * e;
  pins[2 * e] = u;
  pins[2 * e + 1] = v;
  vnets[t] = e;
  // position of u in the (ascending) adjacency of v
  int32_t lo = adj_ptr[v], hi = adj_ptr[v + 1];
  while (lo < hi) {
    int32_t mid = (lo + hi) >> 1;
    if (adj[mid] < u) lo = mid + 1; else hi = mid;
  }
  vnets[lo] = e;
}

__global__ void net_ptr_last_kernel(int32_t* net_ptr, const int32_t* nedges) { net_ptr[*nedges] = 2 * *nedges; }

// ----------------------------- components ----------------------------------
// Union-find on the labels: a root points at itself, every other vertex at a
// smaller one, so a tree's root is its smallest vertex.  Links are lossless
// (a compare-and-swap on the larger root, repeated from its new parent when
// another thread was first), so one pass over the nets finds the components
// and no round has to be checked on the host.  Labels are read through L1: every search
// ends at one of a few roots, and their L2 sectors would be the time of the
// pass; an outdated label is still an ancestor (equal ones still mean one tree),
// and the compare-and-swap on a root that no longer is one returns the new label.

// Joins the trees of u and v: the search whose label is larger moves up, until
// its label is a root, which is put below the other label, whether that one is a
// root or not (a label is never below a smaller one, so no cycle can form).  Only
// one of the two paths is climbed, and not beyond the other's labels: the edges of
// a path graph all link at once, where searches for both roots climbed half a
// chain each (bipartite model of a tridiagonal pattern of 10^6 rows, the whole
// call: 7.7 ms, now 0.18 ms).  A path is split behind the search (every
// vertex passed gets its grandparent; only vertices that are no roots are written,
// each with an ancestor of its own).  ALL: until they are joined; else for at
// most kCcClimb steps, in a pass that another one follows after the paths have
// been flattened (searches that climb a growing chain to its end take 80 ms of
// that pattern's call).
constexpr int kCcClimb = 8;

template <bool ALL>
__device__ inline void cc_link(int32_t u, int32_t v, int32_t* p) {
  int32_t a = __ldca(p + u), b = __ldca(p + v);
  for (int step = 0; a != b && (ALL || step < kCcClimb); ++step) {
    if (a < b) {
      int32_t t = a;
      a = b;
      b = t;
      t = u;
      u = v;
      v = t;
    }
    int32_t q = step < 2 ? __ldca(p + a) : __ldcg(p + a);
    if (q == a) {
      q = atomicCAS(p + a, a, b);
      if (q == a) return;
    }
    if (a != u) p[u] = q;
    u = a;
    a = q;
  }
}

// Graph models start from every vertex's smallest neighbour (its own label if
// that is larger): most vertices then hang below a common root before the pass
// over the edges, which finds nearly every edge inside a tree (rows ascend, so
// it is the row's first entry).
__global__ void cc_init_kernel(const int32_t* __restrict__ adj_ptr, const int32_t* __restrict__ adj,
                               int32_t* __restrict__ p, int32_t k) {
  int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= k) return;
  int32_t q = v;
  if (adj_ptr && adj_ptr[v + 1] > adj_ptr[v]) q = min(v, adj[adj_ptr[v]]);
  p[v] = q;
}

// Links every stride-th vertex to its largest neighbour, unless they have one
// label: a 64th of the vertices first, then a 16th, a quarter and all, with the
// paths flattened in between.  Where every vertex links at once, half a
// million threads chase the same few roots (1.1 ms for the 400k x 300k
// bipartite pattern and 0.27 ms for 500,000 power-law rows; the four
// launches 0.13 and 0.04 ms).
constexpr int kCcSample = 64;

__global__ void cc_neighbour_kernel(const int32_t* __restrict__ adj_ptr, const int32_t* __restrict__ adj, int32_t* p,
                                    int32_t k, int stride) {
  const int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * stride;
  if (v >= k || adj_ptr[v + 1] == adj_ptr[v]) return;
  const int32_t u = adj[adj_ptr[v + 1] - 1];
  if (__ldca(p + v) != __ldca(p + u)) cc_link<false>((int32_t)v, u, p);
}

// Marks the last pin of every net (the pins that start no consecutive pair).
__global__ void cc_last_kernel(const int32_t* __restrict__ net_ptr, int64_t l, uint8_t* __restrict__ last) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= l) return;
  const int32_t b = net_ptr[e + 1];
  if (b > net_ptr[e]) last[b - 1] = 1;
}

// Links the consecutive pins of every net, first with short searches and, the
// paths flattened, again to the end (row nets of a 5-point grid of 10^6 rows: 820 us in
// one pass, 440 in two; of a path in random order 160 and 190).
template <bool ALL>
__global__ void cc_pins_kernel(const int32_t* __restrict__ pins, const uint8_t* __restrict__ last, int64_t npins,
                               int32_t* p) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t + 1 >= npins || last[t]) return;  // the last pin of a net pairs with no next pin
  cc_link<ALL>(pins[t], pins[t + 1], p);
}

// Links the two ends of every edge; most edges already have one label.
__global__ void cc_edges_kernel(const int2* __restrict__ edge, int64_t l, int32_t* p) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= l) return;
  const int2 uv = edge[e];
  if (__ldca(p + uv.x) != __ldca(p + uv.y)) cc_link<true>(uv.x, uv.y, p);
}

// Labels to their roots.  Every thread writes its label as it climbs, past L1
// after two steps, so that the threads of a long path climb on each other's
// steps and the path is flat after about as many as its length has bits (with
// searches that wrote their end only, the path graph of 10^6 vertices in order
// took 1,050 us, now 36 us).  Nothing is linked meanwhile: a root stays one, and
// no thread writes another's label.
__global__ void cc_compress_kernel(int32_t* p, int32_t k) {
  const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= k) return;
  int32_t a = __ldca(p + v);
  for (int step = 0;; ++step) {
    const int32_t q = step < 2 ? __ldca(p + a) : __ldcg(p + a);
    if (q == a) return;
    __stcg(p + v, q);
    a = q;
  }
}

// ------------------------------- cut size ----------------------------------
// One warp per net.  nparts <= 64: union of part bitmasks; otherwise a pin is
// counted when no earlier pin of the net has its part.
__global__ void cut_kernel(const int32_t* __restrict__ net_ptr, const int32_t* __restrict__ pins, int64_t l,
                           const int32_t* __restrict__ part, int32_t nparts, unsigned long long* __restrict__ out) {
  int64_t e = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int lane = lane_id();
  if (e >= l) return;
  int32_t a = net_ptr[e], b = net_ptr[e + 1];
  uint32_t lam;
  if (nparts <= 64) {
    uint64_t mask = 0;
    for (int32_t t = a + lane; t < b; t += 32) mask |= 1ull << part[pins[t]];
    uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)mask);
    uint32_t hi = __reduce_or_sync(0xffffffffu, (uint32_t)(mask >> 32));
    lam = __popc(lo) + __popc(hi);
  } else {
    uint32_t cnt = 0;
    for (int32_t t = a + lane; t < b; t += 32) {
      int32_t pt = part[pins[t]];
      bool first = true;
      for (int32_t u = a; u < t; ++u)
        if (part[pins[u]] == pt) { first = false; break; }
      cnt += first ? 1u : 0u;
    }
    lam = __reduce_add_sync(0xffffffffu, cnt);
  }
  if (lane == 0 && lam > 1) {
    atomicAdd(out, 1ull);
    atomicAdd(out + 1, (unsigned long long)(lam - 1));
  }
}

}  // namespace

static void validate_launch(const vmo_csr* a, int32_t* bad, int32_t* steps, cudaStream_t s) {
  const int64_t n = std::max<int64_t>(a->m, (a->nnz + 3) / 4);
  launch(validate_csr_kernel, (unsigned)std::min<int64_t>(grid_for(n + 1, 256), 152 * 8), 256, 0, s, a->rowptr, a->colidx,
         a->m, a->n, a->nnz, bad, steps);
}

vmo_status validate_csr(const vmo_csr* a, bool* ascending, cudaStream_t s, Scratch& sc) {
  if (!a || a->m < 0 || a->n < 0 || a->nnz < 0) return invalid("csr: negative size or null");
  if (!a->rowptr || (a->nnz > 0 && !a->colidx)) return invalid("csr: null pointer");
  if (a->nnz > INT32_MAX) return unsupported("csr: more than 2^31-1 nonzeros");
  int32_t* bad;  // error bits, steps
  VMO_TRY(sc.alloc(&bad, 3));
  VMO_CUDA(cudaMemsetAsync(bad, 0, 12, s));
  validate_launch(a, bad, bad + 1, s);
  VMO_LAUNCHED("validate_csr");
  int32_t hb[3] = {0, 0, 0};
  VMO_CUDA(cudaMemcpyAsync(hb, bad, 12, cudaMemcpyDeviceToHost, s));
  VMO_CUDA(cudaStreamSynchronize(s));
  const int32_t h = hb[0];
  if (h & 2) return invalid("csr: rowptr[0] != 0 or rowptr[m] != nnz");
  if (h & 1) return invalid("csr: rowptr not monotone");
  if (h & 4) return invalid("csr: column index out of range");
  *ascending = hb[1] == hb[2];
  return VMO_OK;
}

__global__ void fg_vnets_kernel(const int32_t* rptr, const int32_t* cidx, int32_t m, int32_t* vtx_ptr, int32_t* vnets);
__global__ void fg_nets_kernel(const int32_t* rptr, int32_t m, const int32_t* cptr, const int32_t* cpins, int32_t n,
                               int64_t u, int32_t* net_ptr, int32_t* pins);

// Entries of a pattern with ascending rows in column order: their entry
// numbers (order) and rows (by entry number), and the column starts + add in
// ptr (n + 1).
static vmo_status column_order(const vmo_csr* a, int32_t add, int32_t* ptr, uint32_t** order, int32_t** row,
                               cudaStream_t s, Scratch& sc) {
  const int64_t nnz = a->nnz;
  uint32_t *k1, *k2, *v1;
  VMO_TRY(sc.alloc(&k1, (size_t)std::max<int64_t>(nnz, 1)));
  VMO_TRY(sc.alloc(&k2, (size_t)std::max<int64_t>(nnz, 1)));
  VMO_TRY(sc.alloc(&v1, (size_t)std::max<int64_t>(nnz, 1)));
  VMO_TRY(sc.alloc(order, (size_t)std::max<int64_t>(nnz, 1)));
  VMO_TRY(sc.alloc(row, (size_t)std::max<int64_t>(nnz, 1)));
  if (nnz > 0) {
    launch(entry_rows_kernel, grid_for(nnz, kRowTile), 256, 0, s, a->rowptr, a->colidx, a->m, nnz, k1, v1, *row);
    VMO_LAUNCHED("entry_rows");
    VMO_TRY(radix_sort_u32(k1, v1, k2, *order, nnz, bits_for((uint64_t)std::max(a->n - 1, 0)), s, sc));
  }
  launch(column_starts_kernel, grid_for((int64_t)a->n + 1, 256), 256, 0, s, k2, nnz, a->n, add, ptr);
  VMO_LAUNCHED("column_starts");
  return VMO_OK;
}

// Models of a pattern with strictly ascending rows (see the head of the
// file); *done is false for a symmetric model of an unsymmetric pattern.
static vmo_status build_ascending(const vmo_csr* a, vmo_model model, vmo_hg_s* h, bool* done, cudaStream_t s,
                                  Scratch& sc) {
  const int32_t m = a->m, n = a->n;
  const int64_t nnz = a->nnz, cap = std::max<int64_t>(nnz, 1);
  const unsigned ge = grid_for(nnz, 256);
  uint32_t* order;
  int32_t* row;
  *done = true;
  if (model == VMO_SYMMETRIC) {
    int32_t *dpre, *rpre, *missing;
    VMO_TRY(sc.alloc(&dpre, (size_t)m + 1));
    VMO_TRY(sc.alloc(&rpre, (size_t)m + 1));
    VMO_TRY(sc.alloc(&missing, 1));
    VMO_CUDA(cudaMemsetAsync(missing, 0, 4, s));
    if (m > 0) {
      launch(row_parts_kernel, grid_for(m, 256), 256, 0, s, a->rowptr, a->colidx, m, dpre, rpre);
      VMO_LAUNCHED("row_parts");
    }
    VMO_TRY(scan_exclusive<int32_t>(dpre, dpre, m, dpre + m, s, sc));
    VMO_TRY(scan_exclusive<int32_t>(rpre, rpre, m, rpre + m, s, sc));
    int32_t diag = 0, right = 0;
    VMO_CUDA(cudaMemcpyAsync(&diag, dpre + m, 4, cudaMemcpyDeviceToHost, s));
    VMO_CUDA(cudaMemcpyAsync(&right, rpre + m, 4, cudaMemcpyDeviceToHost, s));
    VMO_CUDA(cudaStreamSynchronize(s));
    const int64_t nadj = nnz - diag;
    if (nadj != 2 * (int64_t)right) {  // more entries on one side of the diagonal
      *done = false;
      return VMO_OK;
    }
    h->k = m;
    h->nadj = h->npins = h->nvnets = nadj;
    h->l = right;
    VMO_TRY(h->adj_ptr.resize((size_t)m + 1));
    VMO_TRY(h->vtx_ptr.resize((size_t)m + 1));
    VMO_TRY(h->adj.resize((size_t)std::max<int64_t>(nadj, 1)));
    VMO_TRY(h->vnets.resize((size_t)std::max<int64_t>(nadj, 1)));
    VMO_TRY(h->pins.resize((size_t)std::max<int64_t>(nadj, 1)));
    VMO_TRY(h->net_ptr.resize((size_t)right + 1));
    if (nnz > 0) {
      int2* head;
      VMO_TRY(sc.alloc(&head, (size_t)m + 1));
      launch(row_heads_kernel, grid_for((int64_t)m + 1, 256), 256, 0, s, a->rowptr, dpre, m, head);
      launch(symmetric_kernel, grid_for(nnz, kRowTile), 256, 0, s, a->rowptr, a->colidx, m, nnz, head, rpre,
             h->adj.ptr, h->vnets.ptr, h->net_ptr.ptr, (int2*)h->pins.ptr, missing);
      VMO_LAUNCHED("symmetric");
    }
    launch(symmetric_ptr_kernel, grid_for((int64_t)m + 1, 256), 256, 0, s, a->rowptr, dpre, m, right, h->adj_ptr.ptr,
           h->vtx_ptr.ptr, h->net_ptr.ptr);
    VMO_LAUNCHED("symmetric_ptr");
    int32_t hm = 0;
    VMO_CUDA(cudaMemcpyAsync(&hm, missing, 4, cudaMemcpyDeviceToHost, s));
    VMO_CUDA(cudaStreamSynchronize(s));
    *done = hm == 0;
    return VMO_OK;
  }
  if (model == VMO_BIPARTITE) {
    h->k = m + n;
    h->nadj = h->npins = h->nvnets = 2 * nnz;
    h->l = nnz;
    VMO_TRY(h->adj_ptr.resize((size_t)h->k + 1));
    VMO_TRY(h->vtx_ptr.resize((size_t)h->k + 1));
    VMO_TRY(h->adj.resize((size_t)2 * cap));
    VMO_TRY(h->vnets.resize((size_t)2 * cap));
    VMO_TRY(h->pins.resize((size_t)2 * cap));
    VMO_TRY(h->net_ptr.resize((size_t)nnz + 1));
    VMO_TRY(column_order(a, (int32_t)nnz, h->adj_ptr.ptr + m, &order, &row, s, sc));
    if (m > 0) VMO_CUDA(cudaMemcpyAsync(h->adj_ptr.ptr, a->rowptr, m * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    VMO_CUDA(cudaMemcpyAsync(h->vtx_ptr.ptr, h->adj_ptr.ptr, ((size_t)h->k + 1) * sizeof(int32_t),
                             cudaMemcpyDeviceToDevice, s));
    launch(bipartite_rows_kernel, grid_for(nnz + 1, 256), 256, 0, s, a->colidx, row, m, nnz, h->adj.ptr, h->vnets.ptr,
           h->net_ptr.ptr, (int2*)h->pins.ptr);
    if (nnz > 0)
      launch(column_entries_kernel, ge, 256, 0, s, order, row, nnz, h->adj.ptr + nnz, h->vnets.ptr + nnz);
    VMO_LAUNCHED("bipartite");
  } else if (model == VMO_ROWNET || model == VMO_COLNET) {
    const bool rn = model == VMO_ROWNET;
    h->k = rn ? n : m;
    h->l = rn ? m : n;
    h->npins = h->nvnets = nnz;
    DevArray<int32_t>&rp = rn ? h->net_ptr : h->vtx_ptr, &ri = rn ? h->pins : h->vnets;
    DevArray<int32_t>&cp = rn ? h->vtx_ptr : h->net_ptr, &ci = rn ? h->vnets : h->pins;
    VMO_TRY(rp.resize((size_t)m + 1));
    VMO_TRY(ri.resize((size_t)cap));
    VMO_TRY(cp.resize((size_t)n + 1));
    VMO_TRY(ci.resize((size_t)cap));
    VMO_TRY(column_order(a, 0, cp.ptr, &order, &row, s, sc));
    VMO_CUDA(cudaMemcpyAsync(rp.ptr, a->rowptr, ((size_t)m + 1) * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    if (nnz > 0) {
      VMO_CUDA(cudaMemcpyAsync(ri.ptr, a->colidx, nnz * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
      launch(column_entries_kernel, ge, 256, 0, s, order, row, nnz, ci.ptr, (int32_t*)nullptr);
      VMO_LAUNCHED("column_entries");
    }
  } else {  // finegrain: vertices are the entries
    if (2 * nnz > INT32_MAX) return unsupported("too many entries");
    h->k = (int32_t)nnz;
    h->l = (int64_t)m + n;
    h->npins = h->nvnets = 2 * nnz;
    VMO_TRY(h->vtx_ptr.resize((size_t)nnz + 1));
    VMO_TRY(h->vnets.resize((size_t)2 * cap));
    VMO_TRY(h->net_ptr.resize((size_t)m + n + 1));
    VMO_TRY(h->pins.resize((size_t)2 * cap));
    int32_t* cptr;
    VMO_TRY(sc.alloc(&cptr, (size_t)n + 1));
    VMO_TRY(column_order(a, 0, cptr, &order, &row, s, sc));
    VMO_CUDA(cudaMemsetAsync(h->vtx_ptr.ptr, 0, sizeof(int32_t), s));
    if (m > 0) launch(fg_vnets_kernel, grid_for(m, 256), 256, 0, s, a->rowptr, a->colidx, m, h->vtx_ptr.ptr, h->vnets.ptr);
    const int64_t span = std::max<int64_t>(std::max<int64_t>(nnz, (int64_t)m + 1), (int64_t)n);
    launch(fg_nets_kernel, grid_for(span, 256), 256, 0, s, a->rowptr, m, cptr, (const int32_t*)order, n, nnz,
           h->net_ptr.ptr, h->pins.ptr);
    VMO_LAUNCHED("finegrain");
  }
  VMO_CUDA(cudaStreamSynchronize(s));
  return VMO_OK;
}

// Sorted-unique CSR of `nrows` rows from pair keys row*ncols+col (keys with
// value >= nrows*ncols are dropped).  Allocates ptr (nrows+1) and idx.
static vmo_status csr_from_keys(uint64_t* keys, int64_t nkeys, int64_t nrows, int64_t ncols, DevArray<int32_t>& ptr,
                                DevArray<int32_t>& idx, int64_t* nout, cudaStream_t s, Scratch& sc) {
  uint64_t sentinel = (uint64_t)nrows * (uint64_t)ncols;
  int bits = bits_for(sentinel);
  uint64_t* sorted;
  int32_t *flag, *pos, *total;
  VMO_TRY(sc.alloc(&sorted, (size_t)std::max<int64_t>(nkeys, 1)));
  VMO_TRY(sc.alloc(&flag, (size_t)std::max<int64_t>(nkeys, 1)));
  VMO_TRY(sc.alloc(&pos, (size_t)std::max<int64_t>(nkeys, 1)));
  VMO_TRY(sc.alloc(&total, 1));
  VMO_TRY(radix_sort_u64(keys, nullptr, sorted, nullptr, nkeys, bits, s, sc));
  if (nkeys > 0) {
    launch(unique_flags_kernel, grid_for(nkeys, 256), 256, 0, s, sorted, nkeys, sentinel, flag);
    VMO_LAUNCHED("unique_flags");
  }
  VMO_TRY(scan_exclusive<int32_t>(flag, pos, nkeys, total, s, sc));
  int32_t h_total = 0;
  VMO_CUDA(cudaMemcpyAsync(&h_total, total, 4, cudaMemcpyDeviceToHost, s));
  VMO_CUDA(cudaStreamSynchronize(s));
  VMO_TRY(ptr.resize((size_t)nrows + 1));
  VMO_TRY(idx.resize((size_t)std::max<int32_t>(h_total, 1)));
  VMO_CUDA(cudaMemsetAsync(ptr.ptr, 0, (nrows + 1) * sizeof(int32_t), s));
  if (nkeys > 0) {
    launch(emit_csr_kernel, grid_for(nkeys, 256), 256, 0, s, sorted, nkeys, flag, pos, (uint64_t)ncols, idx.ptr, ptr.ptr);
    VMO_LAUNCHED("emit_csr");
  }
  VMO_TRY(scan_exclusive<int32_t>(ptr.ptr, ptr.ptr, nrows, total, s, sc));
  launch(set_last_kernel, 1, 1, 0, s, ptr.ptr, nrows, total);
  VMO_LAUNCHED("set_last");
  *nout = h_total;
  return VMO_OK;
}

// Finegrain incidence: vertex t (the t-th distinct entry, in row i) lies on
// row net i and column net m + col(t).
__global__ void fg_vnets_kernel(const int32_t* __restrict__ rptr, const int32_t* __restrict__ cidx, int32_t m,
                                int32_t* __restrict__ vtx_ptr, int32_t* __restrict__ vnets) {
  int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  for (int32_t t = rptr[i]; t < rptr[i + 1]; ++t) {
    vtx_ptr[t] = 2 * t;
    vnets[2 * t] = i;
    vnets[2 * t + 1] = m + cidx[t];
  }
  if (i == m - 1) vtx_ptr[rptr[m]] = 2 * rptr[m];
}

// Column keys col * u + t of the u distinct entries (row-major vertex ids).
__global__ void fg_col_keys_kernel(const int32_t* __restrict__ cidx, int64_t u, uint64_t* __restrict__ keys) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < u) keys[t] = (uint64_t)cidx[t] * (uint64_t)u + (uint64_t)t;
}

// Nets of the finegrain model: the row nets (vertex ranges of the row CSR)
// followed by the column nets.
__global__ void fg_nets_kernel(const int32_t* __restrict__ rptr, int32_t m, const int32_t* __restrict__ cptr,
                               const int32_t* __restrict__ cpins, int32_t n, int64_t u, int32_t* __restrict__ net_ptr,
                               int32_t* __restrict__ pins) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t <= m) net_ptr[t] = rptr[t];
  if (t < n) net_ptr[m + 1 + t] = (int32_t)u + cptr[t + 1];
  if (t < u) {
    pins[t] = (int32_t)t;
    pins[u + t] = cpins[t];
  }
}

vmo_status build_model(const vmo_csr* a, vmo_model model, vmo_hg_s* h, cudaStream_t s) {
  Scratch sc(s);
  bool ascending = false;
  VMO_TRY(validate_csr(a, &ascending, s, sc));
  const int32_t m = a->m, n = a->n;
  const int64_t nnz = a->nnz;
  h->model = model;
  h->m = m;
  h->n = n;
  if (model == VMO_SYMMETRIC && m != n) return invalid("symmetric model needs a square pattern");
  if (model == VMO_SYMMETRIC || model == VMO_BIPARTITE) {
    if ((model == VMO_SYMMETRIC ? (int64_t)m : (int64_t)m + n) > INT32_MAX / 2) return unsupported("too many vertices");
  }
  if (model == VMO_FINEGRAIN && (int64_t)m + n > INT32_MAX) return unsupported("too many nets");
  if (ascending && model >= VMO_SYMMETRIC && model <= VMO_FINEGRAIN && (model != VMO_BIPARTITE || 2 * nnz <= INT32_MAX)) {
    bool done = false;
    VMO_TRY(build_ascending(a, model, h, &done, s, sc));
    if (done) return VMO_OK;
  }
  if (model == VMO_SYMMETRIC || model == VMO_BIPARTITE) {
    int64_t K = (model == VMO_SYMMETRIC) ? m : (int64_t)m + n;
    h->k = (int32_t)K;
    uint64_t* keys;
    VMO_TRY(sc.alloc(&keys, (size_t)std::max<int64_t>(2 * nnz, 1)));
    uint64_t sentinel = (uint64_t)K * (uint64_t)K;
    if (nnz > 0) {
      launch(graph_keys_kernel, grid_for(nnz, 256), 256, 0, s, a->rowptr, a->colidx, m, nnz, model == VMO_BIPARTITE,
                                                           (uint64_t)K, sentinel, keys);
      VMO_LAUNCHED("graph_keys");
    }
    VMO_TRY(csr_from_keys(keys, 2 * nnz, K, K, h->adj_ptr, h->adj, &h->nadj, s, sc));
    // nets = edges u < v
    int64_t nadj = h->nadj;
    int32_t *flag, *pos, *tot;
    VMO_TRY(sc.alloc(&flag, (size_t)std::max<int64_t>(nadj, 1)));
    VMO_TRY(sc.alloc(&pos, (size_t)std::max<int64_t>(nadj, 1)));
    VMO_TRY(sc.alloc(&tot, 1));
    if (nadj > 0) {
      launch(forward_flags_kernel, grid_for(nadj, 256), 256, 0, s, h->adj_ptr.ptr, h->adj.ptr, h->k, nadj, flag);
      VMO_LAUNCHED("forward_flags");
    }
    VMO_TRY(scan_exclusive<int32_t>(flag, pos, nadj, tot, s, sc));
    int64_t ne = nadj / 2;
    h->l = ne;
    h->npins = 2 * ne;
    h->nvnets = nadj;
    VMO_TRY(h->net_ptr.resize((size_t)ne + 1));
    VMO_TRY(h->pins.resize((size_t)std::max<int64_t>(2 * ne, 1)));
    VMO_TRY(h->vnets.resize((size_t)std::max<int64_t>(nadj, 1)));
    VMO_TRY(h->vtx_ptr.resize((size_t)K + 1));
    VMO_CUDA(cudaMemcpyAsync(h->vtx_ptr.ptr, h->adj_ptr.ptr, (K + 1) * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    if (nadj > 0) {
      launch(emit_edges_kernel, grid_for(nadj, 256), 256, 0, s, h->adj_ptr.ptr, h->adj.ptr, h->k, nadj, flag, pos,
                                                            h->net_ptr.ptr, h->pins.ptr, h->vnets.ptr);
      VMO_LAUNCHED("emit_edges");
    }
    launch(net_ptr_last_kernel, 1, 1, 0, s, h->net_ptr.ptr, tot);
    VMO_LAUNCHED("net_ptr_last");
    VMO_CUDA(cudaStreamSynchronize(s));
    return VMO_OK;
  }
  if (model == VMO_ROWNET || model == VMO_COLNET) {
    uint64_t* keys;
    VMO_TRY(sc.alloc(&keys, (size_t)std::max<int64_t>(nnz, 1)));
    DevArray<int32_t>* rows_ptr = (model == VMO_ROWNET) ? &h->net_ptr : &h->vtx_ptr;
    DevArray<int32_t>* rows_idx = (model == VMO_ROWNET) ? &h->pins : &h->vnets;
    DevArray<int32_t>* cols_ptr = (model == VMO_ROWNET) ? &h->vtx_ptr : &h->net_ptr;
    DevArray<int32_t>* cols_idx = (model == VMO_ROWNET) ? &h->vnets : &h->pins;
    int64_t cnt_r = 0, cnt_c = 0;
    if (nnz > 0) {
      launch(pattern_keys_kernel, grid_for(nnz, 256), 256, 0, s, a->rowptr, a->colidx, m, n, nnz, 0, keys);
      VMO_LAUNCHED("pattern_keys");
    }
    VMO_TRY(csr_from_keys(keys, nnz, m, n, *rows_ptr, *rows_idx, &cnt_r, s, sc));
    if (nnz > 0) {
      launch(pattern_keys_kernel, grid_for(nnz, 256), 256, 0, s, a->rowptr, a->colidx, m, n, nnz, 1, keys);
      VMO_LAUNCHED("pattern_keys");
    }
    VMO_TRY(csr_from_keys(keys, nnz, n, m, *cols_ptr, *cols_idx, &cnt_c, s, sc));
    if (model == VMO_ROWNET) {
      h->k = n; h->l = m; h->npins = cnt_r; h->nvnets = cnt_c;
    } else {
      h->k = m; h->l = n; h->npins = cnt_c; h->nvnets = cnt_r;
    }
    VMO_CUDA(cudaStreamSynchronize(s));
    return VMO_OK;
  }
  if (model == VMO_FINEGRAIN) {
    uint64_t* keys;
    VMO_TRY(sc.alloc(&keys, (size_t)std::max<int64_t>(nnz, 1)));
    if (nnz > 0) {
      launch(pattern_keys_kernel, grid_for(nnz, 256), 256, 0, s, a->rowptr, a->colidx, m, n, nnz, 0, keys);
      VMO_LAUNCHED("pattern_keys");
    }
    DevArray<int32_t> rptr, cidx, cptr, cpins;
    int64_t u = 0, uc = 0;
    VMO_TRY(csr_from_keys(keys, nnz, m, n, rptr, cidx, &u, s, sc));
    if (2 * u > INT32_MAX) return unsupported("too many entries");
    h->k = (int32_t)u;
    h->l = (int64_t)m + n;
    h->npins = 2 * u;
    h->nvnets = 2 * u;
    VMO_TRY(h->vtx_ptr.resize((size_t)u + 1));
    VMO_TRY(h->vnets.resize((size_t)std::max<int64_t>(2 * u, 1)));
    VMO_TRY(h->net_ptr.resize((size_t)m + n + 1));
    VMO_TRY(h->pins.resize((size_t)std::max<int64_t>(2 * u, 1)));
    VMO_CUDA(cudaMemsetAsync(h->vtx_ptr.ptr, 0, sizeof(int32_t), s));
    if (m > 0) {
      launch(fg_vnets_kernel, grid_for(m, 256), 256, 0, s, rptr.ptr, cidx.ptr, m, h->vtx_ptr.ptr, h->vnets.ptr);
      VMO_LAUNCHED("fg_vnets");
    }
    uint64_t* ckeys;
    VMO_TRY(sc.alloc(&ckeys, (size_t)std::max<int64_t>(u, 1)));
    if (u > 0) {
      launch(fg_col_keys_kernel, grid_for(u, 256), 256, 0, s, cidx.ptr, u, ckeys);
      VMO_LAUNCHED("fg_col_keys");
    }
    VMO_TRY(csr_from_keys(ckeys, u, n, std::max<int64_t>(u, 1), cptr, cpins, &uc, s, sc));
    const int64_t span = std::max<int64_t>(std::max<int64_t>(u, (int64_t)m + 1), (int64_t)n);
    launch(fg_nets_kernel, grid_for(span, 256), 256, 0, s, rptr.ptr, m, cptr.ptr, cpins.ptr, n, u, h->net_ptr.ptr,
           h->pins.ptr);
    VMO_LAUNCHED("fg_nets");
    VMO_CUDA(cudaStreamSynchronize(s));
    return VMO_OK;
  }
  return invalid("unknown model");
}

// Finegrain layout from the bipartite one (Sec. 4.2): entry t at the mean of
// its row's and its column's points.
__global__ void fg_coords_kernel(const int32_t* __restrict__ vnets, int32_t k, const float4* __restrict__ xb,
                                 float4* __restrict__ xf) {
  int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= k) return;
  const float4 a = xb[vnets[2 * t]], b = xb[vnets[2 * t + 1]];
  xf[t] = make_float4(0.5f * (a.x + b.x), 0.5f * (a.y + b.y), 0.5f * (a.z + b.z), 0.5f * (a.w + b.w));
}

vmo_status finegrain_coords(const vmo_hg_s* h, const float* xb, float* xf, cudaStream_t s) {
  if (h->k > 0) {
    launch(fg_coords_kernel, grid_for(h->k, 256), 256, 0, s, h->vnets.ptr, h->k, (const float4*)xb, (float4*)xf);
    VMO_LAUNCHED("fg_coords");
  }
  VMO_CUDA(cudaStreamSynchronize(s));
  return VMO_OK;
}

vmo_status components(const vmo_hg_s* h, int32_t* labels, cudaStream_t s) {
  if (h->k == 0) return VMO_OK;
  Scratch sc(s);
  const bool graph = h->model == VMO_SYMMETRIC || h->model == VMO_BIPARTITE;
  const unsigned gv = grid_for(h->k, 256);
  launch(cc_init_kernel, gv, 256, 0, s, graph ? h->adj_ptr.ptr : (const int32_t*)nullptr, h->adj.ptr, labels, h->k);
  if (graph && h->l > 0) {
    launch(cc_compress_kernel, gv, 256, 0, s, labels, h->k);
    for (int stride = kCcSample; stride >= 1; stride /= 4) {
      launch(cc_neighbour_kernel, grid_for((h->k + stride - 1) / stride, 256), 256, 0, s, h->adj_ptr.ptr, h->adj.ptr,
             labels, h->k, stride);
      launch(cc_compress_kernel, gv, 256, 0, s, labels, h->k);
    }
    launch(cc_edges_kernel, grid_for(h->l, 256), 256, 0, s, (const int2*)h->pins.ptr, h->l, labels);
  } else if (!graph && h->npins > 1) {
    uint8_t* last;
    VMO_TRY(sc.alloc(&last, h->npins));
    VMO_CUDA(cudaMemsetAsync(last, 0, h->npins, s));
    if (h->l > 0) launch(cc_last_kernel, grid_for(h->l, 256), 256, 0, s, h->net_ptr.ptr, h->l, last);
    launch(cc_pins_kernel<false>, grid_for(h->npins, 256), 256, 0, s, h->pins.ptr, last, h->npins, labels);
    launch(cc_compress_kernel, gv, 256, 0, s, labels, h->k);
    launch(cc_pins_kernel<true>, grid_for(h->npins, 256), 256, 0, s, h->pins.ptr, last, h->npins, labels);
  }
  launch(cc_compress_kernel, gv, 256, 0, s, labels, h->k);
  VMO_LAUNCHED("components");
  return VMO_OK;
}

vmo_status cut_size(const vmo_hg_s* h, const int32_t* part, int32_t nparts, int64_t* cutnet, int64_t* lambda1,
                    cudaStream_t s) {
  if (nparts < 1) return invalid("cut_size: nparts < 1");
  if (!part && h->k > 0) return invalid("cut_size: part is null");
  Scratch sc(s);
  unsigned long long* acc;
  VMO_TRY(sc.alloc(&acc, 2));
  VMO_CUDA(cudaMemsetAsync(acc, 0, 16, s));
  if (h->l > 0) {
    launch(cut_kernel, grid_for(h->l * 32, 256), 256, 0, s, h->net_ptr.ptr, h->pins.ptr, h->l, part, nparts, acc);
    VMO_LAUNCHED("cut");
  }
  unsigned long long host[2];
  VMO_CUDA(cudaMemcpyAsync(host, acc, 16, cudaMemcpyDeviceToHost, s));
  VMO_CUDA(cudaStreamSynchronize(s));
  if (cutnet) *cutnet = (int64_t)host[0];
  if (lambda1) *lambda1 = (int64_t)host[1];
  return VMO_OK;
}

}  // namespace vmo
