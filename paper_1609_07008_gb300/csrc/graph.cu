// Graph construction: upload of the CSR adjacency (Sec. 2.1; the paper's
// bulk Tensor::write of the input, Sec. 6.1), validation on the device, the
// transposed adjacency A^T that Algorithm 2's products use, and the work-item
// lists of the level kernels.
//
// Validation (a graph that fails any check is rejected with INVALID):
//   rowptr[0] == 0, non-decreasing, rowptr[n] == nnz;
//   0 <= col < n, strictly increasing within a row (no duplicate arcs),
//   no self-loops, weights >= 1;
//   UNDIRECTED: every arc v->u has a reverse arc u->v of equal weight.
// Distances are int32, so (n-1)*max_w + max_w must stay below INT32_MAX
// (OVERFLOW otherwise): every finite distance and every candidate tau + w of
// the MFBF product then fits.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "internal.cuh"

namespace mfbc {

struct ValFlags {
  unsigned int bad_rowptr, bad_col, unsorted, self_loop, bad_weight, asym, non_unit;
  int wmax;
  unsigned long long looked_up;        // arcs whose reverse was searched for
};

__global__ void k_check_rowptr(int32_t n, int64_t nnz, const int64_t* __restrict__ rowptr, ValFlags* f) {
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v > n) return;
  int64_t r = rowptr[v];
  bool bad = (r < 0 || r > nnz) || (v == 0 && r != 0) || (v == n && r != nnz) ||
             (v < n && rowptr[v + 1] < r);
  if (bad) atomicOr(&f->bad_rowptr, 1u);
}

// First index in [lo, hi) of a non-decreasing array whose value is above x, or hi.
template <class T>
__device__ __forceinline__ int64_t first_above(const T* a, int64_t lo, int64_t hi, T x) {
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (a[mid] <= x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// The arcs' checks, CHECK_ARCS consecutive arcs to a block at a time, whatever
// rows they lie in.  (One warp per row left R-MAT 18's time to the warp that had
// the longest row: 1.75 ms of the 2.5 that creating the graph took.)
// An undirected arc v->u needs u->v.  Of the two, only the one that leaves the
// row with more arcs (ties: the higher vertex) looks the other up, in the shorter
// row.  Where all of them are found and they are half of the arcs, the arcs
// found, one for each, are the other half: no arc is left without its reverse.
// (Rows with repeated columns could break that count; they are flagged as
// unsorted, which is reported first.)
constexpr int CHECK_THREADS = 256, CHECK_ARCS = 1024;
__global__ void __launch_bounds__(CHECK_THREADS) k_check_arcs(int32_t n, int64_t nnz, const int64_t* __restrict__ rowptr,
                                                             const int32_t* __restrict__ col,
                                                             const int32_t* __restrict__ w, bool undirected, ValFlags* f) {
  __shared__ int64_t row[2];
  int wmax = 1;
  unsigned bc = 0, uns = 0, sl = 0, bw = 0, asy = 0, nu = 0, looked = 0;
  for (int64_t base = (int64_t)blockIdx.x * CHECK_ARCS; base < nnz; base += (int64_t)gridDim.x * CHECK_ARCS) {
    const int64_t last = min(base + CHECK_ARCS, nnz);
    __syncthreads();
    // the row of arc k is the last one that begins at or before k
    if (threadIdx.x < 2) row[threadIdx.x] = first_above(rowptr, 0, (int64_t)n, threadIdx.x ? last - 1 : base);
    __syncthreads();
    const int64_t r0 = row[0] - 1, r1 = row[1];
    for (int64_t k = base + threadIdx.x; k < last; k += CHECK_THREADS) {
      const int32_t c = col[k];
      if (c < 0 || c >= n) { bc = 1; continue; }
      const int32_t v = (int32_t)(first_above(rowptr, r0, r1, k) - 1);
      const int64_t beg = rowptr[v];
      if (c == v) sl = 1;
      if (k > beg && col[k - 1] >= c) uns = 1;
      int32_t wk = 1;
      if (w) {
        wk = w[k];
        if (wk < 1) { bw = 1; continue; }
        if (wk != 1) nu = 1;
        wmax = max(wmax, wk);
      }
      if (undirected) {
        const int64_t mine = rowptr[v + 1] - beg, lo = rowptr[c], hi = rowptr[c + 1];
        if (mine < hi - lo || (mine == hi - lo && v < c)) continue;
        looked++;
        const int64_t at = first_above(col, lo, hi, v) - 1;
        if (at < lo || col[at] != v || (w && w[at] != wk)) asy = 1;
      }
    }
  }
  if (bc) atomicOr(&f->bad_col, 1u);
  if (uns) atomicOr(&f->unsorted, 1u);
  if (sl) atomicOr(&f->self_loop, 1u);
  if (bw) atomicOr(&f->bad_weight, 1u);
  if (asy) atomicOr(&f->asym, 1u);
  nu = __any_sync(0xffffffffu, nu);
  looked = __reduce_add_sync(0xffffffffu, looked);
  wmax = __reduce_max_sync(0xffffffffu, wmax);
  if ((threadIdx.x & 31u) == 0u) {
    if (nu) atomicOr(&f->non_unit, 1u);
    if (w) atomicMax(&f->wmax, wmax);
    if (looked) atomicAdd(&f->looked_up, (unsigned long long)looked);
  }
}

template <class T>
static mfbc_status dev_alloc(DevGraph* g, T** p, size_t count, std::string* err) {
  *p = nullptr;
  if (count == 0) count = 1;
  cudaError_t e = cudaMalloc((void**)p, count * sizeof(T));
  if (e != cudaSuccess) {
    if (err) *err = std::string("cudaMalloc(graph): ") + cudaGetErrorString(e);
    cudaGetLastError();
    return MFBC_ERR_OOM;
  }
  g->owned.push_back((void*)*p);
  return MFBC_OK;
}

#define TRY(x)                  \
  do {                          \
    mfbc_status _s = (x);       \
    if (_s != MFBC_OK) return _s; \
  } while (0)

// Columns and, weighted, weights and packed arcs (see pack_arcs).  Up to
// JOINED_ARCS arcs they share one allocation, whose calls are what creating a
// small weighted graph spends most on; beyond, packed arcs are allocated only
// once the weights are known to differ from 1.
constexpr int64_t JOINED_ARCS = 1 << 22;
static mfbc_status alloc_arcs(DevGraph* g, bool weighted, int32_t** col, int32_t** w, uint32_t** pk, std::string* err) {
  const size_t nnz = (size_t)g->nnz, stride = (nnz + 63) & ~(size_t)63;
  if (!weighted || g->nnz > JOINED_ARCS) {
    TRY(dev_alloc(g, col, nnz, err));
    return weighted ? dev_alloc(g, w, nnz, err) : MFBC_OK;
  }
  TRY(dev_alloc(g, col, 3 * stride, err));
  *w = *col + stride;
  *pk = reinterpret_cast<uint32_t*>(*col + 2 * stride);
  return MFBC_OK;
}

// empty_rows: give every row without arcs one empty item.  The MFBr gather
// must visit DAG sinks too (their frontier value 1/sigma_bar is written by
// that visit); in an undirected graph a vertex without arcs can only be a
// source, so only directed graphs need it.
static mfbc_status build_items(DevGraph* g, const int64_t* rp, ItemList* L, bool empty_rows, cudaStream_t st,
                               std::string* err) {
  const int32_t n = g->n;
  if (rp[n] >= (1ll << 40)) { *err = "graphs with 2^40 or more arcs are not supported"; return MFBC_ERR_INVALID; }
  std::vector<int32_t> iv;
  std::vector<int64_t> ib;
  std::vector<int32_t> hub_of((size_t)n, -1), hubs;
  for (int32_t v = 0; v < n; v++) {
    const int64_t deg = rp[v + 1] - rp[v];
    if (deg > CHUNK) { hub_of[v] = (int32_t)hubs.size(); hubs.push_back(v); }
    // item metadata: first arc (bits 0..39), arc count (40..45), multi-item row (46)
    const int64_t multi = deg > CHUNK ? (1ll << 46) : 0;
    for (int64_t b = rp[v]; b < rp[v + 1]; b += CHUNK) {
      iv.push_back(v);
      ib.push_back(b | (std::min<int64_t>(CHUNK, rp[v + 1] - b) << 40) | multi);
    }
    if (deg == 0 && empty_rows) { iv.push_back(v); ib.push_back(rp[v]); }
  }
  L->count = (int64_t)iv.size();
  L->nhub = (int32_t)hubs.size();
  TRY(dev_alloc(g, &L->v, iv.size(), err));
  TRY(dev_alloc(g, &L->beg, ib.size(), err));
  TRY(dev_alloc(g, &L->hub_of, (size_t)n, err));
  TRY(dev_alloc(g, &L->hubs, hubs.size(), err));
  MFBC_CUDA_TRY(cudaMemcpyAsync(L->v, iv.data(), sizeof(int32_t) * iv.size(), cudaMemcpyHostToDevice, st), err);
  MFBC_CUDA_TRY(cudaMemcpyAsync(L->beg, ib.data(), sizeof(int64_t) * ib.size(), cudaMemcpyHostToDevice, st), err);
  MFBC_CUDA_TRY(cudaMemcpyAsync(L->hub_of, hub_of.data(), sizeof(int32_t) * (size_t)n, cudaMemcpyHostToDevice, st), err);
  if (!hubs.empty())
    MFBC_CUDA_TRY(cudaMemcpyAsync(L->hubs, hubs.data(), sizeof(int32_t) * hubs.size(), cudaMemcpyHostToDevice, st), err);
  // the host vectors die at return: finish the copies first
  MFBC_CUDA_TRY(cudaStreamSynchronize(st), err);
  return MFBC_OK;
}

// Order of the landmarks: by degree descending, then id.
struct HigherDegree {
  const int64_t* rp;
  bool operator()(int32_t a, int32_t b) const {
    const int64_t da = rp[a + 1] - rp[a], db = rp[b + 1] - rp[b];
    return da != db ? da > db : a < b;
  }
};

// Targets where the push products' candidates meet often enough for the
// hash accumulator to combine them in shared memory: vertices whose row in
// rp (in-arcs for MFBF targets, out-arcs for MFBr targets) holds at least
// max(16, 2 x the average degree) arcs.  One bit per vertex.
static int64_t hot_degree(const DevGraph* g) { return std::max<int64_t>(16, g->n ? 2 * g->nnz / g->n : 0); }
static mfbc_status upload_hot_targets(DevGraph* g, const int64_t* rp, uint32_t** out, cudaStream_t st,
                                      std::string* err) {
  const int32_t n = g->n;
  const int64_t thr = hot_degree(g);
  std::vector<uint32_t> bits(((size_t)n + 31) / 32 + 1, 0u);
  for (int32_t v = 0; v < n; v++)
    if (rp[(size_t)v + 1] - rp[v] >= thr) bits[(size_t)v >> 5] |= 1u << (v & 31);
  TRY(dev_alloc(g, out, bits.size(), err));
  MFBC_CUDA_TRY(cudaMemcpyAsync(*out, bits.data(), sizeof(uint32_t) * bits.size(), cudaMemcpyHostToDevice, st), err);
  MFBC_CUDA_TRY(cudaStreamSynchronize(st), err);
  return MFBC_OK;
}

// out[k] = col[k] | w[k] << bits
__global__ void k_pack_arcs(const int32_t* __restrict__ col, const int32_t* __restrict__ w, int64_t nnz, int bits,
                            uint32_t* __restrict__ out) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nnz; k += stride)
    out[k] = (uint32_t)col[k] | ((uint32_t)w[k] << bits);
}

// Column and weight of a weighted graph's arc in one word, for the source
// kernel (half the bytes and one load an arc).  They always fit: distances are
// int32, so n * w_max < 2^31, and with n > 2^(cb-1), w_max >= 2^(wb-1) the bits
// cb + wb are at most 32.  Graphs that no call runs by source (see source_graph)
// go without them, and so do graphs that the device has no room left for them:
// their calls run on the families' kernels.
static void pack_arcs(DevGraph* g, cudaStream_t st) {
  int cb = 1;
  while ((1ll << cb) < g->n) cb++;
  bool room = g->w && source_graph(*g);
  if (room && !g->pk) room = dev_alloc(g, &g->pk, (size_t)g->nnz, nullptr) == MFBC_OK;
  if (room && g->directed && !g->pk_t) {
    room = dev_alloc(g, &g->pk_t, (size_t)g->nnz, nullptr) == MFBC_OK;
    if (!room && g->nnz > JOINED_ARCS) {         // (the last allocation made: pk)
      cudaFree(g->pk);
      g->owned.pop_back();
    }
  }
  if (!room) {
    g->pk = g->pk_t = nullptr;
    return;
  }
  g->pk_bits = cb;
  const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((g->nnz + 255) / 256, 152 * 16));
  k_pack_arcs<<<blocks, 256, 0, st>>>(g->col, g->w, g->nnz, cb, g->pk);
  if (!g->directed) g->pk_t = g->pk;
  else k_pack_arcs<<<blocks, 256, 0, st>>>(g->col_t, g->w_t, g->nnz, cb, g->pk_t);
}

// About how many arcs the far ends of the graph are apart, from the breadth-first
// ball of up to BALL vertices around a vertex of high degree.  A ball that needs
// more levels than doubling would (with some room) grows like a power of its
// radius, as on lattices and road networks, and is carried on with that power;
// otherwise it grows by a factor a level.  Only api.cu's choice between kernels of
// equal results depends on it, and only for graphs of HOPS_ROWS vertices and more.
// It takes 10-20 us on the host, of the 400 and more of creating such a graph.  (A
// ball of 4096 would tell three-dimensional lattices from graphs of degree 2 that
// double, but takes ten times as long; one of 256 takes lattices of degree 8 for
// random graphs.)
constexpr int32_t HOPS_ROWS = 1 << 15;
static double estimate_hops(int32_t n, const int64_t* rp, const int32_t* col, const std::vector<int32_t>& roots) {
  constexpr int BALL = 512, SLOTS = 4 * BALL, ARCS = 1 << 13;
  const size_t target = BALL;
  std::vector<int32_t> slots, order;
  std::vector<size_t> size, best;      // vertices within l levels
  for (size_t r = 0; r < std::min<size_t>(roots.size(), 4); r++) {       // (a root's component may be small)
    slots.assign(SLOTS, -1);
    order.clear();
    size.clear();
    auto visit = [&](int32_t v) {
      if (v < 0 || v >= n) return;
      uint32_t h = ((uint32_t)v * 2654435769u) >> 21;                     // 11 bits
      while (slots[h] != v && slots[h] != -1) h = (h + 1) % SLOTS;
      if (slots[h] == v) return;
      slots[h] = v;
      order.push_back(v);
    };
    visit(roots[r]);
    size.push_back(1);
    int64_t arcs = 0;
    for (size_t at = 0; order.size() < target && arcs < ARCS && at < order.size();) {
      for (const size_t end = order.size(); at < end && order.size() < target && arcs < ARCS; at++)
        for (int64_t k = rp[order[at]]; k < rp[order[at] + 1] && order.size() < target && arcs < ARCS; k++, arcs++)
          visit(col[k]);
      if (order.size() > size.back()) size.push_back(order.size());
    }
    if (best.empty() || size.back() > best.back()) best = size;
    if (best.back() >= target || arcs >= ARCS) break;
  }
  if (best.size() < 2) return 1.0;
  const double L = (double)best.size() - 1.0, B = (double)best.back();
  if (best.back() < target) return L;                                     // the whole component
  if (L > 1.15 * std::log2(B)) {
    const size_t half = best.size() / 2;
    const double power = std::max(1.0, std::log(B / (double)best[half]) / std::log(L / (double)half));
    return L * std::pow(n / B, 1.0 / power);
  }
  const double deg = std::max(2.0, (double)rp[n] / n), inner = (double)best[best.size() - 2];
  return std::max(1.0, std::min(L, L - 1.0 + std::log(B / inner) / std::log(deg)) * std::log((double)n) / std::log(B));
}

// ------------------------------------------------- row structure on the device
// Work items, hub lists and the highest-degree vertices from the row pointers.
// On the host these are passes over the vertices with growing vectors and a
// selection by degree (R-MAT 20: 9.5 + 9.7 + 1.1 of the 21 ms that creating the
// graph took); here a scan over the rows gives every row its first item and hub
// index, and a degree histogram the degree that the HOT_ROWS highest reach.
// Creating a graph, host rows against device rows, in ms: R-MAT 10 0.24 / 0.35,
// 12 0.30 / 0.41, 13 (8192 vertices) 0.44 / 0.47, uniform 10 000 0.47 / 0.35,
// R-MAT 14 0.70 / 0.64, 16 1.54 / 1.08, 18 6.4 / 2.5, 20 20.7 / 10.6.  So graphs of
// up to HOST_ROWS vertices stay on the host.
constexpr int32_t HOST_ROWS = 1 << 13;
constexpr int ROWS_PER_BLOCK = 1024;
constexpr int DEG_BINS = 16384;        // degrees from DEG_BINS - 1 share the last bin
constexpr int TOP_ROWS = ORDER_LANDMARKS > HOT_ROWS ? ORDER_LANDMARKS : HOT_ROWS;
// Items and hubs share a 64-bit sum: with fewer arcs than this there are fewer
// than 2^33 items (nnz / 32 + n) and 2^31 hubs.
constexpr int64_t DEVICE_ARCS = 1ll << 36;

struct RowTotals {
  unsigned long long items, max_deg;
  unsigned int hubs, top;              // multi-item rows; vertices collected by k_top_rows
};

struct RowScratch {                    // freed when the graph is built
  RowTotals* tot;
  unsigned long long* bsum;            // per block of rows
  unsigned int* hist;                  // [DEG_BINS]
  int32_t* top;                        // [TOP_ROWS]
};

__device__ __forceinline__ uint32_t row_items(int64_t deg, bool empty_rows) {
  return deg ? (uint32_t)((deg + CHUNK - 1) / CHUNK) : (empty_rows ? 1u : 0u);
}

// Exclusive scan over a block of 1024 threads of x (64 bits); *total: the sum.
__device__ __forceinline__ unsigned long long block_scan(unsigned long long x, unsigned long long* total) {
  __shared__ unsigned long long w[32];
  const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  unsigned long long in = x;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, in, o);
    if ((int)lane >= o) in += y;
  }
  __syncthreads();                     // (the previous scan's sums are read)
  if (lane == 31) w[wid] = in;
  __syncthreads();
  unsigned long long before = 0, sum = 0;
  for (unsigned k = 0; k < 32; k++) {
    if (k < wid) before += w[k];
    sum += w[k];
  }
  *total = sum;
  return before + in - x;
}

// Items in bits 0..32, hubs above: both scans in one.
constexpr unsigned long long ONE_HUB = 1ull << 33;
__device__ __forceinline__ unsigned long long row_counts(const int64_t* rp, int64_t v, int32_t n, bool empty_rows,
                                                         int64_t* deg) {
  *deg = v < n ? rp[v + 1] - rp[v] : 0;
  if (v >= n) return 0ull;
  return row_items(*deg, empty_rows) + (*deg > CHUNK ? ONE_HUB : 0ull);
}

// Per block of rows: its items and hubs; over all: the largest degree and, with
// hist, the number of vertices of each degree.
__global__ void __launch_bounds__(ROWS_PER_BLOCK) k_row_stats(int32_t n, const int64_t* __restrict__ rp, bool empty_rows,
                                                             unsigned long long* bsum, unsigned int* hist,
                                                             RowTotals* tot) {
  __shared__ unsigned int low[1024];
  low[threadIdx.x] = 0u;
  const int64_t v = (int64_t)blockIdx.x * ROWS_PER_BLOCK + threadIdx.x;
  int64_t deg;
  unsigned long long total;
  block_scan(row_counts(rp, v, n, empty_rows, &deg), &total);
  if (threadIdx.x == 0) bsum[blockIdx.x] = total;
  unsigned long long m = (unsigned long long)deg;
  for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31u) == 0u && m) atomicMax(&tot->max_deg, m);
  if (!hist) return;
  if (v < n) {
    const int64_t b = deg < DEG_BINS ? deg : DEG_BINS - 1;
    if (b < 1024) atomicAdd(&low[b], 1u);
    else atomicAdd(&hist[b], 1u);
  }
  __syncthreads();
  if (low[threadIdx.x]) atomicAdd(&hist[threadIdx.x], low[threadIdx.x]);
}

// One block: the blocks' counts become their exclusive sums.
__global__ void __launch_bounds__(1024) k_scan_sums(unsigned long long* sum, int64_t count, RowTotals* tot) {
  unsigned long long run = 0;
  for (int64_t b = 0; b < count; b += 1024) {
    const int64_t i = b + threadIdx.x;
    const unsigned long long x = i < count ? sum[i] : 0ull;
    unsigned long long total;
    const unsigned long long ex = block_scan(x, &total);
    if (i < count) sum[i] = run + ex;
    run += total;
  }
  if (threadIdx.x == 0 && tot) {
    tot->items = run & (ONE_HUB - 1ull);
    tot->hubs = (unsigned int)(run / ONE_HUB);
  }
}

// The rows' items (first arc, arc count, multi-item bit) and hub indices.
__global__ void __launch_bounds__(ROWS_PER_BLOCK) k_fill_items(int32_t n, const int64_t* __restrict__ rp, bool empty_rows,
                                                              const unsigned long long* __restrict__ bsum,
                                                              int32_t* item_v, int64_t* item_beg, int32_t* hub_of,
                                                              int32_t* hubs) {
  const int64_t v = (int64_t)blockIdx.x * ROWS_PER_BLOCK + threadIdx.x;
  int64_t deg;
  unsigned long long total;
  const unsigned long long at = bsum[blockIdx.x] + block_scan(row_counts(rp, v, n, empty_rows, &deg), &total);
  if (v >= n) return;
  int64_t i = (int64_t)(at & (ONE_HUB - 1ull));
  const int32_t h = (int32_t)(at / ONE_HUB);
  const bool multi = deg > CHUNK;
  hub_of[v] = multi ? h : -1;
  if (multi) hubs[h] = (int32_t)v;
  const int64_t b = rp[v];
  if (deg == 0 && empty_rows) {
    item_v[i] = (int32_t)v;
    item_beg[i] = b;
  }
  for (int64_t k = 0; k < deg; k += CHUNK, i++) {
    item_v[i] = (int32_t)v;
    item_beg[i] = (b + k) | (min((int64_t)CHUNK, deg - k) << 40) | (multi ? 1ll << 46 : 0ll);
  }
}

// Vertices of degree above `above`, in any order, and the number of vertices of
// exactly that degree in each block of rows (for the ties, taken by lowest id).
__global__ void __launch_bounds__(ROWS_PER_BLOCK) k_top_rows(int32_t n, const int64_t* __restrict__ rp, int64_t above,
                                                            int32_t* list, unsigned int cap, RowTotals* tot,
                                                            unsigned long long* ties) {
  const int64_t v = (int64_t)blockIdx.x * ROWS_PER_BLOCK + threadIdx.x;
  const int64_t deg = v < n ? rp[v + 1] - rp[v] : -1;
  if (deg > above) {
    const unsigned int k = atomicAdd(&tot->top, 1u);
    if (k < cap) list[k] = (int32_t)v;
  }
  const unsigned int t = (unsigned int)__syncthreads_count(deg == above);
  if (threadIdx.x == 0) ties[blockIdx.x] = t;
}
// The `need` vertices of lowest id among those of degree `tie`.
__global__ void __launch_bounds__(ROWS_PER_BLOCK) k_tied_rows(int32_t n, const int64_t* __restrict__ rp, int64_t tie,
                                                             const unsigned long long* __restrict__ ties, unsigned int need,
                                                             int32_t* list) {
  if (ties[blockIdx.x] >= need) return;                  // (uniform)
  const int64_t v = (int64_t)blockIdx.x * ROWS_PER_BLOCK + threadIdx.x;
  const bool mine = v < n && rp[v + 1] - rp[v] == tie;
  unsigned long long total;
  const unsigned long long k = ties[blockIdx.x] + block_scan(mine ? 1ull : 0ull, &total);
  if (mine && k < need) list[k] = (int32_t)v;
}
// bits[v] = the row holds at least thr arcs
__global__ void k_row_bits(int32_t n, const int64_t* __restrict__ rp, int64_t thr, uint32_t* bits) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t m = __ballot_sync(0xffffffffu, v < n && rp[v + 1] - rp[v] >= thr);
  if ((threadIdx.x & 31u) == 0u && v < n) bits[v >> 5] = m;
}
__global__ void k_set_bits(const int32_t* __restrict__ list, int count, uint32_t* bits) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) atomicOr(&bits[list[i] >> 5], 1u << (list[i] & 31));
}

// Work items of the device rows rp, their largest degree, the hash accumulator's
// target bits and, with top, the TOP_ROWS highest-degree vertices (by degree
// descending, then id, isolated ones excluded; as a set, in any order).
static mfbc_status device_rows(DevGraph* g, const RowScratch& x, const int64_t* rp, const int64_t* h_rp, ItemList* L,
                               bool empty_rows, int64_t* max_deg, uint32_t** hot_targets, std::vector<int32_t>* top,
                               cudaStream_t st, std::string* err) {
  const int32_t n = g->n;
  const unsigned blocks = (unsigned)(((int64_t)n + ROWS_PER_BLOCK - 1) / ROWS_PER_BLOCK);
  MFBC_CUDA_TRY(cudaMemsetAsync(x.tot, 0, sizeof(RowTotals), st), err);
  if (top) MFBC_CUDA_TRY(cudaMemsetAsync(x.hist, 0, sizeof(unsigned int) * DEG_BINS, st), err);
  k_row_stats<<<blocks, ROWS_PER_BLOCK, 0, st>>>(n, rp, empty_rows, x.bsum, top ? x.hist : nullptr, x.tot);
  k_scan_sums<<<1, 1024, 0, st>>>(x.bsum, blocks, x.tot);
  RowTotals ht;
  std::vector<unsigned int> hist(top ? DEG_BINS : 0);
  MFBC_CUDA_TRY(cudaMemcpyAsync(&ht, x.tot, sizeof(ht), cudaMemcpyDeviceToHost, st), err);
  if (top)
    MFBC_CUDA_TRY(cudaMemcpyAsync(hist.data(), x.hist, sizeof(unsigned int) * DEG_BINS, cudaMemcpyDeviceToHost, st), err);
  MFBC_CUDA_TRY(cudaStreamSynchronize(st), err);
  *max_deg = (int64_t)ht.max_deg;
  L->count = (int64_t)ht.items;
  L->nhub = (int32_t)ht.hubs;
  TRY(dev_alloc(g, &L->v, (size_t)L->count, err));
  TRY(dev_alloc(g, &L->beg, (size_t)L->count, err));
  TRY(dev_alloc(g, &L->hub_of, (size_t)n, err));
  TRY(dev_alloc(g, &L->hubs, (size_t)L->nhub, err));
  TRY(dev_alloc(g, hot_targets, ((size_t)n + 31) / 32 + 1, err));
  k_fill_items<<<blocks, ROWS_PER_BLOCK, 0, st>>>(n, rp, empty_rows, x.bsum, L->v, L->beg, L->hub_of, L->hubs);
  k_row_bits<<<blocks, ROWS_PER_BLOCK, 0, st>>>(n, rp, hot_degree(g), *hot_targets);
  if (!top) return MFBC_OK;
  // the highest degree that at least TOP_ROWS vertices reach (1 where fewer have
  // arcs): every vertex above it and, of the ties, the lowest ids
  int64_t tie = DEG_BINS - 1, above = 0;
  for (; tie > 1 && above + hist[(size_t)tie] < TOP_ROWS; tie--) above += hist[(size_t)tie];
  if (tie == DEG_BINS - 1) {           // they all share the open last bin
    for (int32_t v = 0; v < n; v++)
      if (h_rp[v + 1] - h_rp[v] >= tie) top->push_back(v);
    std::nth_element(top->begin(), top->begin() + TOP_ROWS, top->end(), HigherDegree{h_rp});
    top->resize(TOP_ROWS);
    return MFBC_OK;
  }
  const unsigned need = (unsigned)std::min<int64_t>(TOP_ROWS - above, hist[(size_t)tie]);
  k_top_rows<<<blocks, ROWS_PER_BLOCK, 0, st>>>(n, rp, tie, x.top, TOP_ROWS, x.tot, x.bsum);
  k_scan_sums<<<1, 1024, 0, st>>>(x.bsum, blocks, nullptr);
  k_tied_rows<<<blocks, ROWS_PER_BLOCK, 0, st>>>(n, rp, tie, x.bsum, need, x.top + above);
  top->resize((size_t)above + need);
  MFBC_CUDA_TRY(cudaMemcpyAsync(top->data(), x.top, sizeof(int32_t) * top->size(), cudaMemcpyDeviceToHost, st), err);
  MFBC_CUDA_TRY(cudaStreamSynchronize(st), err);
  return MFBC_OK;
}

mfbc_status graph_build(int32_t n, int64_t nnz, const int64_t* h_rowptr, const int32_t* h_col,
                        const int32_t* h_w, uint32_t flags, cudaStream_t st, DevGraph* g,
                        std::string* err) {
  g->n = n;
  g->nnz = nnz;
  g->directed = !(flags & MFBC_UNDIRECTED);
  TRY(dev_alloc(g, &g->rowptr, (size_t)n + 1, err));
  TRY(alloc_arcs(g, h_w != nullptr, &g->col, &g->w, &g->pk, err));
  ValFlags* d_f;
  TRY(dev_alloc(g, &d_f, 1, err));
  MFBC_CUDA_TRY(cudaMemcpyAsync(g->rowptr, h_rowptr, sizeof(int64_t) * ((size_t)n + 1), cudaMemcpyHostToDevice, st), err);
  if (nnz) MFBC_CUDA_TRY(cudaMemcpyAsync(g->col, h_col, sizeof(int32_t) * (size_t)nnz, cudaMemcpyHostToDevice, st), err);
  if (h_w && nnz) MFBC_CUDA_TRY(cudaMemcpyAsync(g->w, h_w, sizeof(int32_t) * (size_t)nnz, cudaMemcpyHostToDevice, st), err);
  MFBC_CUDA_TRY(cudaMemsetAsync(d_f, 0, sizeof(ValFlags), st), err);
  k_check_rowptr<<<(unsigned)((n + 1 + 255) / 256), 256, 0, st>>>(n, nnz, g->rowptr, d_f);
  ValFlags f;
  MFBC_CUDA_TRY(cudaMemcpyAsync(&f, d_f, sizeof(f), cudaMemcpyDeviceToHost, st), err);
  MFBC_CUDA_TRY(cudaStreamSynchronize(st), err);
  if (f.bad_rowptr) { *err = "rowptr must start at 0, be non-decreasing and end at nnz"; return MFBC_ERR_INVALID; }
  if (nnz) {
    const unsigned blocks = (unsigned)std::min<int64_t>((nnz + CHECK_ARCS - 1) / CHECK_ARCS, 152 * 8);
    k_check_arcs<<<blocks, CHECK_THREADS, 0, st>>>(n, nnz, g->rowptr, g->col, g->w, !g->directed, d_f);
  }
  // What depends on the (already checked) row pointers alone; the result of the
  // arcs' check is read further down.
  const int64_t* rp = h_rowptr;
  const bool on_device = n > HOST_ROWS && nnz < DEVICE_ARCS;
  RowScratch x{};
  std::vector<int32_t> top;            // the TOP_ROWS highest out-degree vertices, isolated ones excluded
  if (on_device) {
    const size_t blocks = ((size_t)n + ROWS_PER_BLOCK - 1) / ROWS_PER_BLOCK;
    char* mem;
    TRY(dev_alloc(g, &mem, sizeof(RowTotals) + 8 * blocks + sizeof(unsigned int) * DEG_BINS + sizeof(int32_t) * TOP_ROWS,
                  err));
    x.tot = (RowTotals*)mem;
    x.bsum = (unsigned long long*)(x.tot + 1);
    x.hist = (unsigned int*)(x.bsum + blocks);
    x.top = (int32_t*)(x.hist + DEG_BINS);
    TRY(device_rows(g, x, g->rowptr, rp, &g->items_out, g->directed, &g->max_deg, &g->hot_out, &top, st, err));
  } else {
    top.reserve((size_t)n);
    for (int32_t v = 0; v < n; v++) {
      if (rp[v + 1] > rp[v]) top.push_back(v);
      g->max_deg = std::max<int64_t>(g->max_deg, rp[v + 1] - rp[v]);
    }
    if (top.size() > (size_t)TOP_ROWS) {
      std::nth_element(top.begin(), top.begin() + TOP_ROWS, top.end(), HigherDegree{rp});
      top.resize(TOP_ROWS);
    }
  }
  // landmarks for source ordering: the highest of them, in order; the HOT_ROWS
  // highest also mark the rows the level gathers ask the L2 to keep (their values
  // are read along most DAG arcs)
  static_assert(TOP_ROWS == HOT_ROWS, "the hot rows are all of top");
  const size_t nland = std::min<size_t>(top.size(), (size_t)ORDER_LANDMARKS);
  std::partial_sort(top.begin(), top.begin() + nland, top.end(), HigherDegree{rp});
  g->landmarks.assign(top.begin(), top.begin() + nland);
  const size_t hot_words = ((size_t)n + 31) / 32 + 1;
  std::vector<uint32_t> hot(on_device ? 0 : hot_words, 0u);
  TRY(dev_alloc(g, &g->hot, hot_words, err));
  if (on_device) {
    const int count = (int)top.size();
    MFBC_CUDA_TRY(cudaMemsetAsync(g->hot, 0, sizeof(uint32_t) * hot_words, st), err);
    if (count) {
      MFBC_CUDA_TRY(cudaMemcpyAsync(x.top, top.data(), sizeof(int32_t) * top.size(), cudaMemcpyHostToDevice, st), err);
      k_set_bits<<<(count + 255) / 256, 256, 0, st>>>(x.top, count, g->hot);
    }
  } else {
    for (int32_t v : top) hot[(size_t)v >> 5] |= 1u << (v & 31);
    MFBC_CUDA_TRY(cudaMemcpyAsync(g->hot, hot.data(), sizeof(uint32_t) * hot.size(), cudaMemcpyHostToDevice, st), err);
  }
  if (!g->directed) {
    g->max_in_deg = g->max_deg;
    if (!on_device) {
      TRY(build_items(g, rp, &g->items_out, false, st, err));      // (waits for the stream)
      TRY(upload_hot_targets(g, rp, &g->hot_out, st, err));
    }
    g->items_in = g->items_out;
    g->hot_in = g->hot_out;
  }
  // (on the host while the device works; the arcs are not known to be valid yet.
  // Rows of hundreds of arcs settle the choice without it.)
  if (h_w && n >= HOPS_ROWS && g->max_deg <= std::max<int64_t>(64, 4 * (nnz / n))) g->hops = estimate_hops(n, h_rowptr, h_col, g->landmarks);
  MFBC_CUDA_TRY(cudaMemcpyAsync(&f, d_f, sizeof(f), cudaMemcpyDeviceToHost, st), err);
  MFBC_CUDA_TRY(cudaStreamSynchronize(st), err);
  MFBC_CUDA_TRY(cudaGetLastError(), err);
  if (f.bad_col) { *err = "column index out of range [0, n)"; return MFBC_ERR_INVALID; }
  if (f.self_loop) { *err = "self-loops are not allowed"; return MFBC_ERR_INVALID; }
  if (f.unsorted) { *err = "rows must be sorted by column without duplicate arcs"; return MFBC_ERR_INVALID; }
  if (f.bad_weight) { *err = "weights must be integers >= 1"; return MFBC_ERR_INVALID; }
  if (f.asym || (!g->directed && 2 * f.looked_up != (unsigned long long)nnz)) { *err = "UNDIRECTED graph is not symmetric with symmetric weights"; return MFBC_ERR_INVALID; }
  g->wmax = h_w ? std::max(1, f.wmax) : 1;
  if ((int64_t)n * (int64_t)g->wmax >= (int64_t)INF) {
    *err = "(n-1)*max_w + max_w must be below 2^31-1 for int32 distances";
    return MFBC_ERR_OVERFLOW;
  }
  g->unit = !f.non_unit;
  if (g->unit) g->hops = 0.0;
  if (g->unit && g->w) { g->w = nullptr; g->pk = nullptr; }   // all ones: treat as unweighted (arrays still owned)
  if (g->directed) {
    // A^T by a stable counting sort on the host: rows of A^T are sorted by
    // source vertex, so the transposed graph is deterministic.
    std::vector<int64_t> rpt((size_t)n + 1, 0);
    for (int64_t k = 0; k < nnz; k++) rpt[(size_t)h_col[k] + 1]++;
    for (int32_t v = 0; v < n; v++) {
      g->max_in_deg = std::max<int64_t>(g->max_in_deg, rpt[v + 1]);
      rpt[v + 1] += rpt[v];
    }
    std::vector<int32_t> ct((size_t)nnz), wtv(g->w ? (size_t)nnz : 0);
    std::vector<int64_t> pos(rpt.begin(), rpt.end() - 1);
    for (int32_t v = 0; v < n; v++)
      for (int64_t k = rp[v]; k < rp[v + 1]; k++) {
        int64_t p = pos[h_col[k]]++;
        ct[p] = v;
        if (g->w) wtv[p] = h_w[k];
      }
    TRY(dev_alloc(g, &g->rowptr_t, (size_t)n + 1, err));
    TRY(alloc_arcs(g, g->w != nullptr, &g->col_t, &g->w_t, &g->pk_t, err));
    MFBC_CUDA_TRY(cudaMemcpyAsync(g->rowptr_t, rpt.data(), sizeof(int64_t) * rpt.size(), cudaMemcpyHostToDevice, st), err);
    if (nnz) MFBC_CUDA_TRY(cudaMemcpyAsync(g->col_t, ct.data(), sizeof(int32_t) * ct.size(), cudaMemcpyHostToDevice, st), err);
    if (g->w && nnz) MFBC_CUDA_TRY(cudaMemcpyAsync(g->w_t, wtv.data(), sizeof(int32_t) * wtv.size(), cudaMemcpyHostToDevice, st), err);
    MFBC_CUDA_TRY(cudaStreamSynchronize(st), err);
    if (on_device) {
      int64_t deg;                     // (max_in_deg is known)
      TRY(device_rows(g, x, g->rowptr_t, nullptr, &g->items_in, false, &deg, &g->hot_in, nullptr, st, err));
    } else {
      TRY(build_items(g, rpt.data(), &g->items_in, false, st, err));
      TRY(build_items(g, rp, &g->items_out, true, st, err));
      TRY(upload_hot_targets(g, rpt.data(), &g->hot_in, st, err));
      TRY(upload_hot_targets(g, rp, &g->hot_out, st, err));
    }
  } else {
    g->rowptr_t = g->rowptr;
    g->col_t = g->col;
    g->w_t = g->w;
  }
  pack_arcs(g, st);
  // (calls on the graph may come on any stream: everything is there at return)
  MFBC_CUDA_TRY(cudaStreamSynchronize(st), err);
  MFBC_CUDA_TRY(cudaGetLastError(), err);
  if (x.tot) {
    g->owned.erase(std::find(g->owned.begin(), g->owned.end(), (void*)x.tot));
    cudaFree(x.tot);
  }
  return MFBC_OK;
}

void graph_free(DevGraph* g) {
  for (void* p : g->owned) cudaFree(p);
  g->owned.clear();
}

}  // namespace mfbc
