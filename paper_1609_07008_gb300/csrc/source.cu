// Source path: MFBF (Algorithm 1) and MFBr (Algorithm 2) with one thread block
// per source, for weighted graphs (distance order) and small unit-weight
// graphs (breadth-first order).
//
// With integer weights >= 1, every (s,v) at distance d has all its shortest-
// path predecessors at distances < d and all its DAG successors at distances
// > d.  So a source can step over the distance values that occur, in
// increasing order:
//   * the vertices with tentative distance d are final (no later step can
//     offer less than d + 1);
//   * sigma_bar(s,v) = sum of sigma_bar(s,u) over in-neighbours u with
//     tau(s,u) + w(u,v) = d, all final (a pull: no multiplicity atomics);
//   * each pushes candidates d + w to its out-neighbours (atomicMin on the
//     tentative distance), which can only land on values d+1 .. d+w_max.
// MFBr walks the same steps backwards: zeta(s,v) is the sum over
// out-neighbours x with tau(s,x) = d + w(v,x) of zeta(s,x) + 1/sigma_bar(s,x)
// (Sec. 4.2.1), lambda(v) += zeta * sigma_bar (Algorithm 3), and the slot of
// (s,v) takes the value zeta + 1/sigma_bar.  Over unit weights the steps are
// the breadth-first levels.
//
// Why a block per source.  A step of one source is a few dozen to a few
// thousand vertices, and the sources of a batch are independent, so a step
// shared by all sources pays a launch (or a grid-wide wait) to synchronise
// work that never meets: a weighted 256^2 grid has about 2200 distance values
// and took 2 x 2200 launches of 14-18 us.  Here a step ends at the block's own
// barrier, sources advance at their own pace, and a block that finishes a
// source takes the next one from a queue; the GPU is filled by the sources in
// flight rather than by one step's vertices.
//
// What bounds it: the latency of a step (a chain of five or six dependent loads
// and one atomic, 2.5 us) where steps are narrow; the instructions of the walk
// over the arcs (44 a warp and 32 arcs) where they are wide.  MFBr does not
// walk the arcs again: MFBF records every DAG arc it finds, and MFBr replays
// them backwards, so that only zeta of a vertex is loaded in a step's chain.
//
// Measured, one call, against one launch per step for all sources (distance
// kernels), Bellman-Ford products (general kernels) and block groups that meet
// at a barrier after each level of 128 sources (small-graph kernel): weighted
// 256^2 grid, 512 sources 67.0 -> 11.9 ms; uniform n = 2^15, k = 512, weights
// <= 100, 300 sources 47.6 -> 8.7 ms (5 * 10^9 arcs, each read once: 2.3 TB/s
// of packed arcs out of the L2); directed R-MAT 16, weights <= 255, 2048
// sources 209 -> 48 ms; uniform n = 1024, k = 8, all sources 0.58 -> 0.21 ms;
// R-MAT 13, 500 sources 5.3 -> 1.0 ms; unit-weight 60^2 grid, 500 sources 111 ->
// 1.2 ms (its batches were too deep or their counts too large for the
// small-graph kernel and went to the general kernels).
//
// Tried and not kept: a chunk of a step's rows laid end to end and cut into
// equal spans for the block's warps (no hub rows, perfect balance): R-MAT 14
// unit weights 3.3 -> 5.2 ms, directed weighted R-MAT 16 47 -> 53 ms, weighted
// 256^2 grid 11.9 -> 11.5 ms; the rows' scan, two barriers and the per-arc row
// search cost more than the balance gives.  One block of 128-512 threads and
// several sources an SM with tau in global memory on power-law graphs (139 ms
// against 48): the sources' tau rows fall out of the L2.
#include <algorithm>
#include <type_traits>

#include "dfloat.cuh"
#include "internal.cuh"
#include "pieces.h"

namespace mfbc {

constexpr int SRC_HUB_ARCS = 512;      // longer rows are cut into pieces (pieces.h) for the block's warps
constexpr int SRC_HUBS = 64;           // such rows a step can list (more are walked by their own warp)
constexpr int SRC_BIG_ARCS = 64;       // rows from here on are walked whole, shorter ones as one flat list
constexpr int SRC_SMEM_MAX = 226 * 1024;
constexpr int SRC_SMS = 152;
__host__ __device__ constexpr size_t src_al16(size_t b) { return (b + 15) & ~size_t(15); }

// Where tau lives (DM): 32 bits in global memory; 32, 16 or, for unit weights, 8
// bits in shared memory (a source with a distance past 65534 or 254 is redone).
constexpr int DM_GLOBAL = 0, DM_SMEM32 = 1, DM_SMEM16 = 2, DM_SMEM8 = 3;
// How arcs are stored (AM): column only (unit weights), or column and weight
// packed in 32 bits.
constexpr int AM_UNIT = 0, AM_PACKED = 1;

// Fixed shared memory of a block; bucket counts, per-warp buffers and, when
// they fit, the distances and values follow it.
struct SrcShared {
  double hacc[SRC_HUBS];               // hub rows: the step's sum
  unsigned long long hcnt[SRC_HUBS];   // hub rows: the step's 64-bit count
  int32_t hv[SRC_HUBS];
  uint32_t hbase[SRC_HUBS];            // hub rows: first of the row's pieces
  unsigned long long nhub;             // hub rows listed << 40 | their pieces
  uint32_t tail;                       // vertices settled (weighted) or queued (unit weights)
  uint32_t dtail;                      // weighted: DAG arcs recorded
  uint32_t steps;                      // weighted: steps that settled vertices, and the
  uint32_t mark;                       //   tail after the last of them
  int32_t next;                        // next distance value, -1 none
  uint32_t src;                        // queue index of the block's source
  uint32_t redo;                       // the source needs the wide form (count >= 2^58 or distance > 65534)
};

struct SrcArgs {
  int32_t n;
  const int64_t* rp; const uint32_t* arc;    // A (out-arcs): columns, or packed columns and weights
  const int64_t* rpt; const uint32_t* arct;  // A^T (in-arcs)
  int cb;                              // packed arcs: column bits
  const int32_t* src;                  // sources
  const int32_t* row;                  // lambda row of each source, or null: row 0
  const int32_t* list;                 // indices of the sources to run, or null: all
  uint32_t nsrc;
  double* lambda;                      // rows of n; null: MFBF only
  uint32_t copy_mask;                  // row 0 stands for so many rows less one, one per block in turn
  int32_t* dist_out;                   // [nsrc][n], or null
  double* sigma_out;
  char* slots;                         // [gridDim.x] block states, slot_bytes apart
  size_t slot_bytes;
  size_t o_dist, o_cell, o_order, o_ring, o_dag;  // offsets within a slot
  uint32_t dcap;                       // DAG arcs a slot holds
  int B;                               // buckets (weighted): w_max + 1
  uint32_t scap, cap;                  // entries of a bucket in shared memory, and in all
  SrcCtl* ctl;
  int32_t* redo;                       // sources for the wide form
  unsigned long long* bytes;           // algorithmic bytes (counting runs), or null
};

// A vertex's reduction in one step, kept in 8 bytes of shared memory: FP64 sums
// (values, and path counts of weighted graphs: integers below 2^53, exact in any
// order) or exact 64-bit counts (unit weights).
// Counts of 2^58 send the source to the FP64 form, and every sum is looked at as
// it grows, not only when it is complete: a vertex with more than 64 predecessors
// of almost 2^58 paths each could pass 2^64 and come back small.  The counts that
// a batch of 32 arcs or a piece of a hub row adds are below 2^58 each, so no sum
// wraps before one of at least 2^58 was seen.
struct SumF64 {
  double s = 0.0;
  __device__ __forceinline__ static SumF64 of_count(uint64_t x) { return {__longlong_as_double((long long)x)}; }
  __device__ __forceinline__ static SumF64 of_value(uint64_t x) { return {__longlong_as_double((long long)x)}; }
  __device__ __forceinline__ static uint64_t one() { return (uint64_t)__double_as_longlong(1.0); }
  __device__ __forceinline__ uint64_t bits() const { return (uint64_t)__double_as_longlong(s); }
  __device__ __forceinline__ void add(const SumF64& o) { s += o.s; }
  __device__ __forceinline__ bool wide() const { return false; }
  __device__ __forceinline__ SumF64 up(int o) const { return {__shfl_up_sync(0xffffffffu, s, o)}; }
};
struct SumU64 {
  uint64_t i = 0;
  __device__ __forceinline__ static SumU64 of_count(uint64_t x) { return {x}; }
  __device__ __forceinline__ static uint64_t one() { return 1ull; }
  __device__ __forceinline__ uint64_t bits() const { return i; }
  __device__ __forceinline__ void add(const SumU64& o) { i += o.i; }
  __device__ __forceinline__ bool wide() const { return i >= (1ull << 58); }
  __device__ __forceinline__ SumU64 up(int o) const { return {__shfl_up_sync(0xffffffffu, i, o)}; }
};
template <int ILP>
struct SrcWarp {
  uint64_t acc[32];                    // sums of the batch's 32 vertices
  int32_t y[32 + 32 * ILP];            // tight arcs waiting for their values: far end
  uint8_t t[32 + 32 * ILP];            //   and the vertex's place in the batch
};

// sigma_bar (an integer or an FP64 count; in the pulled form of MFBr later the
// value zeta + 1/sigma_bar) and zeta of a vertex, side by side: a vertex costs
// one 32-byte sector of the L2 rather than one for each.
struct SrcCell {
  uint64_t sv;
  double z;
};

// The state of one source in one block.
template <int DM>
struct SrcState {
  using D = typename std::conditional<DM == DM_SMEM8, uint8_t,
                                      typename std::conditional<DM == DM_SMEM16, uint16_t, int32_t>::type>::type;
  static constexpr int32_t NONE = DM == DM_SMEM8 ? 0xff : DM == DM_SMEM16 ? 0xffff : INF;   // unreached
  SrcShared& sh;
  uint32_t* cnt;                       // bucket counts (weighted)
  int32_t* sring;                      // [B][scap] first entries of each bucket
  D* dist;                             // tau
  SrcCell* cell;                       // sigma_bar and zeta
  int32_t* order;                      // vertices in settling order
  uint2* off;                          // first entries of each step in order and dag
  int32_t* ring;                       // [B][cap - scap] further bucket entries (weighted)
  // DAG arcs as (vertex, predecessor), in step order; two 16-bit ids in a word
  // where every id fits (dag16)
  uint32_t* dag;
  bool dag16;
  __device__ __forceinline__ void put_arc(uint32_t at, int32_t v, int32_t u) {
    if (dag16) dag[at] = (uint32_t)v | ((uint32_t)u << 16);
    else reinterpret_cast<int2*>(dag)[at] = make_int2(v, u);
  }
  __device__ __forceinline__ int2 arc(uint32_t at) const {
    if (!dag16) return reinterpret_cast<const int2*>(dag)[at];
    const uint32_t x = dag[at];
    return make_int2((int32_t)(x & 0xffffu), (int32_t)(x >> 16));
  }
  __device__ __forceinline__ int32_t tau(int32_t v) const {
    const int32_t x = (int32_t)dist[v];
    return x == NONE ? INF : x;
  }
  // unit weights: gives v the level l unless it has one; true for the caller
  // that did.  Every caller of a step offers the same level, so clearing the
  // bits that l lacks from an unreached entry (all ones) sets it once.
  __device__ __forceinline__ bool claim(int32_t v, int32_t l) {
    if constexpr (DM == DM_SMEM8 || DM == DM_SMEM16) {
      constexpr int per = 4 / (int)sizeof(D);
      uint32_t* word = reinterpret_cast<uint32_t*>(dist) + v / per;
      const int shift = (v % per) * 8 * (int)sizeof(D);
      const uint32_t old = atomicAnd(word, ~((uint32_t)(NONE ^ l) << shift));
      return ((old >> shift) & (uint32_t)NONE) == (uint32_t)NONE;
    } else {
      return atomicMin(&dist[v], l) > l;
    }
  }
  // lowers tau(v) to cand; true for the caller that did
  __device__ __forceinline__ bool lower(int32_t v, int32_t cand) {
    if constexpr (DM == DM_SMEM16) {
      unsigned short* p = reinterpret_cast<unsigned short*>(&dist[v]);
      unsigned short old = *reinterpret_cast<volatile unsigned short*>(p);
      while ((int32_t)old > cand) {
        const unsigned short seen = atomicCAS(p, old, (unsigned short)cand);
        if (seen == old) return true;
        old = seen;
      }
      return false;
    } else if constexpr (DM == DM_SMEM8) {
      return false;                    // unit weights only: see claim
    } else {
      return atomicMin(&dist[v], cand) > cand;
    }
  }
};

// Sums the list's first 32 entries (qn of them when fewer) into the batch's
// accumulators.  Entries are grouped by vertex.
template <class Sum, bool COUNT, int ILP, class S>
__device__ __forceinline__ void src_flush(const SrcArgs& a, SrcWarp<ILP>& wb, S& st, int q0, int qn, int32_t mv) {
  const unsigned lane = lane_id();
  const bool has = (int)lane < qn;
  const int t = has ? (int)wb.t[q0 + lane] : 64;
  Sum x;
  const int32_t y = has ? wb.y[q0 + lane] : 0;
  if (COUNT) {                         // MFBF: the DAG arc, for MFBr
    uint32_t at = 0;
    if (lane == 0) at = atomicAdd(&st.sh.dtail, (uint32_t)qn);
    at = __shfl_sync(0xffffffffu, at, 0) + lane;
    const int32_t v = __shfl_sync(0xffffffffu, mv, t & 31);
    if (has && at < a.dcap) st.put_arc(at, v, y);
  }
  if (has) {
    const uint64_t b = st.cell[y].sv;
    if constexpr (COUNT) x = Sum::of_count(b);
    else x = Sum::of_value(b);
  }
  // sum of each run of one vertex, on the run's last lane, in as many steps as
  // the longest run needs
  const int tp = __shfl_up_sync(0xffffffffu, t, 1);
  const uint32_t heads = __ballot_sync(0xffffffffu, lane == 0 || tp != t) | 1u;
  const int back = (int)lane - (31 - __clz(heads & (0xffffffffu >> (31u - lane))));   // lanes to the run's first
  const int longest = (int)__reduce_max_sync(0xffffffffu, has ? (unsigned)back : 0u);
  for (int o = 1; o <= longest; o <<= 1) {
    const Sum x2 = x.up(o);
    if (back >= o) x.add(x2);
  }
  if (has && ((int)lane == qn - 1 || ((heads >> (lane + 1)) & 1u))) {
    Sum sum;
    if constexpr (COUNT) sum = Sum::of_count(wb.acc[t]);
    else sum = Sum::of_value(wb.acc[t]);
    sum.add(x);
    wb.acc[t] = sum.bits();
    if (sum.wide()) st.sh.redo = 1u;
  }
  __syncwarp();
}

// One round of a warp's walk: 32 * ILP arcs.
template <int ILP>
struct SrcRound {
  uint32_t p[ILP];                     // the arcs' words
  uint32_t t;                          // their rows' places in the batch, 8 bits each
  __device__ __forceinline__ int row(int r) const { return (int)((t >> (8 * r)) & 31u); }
};

// The rows of a batch: lane i holds row i (first arc, length; 0 when it has
// none to walk).  Rows of SRC_BIG_ARCS arcs and more are walked one after the
// other by the whole warp, the others as one flat list of arcs found by a
// search over the lengths' prefix sums, so that short rows still fill the
// lanes.  f(round, left) is called by the whole warp; lane l's arc r is there
// when 32 r + l < left (left is a constant for whole rounds of big rows).
template <int ILP, class F>
__device__ __forceinline__ void src_walk(const uint32_t* __restrict__ arc, int64_t beg, int32_t len, F f) {
  const unsigned lane = lane_id();
  SrcRound<ILP> x;
  uint32_t big = __ballot_sync(0xffffffffu, len >= SRC_BIG_ARCS);
  while (big) {
    const int t = __ffs(big) - 1;
    big &= big - 1;
    const uint32_t* a0 = arc + __shfl_sync(0xffffffffu, beg, t) + lane;
    const int32_t n = __shfl_sync(0xffffffffu, len, t);
    x.t = (uint32_t)t * 0x01010101u;
    int32_t k = 0;
    for (; k + 32 * ILP <= n; k += 32 * ILP) {
#pragma unroll
      for (int r = 0; r < ILP; r++) x.p[r] = __ldg(a0 + k + 32 * r);
      f(x, std::integral_constant<int, 32 * ILP>());
    }
    if (k < n) {
#pragma unroll
      for (int r = 0; r < ILP; r++) x.p[r] = k + 32 * r + (int32_t)lane < n ? __ldg(a0 + k + 32 * r) : 0u;
      f(x, n - k);
    }
  }
  const int32_t sl = len < SRC_BIG_ARCS ? len : 0;
  int32_t incl = sl;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t z = __shfl_up_sync(0xffffffffu, incl, o);
    if ((int)lane >= o) incl += z;
  }
  const int32_t excl = incl - sl;
  const int32_t T = __shfl_sync(0xffffffffu, incl, 31);
  for (int32_t p0 = 0; p0 < T; p0 += 32 * ILP) {
    x.t = 0u;
#pragma unroll
    for (int r = 0; r < ILP; r++) {
      const int32_t p = p0 + 32 * r + (int32_t)lane;
      x.p[r] = 0u;
      if (p0 + 32 * r >= T) continue;                    // (uniform)
      int t = 0;
#pragma unroll
      for (int step = 16; step; step >>= 1)              // the last row that starts at or before p
        if (__shfl_sync(0xffffffffu, excl, t + step) <= p) t += step;
      const int32_t e = __shfl_sync(0xffffffffu, excl, t);
      const int64_t b = __shfl_sync(0xffffffffu, beg, t);
      if (p < T) x.p[r] = __ldg(arc + (b + (p - e)));
      x.t |= (uint32_t)t << (8 * r);
    }
    f(x, T - p0);
  }
}

// A kernel block's shared context of one warp.
template <bool UNIT, int DM, int AM, int ILP>
struct SrcCtx {
  const SrcArgs& a;
  SrcState<DM>& st;
  SrcWarp<ILP>& wb;
  int qn;                              // tight arcs listed
  int32_t mv;                          // this lane's vertex of the batch
  unsigned long long nbytes;

  __device__ __forceinline__ int32_t head(uint32_t p) const {
    return (int32_t)(AM == AM_UNIT ? p : p & ((1u << a.cb) - 1u));
  }
  __device__ __forceinline__ int32_t weight(uint32_t p) const { return AM == AM_UNIT ? 1 : (int32_t)(p >> a.cb); }
  template <class Sum, bool COUNT>
  __device__ __forceinline__ void drain(bool all) {
    if (qn < 32 && !(all && qn)) return;
    __syncwarp();
    int q = 0;
    while (qn - q >= 32) { src_flush<Sum, COUNT>(a, wb, st, q, 32, mv); q += 32; }
    if (all) {
      if (qn - q) src_flush<Sum, COUNT>(a, wb, st, q, qn - q, mv);
      qn = 0;
      return;
    }
    const unsigned lane = lane_id();
    int32_t y = 0;
    uint8_t t = 0;
    if ((int)lane < qn - q) { y = wb.y[q + lane]; t = wb.t[q + lane]; }
    __syncwarp();
    if ((int)lane < qn - q) { wb.y[lane] = y; wb.t[lane] = t; }
    qn -= q;
    __syncwarp();
  }
  __device__ __forceinline__ void list(bool tight, int32_t y, int t) {
    const uint32_t m = __ballot_sync(0xffffffffu, tight);
    if (!m) return;
    if (tight) {
      const int at = qn + __popc(m & ((1u << lane_id()) - 1u));
      wb.y[at] = y;
      wb.t[at] = (uint8_t)t;
    }
    qn += __popc(m);
    if (a.bytes && lane_id() == 0) nbytes += 8ull * __popc(m);
  }
  // Offer cand to y (tentative distance dy): the lane that improves it queues
  // y.  A vertex enters a bucket at most once, as its distance only falls.
  // Entries past the bucket's room are not stored: the count tells the step to
  // look through all distances instead.
  __device__ __forceinline__ void offer(int32_t y, int32_t w, int32_t cand, int slot) {
    if (UNIT) {
      if (st.claim(y, cand)) st.order[atomicAdd(&st.sh.tail, 1u)] = y;
    } else if (st.lower(y, cand)) {
      int b = slot + w;
      if (b >= a.B) b -= a.B;
      const uint32_t at = atomicAdd(&st.cnt[b], 1u);
      if (at < a.scap) st.sring[(size_t)b * a.scap + at] = y;
      else if (at < a.cap) st.ring[(size_t)b * (a.cap - a.scap) + (at - a.scap)] = y;
    }
  }
  // MFBF rows of vertices settled at distance d: PULL lists the tight in-arcs,
  // PUSH offers d + w along the out-arcs; an undirected row serves both.
  template <bool PULL, bool PUSH, class Sum>
  __device__ __forceinline__ void fwd(const uint32_t* arc, int64_t beg, int32_t len, int32_t d, int slot) {
    if (a.bytes) nbytes += 8ull * (unsigned long long)len;
    src_walk<ILP>(arc, beg, len, [&](const SrcRound<ILP>& x, auto left) {
      int32_t dy[ILP];
      bool tight = false, nearer = false;
#pragma unroll
      for (int r = 0; r < ILP; r++) {                   // -2: neither tight nor improved
        dy[r] = 32 * r + (int)lane_id() < left ? (int32_t)st.dist[head(x.p[r])] : -2;
        tight |= dy[r] + weight(x.p[r]) == d;           // (unreached entries pass no test, see redo)
        nearer |= d + weight(x.p[r]) < dy[r];
      }
      if (PULL && __any_sync(0xffffffffu, tight)) {
#pragma unroll
        for (int r = 0; r < ILP; r++) list(dy[r] + weight(x.p[r]) == d, head(x.p[r]), x.row(r));
      }
      if (PUSH && nearer) {
#pragma unroll
        for (int r = 0; r < ILP; r++)
          if (d + weight(x.p[r]) < dy[r]) offer(head(x.p[r]), weight(x.p[r]), d + weight(x.p[r]), slot);
      }
      if (PULL) {
        __syncwarp();
        drain<Sum, true>(false);
      }
    });
  }
  // MFBr rows: this lane's vertex is at distance d.
  template <class Sum>
  __device__ __forceinline__ void bwd(int64_t beg, int32_t len, int32_t d) {
    if (a.bytes) nbytes += 8ull * (unsigned long long)len;
    src_walk<ILP>(a.arc, beg, len, [&](const SrcRound<ILP>& x, auto left) {
      int32_t dy[ILP];
#pragma unroll
      for (int r = 0; r < ILP; r++) dy[r] = 32 * r + (int)lane_id() < left ? st.tau(head(x.p[r])) : -1;
#pragma unroll
      for (int r = 0; r < ILP; r++) {
        const int32_t dv = __shfl_sync(0xffffffffu, d, x.row(r));
        list(dy[r] == dv + weight(x.p[r]), head(x.p[r]), x.row(r));
      }
      drain<Sum, false>(false);
    });
  }
};

// sigma_bar as FP64.
template <bool UNIT>
__device__ __forceinline__ double src_sigma(uint64_t sv) {
  return UNIT ? (double)sv : __longlong_as_double((long long)sv);
}
// sigma_bar of a settled vertex: stored beside a zeta of 0, and checked against
// 2^53 (FP64 output inexact).
__device__ __forceinline__ void src_put(SrcCell* c, uint64_t sv) {
  *reinterpret_cast<ulonglong2*>(c) = make_ulonglong2(sv, 0ull);
}
template <class S>
__device__ __forceinline__ void src_put_count(const SrcArgs& a, S& st, int32_t v, const SumF64& x) {
  src_put(&st.cell[v], x.bits());
  if (x.s >= 9007199254740992.0) atomicOr(&a.ctl->flags, FLAG_SIGMA_INEXACT);
}
template <class S>
__device__ __forceinline__ void src_put_count(const SrcArgs& a, S& st, int32_t v, const SumU64& x) {
  src_put(&st.cell[v], x.i);
  if (x.i >= (1ull << 53)) atomicOr(&a.ctl->flags, FLAG_SIGMA_INEXACT);
}
// zeta of a vertex (pulled form): its lambda term, and the value zeta +
// 1/sigma_bar in the place of the count.
template <bool UNIT>
__device__ __forceinline__ void src_put_value(SrcCell* c, double* lam, const SumF64& x) {
  const double sg = src_sigma<UNIT>(c->sv);
  if (x.s != 0.0) atomicAdd(lam, x.s * sg);
  c->sv = (uint64_t)__double_as_longlong(x.s + 1.0 / sg);
}

// Hub rows: a warp's share of the row's sum joins the total; the total read back.
__device__ __forceinline__ void src_hub_add(SrcShared& sh, int h, const SumF64& x) { atomicAdd(&sh.hacc[h], x.s); }
__device__ __forceinline__ void src_hub_add(SrcShared& sh, int h, SumU64 x) {
  x.add(SumU64{atomicAdd(&sh.hcnt[h], (unsigned long long)x.i)});
  if (x.wide()) sh.redo = 1u;
}
__device__ __forceinline__ void src_hub_get(const SrcShared& sh, int h, SumF64& x) { x.s = sh.hacc[h]; }
__device__ __forceinline__ void src_hub_get(const SrcShared& sh, int h, SumU64& x) { x.i = sh.hcnt[h]; }
// Lists v as a hub row of the step, cut into `pieces`; false when the list is
// full.  One atomic gives the place and the first piece, so both grow together.
__device__ __forceinline__ bool src_list_hub(SrcShared& sh, int32_t v, uint32_t pieces) {
  const unsigned long long o = atomicAdd(&sh.nhub, (1ull << 40) | pieces);
  const uint32_t h = (uint32_t)(o >> 40);
  if (h >= SRC_HUBS) return false;
  sh.hv[h] = v;
  sh.hbase[h] = (uint32_t)o;
  sh.hacc[h] = 0.0;
  sh.hcnt[h] = 0ull;
  return true;
}
// The hub row that piece p belongs to: the last of the nh listed rows whose
// first piece is at most p (whole warp).
__device__ __forceinline__ uint32_t src_piece_row(const SrcShared& sh, uint32_t nh, uint32_t p) {
  const unsigned lane = lane_id();
  uint32_t h = (uint32_t)__popc(__ballot_sync(0xffffffffu, lane < nh && sh.hbase[lane] <= p));
  if (nh > 32) h += (uint32_t)__popc(__ballot_sync(0xffffffffu, lane + 32 < nh && sh.hbase[lane + 32] <= p));
  return h - 1u;
}

// Items a warp takes at a time: 32, or fewer (a power of two) when the step
// is too short to give every warp that many.
__device__ __forceinline__ uint32_t src_batch(uint32_t items, int nwarp) {
  uint32_t bs = 32;
  while (bs > 4 && bs * (uint32_t)nwarp >= 2 * items) bs >>= 1;
  return bs;
}

// UNIT: unit weights by levels, 64-bit counts; otherwise integer weights (or
// none, AM_UNIT) by distance, FP64 counts.  SYM: undirected.
template <bool UNIT, int DM, int AM, bool SYM>
__global__ void __launch_bounds__(1024) k_src_bc(SrcArgs a) {
  constexpr int ILP = 4;
  using Cnt = typename std::conditional<UNIT, SumU64, SumF64>::type;
  using Val = SumF64;
  using D = typename SrcState<DM>::D;
  extern __shared__ __align__(16) unsigned char src_raw[];
  SrcShared& sh = *reinterpret_cast<SrcShared*>(src_raw);
  char* slot_mem = a.slots + (size_t)blockIdx.x * a.slot_bytes;
  const int wid = (int)threadIdx.x >> 5, nwarp = (int)blockDim.x >> 5;
  const size_t n8 = ((size_t)a.n + 15) & ~size_t(15);
  unsigned char* sp = src_raw + src_al16(sizeof(SrcShared));
  SrcWarp<ILP>& wb = reinterpret_cast<SrcWarp<ILP>*>(sp)[wid];
  sp += src_al16(sizeof(SrcWarp<ILP>) * nwarp);
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(sp);
  if (!UNIT) sp += src_al16((size_t)a.B * 4);
  int32_t* s_ring = reinterpret_cast<int32_t*>(sp);
  if (!UNIT) sp += src_al16((size_t)a.B * a.scap * 4);
  SrcState<DM> st{sh, s_cnt, s_ring,
                  DM != DM_GLOBAL ? reinterpret_cast<D*>(sp) : reinterpret_cast<D*>(slot_mem + a.o_dist),
                  reinterpret_cast<SrcCell*>(slot_mem + a.o_cell),
                  reinterpret_cast<int32_t*>(slot_mem + a.o_order),
                  reinterpret_cast<uint2*>(slot_mem + a.o_order + 4 * n8),
                  reinterpret_cast<int32_t*>(slot_mem + a.o_ring),
                  reinterpret_cast<uint32_t*>(slot_mem + a.o_dag), a.n <= 65536};
  SrcCtx<UNIT, DM, AM, ILP> cx{a, st, wb, 0, 0, 0ull};
  const unsigned lane = lane_id();
  const uint32_t lt = (1u << lane) - 1u;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      sh.src = atomicAdd(&a.ctl->head, 1u);
      sh.nhub = 0ull;
      sh.redo = 0u;
      sh.tail = UNIT ? 1u : 0u;
      sh.steps = sh.mark = sh.dtail = 0u;
    }
    __syncthreads();
    if (sh.src >= a.nsrc) break;
    const uint32_t si = a.list ? (uint32_t)a.list[sh.src] : sh.src;
    const int32_t s = a.src[si];
    if (s < 0 || s >= a.n) {                            // the caller refuses the call; nothing is indexed with s
      if (threadIdx.x == 0) atomicOr(&a.ctl->flags, FLAG_BAD_SOURCE);
      continue;
    }
    if (DM == DM_SMEM16 || DM == DM_SMEM8) {
      for (uint32_t i = threadIdx.x; i < (uint32_t)(n8 * sizeof(D) / 16); i += blockDim.x)
        reinterpret_cast<uint4*>(st.dist)[i] = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
    } else {
      for (int32_t v = (int32_t)threadIdx.x; v < a.n; v += (int32_t)blockDim.x) st.dist[v] = (D)INF;
    }
    if (!UNIT)
      for (int b = (int)threadIdx.x; b < a.B; b += (int)blockDim.x) st.cnt[b] = 0u;
    __syncthreads();
    if (threadIdx.x == 0) {
      st.dist[s] = 0;
      st.off[0] = make_uint2(0u, 0u);
      if (UNIT) st.order[0] = s;
      else {
        st.cnt[0] = 1u;
        if (a.scap) st.sring[0] = s;
        else st.ring[0] = s;
      }
    }
    __syncthreads();

    // ---- MFBF: one step per distance value
    int32_t d = 0;
    int slot = 0;
    uint32_t k = 0;                                     // steps done
    uint32_t q0 = 0, q1 = 1;                            // unit weights: the level's part of the queue
    bool redo = false;
    for (;;) {
      const uint32_t m = UNIT ? q1 - q0 : st.cnt[slot];
      const bool scan = !UNIT && m > a.cap;             // entries were dropped: look through every vertex
      const uint32_t items = scan ? (uint32_t)a.n : m;
      const uint32_t bs = src_batch(items, nwarp);
      bool hub = false;
      for (uint32_t i0 = (uint32_t)wid * bs; i0 < items; i0 += (uint32_t)nwarp * bs) {
        const uint32_t i = i0 + lane;
        bool on = lane < bs && i < items;
        int32_t v = 0;
        if (on) {
          if (UNIT) v = st.order[q0 + i];
          else if (scan) v = (int32_t)i;
          else v = i < a.scap ? st.sring[(size_t)slot * a.scap + i]
                              : st.ring[(size_t)slot * (a.cap - a.scap) + (i - a.scap)];
        }
        int64_t b = 0, bt = 0;
        int32_t len = 0, lent = 0;
        if (on && !(scan && st.tau(v) != d)) {          // (a row's ends are loaded beside its tau)
          const int64_t e = __ldg(&a.rp[v + 1]);
          b = __ldg(&a.rp[v]);
          int64_t et = 0;
          if (!SYM) { bt = __ldg(&a.rpt[v]); et = __ldg(&a.rpt[v + 1]); }
          if (!UNIT) on = st.tau(v) == d;               // otherwise improved since it was queued
          if (on) {
            len = (int32_t)(e - b);
            if (!SYM) lent = (int32_t)(et - bt);
          }
        } else {
          on = false;
        }
        const uint32_t mm = __ballot_sync(0xffffffffu, on);
        if (!mm) continue;
        if (!UNIT) {
          uint32_t at = 0;
          if (lane == 0) at = atomicAdd(&sh.tail, (uint32_t)__popc(mm));
          at = __shfl_sync(0xffffffffu, at, 0) + __popc(mm & lt);
          if (on) st.order[at] = v;
        }
        bool mine = on;                                 // rows this warp walks and finishes
        if (on && (len > SRC_HUB_ARCS || lent > SRC_HUB_ARCS) &&
            src_list_hub(sh, v, src_pieces(len) + src_pieces(lent))) {
          hub = true;
          mine = false;
          len = lent = 0;
        }
        wb.acc[lane] = 0ull;
        cx.mv = v;
        __syncwarp();
        if (SYM) {
          cx.template fwd<true, true, Cnt>(a.arc, b, len, d, slot);
        } else {
          cx.template fwd<true, false, Cnt>(a.arct, bt, lent, d, slot);
          cx.template fwd<false, true, Cnt>(a.arc, b, len, d, slot);
        }
        cx.template drain<Cnt, true>(true);
        __syncwarp();
        if (mine) src_put_count(a, st, v, Cnt::of_count(d == 0 ? Cnt::one() : wb.acc[lane]));
        __syncwarp();
      }
      const bool hubs = __syncthreads_or(hub);          // the same answer for every thread
      if (hubs) {
        const uint32_t nh = min((uint32_t)(sh.nhub >> 40), (uint32_t)SRC_HUBS), np = (uint32_t)sh.nhub;
        for (uint32_t p = (uint32_t)wid; p < np; p += (uint32_t)nwarp) {
          const uint32_t h = src_piece_row(sh, nh, p);
          const int32_t v = sh.hv[h];
          const int64_t b = __ldg(&a.rp[v]);
          const int32_t len = (int32_t)(__ldg(&a.rp[v + 1]) - b);
          int64_t bt = 0;
          int32_t lent = 0;
          if (!SYM) {
            bt = __ldg(&a.rpt[v]);
            lent = (int32_t)(__ldg(&a.rpt[v + 1]) - bt);
          }
          const HubPiece hp = src_hub_piece(len, lent, p - sh.hbase[h]);
          if (!hp.count) continue;                      // (pieces of a row not listed)
          if (lane == 0) wb.acc[0] = 0ull;
          cx.mv = v;
          __syncwarp();
          if (!hp.in)
            cx.template fwd<SYM, true, Cnt>(a.arc, b + hp.first, lane == 0 ? hp.count : 0, d, slot);
          else if (!SYM)
            cx.template fwd<true, false, Cnt>(a.arct, bt + hp.first, lane == 0 ? hp.count : 0, d, slot);
          cx.template drain<Cnt, true>(true);
          __syncwarp();
          if (lane == 0 && wb.acc[0]) src_hub_add(sh, (int)h, Cnt::of_count(wb.acc[0]));
          __syncwarp();
        }
        __syncthreads();
        for (uint32_t h = threadIdx.x; h < nh; h += blockDim.x) {
          Cnt x;
          src_hub_get(sh, (int)h, x);
          src_put_count(a, st, sh.hv[h], d == 0 ? Cnt::of_count(Cnt::one()) : x);
        }
        if (threadIdx.x == 0) sh.nhub = 0ull;
      }
      if (UNIT) {
        if (hubs) __syncthreads();                      // the hubs' sums are stored
        q0 = q1;
        q1 = sh.tail;
        // (a count past 2^58, or a level past which a narrow tau cannot go)
        redo = sh.redo != 0u || (DM != DM_GLOBAL && d + 2 >= SrcState<DM>::NONE);
        k++;
        if (threadIdx.x == 0) st.off[k] = make_uint2(q0, sh.dtail);
        __syncthreads();                                // every thread has read tail and redo
        d++;
        if (q1 == q0 || redo) break;
      } else {
        // the next distance value with entries, 32 buckets at a time
        if (wid == 0) {
          int32_t nd = -1;
          for (int j0 = 1; j0 < a.B; j0 += 32) {
            int b = slot + j0 + (int)lane;
            if (b >= a.B) b -= a.B;
            const bool hit = j0 + (int)lane < a.B && st.cnt[b] != 0u;
            const uint32_t bal = __ballot_sync(0xffffffffu, hit);
            if (bal) { nd = d + j0 + __ffs(bal) - 1; break; }
          }
          if (lane == 0) {
            // distances of the next step's offers must stay below an unreached entry's
            if (DM == DM_SMEM16 && nd >= SrcState<DM>::NONE - a.B) { sh.redo = 1u; nd = -1; }
            sh.next = nd;
            st.cnt[slot] = 0u;
            if (sh.tail != sh.mark) {                   // a step of stale entries settles nothing
              sh.mark = sh.tail;
              st.off[++sh.steps] = make_uint2(sh.tail, sh.dtail);
            }
          }
        }
        __syncthreads();
        k = sh.steps;
        const int32_t nd = sh.next;
        if (nd < 0) break;
        slot += nd - d;
        if (slot >= a.B) slot -= a.B;
        d = nd;
      }
    }
    if (!UNIT && DM == DM_SMEM16) {
      __syncthreads();
      redo = sh.redo != 0u;
    }
    if (threadIdx.x == 0) atomicMax(&a.ctl->steps, k);
    if (redo) {                                         // the wide form takes this source
      if (threadIdx.x == 0) a.redo[atomicAdd(&a.ctl->nredo, 1u)] = (int32_t)si;
      continue;
    }
    if (a.dist_out) {                                   // MFBF alone: the source's row of tau and sigma_bar
      for (int32_t v = (int32_t)threadIdx.x; v < a.n; v += (int32_t)blockDim.x) {
        const int32_t x = st.tau(v);
        a.dist_out[(size_t)si * a.n + v] = x;
        if (a.sigma_out)
          a.sigma_out[(size_t)si * a.n + v] =
              x == INF ? 0.0 : src_sigma<UNIT>(st.cell[v].sv);
      }
    }
    if (!a.lambda) continue;
    // ---- MFBr: the same steps backwards (step 0 is the source)
    double* lam = a.lambda + (size_t)(a.row ? (uint32_t)a.row[si] : blockIdx.x & a.copy_mask) * a.n;
    if (sh.dtail <= a.dcap) {
      // over the recorded DAG arcs (v, u): zeta(u) += zeta(v) + 1/sigma_bar(v).
      // Only zeta(v) depends on the step before, so a step's first arcs and
      // their 1/sigma_bar are loaded one step ahead.
      const uint32_t tid = threadIdx.x, T = blockDim.x;
      uint32_t e1 = st.off[k].y, e0 = st.off[k - 1].y, em = k > 1 ? st.off[k - 2].y : 0u;
      int2 cur = make_int2(s, s);
      double rs = 0.0;
      if (e0 + tid < e1) {
        cur = st.arc(e0 + tid);
        rs = 1.0 / src_sigma<UNIT>(st.cell[cur.x].sv);
      }
      for (uint32_t t = k; t-- > 1;) {
        const uint32_t en = t > 1 ? st.off[t - 2].y : 0u;
        int2 nxt = make_int2(s, s);
        double nrs = 0.0;
        if (t > 1 && em + tid < e0) nxt = st.arc(em + tid);
        if (cur.y != s) atomicAdd(&st.cell[cur.y].z, __ldcg(&st.cell[cur.x].z) + rs);
        for (uint32_t e = e0 + tid + T; e < e1; e += ILP * T) {
          int2 x[ILP];
          double z[ILP], sg[ILP];
#pragma unroll
          for (int r = 0; r < ILP; r++) x[r] = e + r * T < e1 ? st.arc(e + r * T) : make_int2(s, s);
#pragma unroll
          for (int r = 0; r < ILP; r++)
            if (x[r].y != s) {
              z[r] = __ldcg(&st.cell[x[r].x].z);
              sg[r] = src_sigma<UNIT>(st.cell[x[r].x].sv);
            }
#pragma unroll
          for (int r = 0; r < ILP; r++)
            if (x[r].y != s) atomicAdd(&st.cell[x[r].y].z, z[r] + 1.0 / sg[r]);
        }
        if (nxt.y != s) nrs = 1.0 / src_sigma<UNIT>(st.cell[nxt.x].sv);
        if (a.bytes) cx.nbytes += e0 + tid < e1 ? 32ull * ((e1 - e0 - tid + T - 1) / T) : 0ull;
        __syncthreads();
        e1 = e0;
        e0 = em;
        em = en;
        cur = nxt;
        rs = nrs;
      }
      for (uint32_t i = 1 + tid; i < sh.tail; i += ILP * T) {  // (entry 0 is the source)
        int32_t v[ILP];
        double z[ILP], sg[ILP];
#pragma unroll
        for (int r = 0; r < ILP; r++) v[r] = i + r * T < sh.tail ? st.order[i + r * T] : -1;
#pragma unroll
        for (int r = 0; r < ILP; r++) {
          z[r] = v[r] >= 0 ? __ldcg(&st.cell[v[r]].z) : 0.0;
          sg[r] = v[r] >= 0 ? src_sigma<UNIT>(st.cell[v[r]].sv) : 0.0;
        }
#pragma unroll
        for (int r = 0; r < ILP; r++)
          if (z[r] != 0.0) atomicAdd(&lam[v[r]], z[r] * sg[r]);
      }
      if (a.bytes && tid == 0) cx.nbytes += 28ull * sh.tail;
      continue;
    }
    // more DAG arcs than recorded: pulled over the out-arcs
    for (uint32_t t = k; t-- > 1;) {
      const uint32_t o0 = st.off[t].x, items = st.off[t + 1].x - o0;
      const uint32_t bs = src_batch(items, nwarp);
      bool hub = false;
      for (uint32_t i0 = (uint32_t)wid * bs; i0 < items; i0 += (uint32_t)nwarp * bs) {
        const uint32_t i = i0 + lane;
        const bool on = lane < bs && i < items;
        int32_t v = 0, len = 0, dv = 0;
        int64_t b = 0;
        if (on) {
          v = st.order[o0 + i];
          b = __ldg(&a.rp[v]);
          len = (int32_t)(__ldg(&a.rp[v + 1]) - b);
          dv = st.tau(v);
        }
        bool mine = on;
        if (len > SRC_HUB_ARCS && src_list_hub(sh, v, src_pieces(len))) {
          hub = true;
          mine = false;
          len = 0;
        }
        wb.acc[lane] = 0ull;
        __syncwarp();
        cx.template bwd<Val>(b, len, dv);
        cx.template drain<Val, false>(true);
        __syncwarp();
        if (mine) src_put_value<UNIT>(&st.cell[v], &lam[v], Val::of_value(wb.acc[lane]));
        if (a.bytes && mine) cx.nbytes += 24;
        __syncwarp();
      }
      if (__syncthreads_or(hub)) {
        const uint32_t nh = min((uint32_t)(sh.nhub >> 40), (uint32_t)SRC_HUBS), np = (uint32_t)sh.nhub;
        for (uint32_t p = (uint32_t)wid; p < np; p += (uint32_t)nwarp) {
          const uint32_t h = src_piece_row(sh, nh, p);
          const int32_t v = sh.hv[h];
          const int64_t b = __ldg(&a.rp[v]);
          const int32_t len = (int32_t)(__ldg(&a.rp[v + 1]) - b);
          const HubPiece hp = src_hub_piece(len, 0, p - sh.hbase[h]);
          if (!hp.count) continue;                      // (pieces of a row not listed)
          if (lane == 0) wb.acc[0] = 0ull;
          __syncwarp();
          cx.template bwd<Val>(b + hp.first, lane == 0 ? hp.count : 0, st.tau(v));
          cx.template drain<Val, false>(true);
          __syncwarp();
          if (lane == 0 && wb.acc[0]) src_hub_add(sh, (int)h, Val::of_value(wb.acc[0]));
          __syncwarp();
        }
        __syncthreads();
        for (uint32_t h = threadIdx.x; h < nh; h += blockDim.x) {
          Val x;
          src_hub_get(sh, (int)h, x);
          src_put_value<UNIT>(&st.cell[sh.hv[h]], &lam[sh.hv[h]], x);
        }
        if (threadIdx.x == 0) sh.nhub = 0ull;
        __syncthreads();
      }
    }
  }
  if (a.bytes) {
    unsigned long long nb = cx.nbytes;
    for (int o = 16; o; o >>= 1) nb += __shfl_xor_sync(0xffffffffu, nb, o);
    if (lane == 0 && nb) atomicAdd(a.bytes, nb);
  }
}

// ------------------------------------------------------------------ driver
template <bool UNIT, int DM, int AM>
static const void* src_pick(bool sym) {
  return sym ? (const void*)k_src_bc<UNIT, DM, AM, true> : (const void*)k_src_bc<UNIT, DM, AM, false>;
}
static const void* src_kernel(const SourcePlan& p, bool sym) {
  if (p.unit) {
    if (p.dm == DM_SMEM16) return src_pick<true, DM_SMEM16, AM_UNIT>(sym);
    if (p.dm == DM_SMEM8) return src_pick<true, DM_SMEM8, AM_UNIT>(sym);
    return src_pick<true, DM_GLOBAL, AM_UNIT>(sym);
  }
  if (p.am == AM_UNIT) return src_pick<false, DM_GLOBAL, AM_UNIT>(sym);
  if (p.dm == DM_SMEM16) return src_pick<false, DM_SMEM16, AM_PACKED>(sym);
  if (p.dm == DM_SMEM32) return src_pick<false, DM_SMEM32, AM_PACKED>(sym);
  return src_pick<false, DM_GLOBAL, AM_PACKED>(sym);
}

static int pow2_floor(int64_t x) {
  int p = 1;
  while (2 * (int64_t)p <= x) p *= 2;
  return p;
}

// unit: by levels, 64-bit counts.  wide: FP64 counts and distances in 32 bits,
// the form that sources are redone in.
void source_plan(const DevGraph& g, int cols, bool unit, bool wide, SourcePlan& p) {
  const int64_t n = std::max(g.n, 1);
  const int64_t n8 = (n + 15) & ~int64_t(15);
  const int64_t avg = g.nnz / n;
  int64_t per_sm = std::max<int64_t>(1, (cols + SRC_SMS - 1) / SRC_SMS);         // sources an SM should hold
  p = SourcePlan{};
  p.unit = unit && !wide;
  p.B = p.unit ? 0 : g.wmax + 1;
  p.am = g.w ? AM_PACKED : AM_UNIT;
  p.scap = p.unit ? 0u : (uint32_t)std::min<int64_t>(64, 8192 / (4 * p.B));
  if (!p.unit) {
    p.cap = (uint32_t)std::min<int64_t>(n, std::max<int64_t>(512, std::min<int64_t>(n / 8, 16 * n / p.B)));
    p.cap = std::max(p.cap, p.scap + 1);
  }
  // DAG arcs for MFBr: all there can be (an undirected edge is one in at most
  // one direction), or 32 per vertex; sources with more pull instead
  p.dcap = (uint32_t)std::min<int64_t>(g.directed ? g.nnz : g.nnz / 2, 32 * n8);
  auto layout = [&](bool tau) {
    Carver c(nullptr, 0);
    p.o_cell = c.off; c.take<ulonglong2>((size_t)n8);    // (SrcCell)
    p.o_dist = c.off; c.take<int32_t>(tau ? (size_t)n8 : 0);
    p.o_order = c.off; c.take<int32_t>((size_t)(3 * n8 + 16));
    p.o_ring = c.off; c.take<int32_t>((size_t)p.B * (p.cap - p.scap));
    p.o_dag = c.off; c.take<uint32_t>((size_t)p.dcap * (n <= 65536 ? 1 : 2));
    return c.off;
  };
  // unit-weight graphs: two sources an SM, or as many as 256 MB of block states
  // hold.  (Two take what they need: 152 sources of a graph of 10^7 vertices and
  // 10^6 arcs 49 GB, where the level kernels' state takes 38 GB and the call 3.7 ms
  // instead of 1.3.  Calls cut the blocks down to the scratch there is.)
  if (p.unit)
    per_sm = std::min(per_sm, std::max<int64_t>(2, (256ll << 20) / (int64_t)layout(false) / SRC_SMS));
  const int64_t ring = (int64_t)src_al16((size_t)p.B * 4) + (int64_t)src_al16((size_t)p.B * p.scap * 4);
  auto fixed = [&](int threads) {
    return (int64_t)src_al16(sizeof(SrcShared)) + (int64_t)src_al16(sizeof(SrcWarp<4>) * (threads / 32)) + ring;
  };
  // Distances in shared memory where an SM then still holds as many sources as
  // it should, or where the walk over the arcs dominates and one block's warps
  // fill the SM.
  const int64_t share = std::min<int64_t>(per_sm, 8);
  auto room = [&](int threads, int64_t db) { return SRC_SMEM_MAX / (fixed(threads) + db * n8 + 1024); };
  auto threads_for = [&](int64_t blocks) { return std::max(128, pow2_floor(1024 / std::max<int64_t>(1, blocks))); };
  p.dm = DM_GLOBAL;
  p.threads = std::max(g.max_deg, g.max_in_deg) <= 8 ? threads_for(share) : 1024;
  int64_t db = 0;
  const int form[2] = {p.unit ? DM_SMEM16 : DM_SMEM32, p.unit ? DM_SMEM8 : DM_SMEM16};
  const int forms = p.unit ? 2 : p.am != AM_PACKED ? 0 : wide ? 1 : 2;
  for (int f = 0; f < forms && p.dm == DM_GLOBAL; f++) {
    const int64_t bytes = (p.unit ? 2 : 4) >> f;
    if (room(threads_for(share), bytes) >= share) {
      p.dm = form[f];
      db = bytes;
      p.threads = threads_for(share);
    } else if (avg >= 8 && room(512, bytes) >= 1) {
      p.dm = form[f];
      db = bytes;
      p.threads = room(1024, bytes) >= 1 ? 1024 : 512;
      while (p.threads > 128 && room(p.threads / 2, bytes) > room(p.threads, bytes) &&
             room(p.threads / 2, bytes) <= share)
        p.threads /= 2;
    }
  }
  const int64_t smem = fixed(p.threads) + db * n8;
  const int64_t resident =
      std::max<int64_t>(1, std::min({room(p.threads, db), (int64_t)(1024 / p.threads), p.unit ? per_sm : int64_t(8)}));
  p.slots = (int)std::max<int64_t>(1, std::min<int64_t>(cols, SRC_SMS * resident));
  p.smem = (size_t)smem;
  p.slot_bytes = layout(p.dm == DM_GLOBAL);
}

// lambda of a call with one row is summed in 8 to 32 copies, added up at the end:
// a sum of thousands of terms one by one is less accurate than a sum of sums.
// Against 64-bit Brandes, relative to the largest: directed weighted R-MAT 16,
// 2048 sources 1.3e-15 -> 1.8e-16, weighted 256^2 grid, 512 sources 1.2e-15 ->
// 1.5e-16, uniform n = 1024, all sources 8e-16 -> 1.5e-16 (and 0.204 -> 0.201 ms,
// as fewer sources in lock step meet at an address).  A copy serves four blocks
// at least, and all of them take 64 MB at most.
int source_copies(const SourcePlan& p, int32_t n) {
  int k = 32;
  while (k > 4 && (4 * k > p.slots || (size_t)k * n > (8u << 20))) k >>= 1;
  return k > 4 ? k : 0;
}
__global__ void k_src_sum_copies(const double* __restrict__ lam, int copies, int32_t n, double* lambda) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  double s = 0.0;
  for (int k = 0; k < copies; k += 8) {
    double x[8];
#pragma unroll
    for (int i = 0; i < 8; i++) x[i] = lam[(size_t)(k + i) * n + v];
    s += ((x[0] + x[1]) + (x[2] + x[3])) + ((x[4] + x[5]) + (x[6] + x[7]));
  }
  lambda[v] += s;
}

void source_carve(Carver& c, const SourcePlan& p, int32_t nredo, size_t lam, SourceState& s) {
  s.ctl = c.take<SrcCtl>(1);
  s.lam = c.take<double>(lam);
  s.redo = c.take<int32_t>((size_t)nredo);
  s.ctr = c.take<Counters>(1);
  s.slots = c.take<char>(p.slot_bytes * (size_t)p.slots);   // last: its size is the form's
}

size_t source_bytes(const SourcePlan& p, int32_t nredo, size_t lam) {
  Carver c(nullptr, 0);
  SourceState s;
  source_carve(c, p, nredo, lam, s);
  return c.off;
}

mfbc_status source_run(RunCtx& rc, const SourcePlan& p, SourceState& s, const int32_t* d_src, const int32_t* d_row,
                       const int32_t* d_list, int32_t nsrc, double* lambda, int copies, int32_t* dist_out,
                       double* sigma_out, KId id) {
  const DevGraph& g = *rc.g;
  if (g.n == 0 || nsrc == 0) return MFBC_OK;
  SrcArgs a;
  a.n = g.n;
  a.rp = g.rowptr;
  a.rpt = g.rowptr_t;
  a.arc = p.am == AM_PACKED ? g.pk : reinterpret_cast<const uint32_t*>(g.col);
  a.arct = p.am == AM_PACKED ? g.pk_t : reinterpret_cast<const uint32_t*>(g.col_t);
  a.cb = g.pk_bits;
  a.src = d_src;
  a.row = d_row;
  a.list = d_list;
  a.nsrc = (uint32_t)nsrc;
  a.lambda = lambda && copies ? s.lam : lambda;
  a.copy_mask = copies ? (uint32_t)copies - 1u : 0u;
  a.dist_out = dist_out;
  a.sigma_out = sigma_out;
  a.slots = s.slots;
  a.slot_bytes = p.slot_bytes;
  a.o_dist = p.o_dist; a.o_cell = p.o_cell; a.o_order = p.o_order;
  a.o_ring = p.o_ring; a.o_dag = p.o_dag;
  a.dcap = lambda ? p.dcap : 0u;
  a.B = p.B;
  a.scap = p.scap;
  a.cap = p.cap;
  a.ctl = s.ctl;
  a.redo = s.redo;
  a.bytes = rc.prof->count_bytes ? &s.ctr->bytes[id] : nullptr;
  const void* k = src_kernel(p, !g.directed);
  // (the limit is the kernel's, not the launch's: calls on other threads must not
  // lower it between here and the launch)
  MFBC_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SRC_SMEM_MAX), rc.err);
  MFBC_CUDA_TRY(cudaMemsetAsync(&s.ctl->head, 0, sizeof(uint32_t), rc.stream), rc.err);
  if (lambda && copies)
    MFBC_CUDA_TRY(cudaMemsetAsync(s.lam, 0, sizeof(double) * (size_t)copies * g.n, rc.stream), rc.err);
  void* args[] = {&a};
  rc.prof->begin(id);
  const cudaError_t e = cudaLaunchKernel(k, dim3((unsigned)std::min(p.slots, nsrc)), dim3((unsigned)p.threads), args,
                                         p.smem, rc.stream);
  rc.prof->end(id);
  if (e != cudaSuccess) return cuda_fail(rc.err, "launch of the source kernel", e);
  if (lambda && copies) {
    rc.prof->begin(K_LAMBDA);
    k_src_sum_copies<<<(unsigned)((g.n + 255) / 256), 256, 0, rc.stream>>>(s.lam, copies, g.n, lambda);
    rc.prof->end(K_LAMBDA);
  }
  return MFBC_OK;
}

}  // namespace mfbc
