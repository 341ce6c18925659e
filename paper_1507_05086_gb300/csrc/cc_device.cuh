// cc_device.cuh -- device-side building blocks shared by the library's kernels:
// the permutation hash, bounded waits, warp/block scans and the edge-balanced
// walks over adjacency rows: row_walk (the round kernel, the objective above 2^24
// vertices), unit_walk (the objective below) and lbs_for_each (validation, graphs
// with short rows, C4 without rounds).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace ccg {

constexpr unsigned FULL = 0xFFFFFFFFu;

// Status codes, mirrored from include/cc.h.
constexpr int kOk = 0;
constexpr int kErrTimeout = -5;
constexpr int kErrInternal = -7;

// ---------------------------------------------------------------------------
// Permutation hash: the SplitMix64 output function (Steele, Lea & Flood,
// OOPSLA 2014) applied to seed ^ v.  pi orders vertices by (key, v).
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ uint64_t perm_key(uint64_t seed, uint64_t v) {
  uint64_t z = (seed ^ v) + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// ---------------------------------------------------------------------------
// Memory access helpers.  Data that other blocks of the same persistent
// kernel write is read at L2 (ld.cg); L1 is not coherent across SMs.
// ---------------------------------------------------------------------------
template <class T>
__device__ __forceinline__ T ldcg(const T* p) { return __ldcg(p); }

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ uint32_t ld_relaxed_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ int ld_volatile_int(const int* p) {
  return *reinterpret_cast<const volatile int*>(p);
}
__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounds checks of the debug build (nvcc -DCC_DEBUG; build(debug=True)): an
// index outside [0, cap) records CC_ERR_INTERNAL in the kernel's error word
// and the access is skipped, so a bookkeeping mistake reports an error
// instead of touching memory out of range.  Release builds compile the
// checks away.
#ifdef CC_DEBUG
constexpr bool kDebugChecks = true;
#else
constexpr bool kDebugChecks = false;
#endif
__device__ __forceinline__ bool in_bounds(int64_t i, int64_t cap, int* err) {
  if (!kDebugChecks) return true;
  if (i >= 0 && i < cap) return true;
  if (err) atomicCAS(err, kOk, kErrInternal);
  return false;
}
// The checks as written at the access sites: in release builds the macro is
// the constant true and its arguments are not compiled at all, so the kernels
// are the same code as without the checks (register allocation included).
#ifdef CC_DEBUG
#define CC_IN_BOUNDS(i, cap, err) in_bounds((i), (cap), (err))
#define CC_ROWLIST_CHECK(cap, err) , (cap), (err)
#else
#define CC_IN_BOUNDS(i, cap, err) true
#define CC_ROWLIST_CHECK(cap, err)
#endif

// Every spin-wait of the kernels is bounded: after kBarrierLimitNs the waiter
// records kErrTimeout in the error word and the kernel unwinds.
constexpr uint64_t kBarrierLimitNs = 4000000000ull;   // 4 s

// ---------------------------------------------------------------------------
// Scans
// ---------------------------------------------------------------------------
template <class T>
__device__ __forceinline__ T warp_inclusive_sum(T x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T y = __shfl_up_sync(FULL, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// The same as a loop: a quarter of the code, for sums whose code runs once per
// pass and so is fetched rather than found in the instruction cache.
__device__ __forceinline__ int64_t warp_inclusive_sum_rolled(int64_t x) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(FULL, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

template <class T>
__device__ __forceinline__ T warp_sum(T x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
  return x;
}

__device__ __forceinline__ int32_t warp_min_i32(int32_t x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const int32_t y = __shfl_xor_sync(FULL, x, o);
    x = y < x ? y : x;
  }
  return x;
}

template <class T>
__device__ __forceinline__ T warp_max(T x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    T y = __shfl_xor_sync(FULL, x, o);
    x = y > x ? y : x;
  }
  return x;
}

// Block-wide exclusive sum; *total receives the block total.  scratch must
// hold 33 elements.  All threads of the block must call it.
template <class T>
__device__ __forceinline__ T block_exclusive_sum(T x, T* scratch, T* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = (blockDim.x + 31) >> 5;
  const T inc = warp_inclusive_sum(x);
  __syncthreads();                       // earlier readers of scratch
  if (lane == 31) scratch[warp] = inc;
  __syncthreads();
  // every warp scans the warps' totals itself: no third barrier
  const T w = lane < nwarps ? scratch[lane] : T(0);
  const T wi = warp_inclusive_sum(w);
  *total = __shfl_sync(FULL, wi, 31);
  return __shfl_sync(FULL, wi - w, warp) + inc - x;
}

template <class T>
__device__ __forceinline__ T block_sum(T x, T* scratch) {
  T tot;
  block_exclusive_sum(x, scratch, &tot);
  return tot;
}

__device__ __forceinline__ int32_t block_max_i32(int32_t x, int32_t* scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  x = __reduce_max_sync(FULL, x);
  __syncthreads();
  if (lane == 0) scratch[warp] = x;
  __syncthreads();
  return __reduce_max_sync(FULL, lane < (int)((blockDim.x + 31) >> 5) ? scratch[lane] : INT32_MIN);
}

__device__ __forceinline__ int32_t block_sum_i32(int32_t x, int32_t* scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  x = __reduce_add_sync(FULL, x);
  __syncthreads();
  if (lane == 0) scratch[warp] = x;
  __syncthreads();
  return __reduce_add_sync(FULL, lane < (int)((blockDim.x + 31) >> 5) ? scratch[lane] : 0);
}

// ---------------------------------------------------------------------------
// 4-bit signatures of cluster ids (objective): equal ids have equal ones.
// pack_sig8: the eight signatures of lanes 8 i .. 8 i + 7 in one word (valid
// in the first of the eight lanes).  All lanes must call it.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_sig(uint32_t id) { return (id * 0x9E3779B1u) >> 28; }
__device__ __forceinline__ uint32_t pack_sig8(uint32_t sig) {
  uint32_t x = sig << ((threadIdx.x & 7) * 4);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) x |= __shfl_xor_sync(FULL, x, o);
  return x;
}

// ---------------------------------------------------------------------------
// Edge-balanced walk over a list of adjacency rows.
//
// Item j of the list owns the virtual edges [epos[j], epos[j+1]) (epos[j] is
// non-decreasing in j and every item owns at least one edge); E is the total.
// Warps take chunks of kLbsBatches * kLbsW consecutive virtual edges, so a hub
// row is spread over many warps and short rows are packed together.  Within a
// chunk a warp handles kLbsW = 32 * kLbsK edges at a time: each lane gets kLbsK
// edges (e = base + lane + 32 t), so kLbsK independent loads per lane are in
// flight instead of one.  f(L) receives an Lbs view of the batch (item, virtual
// edge and position in the item of each of the lane's edges); all 32 lanes
// call f together (edges with L.ok(t) == false must be skipped, but their
// lanes still take part in warp collectives).
// ---------------------------------------------------------------------------
constexpr int kLbsK = 4;
#ifndef CC_LBS_PF_AHEAD
#define CC_LBS_PF_AHEAD 2
#endif
constexpr int kLbsPfAhead = CC_LBS_PF_AHEAD;   // batches of a long row prefetched into L2 ahead

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}
constexpr int kLbsW = 32 * kLbsK;
#ifndef CC_LBS_BATCHES
#define CC_LBS_BATCHES 4
#endif
constexpr int kLbsBatches = CC_LBS_BATCHES;   // batches per chunk of a long walk

// Run-time shape of a walk (the defaults above unless a tuning says
// otherwise): batches per chunk (1..8) and batches of a long row prefetched
// ahead (0..8).  Neither changes what a walk visits, only its schedule.
struct WalkShape {
  int batches = kLbsBatches;
  int pf_ahead = kLbsPfAhead;
};

struct LbsWarp {
  int32_t mark[kLbsW];   // relative item index per position
  int32_t rel[kLbsW];    // item start relative to the batch base
  int64_t dlt[kLbsW];    // per-item CSR delta (prefetched when given)
  int32_t vtx[kLbsW];    // per-item vertex or payload (prefetched when given)
  int32_t next;          // relative index of the item starting the next batch
  int32_t pad;
};

// One batch of kLbsW virtual edges as seen by one lane.
struct Lbs {
  int64_t j0, base;
  const LbsWarp* ws;
  int32_t ri[kLbsK];
  unsigned valid;
  __device__ __forceinline__ bool ok(int t) const { return (valid >> t) & 1u; }
  __device__ __forceinline__ int64_t item(int t) const { return j0 + ri[t]; }
  __device__ __forceinline__ int64_t edge(int t) const { return base + (threadIdx.x & 31) + 32 * t; }
  // index of the edge inside its item's row
  __device__ __forceinline__ int64_t in_row(int t) const {
    return (int64_t)((threadIdx.x & 31) + 32 * t) - ws->rel[ri[t]];
  }
  // prefetched per-item data (only when the walk was given the arrays)
  __device__ __forceinline__ int64_t csr(int t) const { return edge(t) + ws->dlt[ri[t]]; }
  __device__ __forceinline__ int32_t vtx(int t) const { return ws->vtx[ri[t]]; }
};

// Number of elements of the sorted array a[0..n) that are <= x, by a 33-ary
// search of the whole warp (about log_33(n) dependent loads).
__device__ __forceinline__ int64_t warp_upper_bound(const int64_t* a, int64_t n, int64_t x) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, hi = n;
  while (hi - lo > 32) {
    const int64_t span = hi - lo;
    const int64_t p = lo + (span * (lane + 1)) / 33;
    const unsigned b = __ballot_sync(FULL, ldcg(a + p) <= x);
    const int c = __popc(b);
    const int64_t pp = __shfl_sync(FULL, p, c > 0 ? c - 1 : 0);
    const int64_t pn = __shfl_sync(FULL, p, c < 32 ? c : 31);
    lo = c > 0 ? pp + 1 : lo;
    hi = c < 32 ? pn : hi;
  }
  const int64_t p = lo + lane;
  const bool le = p < hi && ldcg(a + p) <= x;
  return lo + __popc(__ballot_sync(FULL, le));
}

// One chunk [c0, cend) of the walk: find the item holding c0, then batches
// of kLbsW virtual edges.  A batch that lies inside one item (a long row)
// needs none of the per-item loads: the warp keeps the range, delta and
// vertex of its current item, taken from the previous batch's loads, and
// only a batch that crosses an item boundary loads and scans item starts,
// in groups of 32 items: a group is loaded only while the previous one ends
// inside the batch, so a batch spanning a few rows costs one group, not
// kLbsK (every item owns at least one edge, so kLbsK groups always suffice,
// and the item after the batch's last one is always among those loaded).
//
// With colp (the CSR column array; the walk's CSR position of virtual edge e
// of item j is e + delta[j], or e without delta), the column ids of the
// batch kLbsPfAhead ahead in the current row are prefetched into L2, so a
// long row streams from DRAM ahead of its use.  E: the walk's end.
template <class F>
__device__ __forceinline__ void lbs_chunk(const int64_t* epos, int64_t nitems, int64_t c0, int64_t cend, LbsWarp* ws,
                                          F& f, const int64_t* delta, const int32_t* vtx,
                                          const int32_t* colp, int64_t E) {
  const int lane = threadIdx.x & 31;
  int64_t j0 = warp_upper_bound(epos, nitems, c0) - 1;
  // cached item (warp-uniform): valid when cur_j == j0
  int64_t cur_j = -1, cur_start = 0, cur_end = 0, cur_dlt = 0;
  int32_t cur_vtx = 0;
  for (int64_t base = c0; base < cend; base += kLbsW) {
    Lbs L;
    L.j0 = j0;
    L.base = base;
    L.ws = ws;
    L.valid = 0;
    if (cur_j == j0 && cur_end >= base + kLbsW) {
      // the whole batch belongs to item j0
      if (lane == 0) {
        ws->rel[0] = (int32_t)(cur_start - base);
        ws->dlt[0] = cur_dlt;
        ws->vtx[0] = cur_vtx;
      }
      __syncwarp();
#pragma unroll
      for (int t = 0; t < kLbsK; ++t) {
        L.ri[t] = 0;
        if (base + lane + 32 * t < cend) L.valid |= 1u << t;
      }
      if (colp && kLbsPfAhead > 0 && lane < kLbsW / 32) {
        const int64_t pe = base + (int64_t)kLbsPfAhead * kLbsW + 32 * lane;
        if (pe < cur_end && pe < E) prefetch_l2(colp + pe + cur_dlt);
      }
      f(L);
      __syncwarp();
      if (cur_end == base + kLbsW) ++j0;          // the next batch starts the next item
      continue;
    }
    int64_t s[kLbsK];
#pragma unroll
    for (int t = 0; t < kLbsK; ++t) {
      s[t] = INT64_MAX;
      ws->mark[lane + 32 * t] = -1;
    }
#pragma unroll
    for (int t = 0; t < kLbsK; ++t) {
      // a group of 32 items is needed while the previous group's last item
      // starts inside the batch or at its end
      if (t > 0 && __shfl_sync(FULL, s[t - 1], 31) > base + kLbsW) break;
      const int64_t jj = j0 + lane + 32 * t;
      const bool in = jj < nitems;
      s[t] = in ? ldcg(epos + jj) : INT64_MAX;
      // per-item data loads issue together with the start offsets
      if (delta) ws->dlt[lane + 32 * t] = in ? ldcg(delta + jj) : 0;
      if (vtx) ws->vtx[lane + 32 * t] = in ? ldcg(vtx + jj) : 0;
    }
    if (lane == 0) ws->next = -1;
    __syncwarp();
#pragma unroll
    for (int t = 0; t < kLbsK; ++t) {
      const int i = lane + 32 * t;
      // start relative to the batch, clamped to int32 (items past the end of
      // the list, or starting 2^31 edges later, read as INT32_MAX)
      const int64_t r = s[t] - base;
      ws->rel[i] = s[t] == INT64_MAX || r > INT32_MAX - 1 ? INT32_MAX : (int32_t)r;
      if (s[t] < base + kLbsW) {
        if (s[t] >= base) ws->mark[s[t] - base] = i;
      } else if (s[t] == base + kLbsW) {
        ws->next = i;                  // the item that starts the next batch
      }
    }
    __syncwarp();
    // segmented max-scan: each position takes the last item starting at or before it
    int v[kLbsK];
    int run = -1;
#pragma unroll
    for (int t = 0; t < kLbsK; ++t) {
      const int m = ws->mark[lane * kLbsK + t];
      run = m > run ? m : run;
      v[t] = run;
    }
    int inc = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, inc, o);
      if (lane >= o) inc = y > inc ? y : inc;
    }
    int exc = __shfl_up_sync(FULL, inc, 1);
    if (lane == 0) exc = -1;
    __syncwarp();
#pragma unroll
    for (int t = 0; t < kLbsK; ++t) {
      int m = v[t] > exc ? v[t] : exc;
      ws->mark[lane * kLbsK + t] = m < 0 ? 0 : m;
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < kLbsK; ++t) {
      const int p = lane + 32 * t;
      L.ri[t] = ws->mark[p];
      if (base + p < cend) L.valid |= 1u << t;
    }
    const int last = ws->mark[kLbsW - 1];
    const int nxt = ws->next;
    // next batch: the item holding its first edge is the last item of this
    // batch or, when an item starts exactly at the next base, that item (the
    // item after `last` is always among the ones loaded here unless `last`
    // is the final loaded slot, in which case one load decides)
    int m = nxt >= 0 ? nxt : last;
    if (nxt < 0 && last == kLbsW - 1 && j0 + kLbsW < nitems && ldcg(epos + j0 + kLbsW) <= base + kLbsW) m = kLbsW;
    // remember the next batch's item when its range is among the loaded ones
    if (m + 1 < kLbsW) {
      const int32_t r1 = ws->rel[m + 1];
      cur_j = j0 + m;
      cur_start = base + ws->rel[m];
      cur_end = r1 == INT32_MAX ? INT64_MAX : base + r1;
      cur_dlt = delta ? ws->dlt[m] : 0;
      cur_vtx = vtx ? ws->vtx[m] : 0;
      // the next batches of that item: start streaming them
      if (colp) {
        for (int a = 1; a <= kLbsPfAhead; ++a) {
          const int64_t pe = base + (int64_t)a * kLbsW + 32 * lane;
          if (lane < kLbsW / 32 && pe >= cur_start && pe < cur_end && pe < E) prefetch_l2(colp + pe + cur_dlt);
        }
      }
    }
    f(L);
    __syncwarp();
    j0 += m;
  }
}

// The walk covers the virtual edges [E0, E); warp w of the grid takes chunks w,
// w + nwarps, ... of up to kLbsBatches batches, fewer when the list is short, so
// that short lists still spread over many warps.
template <class F>
__device__ __forceinline__ void lbs_for_each(const int64_t* epos, int64_t nitems, int64_t E, LbsWarp* ws, F&& f,
                                             const int64_t* delta = nullptr, const int32_t* vtx = nullptr,
                                             int64_t E0 = 0, const int32_t* colp = nullptr) {
  if (E <= E0) return;
  const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int64_t nb = (E - E0) / (nwarps * (int64_t)kLbsW * 2);
  nb = nb < 1 ? 1 : (nb > kLbsBatches ? kLbsBatches : nb);
  const int64_t kChunk = (int64_t)kLbsW * nb;
  for (int64_t c0 = E0 + gwarp * kChunk; c0 < E; c0 += nwarps * kChunk)
    lbs_chunk(epos, nitems, c0, c0 + kChunk < E ? c0 + kChunk : E, ws, f, delta, vtx, colp, E);
}

// ---------------------------------------------------------------------------
// Unit walk: the edge-balanced walk over rows cut into units of 32 entries.
//
// Item j of the list (a row of len >= 1 entries from CSR position row) owns
// the units [pos, pos + units_of(len)); pos counts up over the list, U is the
// total.  Warps take chunks of consecutive units and read kUnitB of them at a
// time, so every lane has kUnitB independent column loads in flight, and the
// item of a unit is known to the whole warp: the warp holds the data of 32
// consecutive items, one per lane, and picks the unit's item by a ballot.
// Against the 128-edge batches of lbs_for_each, which resolve the item of
// every single edge through shared memory, a batch is twice as many entries
// behind half as many dependent steps.  Short rows leave lanes idle (a row of
// 8 entries fills a quarter of its unit), which costs little: the walk is
// bound by latency, not by lanes.
//
// at(j) = pos of item j; load(j) = the item's data, read once per window of
// items; f(X) gets the batch: the column of this lane's entry of each unit
// (-1: none) and, the same in all lanes, the unit's payload.  All 32
// lanes call f together.
// ---------------------------------------------------------------------------
constexpr int kUnitB = 8;
__host__ __device__ __forceinline__ int64_t units_of(int64_t len) { return (len + 31) >> 5; }

struct UnitItem {
  uint32_t pos;          // below 2^33 / 32 + 2^31 units
  int32_t len;
  int64_t row;
  int32_t aux;           // payload
};

struct UnitBatch {
  int32_t w[kUnitB];     // column of this lane's entry, -1 when there is none
  int32_t aux[kUnitB];   // payload of the unit's item
};

// Number of items whose pos is <= x (pos ascending), by a 33-ary search of the warp.
template <class At>
__device__ __forceinline__ int64_t warp_count_upto(const At& at, int64_t n, uint32_t x) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, hi = n;
  while (hi - lo > 32) {
    const int64_t p = lo + ((hi - lo) * (lane + 1)) / 33;
    const int c = __popc(__ballot_sync(FULL, at(p) <= x));
    const int64_t pp = __shfl_sync(FULL, p, c > 0 ? c - 1 : 0);
    const int64_t pn = __shfl_sync(FULL, p, c < 32 ? c : 31);
    lo = c > 0 ? pp + 1 : lo;
    hi = c < 32 ? pn : hi;
  }
  const int64_t p = lo + lane;
  const bool le = p < hi && at(p) <= x;
  return lo + __popc(__ballot_sync(FULL, le));
}

template <class At, class Load, class F>
__device__ __forceinline__ void unit_walk(int64_t gwarp, int64_t nwarps, int64_t nitems, int64_t U,
                                          const int32_t* __restrict__ col, WalkShape shape, const At& at,
                                          const Load& load, F&& f) {
  const int lane = threadIdx.x & 31;
  // up to 4 * shape.batches batches per chunk, fewer when the list is short
  int64_t nb = U / (nwarps * (int64_t)kUnitB * 2);
  nb = nb < 1 ? 1 : (nb > 4 * shape.batches ? 4 * shape.batches : nb);
  const int64_t chunk = nb * kUnitB;
  for (int64_t c0 = gwarp * chunk; c0 < U; c0 += nwarps * chunk) {
    const int64_t cend = c0 + chunk < U ? c0 + chunk : U;
    UnitBatch X;
    int64_t j0 = warp_count_upto(at, nitems, (uint32_t)c0) - 1;
    UnitItem it;
    uint32_t wend = 0;                  // first unit after the window's items
    for (int64_t t = c0; t < cend; t += kUnitB) {
      const int64_t tend = t + kUnitB < cend ? t + kUnitB : cend;
      if (t == c0 || tend > (int64_t)wend) {
        if (t != c0) j0 += __popc(__ballot_sync(FULL, it.pos <= (uint32_t)t)) - 1;
        const int64_t j = j0 + lane;
        it = UnitItem{0xFFFFFFFFu, 0, 0, 0};
        if (j < nitems) it = load(j);
        const uint32_t e = it.pos + (uint32_t)units_of(it.len);
        wend = __shfl_sync(FULL, e, 31);
      }
      int64_t pf = -1;
#pragma unroll
      for (int q = 0; q < kUnitB; ++q) {
        const int64_t x = t + q;
        const int i = __popc(__ballot_sync(FULL, it.pos <= (uint32_t)x)) - 1;
        const uint32_t p = __shfl_sync(FULL, it.pos, i);
        const int32_t len = __shfl_sync(FULL, it.len, i);
        const int64_t row = __shfl_sync(FULL, it.row, i);
        X.aux[q] = __shfl_sync(FULL, it.aux, i);
        const int32_t k = (int32_t)((uint32_t)x - p) * 32 + lane;
        X.w[q] = x < cend && k < len ? __ldg(col + row + k) : -1;
        // lane q looks shape.pf_ahead batches ahead in the same row
        const int32_t kp = k - lane + shape.pf_ahead * kUnitB * 32;
        if (lane == q && shape.pf_ahead > 0 && kp < len) pf = row + kp;
      }
      if (pf >= 0) prefetch_l2(col + pf);
      f(X);
    }
  }
}

// ---------------------------------------------------------------------------
// Row walk: the edge-balanced walk of the round kernel.
//
// Item j of the list is a row of len >= 1 entries from CSR position row; pos(j)
// counts the entries of the items before it, E is the total.  Warps take
// chunks of consecutive entries.  A warp holds a window of 32 items, one per
// lane, in registers, and reads up to kB times 32 entries of the window at a
// time, so every lane has kB independent column loads in flight.  A lane finds
// the item of its entry by a five-step search over the lanes' starts (none
// when the batch lies inside one row), so rows of any length fill the warp.
// lbs_for_each does the same through marks in shared memory and a scan, behind
// twice as many dependent steps.
//
// at(j) = pos of item j; load(j) = the item's data, read once per window;
// f(X) gets a batch, g(j) follows the last batch of a window, with this lane's
// item (j >= nitems: none).  All 32 lanes call f and g together.
// ---------------------------------------------------------------------------
struct RowItem {
  int64_t pos;
  int64_t row;
  int32_t len;
  int32_t aux;           // payload
};

template <int kB>
struct RowBatch {
  int32_t w[kB];         // column of this lane's entry, -1 when there is none
  int32_t aux[kB];       // payload of its item
  int32_t item[kB];      // its item
  int32_t from, to;      // where this lane's window item lies, relative to the batch (from > 32 kB: after it)
};

// The last item whose pos is <= x (pos ascending from 0, x >= 0), by a 32-ary
// search of the warp.
template <class At>
__device__ __forceinline__ int32_t warp_item_at(const At& at, int32_t n, int64_t x) {
  const int lane = threadIdx.x & 31;
  int32_t lo = 0, span = n;
#pragma unroll 1
  while (span > 1) {
    const int32_t step = (int32_t)(((uint32_t)span + 31u) >> 5), p = lane * step;     // p < 2^31 + 31
    const int c = __popc(__ballot_sync(FULL, (uint32_t)p < (uint32_t)span && at(lo + p) <= x));    // >= 1
    lo += (c - 1) * step;
    span = span - (c - 1) * step < step ? span - (c - 1) * step : step;
  }
  return lo;
}

template <int kB, class At, class Load, class F, class G>
__device__ __forceinline__ void row_walk(int gwarp, int nwarps, int32_t nitems, int64_t E,
                                         const int32_t* __restrict__ col, WalkShape shape, const At& at,
                                         const Load& load, F&& f, G&& g) {
  constexpr int32_t kFar = 1 << 30;     // relative positions from here on lie behind the chunk
  const auto near = [](int64_t x) { return (int32_t)(x < -kFar ? -kFar : x < kFar ? x : kFar); };
  constexpr int kW = 32 * kB;
  const int lane = threadIdx.x & 31;
  // up to 2 * shape.batches batches per chunk, fewer when the list is short
  const int64_t most = (int64_t)nwarps * kW * 4 * shape.batches;
  int nb = E >= most ? 2 * shape.batches : (int)((uint32_t)E / (uint32_t)(nwarps * kW * 2));
  nb = nb < 1 ? 1 : nb;
  const int32_t chunk = nb * kW;
  for (int64_t cs = (int64_t)gwarp * chunk; cs < E; cs += (int64_t)nwarps * chunk) {
    const int32_t cend = E - cs < chunk ? (int32_t)(E - cs) : chunk;
    int32_t j0 = nitems > 32 ? warp_item_at(at, nitems, cs) : 0;       // a short list is one window
    for (int32_t e = 0; e < cend; j0 += 32) {
      // the window: starts and ends relative to the chunk, from kFar before it to
      // kFar behind it (a short list's first rows may end 2^31 entries before it)
      int32_t p = kFar, end = kFar, aux = 0;
      int64_t rel = 0;                  // CSR position of the chunk's first entry, were it in this row
      if (j0 + lane < nitems) {
        const RowItem it = load(j0 + lane);
        const int64_t d = it.pos - cs;
        rel = it.row - d;
        aux = it.aux;
        p = near(d);
        end = near(d + it.len);
      }
      int32_t wend = __shfl_sync(FULL, end, 31);
      wend = wend < cend ? wend : cend;
      for (; e < wend; e += kW) {
        const int32_t stop = e + kW < wend ? e + kW : wend;
        RowBatch<kB> X;
        X.from = p - e;
        X.to = (end < stop ? end : stop) - e;
        const int i0 = __popc(__ballot_sync(FULL, p <= e)) - 1;
        const int32_t end0 = __shfl_sync(FULL, end, i0);
#pragma unroll
        for (int q = 0; q < kB; ++q) {
          const int32_t x = e + lane + 32 * q;
          int i = i0;
          if (end0 < stop) {            // warp-uniform: several rows in the batch
            i = 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
              if (__shfl_sync(FULL, p, i + o) <= x) i += o;
          }
          const int64_t at0 = __shfl_sync(FULL, rel, i);
          X.aux[q] = __shfl_sync(FULL, aux, i);
          X.item[q] = j0 + i;
          X.w[q] = x < stop ? __ldg(col + at0 + x) : -1;
        }
        if (kB > 1 && shape.pf_ahead > 0 && end0 >= stop) {       // stream a long row ahead
          const int32_t x = e + shape.pf_ahead * kW + 32 * lane;
          const int64_t at0 = __shfl_sync(FULL, rel, i0);
          if (lane < kB && x < end0) prefetch_l2(col + at0 + x);
        }
        f(X);
      }
      e = wend;
      g(j0 + lane);
    }
  }
}

template <int kB, class At, class Load, class F>
__device__ __forceinline__ void row_walk(int gwarp, int nwarps, int32_t nitems, int64_t E,
                                         const int32_t* __restrict__ col, WalkShape shape, const At& at,
                                         const Load& load, F&& f) {
  row_walk<kB>(gwarp, nwarps, nitems, E, col, shape, at, load, f, [](int32_t) {});
}

// Lists of adjacency rows.  A list counter packs (items << 33 | edges): one
// atomicAdd hands out an item index and the item's first virtual edge, so
// epos stays non-decreasing in the item index.  For every item the list keeps
// its vertex, epos and delta = (CSR row start) - epos, so the CSR position of
// virtual edge e of item j is e + delta[j].
constexpr int kPackShift = 33;
constexpr uint64_t kPackEdgeMask = (1ull << kPackShift) - 1;

struct RowList {
  int32_t* v;
  int64_t* epos;
  int64_t* delta;
  int32_t* aux;                 // optional per-item payload (may be null)
  unsigned long long* counter;  // packed (items << 33 | edges)
#ifdef CC_DEBUG
  int64_t cap;                  // items the arrays hold
  int* err;                     // error word for a failed check
#endif
};

// Warp-aggregated append of one item per lane with want == true.  All 32
// lanes must call it.
__device__ __forceinline__ void warp_append_rows(bool want, int32_t v, int64_t row, int64_t edges, int32_t aux,
                                                 const RowList& L) {
  const int lane = threadIdx.x & 31;
  const unsigned mask = __ballot_sync(FULL, want);
  if (mask == 0) return;
  const int64_t mine = want ? edges : 0;
  const int64_t ex = warp_inclusive_sum<int64_t>(mine) - mine;
  const int64_t tot = __shfl_sync(FULL, ex + mine, 31);
  const int leader = __ffs(mask) - 1;
  unsigned long long old = 0;
  if (lane == leader)
    old = atomicAdd(L.counter, ((unsigned long long)__popc(mask) << kPackShift) | (unsigned long long)tot);
  old = __shfl_sync(FULL, old, leader);
  if (want) {
    const int64_t j = (int64_t)(old >> kPackShift) + __popc(mask & ((1u << lane) - 1u));
    const int64_t ep = (int64_t)(old & kPackEdgeMask) + ex;
    if (!CC_IN_BOUNDS(j, L.cap, L.err)) return;
    L.v[j] = v;
    L.epos[j] = ep;
    L.delta[j] = row - ep;
    if (L.aux) L.aux[j] = aux;
  }
}

}  // namespace ccg
