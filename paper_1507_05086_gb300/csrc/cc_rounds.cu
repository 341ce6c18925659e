// cc_rounds.cu -- the bulk-synchronous rounds of C4 and ClusterWild! (Alg. 2)
// as one persistent cooperative kernel.
//
// All rounds run inside a single launch.  Phases are separated by grid
// barriers; block 0 is the coordinator: at every barrier it waits for all
// blocks, does the serial bookkeeping of the round (Delta walk, batch size,
// selection windows, statistics) on state it keeps in its own shared memory,
// publishes a 128-byte plan, whose words carry the barrier's number and so
// release the others.  Every wait is bounded.  The host is not involved between
// rounds.
//
// Per-vertex state: one 32-bit word st[v]
//   alive ............ kAlive | bound of the residual degree
//   clustered ........ kLab + center rank
//   active ............ kActive / kActCenter / kActNon (undecided or
//                       ClusterWild! center / C4 center / C4 non-center)
// C4 keeps every vertex's rank in arank[v] (above kStateInL2 vertices: an active's).  A center keeps its active marker for
// good (its label is its own rank, arank); the actives of the current round
// are the ones whose rank is >= r0, the round's first active rank.
//
// Attachment (createCluster, concurrency rule 2): a center of rank r lowers
// st[u] with atomicMin(kLab + r).  Alive words compare above every label and
// active markers below, so one compare-then-atomicMin does rule 2 and skips
// clustered and active vertices.
//
// The alive word holds an upper bound of the residual degree: the full degree
// at first, later the exact residual degree as of the vertex's last recount
// (degrees only fall, so a value once exact stays a bound).  Nothing is
// decremented when a vertex leaves; only the few vertices that can hold the
// maximum are recounted, once per round (see co_delta).
// The alive tests of the adjacency passes and of the selection scans read a
// removal tag instead of the state word: 4 bits per vertex, 0 while alive,
// else 1 + (removal round mod 15), an eighth of the state words' footprint, so
// that the random reads mostly hit L2.  A tag equal to the current round's
// only says "maybe removed this round" (a vertex removed 15, 30, ... rounds
// earlier carries it too); the state word decides.
//
// Delta_i (max residual degree, exact every round) comes from a heavy list H
// that holds every alive vertex whose bound was >= tau when H was built: the
// rows of H's vertices with the largest bounds are recounted until the largest
// exact degree found is at least every other bound.  Selection scans pi itself
// from a cursor (entry i is the vertex of rank i) and skips removed vertices
// by their tag; a selected vertex of bound 0 is a singleton center for which
// nothing is written (the label pass reads its alive word of degree 0).
//
// Every adjacency pass is edge-balanced (row_walk), so hub rows of power-law
// graphs are split across many warps.
#include <cstdint>

#include "cc_device.cuh"
#include "cc_internal.h"

namespace ccg {
namespace {

constexpr int kThreads = 512;
constexpr int kRowB = 4;                     // entries in flight per lane (8 spill at 64 registers)
constexpr int kScanU = 4;                    // list entries per thread per scan step
// Windows of up to this many entries per block are selected and attached in one
// pass (select_attach).  ClusterWild!: planted 10^6 at eps 0.1 6.69 -> 5.47 ms
// for 211 rounds, R-MAT 20 3.67 -> 3.19 for 102.  C4: planted 0.7M at eps 0.9
// 1.44 -> 1.23 ms for 22 rounds, R-MAT 24 12.2 -> 11.4 for 145.  Longer windows
// take as long either way (ClusterWild! on R-MAT 26: 17.7 / 17.6 / 17.7 / 17.6
// ms for 0 / 1024 / 2048 / 4096; C4 on R-MAT 24: 11.6 / 11.4 / 11.4 for 1024 /
// 2048 / 8192), and their rows are better shared out by the list of all actives.
constexpr int64_t kFuseWindow = 2048;
constexpr int32_t kLongAttach = 8192;        // rows longer than this are walked by the whole grid
constexpr int kSelU = 2;                     // window entries per thread per selection step
// Up to this many vertices (64 MB of state words, which L2 holds) selection
// also reads the bounds and spares the rows of vertices known to have no alive
// neighbour; above, those rows cost less than a random DRAM read per active.
// C4 holds the inverse of pi up to here: beyond, its random writes (2.4 ms at 2^26)
// and reads cost as much as the phases that it spares (set-up and rounds of C4 on
// R-MAT 25 / 26 16.8 / 25.3 ms, with it 16.7 / 26.2).
constexpr int64_t kStateInL2 = int64_t(1) << 24;
constexpr int kInlineWindow = 1024;          // without it, windows up to this long are selected inside the barrier
constexpr int64_t kDescStride = 16;          // look-back descriptors: one per 128-byte line
constexpr int kAlgoC4 = 1, kAlgoCW = 2;
constexpr int kRun = 0, kDone = 1, kSelect = 2, kAbort = 3, kDrawBatch = 6;   // kRun: the active set is there
constexpr int kRebuildOrder = 7, kRebuildAlive = 8; // heavy list from the degree order, from the alive vertices
constexpr int kRecount = 9, kRecountLong = 10;      // degree recounts
constexpr int kResolve = 11;                 // C4: the round's blocked actives are listed
// where co_delta takes up again, or what it does next
constexpr int kDScan = 0, kDCounted = 1, kDRebuild = 2, kDPlanned = 3, kDDone = 4;
constexpr int kHList = kThreads;             // heavy lists up to this long: every block lists all of them
// Heavy lists up to this long, one read of the block, are looked at inside the
// barrier (10K Erdos-Renyi 583 us of rounds, R-MAT 24 11.2 ms; 8192: 647, 11.5;
// 1024: 589, 11.2, and planted 10^6 5.7 ms against 5.6).
constexpr int kHere = kScanU * kThreads;
constexpr int kHRows = 1024;                 // rows that one block recounts at once
constexpr int kHPick = 4096;                 // vertices that one block picks at once
// Picked rows of more than kManyEdges entries together: about kFewEdges of them are
// recounted first (300 cliques of 300, ClusterWild! at eps 0.05 / 0.01: 5.5 / 18.8 ms
// without, 2.4 / 6.1 with; 16384: 2.3 / 5.8, 49152: 2.9 / 7.8.  Where no row can be
// left out it costs: R-MAT 24 and 26 and batches of Chung-Lu graphs 0.5 %).
constexpr int kManyEdges = 24576, kFewEdges = 2048;
constexpr int kInlineEdges = 8192;           // recounts up to this many entries run inside the barrier
constexpr int32_t kLongRow = 1024;           // rows above this are not recounted by one block alone
constexpr int32_t kTightest = 8;             // heavy lists reach down to 1 - 2^-8 of the largest bound at most
// Defaults of the run-time schedule settings (Tuning; cc_tuning in the C ABI)
constexpr int32_t kInlineH = kHere;          // heavy lists up to this size (and kHere) are looked at by the coordinator
constexpr int32_t kInlineDecide = 4096;      // C4 blocked lists up to this size are decided by the coordinator
constexpr int32_t kInlineRebuild = 8192;     // heavy-list rebuilds over prefixes up to this size run in the coordinator
constexpr int32_t kHeavyShift = 1;           // heavy-list threshold tau = max(1, D >> kHeavyShift)
// C4 blocked actives are resolved one warp each (one grid phase) when every
// one of them has a warp and no blocked row is longer than this
constexpr int32_t kWarpResolveRow = 1024;

// State word of a vertex (uint32):
//   alive ........... kAlive | bound of the residual degree
//   clustered ....... kLab + center rank
//   active this round kActive (undecided, or a ClusterWild! center),
//                     kActCenter / kActNon (C4 center / non-center)
constexpr uint32_t kAlive = 0x80000000u, kDegMask = 0x7FFFFFFFu, kLab = 16;
constexpr uint32_t kActive = 1, kActCenter = 2, kActNon = 3;
constexpr int kTagCycle = 15;                // removal tags 1..15
__device__ __forceinline__ bool is_alive(uint32_t x) { return x >= kAlive; }
__device__ __forceinline__ uint32_t deg_of(uint32_t x) { return x & kDegMask; }
__device__ __forceinline__ bool is_active(uint32_t x) { return x < kLab; }

// The cluster of a member as the objective compares it: its state word; a
// center or singleton matches nothing (member-center edges are counted by
// finish_vertices).
__device__ __forceinline__ uint32_t member_id(uint32_t x) { return x >= kLab && x < kAlive ? x : 0xFFFFFFFFu; }

__device__ __forceinline__ int64_t rtag_words(int64_t n) { return (n >> 3) + 1; }
__device__ __forceinline__ uint32_t rtag_of(const uint32_t* rtag, int32_t v) {
  return (ldcg(rtag + (v >> 3)) >> ((v & 7) * 4)) & 15u;
}
__device__ __forceinline__ void set_rtag(uint32_t* rtag, int32_t v, uint32_t tag) {
  atomicOr(rtag + (v >> 3), tag << ((v & 7) * 4));      // result unused
}

// ---- the practical schedule of Sec. 5 ------------------------------------------
// Delta-hat starts at the maximum degree and halves every P rounds,
// P = (2/eps) ln(n log Delta / delta) with delta = 1/10, in integers: ln x =
// ln 2 log2 x with log2 rounded up to a bit length.  The batch B_i is
// binomial over the n - cursor unprocessed ranks of pi with p = eps /
// Delta-hat_i: the number of the round's SplitMix64 draws (a stream seeded
// from the seed of pi and the round) below T_i = floor(p 2^64).  A_i = the
// alive vertices among the next B_i ranks.
__device__ __forceinline__ int64_t bit_length(uint64_t x) { return x ? 64 - __clzll((long long)x) : 0; }

__device__ __forceinline__ int64_t sec5_period(int64_t n, int64_t max_deg, int64_t eps_ppm) {
  const int64_t l = bit_length((uint64_t)n) + bit_length((uint64_t)bit_length((uint64_t)(max_deg > 2 ? max_deg : 2))) + 4;
  return (int64_t)((2ull * 693147ull * (uint64_t)l + (uint64_t)eps_ppm - 1) / (uint64_t)eps_ppm);
}

__device__ __forceinline__ int64_t sec5_delta_hat(int64_t max_deg, int64_t period, int64_t round) {
  const int64_t h = round / period;
  const int64_t d = h >= 63 ? 0 : (max_deg >> h);
  return d > 1 ? d : 1;
}

// floor(eps_ppm 2^64 / (10^6 dhat)) for eps_ppm < 10^6 dhat: 64 quotient bits
// by long division (12, 12, 12, 12, 12, 4 bits; the remainder stays < 2^51).
__device__ __forceinline__ uint64_t sec5_threshold(int64_t eps_ppm, int64_t dhat, bool* all) {
  const uint64_t den = 1000000ull * (uint64_t)dhat;
  *all = (uint64_t)eps_ppm >= den;
  if (*all) return ~0ull;
  uint64_t r = (uint64_t)eps_ppm, t = 0;
#pragma unroll 1
  for (int s = 0; s < 5; ++s) {
    r <<= 12;
    t = (t << 12) | (r / den);
    r %= den;
  }
  r <<= 4;
  return (t << 4) | (r / den);
}

// Draw j of round i's stream: the j-th output of SplitMix64 seeded with s.
__device__ __forceinline__ uint64_t sec5_draw(uint64_t s, uint64_t j) {
  return perm_key(0, s + j * 0x9E3779B97F4A7C15ull);     // state s + (j+1) gamma, mixed
}

template <class T>
__device__ __forceinline__ T vload(const T* p) { return *reinterpret_cast<const volatile T*>(p); }

__device__ __forceinline__ void atom_add_release(unsigned long long* p, unsigned long long v) {
  asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
constexpr unsigned long long kArriveError = 1ull << 63;

constexpr int kPlanWords = sizeof(Plan) / 4;
// Teams above kPlanAlone blocks wait on kPlanCopies copies of the plan: the 300
// blocks of a grid polling one copy keep its L2 slice busy for longer than a
// copy costs.
constexpr unsigned kPlanAlone = 32;
static_assert(kPlanWords == 32, "one warp reads the plan");

// Coordinator state, in block 0's shared memory for the whole kernel.
struct Coord {
  int64_t n, n_alive, cursor, al_len, k, round, stats_cap, eps_ppm;
  int64_t need, win_lo, win_len, r_edges, fix_iter;
  int64_t h_len;                 // heavy list length
  int64_t nz_len;                // alive non-isolated vertices, as of the last look at all of them
  int32_t tau, delta, max_deg;
  int32_t d_lb;                  // largest exact degree recounted this round (-1: none)
  int32_t d_th;                  // heavy-list vertices of this bound or more are recounted
  int32_t d_other;               // largest bound among the others
  int32_t tight;                 // the heavy list reaches down to ub - (ub >> tight)
  int32_t tau_next;              // the raised tau of a planned look
  int32_t d_top, d_drop;         // largest bound at the first look; how far Delta fell below it lately
  int algo, rebuilds_in_row;
  int delta_zero;                // a rebuild found no alive vertex with an alive neighbour
  int est;                       // the Sec. 5 schedule: Delta-hat and binomial batches
  int64_t period, rank_cursor;   // rounds per halving of Delta-hat; ranks of pi passed
  int ahead;                     // the next batch has been drawn
  int32_t withhold;              // test hook (Ctl::withhold)
  int32_t round_ended;           // this barrier ended a round
  int64_t batch_end;             // rank (index in pi) that ends the round's batch
  unsigned long long t0, round_t0;
  unsigned long long ph_ns[8];
};

// Shared memory of one block (dynamic: larger than the 48 KB static limit).
// Bucket-sort scratch of the in-kernel permutation (batched jobs).
constexpr int kPermCap = 1536;        // vertices per bucket sorted in shared memory
constexpr int kPermSubBits = 10;
constexpr int kPermSub = 1 << kPermSubBits;
constexpr int kPermMaxBuckets = 4096;

struct PermSmem {
  uint64_t sk[kPermCap];
  uint64_t ok[kPermCap];
  int32_t sv[kPermCap];
  int32_t ov[kPermCap];
  int32_t cnt[kPermSub + 1];
  int32_t hist[kPermMaxBuckets];
};

// Round tallies of a block (Shared::tal), added up over the team at the end of
// a round.
enum { kTCenters = 0, kTAttached, kTNonCenter, kTBlocked, kTEdges, kTallies };

// Rows to be recounted (slot order = heavy-list order).
struct HeavyList {
  int64_t pos[kHRows];
  int64_t row[kHRows];
  int32_t len[kHRows];
  int32_t v[kHRows];             // -1: recounted elsewhere
  unsigned cnt[kHRows];          // alive entries found (recount by one block)
  int32_t pick[kHPick];          // vertices whose rows are recounted next
};

// The rows of a tile's actives (select_attach).
struct TileRows {
  int64_t row[kThreads * kSelU];
  int32_t pos[kThreads * kSelU], len[kThreads * kSelU], rank[kThreads * kSelU], v[kThreads * kSelU];
  uint8_t blocked[kThreads * kSelU];
};

struct Shared {
  Plan plan;
  Coord co;
  int ok;
  int failed;                    // this block has recorded an error
  int dec;
  int64_t scr[33];
  int64_t bcast[8];
  unsigned long long tal[kTallies];     // round tallies of the block (flushed at round end)
  int32_t scr32[32];
  // the selection's outcome: alive entries of the window, the round's first
  // active rank, the next cursor, the active list (items << 33 | entries)
  int64_t sel_total, sel_cursor;
  int32_t sel_r0;
  unsigned long long sel_pack;
  int32_t h_picked, h_kept;      // vertices picked for the recount; entries of a compacted list
  int32_t h_best;                // largest exact degree that this block knows of
  int32_t drawn;                 // Sec. 5: the last batch (Plan::drop) that this block drew its share of
  int64_t nz_cnt;                // alive non-isolated vertices of this block's segment (-1: not looked at yet)
  union {
    HeavyList hl;
    PermSmem perm;
    TileRows rows;
  } u;
};

// The blocks that run one clustering job: the whole grid, or a team of
// G blocks inside a batched launch (bid = this block's rank in the team).
// It lives in shared memory: the passes are functions of their own (each with
// its own register allocation), and from there they read a field in one step.
template <int kPerSM>
struct K {
  RoundBuffers B;
  Ctl* C;
  Shared* S;
  unsigned G;
  unsigned bid;
  unsigned epoch;
  int algo;                      // C4 or ClusterWild!
  bool est;                      // by the Sec. 5 schedule

  // One round tally of this block; all lanes of the warp call it.
  __device__ __forceinline__ void tally(int which, int32_t x) {
    const int32_t sum = __reduce_add_sync(FULL, x);
    if (sum && (threadIdx.x & 31) == 0) atomicAdd(&S->tal[which], (unsigned long long)sum);
  }
  // Block-wide sums as one copy of the code (see sync).
  struct Scan {
    int64_t ex, tot;
  };
  __device__ __noinline__ Scan scan(int64_t x) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t inc = warp_inclusive_sum_rolled(x);
    __syncthreads();                       // earlier readers of scr
    if (lane == 31) S->scr[warp] = inc;
    __syncthreads();
    const int64_t w = lane < kThreads / 32 ? S->scr[lane] : 0, wi = warp_inclusive_sum_rolled(w);
    return Scan{__shfl_sync(FULL, wi - w, warp) + inc - x, __shfl_sync(FULL, wi, 31)};
  }
  __device__ __noinline__ int32_t sum_i32(int32_t x) { return block_sum_i32(x, S->scr32); }
  __device__ __noinline__ int32_t max_i32(int32_t x) { return block_max_i32(x, S->scr32); }

  // This warp among the team's warps.
  __device__ __forceinline__ int team_warp() const { return (int)((threadIdx.x >> 5) * G + bid); }
  __device__ __forceinline__ int team_warps() const { return (int)((G * blockDim.x) >> 5); }

  // A walk of the team over the E entries of n rows.  Warps are numbered across
  // the blocks first (warp w of block b is w * G + b), so a short walk spreads
  // over every SM instead of the first few blocks.
  // A walk of at most two batches of 32 entries per warp takes one entry per
  // lane at a time: a third of the code, which such a walk spends its time
  // fetching (f takes either batch).
  template <class At, class Load, class F>
  __device__ __forceinline__ void walk(int64_t n, int64_t E, const At& at, const Load& load, F&& f) {
    const WalkShape shape{B.tune.walk_batches, B.tune.prefetch_ahead};
    if (E <= 64 * (int64_t)team_warps()) row_walk<1>(team_warp(), team_warps(), (int32_t)n, E, B.col, shape, at, load, f);
    else row_walk<kRowB>(team_warp(), team_warps(), (int32_t)n, E, B.col, shape, at, load, f);
  }

  __device__ __forceinline__ const Plan& P() const { return S->plan; }
  // Whether windows can be selected and attached in one pass (C4: by the inverse of pi).
  __device__ __forceinline__ bool fused() const { return algo == kAlgoCW || B.n <= kStateInL2; }
  // The current heavy list (its buffer changes when the grid cuts it down).
  __device__ __forceinline__ int32_t* hv() const { return S->plan.hv_sel ? B.hv2 : B.hv; }
  __device__ __forceinline__ Coord& co() const { return S->co; }
  // Records an error; the coordinator sees it in the arrivals.
  __device__ __noinline__ void fail(int code) {
    if (atomicCAS(&C->err, kOk, code) == kOk) atomicOr(&C->arrive, kArriveError);
    S->failed = 1;
  }

  // ---------------- grid barrier with the coordinator -------------------------
  // All blocks call sync(); block 0 waits for every arrival, books the time
  // since the previous barrier to phase `cat`, runs act() with its whole
  // block (writing S->plan), publishes the plan and releases.  The others
  // wait for the release and copy the plan.  Returns false once the run
  // must stop (error, or the plan says so).
  // The waits are functions of their own: a phase is mostly straight-line code
  // that runs once, so what the phases share should be fetched once.
  template <class A>
  __device__ __forceinline__ bool sync(int cat, A&& act) {
    if (bid != 0) return wait_release();
    if (co_arrived(cat)) act();
    return co_release();
  }

  // Coordinator: waits for every arrival; false after an error.
  __device__ __noinline__ bool co_arrived(int cat) {
    __syncthreads();
    if (threadIdx.x == 0) {
      ++epoch;
      int ok = 1;
      if (G > 1) {
        atom_add_release(&C->arrive, 1ull);
        const unsigned long long target = (unsigned long long)G * epoch;
        const uint64_t t0 = globaltimer_ns();
        unsigned spins = 0;
        unsigned long long x;
        while ((x = ld_relaxed_u64(&C->arrive)) < target) {
          if ((++spins & 63) == 0 && globaltimer_ns() - t0 > kBarrierLimitNs) { fail(kErrTimeout); ok = 0; break; }
        }
        if (x & kArriveError) ok = 0;
        fence_gpu();
      }
      if (S->failed || (kDebugChecks && ld_volatile_int(&C->err) != kOk)) ok = 0;
      const unsigned long long now = globaltimer_ns();
      S->co.ph_ns[cat] += now - S->co.t0;
      S->co.t0 = now;
      S->co.round_ended = 0;
      S->ok = ok;
    }
    __syncthreads();
    return S->ok != 0;
  }

  // Coordinator: publishes the plan.  Every word goes out in one 8-byte store
  // with the barrier's number above it, so whoever sees the number has the
  // word; the fence orders what this block and, through the arrivals, every
  // block wrote before it.
  __device__ __noinline__ bool co_release() {
    __syncthreads();
    if (threadIdx.x == 0) {
      // an error (here or in any block) travels in the plan as the abort state
      if (!S->ok || S->failed || (kDebugChecks && ld_volatile_int(&C->err) != kOk)) S->plan.state = kAbort;
      // test hook: after the chosen round the release is withheld; the other
      // blocks' bounded waits run out (kErrTimeout) and every block unwinds
      if (G > 1 && S->co.round_ended && S->co.withhold != 0 && S->co.round == S->co.withhold) {
        S->plan.state = kAbort;
        S->ok = 2;
      }
    }
    __syncthreads();
    const unsigned copies = G > kPlanAlone ? kPlanCopies : G > 1 ? 1 : 0;
    if (S->ok != 2 && threadIdx.x < kPlanWords * copies) {
      const uint32_t w = reinterpret_cast<const uint32_t*>(&S->plan)[threadIdx.x % kPlanWords];
      fence_gpu();
      st_relaxed_u64(C->plan_ll + threadIdx.x, ((unsigned long long)epoch << 32) | w);
    }
    return S->plan.state != kAbort;
  }

  // The other blocks: arrive, wait for the release and take the plan over.
  __device__ __noinline__ bool wait_release() {
    __syncthreads();
    if (threadIdx.x < kPlanWords) {          // the first warp
      if (threadIdx.x == 0) {
        ++epoch;
        atom_add_release(&C->arrive, 1ull);
      }
      __syncwarp();
      const unsigned long long* const src =
          C->plan_ll + (G > kPlanAlone ? bid % kPlanCopies : 0) * kPlanWords + threadIdx.x;
      const unsigned e = epoch;
      const uint64_t t0 = globaltimer_ns();
      unsigned spins = 0;
      bool released = true;
      unsigned long long x = ld_relaxed_u64(src);
      while (!__all_sync(FULL, (unsigned)(x >> 32) == e)) {
        if ((++spins & 63) == 0) {
          if (ld_volatile_int(&C->err) != kOk) released = false;
          else if (globaltimer_ns() - t0 > kBarrierLimitNs) {
            fail(kErrTimeout);
            released = false;
          }
          if (__any_sync(FULL, !released)) break;
        }
        x = ld_relaxed_u64(src);
      }
      fence_gpu();
      reinterpret_cast<uint32_t*>(&S->plan)[threadIdx.x] = (uint32_t)x;
      __syncwarp();
      // without a release the copy is stale and the state becomes the abort state
      if (__any_sync(FULL, !released) && threadIdx.x == 0) S->plan.state = kAbort;
    }
    __syncthreads();
    return S->plan.state != kAbort;
  }

  __device__ bool sync(int cat) {
    return sync(cat, [] {});
  }

  // blocked actives; the payload initialises each one's pull slot (no center yet)
  __device__ RowList blk_list() const { return RowList{B.b_j, B.b_e, B.b_d, B.pull, &C->blk_pack CC_ROWLIST_CHECK(B.n, &C->err)}; }

  // contiguous slice of [lo, lo+len) for this block
  __device__ __forceinline__ void slice(int64_t lo, int64_t len, int64_t* s, int64_t* e) const {
    const uint32_t chunk = ((uint32_t)len + G - 1) / G;           // len < 2^31
    *s = lo + (int64_t)chunk * bid;
    *e = *s + chunk < lo + len ? *s + chunk : lo + len;
    if (*s > *e) *s = *e;
  }

  // ---------------- coordinator actions ----------------------------------------
  __device__ void co_init() {
    if (threadIdx.x == 0) {
      Coord& c = co();
      c.n = B.n;
      c.n_alive = B.n;
      c.cursor = 0;
      c.al_len = B.n;
      c.max_deg = B.max_deg;
      c.tau = 0x7FFFFFFF;         // empty heavy list: the first round rebuilds it
      c.h_len = 0;
      c.nz_len = B.nz_n;          // non-isolated vertices, from the graph
      c.delta_zero = 0;
      c.d_drop = 0;
      c.tight = 1;
      c.r_edges = 0;
      c.round = 0;
      c.rebuilds_in_row = 0;
      c.algo = vload(&C->algo);
      c.eps_ppm = vload(&C->eps_ppm);
      c.withhold = vload(&C->withhold);
      c.est = c.algo >= 3;                // the Sec. 5 schedule
      if (c.est) c.algo -= 2;
      c.period = c.est ? sec5_period(c.n, c.max_deg, c.eps_ppm) : 0;
      c.rank_cursor = 0;
      c.ahead = 0;
      c.stats_cap = B.stats_cap;
      Plan& p = S->plan;
      p = Plan{};
      p.r0 = -1;
    }
    if (threadIdx.x < kHList) B.h_acc[threadIdx.x] = 0;
    __syncthreads();
    if (threadIdx.x == 0) S->dec = co_next();
    __syncthreads();
    co_go_on();
  }

  // Coordinator: with Delta known, set k and the first selection window.
  __device__ __noinline__ void plan_selection(int32_t delta) {
    if (threadIdx.x == 0) {
      Coord& c = co();
      Plan& p = S->plan;
      int64_t k;
      if (delta <= 0) k = c.n_alive;
      else {
        const unsigned long long num = (unsigned long long)c.eps_ppm * (unsigned long long)c.n_alive;
        const unsigned long long den = 1000000ull * (unsigned long long)delta;
        k = (int64_t)((num + den - 1) / den);
        if (k < 1) k = 1;
        if (k > c.n_alive) k = c.n_alive;
      }
      c.delta = delta;
      c.k = k;
      c.need = k;
      c.win_lo = c.cursor;
      const int64_t avail = c.al_len - c.cursor;
      const int64_t est = (int64_t)((float)k * ((float)avail / (float)c.n_alive) * 1.05f) + 256;   // a guess
      c.win_len = est < avail ? est : avail;
      if (c.est) {
        // Sec. 5: the whole window of the round's batch, every alive entry of it
        c.k = 0;                          // set from the window's alive count
        c.need = INT64_MAX / 4;
        c.win_len = c.batch_end - c.cursor;
        // The next batch depends on the cursor alone, not on what this round
        // removes: it is drawn in this round's first phase.
        if (c.rank_cursor < c.n) plan_draw(c.round + 1);
      }
      C->act_pack = 0; C->blk_pack = 0; C->blk_maxlen = 0;
      C->r_centers = 0; C->r_attached = 0; C->r_noncenter = 0; C->r_blocked = 0; C->r_edges = 0;
      C->r0 = -1;
      S->sel_r0 = -1;
      S->sel_cursor = 0;
      S->sel_pack = 0;
      p.state = kSelect;
      p.k = c.k;
      p.need = c.need;
      p.win_lo = c.win_lo;
      p.win_len = c.win_len;
      p.th = (int32_t)c.cursor;         // labels from this rank on are this round's
      p.r0 = -1;
      p.tag = (int32_t)(c.round % kTagCycle) + 1;
    }
    __syncthreads();
    select_here();
  }

  // Coordinator, at a round boundary (thread 0): finish or draw the Sec. 5 batch
  // (1), a round with Delta known (2), or find Delta (0).
  __device__ __forceinline__ int co_next() {
    Coord& c = co();
    Plan& p = S->plan;
    if (c.n_alive <= 0) { p.state = kDone; return 1; }
    if (c.est) {
      c.delta = (int32_t)sec5_delta_hat(c.max_deg, c.period, c.round);
      if (c.ahead) {                      // drawn during this round's first phase
        c.ahead = 0;
        batch_drawn((int64_t)vload(&C->drawn));
        return 2;
      }
      plan_draw(c.round);                 // the first batch: a phase of its own
      p.state = kDrawBatch;
      return 1;
    }
    if (c.round == 0) {                   // every degree is still the full one
      c.delta = c.max_deg;
      if (c.max_deg <= 0) c.delta_zero = 1;
      return 2;
    }
    if (c.delta_zero) {                   // every alive vertex is isolated: Delta = 0
      c.delta = 0;
      return 2;
    }
    // every bound is at most the last Delta: start a little below it
    c.d_lb = -1;
    c.d_top = -1;
    c.d_th = below(c.delta, c.d_drop);
    return 0;
  }
  // Sec. 5: plans the draws of round `round` (no Delta): trials, threshold bits,
  // stream seed; d_lb = 2: every trial succeeds, else 1.
  __device__ __noinline__ void plan_draw(int64_t round) {
    const Coord& c = co();
    Plan& p = S->plan;
    bool all;
    p.long_E = (int64_t)sec5_threshold(c.eps_ppm, sec5_delta_hat(c.max_deg, c.period, round), &all);
    p.long_n = c.n - c.rank_cursor;
    p.undecided = (int64_t)perm_key(vload(&C->seed) ^ 0x5851F42D4C957F2Dull, (uint64_t)round);
    p.d_lb = all ? 2 : 1;
    p.drop = (int32_t)(round & 0x3FFFFFFF);      // tells the blocks that this batch is a new one
    C->drawn = 0;
  }
  // The batch of b ranks of pi from the cursor on.
  __device__ void batch_drawn(int64_t b) {
    Coord& c = co();
    const int64_t end_rank = c.rank_cursor + b;
    c.batch_end = end_rank < c.al_len ? end_rank : c.al_len;      // entry i of the list has rank i
    c.rank_cursor = end_rank;
    if (end_rank > c.n) fail(kErrInternal);
  }
  __device__ __forceinline__ void co_go_on() {
    const int dec = S->dec;
    if (dec == 2) plan_selection(co().delta);
    else if (dec == 0) co_delta(kDScan);
  }

  // The recount threshold when the largest bound is x: as far below it as
  // Delta fell lately, but by no more than a quarter.
  __device__ static int32_t below(int32_t x, int32_t drop) {
    const int32_t lo = x - (x >> 2);
    const int32_t t = x - drop > lo ? x - drop : lo;
    return t > 1 ? t : 1;
  }

  // Exact Delta without decrements.  Every alive vertex outside H has a bound
  // < tau.  Alive vertices of H with a bound >= some threshold are picked and
  // their degrees recounted; d_lb is the largest exact degree found, d_other
  // the largest bound that was not picked.  Then, until Delta is known:
  //   a bound above d_lb is left: recount those as well;
  //   d_lb >= tau - 1: no vertex can have more, Delta = d_lb;
  //   else H no longer holds the maximum: rebuild it with a lower tau.
  // A pass with threshold d_lb + 1 leaves no larger bound, so each H is
  // recounted at most twice.  The first threshold decides between rows
  // recounted in vain and second passes: taking the recent fall of Delta, the
  // recounted rows hold 0.15-0.6 of the graph's entries over a whole clustering
  // (R-MAT 26 0.15, planted 10^6 0.55, eps 0.5 and 0.1) and 10-15 % of the rounds
  // need a second pass; recounting all of H every round reads 1.6-3.3.
  // Decrementing the neighbours of every removed vertex instead read 0.85-0.9
  // of the entries, with an atomic for half of them.
  // A list of up to kHere vertices is looked at here (inline_heavy), and
  // recounted here while its rows are short: a grid phase would cost a barrier
  // and the same dependent loads.
  __device__ __noinline__ void co_delta(int step) {
    Coord& c = co();
    for (;;) {
      if (step == kDScan) {
        const int64_t hl = c.h_len;
        step = kDPlanned;
        if (hl <= kHere && (hl <= B.tune.inline_heavy || hl == 0)) {
          look_here();
          const int picked = S->h_picked;
          int64_t E = 0;
          if (picked > 0 && picked <= kHRows) E = prepare_rows(0, picked, false);
          if (picked <= kHRows && (E <= kInlineEdges || G == 1)) {
            if (picked > 0) {
              const int32_t best = block_recount(picked, E);
              if (threadIdx.x == 0) {
                c.r_edges += E;
                if (best > c.d_lb) c.d_lb = best;
              }
            }
            step = kDCounted;
          }
        }
        if (step == kDPlanned && threadIdx.x == 0) {
          Plan& p = S->plan;
          p.state = kRecount;
          p.win_len = c.h_len;
          p.pad0 = G > 1 && c.h_len <= kHList ? 1 : 0;       // every block lists all of H
          p.th = c.d_lb < 0 && c.h_len <= kHere && c.d_top > 0 ? below(c.d_top, c.d_drop) : c.d_th;
          p.d_lb = c.d_lb;
          p.drop = c.d_drop;
          p.long_n = 0;
          if (c.h_len > kHere) {
            // the list is too long: keep what the next rounds will ask for (one block
            // as well: 160 jobs on grids of 10^6 vertices at eps 0.1 200 ms without, 81 with)
            if (c.tight < kTightest) c.tight += 1;
            const int32_t d2 = c.delta - 2 * c.d_drop - 1, t = c.delta - (c.delta >> c.tight);
            const int32_t up = d2 < t ? d2 : t;
            c.tau_next = up > c.tau && c.d_lb < 0 && c.rebuilds_in_row == 0 ? up : c.tau;     // not after a rebuild
            p.long_n = c.tau_next;
            C->h_pack = 0;
          }
          reset_looked();
        }
        __syncthreads();
      }
      if (step == kDPlanned) return;
      if (threadIdx.x == 0) {
        int next = kDScan;
        if (c.d_other > c.d_lb && c.d_other > 0) {
          c.d_th = c.d_lb < 0 ? below(c.d_other, c.d_drop) : c.d_lb + 1;
        } else {
          const int32_t D = c.d_lb > 0 ? c.d_lb : 0;
          if (D + 1 >= c.tau) {
            const int32_t fall = c.d_top > D ? c.d_top - D : 0;
            c.d_drop = fall > c.d_drop ? fall : c.d_drop - ((c.d_drop - fall) >> 2);
            if (D <= 0) c.delta_zero = 1;
            c.delta = D;
            next = kDDone;
          } else {
            next = kDRebuild;
          }
        }
        S->dec = next;
      }
      __syncthreads();
      step = S->dec;
      __syncthreads();
      if (step == kDDone) { plan_selection(c.delta); return; }
      if (step == kDRebuild) {
        if (!rebuild()) return;
        step = kDScan;
      }
    }
  }

  // The largest bounds of a look over H (thread 0 of the coordinator).
  __device__ void note_looked(int32_t other, int32_t top) {
    co().d_other = other;
    if (co().d_top <= 0) co().d_top = top;
  }

  // Appends v to S->u.hl.pick where take is set (all lanes call it).
  __device__ __forceinline__ void pick(bool take, int32_t v) {
    const unsigned m = __ballot_sync(FULL, take);
    if (m == 0) return;
    int at = 0;
    if ((threadIdx.x & 31) == 0) at = atomicAdd(&S->h_picked, __popc(m));
    at = __shfl_sync(FULL, at, 0) + __popc(m & ((1u << (threadIdx.x & 31)) - 1u));
    if (take) S->u.hl.pick[at] = v;
  }

  // Coordinator block, a heavy list of up to kHere vertices: picks the alive ones
  // with a bound >= th, th = d_lb + 1 or a little below the largest bound while
  // d_lb < 0, and compacts the list to its alive vertices.
  __device__ __noinline__ void look_here() {
    Coord& c = co();
    const int len = (int)c.h_len;
    int32_t v[kScanU], ub[kScanU], top = 0, alive = 0;
#pragma unroll
    for (int q = 0; q < kScanU; ++q) {
      const int i = q * kThreads + (int)threadIdx.x;
      v[q] = i < len ? ldcg(hv() + i) : -1;
    }
#pragma unroll
    for (int q = 0; q < kScanU; ++q) {
      const uint32_t x = v[q] >= 0 ? ldcg(B.st + v[q]) : 0u;
      ub[q] = is_alive(x) ? (int32_t)deg_of(x) : 0;
      top = ub[q] > top ? ub[q] : top;
      alive += ub[q] > 0 ? 1 : 0;
    }
    if (threadIdx.x == 0) S->h_picked = S->h_kept = 0;
    top = max_i32(top);
    // a second look costs no barrier here: a fraction of the recent fall
    const int32_t th = c.d_lb < 0 ? below(top, c.d_drop >> 2) : c.d_lb + 1;
    const bool pack = sum_i32(alive) < len - (len >> 2);    // a quarter has left (every entry is read by now)
    int32_t other = 0;
#pragma unroll
    for (int q = 0; q < kScanU; ++q) {
      const bool take = v[q] >= 0 && ub[q] >= th;        // th >= 1
      other = !take && ub[q] > other ? ub[q] : other;
      pick(take, v[q]);
      if (!pack) continue;
      const unsigned k = __ballot_sync(FULL, ub[q] > 0);
      int at = 0;
      if (k && (threadIdx.x & 31) == 0) at = atomicAdd(&S->h_kept, __popc(k));
      at = __shfl_sync(FULL, at, 0) + __popc(k & ((1u << (threadIdx.x & 31)) - 1u));
      if (ub[q] > 0) hv()[at] = v[q];
    }
    other = max_i32(other);
    if (threadIdx.x == 0) {
      if (pack) c.h_len = S->h_kept;
      c.d_th = th;
      note_looked(other, top);
    }
    __syncthreads();
  }

  // Block-wide, for a heavy list of len <= kHList vertices: the alive ones with a
  // bound >= th become the rows S->u.hl (in list order: every block makes the
  // same list), th as in look_here.  Returns their number and entries.
  __device__ __noinline__ void list_heavy(int64_t len, int32_t lb, int32_t drop, int64_t* items, int64_t* E) {
    HeavyList& hl = S->u.hl;
    const int32_t v = threadIdx.x < len ? ldcg(hv() + threadIdx.x) : -1;
    const uint32_t x = v >= 0 ? ldcg(B.st + v) : 0u;
    const int32_t ub = is_alive(x) ? (int32_t)deg_of(x) : 0;
    int64_t row = 0, end = 0;
    if (ub > 0) {                          // the row is asked for before the threshold is known
      row = __ldg(B.off + v);
      end = __ldg(B.off + v + 1);
    }
    const int32_t top = max_i32(ub);
    const int32_t th = lb < 0 ? below(top, drop) : lb + 1;
    const bool take = ub >= th;
    const int32_t other = max_i32(take ? 0 : ub);
    const int32_t n = take ? (int32_t)(end - row) : 0;
    const Scan sc = scan(take ? (int64_t(1) << kPackShift) | n : 0);
    if (take) {
      const int j = (int)(sc.ex >> kPackShift);
      hl.pos[j] = sc.ex & (int64_t)kPackEdgeMask;
      hl.len[j] = n;
      hl.row[j] = row;
      hl.v[j] = v;
    }
    if (bid == 0 && threadIdx.x == 0) {    // the coordinator's copy counts
      S->tal[kTEdges] += (unsigned long long)(sc.tot & (int64_t)kPackEdgeMask);
      note_looked(other, top);
    }
    *items = sc.tot >> kPackShift;
    *E = sc.tot & (int64_t)kPackEdgeMask;
    __syncthreads();
  }

  // Block-wide: the rows of pick[base, base + items), items <= kHRows, into
  // S->u.hl; returns their entries.  split: rows above kLongRow go to the
  // grid-wide list instead.
  __device__ __noinline__ int64_t prepare_rows(int base, int items, bool split) {
    constexpr int kPer = kHRows / kThreads;
    HeavyList& hl = S->u.hl;
    int32_t v[kPer], len[kPer];
    int64_t row[kPer];
    int64_t mine = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int i = threadIdx.x * kPer + q;
      v[q] = i < items ? hl.pick[base + i] : -1;
      row[q] = v[q] >= 0 ? __ldg(B.off + v[q]) : 0;
      len[q] = v[q] >= 0 ? (int32_t)(__ldg(B.off + v[q] + 1) - row[q]) : 0;
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      if (split && len[q] > kLongRow) {
        const unsigned long long old = atomicAdd(&C->long_pack, (1ull << kPackShift) | (unsigned long long)len[q]);
        const int64_t j = (int64_t)(old >> kPackShift);
        if (CC_IN_BOUNDS(j, B.n, &C->err)) {
          B.b_j[j] = v[q];
          B.b_e[j] = (int64_t)(old & kPackEdgeMask);
          B.b_d[j] = row[q];
          B.pull[j] = len[q];
          B.act_n[j] = 0;
        }
        v[q] = -1;
        len[q] = 0;
      }
      mine += len[q];
    }
    const Scan sc = scan(mine);
    int64_t ex = sc.ex;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int i = threadIdx.x * kPer + q;
      hl.pos[i] = ex;
      hl.row[i] = row[q];
      hl.len[i] = len[q];
      hl.v[i] = v[q];
      hl.cnt[i] = 0;
      ex += len[q];
    }
    __syncthreads();
    return sc.tot;
  }

  // Block-wide: the rows from `first` on of S->u.hl whose vertex has a bound above
  // `known`, moved to the list's front; returns their entries, *items their number.
  __device__ __noinline__ int64_t drop_known(int first, int items, int32_t known, int* kept) {
    constexpr int kPer = kHRows / kThreads;
    HeavyList& hl = S->u.hl;
    int32_t v[kPer], len[kPer];
    int64_t row[kPer], mine = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int i = first + threadIdx.x * kPer + q;
      v[q] = i < items ? hl.v[i] : -1;
      len[q] = v[q] >= 0 ? hl.len[i] : 0;
      row[q] = v[q] >= 0 ? hl.row[i] : 0;
      if (v[q] >= 0 && (int32_t)deg_of(ldcg(B.st + v[q])) <= known) v[q] = -1;
      mine += v[q] >= 0 ? (int64_t(1) << kPackShift) | len[q] : 0;
    }
    const Scan sc = scan(mine);             // every row has been read by now
    int64_t ex = sc.ex;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      if (v[q] < 0) continue;
      const int j = (int)(ex >> kPackShift);
      hl.pos[j] = ex & (int64_t)kPackEdgeMask;
      hl.row[j] = row[q];
      hl.len[j] = len[q];
      hl.v[j] = v[q];
      hl.cnt[j] = 0;
      ex += (int64_t(1) << kPackShift) | len[q];
    }
    *kept = (int)(sc.tot >> kPackShift);
    __syncthreads();
    return sc.tot & (int64_t)kPackEdgeMask;
  }

  // Block-wide: recount of the picked vertices; the largest degree known to the
  // block, and to the team so far, goes to S->h_best.  Of long lists of entries a few
  // rows are recounted first: where degrees are equal and few of them fall in a round
  // (cliques at small eps), no other vertex's bound is above what these have.
  __device__ __noinline__ void recount_picked() {
    const int n = S->h_picked;
    int32_t best = -1;
    int64_t edges = 0;
    for (int base = 0; base < n; base += kHRows) {
      int items = n - base < kHRows ? n - base : kHRows;
      int64_t E = prepare_rows(base, items, G > 1);
      if (E > kManyEdges) {
        const int few = (int)(items * (int64_t)kFewEdges / E) + 1;
        if (few < items) {
          const int64_t first = S->u.hl.pos[few];
          const int32_t b = block_recount(few, first);
          best = b > best ? b : best;
          edges += first;
          E = drop_known(few, items, best, &items);
        }
      }
      const int32_t b = block_recount(items, E);
      best = b > best ? b : best;
      edges += E;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      S->h_picked = 0;
      if (best > S->h_best) {
        const int32_t old = atomicMax(&C->best, best);
        S->h_best = old > best ? old : best;
      }
      S->tal[kTEdges] += (unsigned long long)edges;
    }
    __syncthreads();
  }

  // Counts the alive entries of `items` rows (lists in shared or global memory)
  // into acc: warp gw of nw takes its share of the E entries.  The alive entries
  // of a batch come as ballots, of which every lane counts the part of its own
  // window item, so an item costs one add per window.
  __device__ __noinline__ void count_alive(int gw, int nw, int32_t items, int64_t E, const int64_t* pos,
                                           const int64_t* row, const int32_t* len, unsigned* acc) {
    const uint32_t* const rtag = B.rtag;
    unsigned cnt = 0;
    const auto at = [&](int32_t j) { return vload(pos + j); };
    const auto load = [&](int32_t j) { return RowItem{vload(pos + j), vload(row + j), vload(len + j), 0}; };
    const auto count = [&](const auto& X) {
      constexpr int kB = sizeof(X.w) / sizeof(int32_t);
      uint32_t tg[kB];
#pragma unroll
      for (int q = 0; q < kB; ++q) {
        const bool in = X.w[q] >= 0 && CC_IN_BOUNDS(X.w[q], B.n, &C->err);
        tg[q] = in ? ldcg(rtag + (X.w[q] >> 3)) >> ((X.w[q] & 7) * 4) : 1u;
      }
#pragma unroll
      for (int q = 0; q < kB; ++q) {
        const unsigned m = __ballot_sync(FULL, (tg[q] & 15u) == 0);
        const int lo = X.from - 32 * q > 0 ? X.from - 32 * q : 0, hi = X.to - 32 * q < 32 ? X.to - 32 * q : 32;
        if (hi > lo) cnt += __popc(m & (0xFFFFFFFFu >> (32 - (hi - lo)) << lo));
      }
    };
    const auto flush = [&](int32_t j) {
      if (cnt) atomicAdd(acc + j, cnt);
      cnt = 0;
    };
    const WalkShape shape{B.tune.walk_batches, B.tune.prefetch_ahead};
    if (E <= 64 * (int64_t)nw) row_walk<1>(gw, nw, items, E, B.col, shape, at, load, count, flush);
    else row_walk<kRowB>(gw, nw, items, E, B.col, shape, at, load, count, flush);
  }

  // Recount of the block's list by the block itself; returns the largest
  // degree found to every thread.
  __device__ __noinline__ int32_t block_recount(int32_t items, int64_t E) {
    HeavyList& hl = S->u.hl;
    count_alive((int)(threadIdx.x >> 5), (int)(blockDim.x >> 5), items, E, hl.pos, hl.row, hl.len, hl.cnt);
    __syncthreads();
    int32_t best = -1;
    for (int i = threadIdx.x; i < items; i += blockDim.x) {
      const int32_t v = hl.v[i], d = (int32_t)hl.cnt[i];
      if (v < 0 || !CC_IN_BOUNDS(v, B.n, &C->err)) continue;
      B.st[v] = kAlive | (uint32_t)d;
      best = d > best ? d : best;
    }
    return max_i32(best);
  }

  // Grid phase over a heavy list of up to kHList vertices: every block makes
  // the same list (no state word changes in this phase), the grid's warps share
  // its entries, and the coordinator writes the degrees inside the barrier.
  // Longer lists: every block picks the vertices to recount out of its share
  // (dealt out by 32 entries: neighbours in the list have similar rows) and
  // recounts them, rows above kLongRow are left to a second phase of the whole
  // grid.  A block that has recounted some raises its threshold to the largest
  // degree known.
  __device__ __noinline__ bool recount_phase() {
    const int64_t len = P().win_len;
    if (P().pad0) {
      int64_t items, E;
      list_heavy(len, P().d_lb, P().drop, &items, &E);
      HeavyList& hl = S->u.hl;
      count_alive(team_warp(), team_warps(), (int32_t)items, E, hl.pos, hl.row, hl.len, B.h_acc);
      return sync(6, [&] {
        int32_t best = -1;
        if (threadIdx.x < items) {
          const int32_t v = hl.v[threadIdx.x];
          best = (int32_t)ldcg(B.h_acc + threadIdx.x);
          B.h_acc[threadIdx.x] = 0;
          if (CC_IN_BOUNDS(v, B.n, &C->err)) B.st[v] = kAlive | (uint32_t)best;
        }
        best = max_i32(best);
        if (threadIdx.x == 0 && best > co().d_lb) co().d_lb = best;
        __syncthreads();
        co_delta(kDCounted);
      });
    }
    Look k = look_begin(P().th);
    const int64_t all = (int64_t)G * blockDim.x;
    const int32_t keep = (int32_t)P().long_n;       // > 0: the list is rewritten with the bounds >= keep
    int32_t* const to = S->plan.hv_sel ? B.hv : B.hv2;
    for (int64_t base = 0; base < len; base += all * kScanU) {
      int32_t v[kScanU];
      uint32_t x[kScanU];
#pragma unroll
      for (int q = 0; q < kScanU; ++q) {
        const int64_t i = base + q * all + (int64_t)(threadIdx.x >> 5) * G * 32 + bid * 32 + (threadIdx.x & 31);
        v[q] = i < len ? ldcg(hv() + i) : -1;
      }
#pragma unroll
      for (int q = 0; q < kScanU; ++q) x[q] = v[q] >= 0 ? ldcg(B.st + v[q]) : 0u;
      if (keep > 0) append_heavy<kScanU>(v, x, keep, to);
      look_step(k, v, x, keep > 0 ? keep : 1, base + all * kScanU >= len);
    }
    look_end(k);
    return sync(6, [&] {
      if (threadIdx.x == 0 && S->plan.long_n > 0) {
        co().h_len = (int64_t)vload(&C->h_pack);
        co().tau = co().tau_next;
        S->plan.hv_sel ^= 1;
      }
      __syncthreads();
      looked();
    });
  }

  // A block's look at its share of the heavy vertices: the vertices of a bound
  // >= th are picked and recounted, at first a small number of them, after
  // which th is the largest degree known + 1.
  struct Look {
    int32_t th, other, top;
    int limit;
  };
  __device__ __forceinline__ Look look_begin(int32_t th) {
    if (threadIdx.x == 0) {
      S->h_picked = 0;
      S->h_best = -1;
    }
    __syncthreads();
    return Look{th, 0, 0, 256};
  }
  // Vertices v with state words x; bounds below tau are not heavy.
  __device__ __forceinline__ void look_step(Look& k, const int32_t* v, const uint32_t* x, int32_t tau, bool last) {
#pragma unroll
    for (int q = 0; q < kScanU; ++q) {
      const int32_t d = is_alive(x[q]) ? (int32_t)deg_of(x[q]) : 0;
      const int32_t ub = d >= tau ? d : 0;
      const bool take = ub >= k.th;         // th >= 1
      k.top = ub > k.top ? ub : k.top;
      k.other = !take && ub > k.other ? ub : k.other;
      pick(take, v[q]);                     // room for a whole step is left (below)
    }
    __syncthreads();
    const int picked = S->h_picked;
    __syncthreads();                        // all have read it: the next step's picks may add to it
    if (picked > k.limit || (last && picked > 0)) {      // the same in every thread: recount_picked has barriers
      recount_picked();
      if (S->h_best >= k.th) k.th = S->h_best + 1;
      k.limit = k.limit * 4 < kHPick / 2 ? k.limit * 4 : kHPick / 2;
    }
  }
  __device__ __forceinline__ void look_end(const Look& k) {
    const int32_t other = __reduce_max_sync(FULL, k.other), top = __reduce_max_sync(FULL, k.top);
    if ((threadIdx.x & 31) == 0) {
      if (other > ld_volatile_int(&C->other_max)) atomicMax(&C->other_max, other);
      if (top > ld_volatile_int(&C->listed_max)) atomicMax(&C->listed_max, top);
    }
  }
  // Coordinator, after the blocks' looks.
  __device__ __forceinline__ void looked() {
    if (threadIdx.x < 4) {
      const int i = threadIdx.x;
      S->bcast[i] = i == 0 ? (int64_t)vload(&C->best) : i == 1 ? (int64_t)vload(&C->other_max)
                    : i == 2 ? (int64_t)vload(&C->listed_max) : (int64_t)vload(&C->long_pack);
    }
    __syncthreads();
    const unsigned long long lp = (unsigned long long)S->bcast[3];
    if (threadIdx.x == 0) {
      note_looked((int32_t)S->bcast[1], (int32_t)S->bcast[2]);
      if ((int32_t)S->bcast[0] > co().d_lb) co().d_lb = (int32_t)S->bcast[0];
      if (lp) {
        S->plan.state = kRecountLong;
        S->plan.long_n = (int64_t)(lp >> kPackShift);
        S->plan.long_E = (int64_t)(lp & kPackEdgeMask);
        co().r_edges += S->plan.long_E;
      }
    }
    __syncthreads();
    if (!lp) co_delta(kDCounted);
  }
  // What a planned look starts from (thread 0 of the coordinator).
  __device__ __forceinline__ void reset_looked() {
    C->best = -1; C->listed_max = 0; C->other_max = 0; C->long_pack = 0;
  }

  // The long rows of a long heavy list, shared by the grid.
  __device__ __noinline__ bool recount_long() {
    unsigned* const acc = reinterpret_cast<unsigned*>(B.act_n);
    count_alive(team_warp(), team_warps(), (int32_t)P().long_n, P().long_E, B.b_e, B.b_d, B.pull, acc);
    return sync(6, [&] {
      int32_t best = -1;
      for (int64_t j = threadIdx.x; j < S->plan.long_n; j += blockDim.x) {
        const int32_t v = ldcg(B.b_j + j), d = (int32_t)ldcg(acc + j);
        if (CC_IN_BOUNDS(v, B.n, &C->err)) B.st[v] = kAlive | (uint32_t)d;
        best = d > best ? d : best;
      }
      best = max_i32(best);
      if (threadIdx.x == 0 && best > co().d_lb) co().d_lb = best;
      __syncthreads();
      co_delta(kDCounted);
    });
  }

  // ---------------- rebuild of the heavy list ----------------------------------
  // A new H of every alive vertex with a bound >= tau, for a lower tau.  All
  // bounds are at most ub = min(the last Delta, the old tau - 1).  tau = ub -
  // (ub >> tight): a long list is costly every round, a short one is soon used
  // up, so tight follows the length (from 1; up while the list is too long for
  // the coordinator, down again when it is very short), and a list that is too
  // long is cut down to a higher tau when the grid looks at it.  (R-MAT 26: with
  // half of ub throughout, rounds below Delta = 100 scanned up to 10M entries
  // each.)  A second rebuild in one round goes down to d_lb, at most to half of
  // ub: only larger bounds matter.
  // A vertex of bound >= tau has full degree >= tau, so the list comes from a
  // prefix of the degree order (dsort): up to inline_rebuild vertices (a tuning
  // setting) are read by the coordinator block inside the barrier, longer
  // prefixes by the grid, and once the prefix exceeds a quarter of the alive
  // non-isolated vertices, the grid reads those instead (vertex order).  True:
  // the list is in place; false: a grid step is planned.
  __device__ __noinline__ bool rebuild() {
    Coord& c = co();
    if (threadIdx.x == 0) {
      Plan& p = S->plan;
      c.rebuilds_in_row += 1;
      if (c.rebuilds_in_row > 64) fail(kErrInternal);     // tau falls every time
      const int32_t ub = c.delta < c.tau ? c.delta : c.tau - 1;     // >= 1: with tau = 1 Delta is known
      const int32_t loose = ub >> B.tune.heavy_shift > 1 ? ub >> B.tune.heavy_shift : 1;
      int32_t t = ub - (ub >> c.tight);
      if (t > ub - 2 * c.d_drop) t = ub - 2 * c.d_drop;      // meant to last for more than a round
      if (t < loose) t = loose;
      if (c.rebuilds_in_row > 1) {
        const int32_t lb = c.d_lb < t ? c.d_lb : t;
        t = lb > loose ? lb : loose;
      }
      c.tau = t;
      c.d_th = c.d_lb < 0 ? below(ub, c.d_drop) : c.d_lb + 1;
      const int64_t prefix = __ldg(B.dge + t);
      int dec = 0;
      if (prefix > B.tune.inline_rebuild) {
        dec = 1;
        p.th = t;
        p.take = c.d_th;                    // the grid looks at the new list while it makes it
        p.win_len = prefix;
        reset_looked();
        p.state = prefix > c.nz_len / 4 ? kRebuildAlive : kRebuildOrder;
        C->h_pack = 0;
        C->nz_pack = 0;
      }
      S->dec = dec;
      S->bcast[0] = prefix;
      S->h_kept = 0;
    }
    __syncthreads();
    if (S->dec) return false;
    const int32_t tau = c.tau;
    const int64_t len = S->bcast[0];
    for (int64_t base = 0; base < len; base += (int64_t)kScanU * blockDim.x) {
      int32_t v[kScanU];
      uint32_t x[kScanU];
#pragma unroll
      for (int q = 0; q < kScanU; ++q) {
        const int64_t i = base + threadIdx.x + (int64_t)q * blockDim.x;
        v[q] = i < len ? __ldg(B.dsort + i) : -1;
      }
#pragma unroll
      for (int q = 0; q < kScanU; ++q) x[q] = v[q] >= 0 ? ldcg(B.st + v[q]) : 0u;
#pragma unroll
      for (int q = 0; q < kScanU; ++q) {
        if (!is_alive(x[q]) || (int32_t)deg_of(x[q]) < tau) continue;
        const int h = atomicAdd(&S->h_kept, 1);
        if (CC_IN_BOUNDS(h, B.n, &C->err)) hv()[h] = v[q];
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      c.h_len = S->h_kept;
      follow_length();
    }
    __syncthreads();
    return true;
  }

  // Thread 0 of the coordinator, with a new heavy list in place.
  __device__ __forceinline__ void follow_length() {
    Coord& c = co();
    if (c.h_len > kHere && c.tight < kTightest) c.tight += 1;
    else if (c.h_len < kHere / 16 && c.tight > 1) c.tight -= 1;
  }

  // Statistics and n_i update after the removal phase, then the next plan.
  __device__ __noinline__ void co_end_round() {
    Coord& c = co();
    if (threadIdx.x < 5) {
      const long long* src[5] = {&C->r_centers, &C->r_attached, &C->r_noncenter, &C->r_blocked, &C->r_edges};
      S->bcast[threadIdx.x] = vload(src[threadIdx.x]);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      const int64_t centers_seen = S->bcast[0], attached = S->bcast[1], noncenter = S->bcast[2];
      const int64_t blocked = S->bcast[3];
      const int64_t k = c.k;
      const int64_t removed = k + attached;
      const int64_t centers = k - noncenter;
      const int64_t r = c.round;
      if (r < c.stats_cap) {
        RoundStat s;
        s.n_alive = c.n_alive; s.delta = c.delta; s.k = k; s.centers = centers;
        s.removed = removed; s.blocked = blocked; s.edges = c.r_edges + S->bcast[4];
        s.ns = (int64_t)(globaltimer_ns() - c.round_t0);
        B.stats[r] = s;
      }
      c.round_t0 = globaltimer_ns();
      c.round_ended = 1;
      c.r_edges = 0;
      if (centers_seen != centers) fail(kErrInternal);
      c.n_alive -= removed;
      if (c.n_alive < 0) fail(kErrInternal);
      c.round = r + 1;
      c.rebuilds_in_row = 0;
      if (!c.est && c.round > c.n + 1) fail(kErrInternal);   // Sec. 5 rounds may hold no active vertex
      S->dec = co_next();
    }
    __syncthreads();
    co_go_on();
  }

  // Coordinator: the centers that nothing blocked have attached their
  // neighbours; the round ends, or the blocked actives are next.
  __device__ __noinline__ void co_blocked() {
    if (threadIdx.x < 2) S->bcast[threadIdx.x] = (int64_t)vload(threadIdx.x == 0 ? &C->blk_pack : &C->blk_maxlen);
    __syncthreads();
    if (threadIdx.x == 0) {
      Plan& p = S->plan;
      const unsigned long long pk = (unsigned long long)S->bcast[0];
      p.b_n = (int64_t)(pk >> kPackShift);
      p.b_E = (int64_t)(pk & kPackEdgeMask);
      p.undecided = p.b_n;
      p.state = kResolve;
      co().fix_iter = 0;
      co().r_edges += 2 * p.b_E;            // first fixpoint scan, blocked attach / pull
      const int64_t warps = (int64_t)G * (blockDim.x >> 5);
      p.by_warp = p.b_n <= warps && S->bcast[1] <= (int64_t)B.tune.warp_resolve_row ? 1 : 0;
    }
    __syncthreads();
    if (P().b_n == 0) co_end_round();
  }

  // ---------------- Sec. 5: the round's binomial batch ------------------------
  // The next batch is drawn in the first phase of the round before, which spares
  // a phase per round (R-MAT 18, 547 rounds: 12.4 -> 10.6 ms).
  // Every block counts its share of the draws below the threshold (plan: long_n
  // trials, long_E = threshold bits, undecided = stream seed, d_lb = 2: every
  // trial succeeds).  The count moves the rank cursor past the batch, whose
  // ranks of pi are the round's single selection window.
  __device__ __noinline__ void draw_batch() {
    const int64_t trials = P().long_n;
    const uint64_t thr = (uint64_t)P().long_E, s = (uint64_t)P().undecided;
    int64_t cnt = 0;
    if (P().d_lb == 2) {
      cnt = bid == 0 && threadIdx.x == 0 ? trials : 0;
    } else {
      for (int64_t j = (int64_t)bid * blockDim.x + threadIdx.x; j < trials; j += (int64_t)G * blockDim.x)
        cnt += sec5_draw(s, (uint64_t)j) < thr ? 1 : 0;
    }
    cnt = block_sum<int64_t>(cnt, S->scr);
    if (threadIdx.x == 0) {
      if (cnt) atomicAdd(&C->drawn, (unsigned long long)cnt);
      S->drawn = P().drop;
      co().ahead = 1;                     // (the coordinator's)
    }
  }

  // ---------------- rebuild of the heavy list: grid passes ---------------------
  // Appends v (with its state word x) to the list `to` where its bound is >= tau.
  template <int kN>
  __device__ __forceinline__ void append_heavy(const int32_t* v, const uint32_t* x, int32_t tau, int32_t* to) {
    int64_t heavy = 0;
#pragma unroll
    for (int q = 0; q < kN; ++q) heavy += is_alive(x[q]) && (int32_t)deg_of(x[q]) >= tau ? 1 : 0;
    const Scan sc = scan(heavy);
    if (sc.tot == 0) return;                // uniform
    if (threadIdx.x == 0) S->bcast[0] = (int64_t)atomicAdd(&C->h_pack, (unsigned long long)sc.tot);
    __syncthreads();
    int64_t ho = S->bcast[0] + sc.ex;
#pragma unroll
    for (int q = 0; q < kN; ++q)
      if (is_alive(x[q]) && (int32_t)deg_of(x[q]) >= tau && CC_IN_BOUNDS(ho, B.n, &C->err)) to[ho++] = v[q];
  }

  // H from the first win_len vertices of the degree order (dealt out by 32, as
  // in recount_phase); the vertices of the largest bounds are recounted at once.
  __device__ __noinline__ bool rebuild_from_order() {
    const int64_t len = P().win_len;
    const int32_t tau = P().th;
    Look k = look_begin((int32_t)P().take);
    const int64_t all = (int64_t)G * blockDim.x;
    for (int64_t base = 0; base < len; base += all * kScanU) {
      int32_t v[kScanU];
      uint32_t x[kScanU];
#pragma unroll
      for (int q = 0; q < kScanU; ++q) {
        const int64_t i = base + q * all + (int64_t)(threadIdx.x >> 5) * G * 32 + bid * 32 + (threadIdx.x & 31);
        v[q] = i < len ? __ldg(B.dsort + i) : -1;
      }
#pragma unroll
      for (int q = 0; q < kScanU; ++q) x[q] = v[q] >= 0 ? ldcg(B.st + v[q]) : 0u;
      append_heavy<kScanU>(v, x, tau, hv());
      look_step(k, v, x, tau, base + all * kScanU >= len);
    }
    look_end(k);
    return sync(1, [&] { rebuilt(); });
  }

  // The same from the alive non-isolated vertices.  Every block keeps its own
  // segment of them (vertex order; of the graph's list at first) and drops from
  // it, in place, those that have left or have no alive neighbour.
  __device__ __noinline__ bool rebuild_from_alive() {
    int64_t s, e;
    slice(0, B.nz_n, &s, &e);
    const bool first = S->nz_cnt < 0;
    const int32_t* const src = first ? B.nz_static : B.nz0;
    if (!first) e = s + S->nz_cnt;
    const int32_t tau = P().th;
    int64_t out = s;
    Look k = look_begin((int32_t)P().take);
    const int64_t step = (int64_t)blockDim.x * kScanU;
    for (int64_t base = s; base < e; base += step) {
      int32_t v[kScanU];
      uint32_t x[kScanU];
      int64_t mine = 0;
#pragma unroll
      for (int q = 0; q < kScanU; ++q) {
        const int64_t i = base + (int64_t)threadIdx.x * kScanU + q;
        v[q] = i < e ? ldcg(src + i) : -1;
      }
#pragma unroll
      for (int q = 0; q < kScanU; ++q) x[q] = v[q] >= 0 ? ldcg(B.st + v[q]) : 0u;
#pragma unroll
      for (int q = 0; q < kScanU; ++q) mine += is_alive(x[q]) && deg_of(x[q]) > 0 ? 1 : 0;
      const Scan sc = scan(mine);           // every entry of the step is read by now
      int64_t o = out + sc.ex;
#pragma unroll
      for (int q = 0; q < kScanU; ++q)
        if (is_alive(x[q]) && deg_of(x[q]) > 0 && CC_IN_BOUNDS(o, B.n, &C->err)) B.nz0[o++] = v[q];
      out += sc.tot;
      append_heavy<kScanU>(v, x, tau, hv());
      look_step(k, v, x, tau, base + step >= e);
    }
    look_end(k);
    __syncthreads();
    if (threadIdx.x == 0) {
      S->nz_cnt = out - s;
      atomicAdd(&C->nz_pack, (unsigned long long)(out - s));
    }
    return sync(0, [&] {
      if (threadIdx.x == 0) co().nz_len = (int64_t)vload(&C->nz_pack);
      rebuilt();
    });
  }

  // Coordinator: the grid has filled H and looked at it.
  __device__ void rebuilt() {
    if (threadIdx.x == 0) {
      co().h_len = (int64_t)vload(&C->h_pack);
      follow_length();
    }
    __syncthreads();
    looked();
  }

  // ---------------- active-set selection (Alg. 2: A = next k alive of pi) ----
  // One tile of the window as one thread sees it: kU consecutive entries of
  // pi from rank `first`, their vertices (-1: none or removed) and rows.
  template <int kU>
  struct SelTile {
    int64_t first;
    int32_t v[kU];
    int32_t len[kU];
    int64_t row[kU];
  };
  // Alive when the round began: not removed, or attached in this round, which
  // select_attach of other blocks may be doing (the tag may also be that of 15k
  // rounds ago, the rank of the label tells).
  __device__ __forceinline__ bool was_alive(int32_t v) const {
    const uint32_t t = rtag_of(B.rtag, v);
    if (t == 0) return true;
    return t == (uint32_t)P().tag && ldcg(B.st + v) >= kLab + (uint32_t)P().th;
  }
  // (pi is read at L2: a batched job writes it in the same kernel, over the order of
  // the job before it)
  template <int kU>
  __device__ __forceinline__ void sel_vertices(SelTile<kU>& T, int64_t base, int64_t e) const {
    T.first = base + (int64_t)threadIdx.x * kU;
#pragma unroll
    for (int q = 0; q < kU; ++q) T.v[q] = T.first + q < e ? ldcg(B.order + T.first + q) : -1;
#pragma unroll
    for (int q = 0; q < kU; ++q)
      if (T.v[q] >= 0 && !was_alive(T.v[q])) T.v[q] = -1;
  }
  template <int kU>
  __device__ __forceinline__ void sel_rows(SelTile<kU>& T) const {
#pragma unroll
    for (int q = 0; q < kU; ++q) {
      T.row[q] = T.v[q] >= 0 ? __ldg(B.off + T.v[q]) : 0;
      T.len[q] = T.v[q] >= 0 ? (int32_t)(__ldg(B.off + T.v[q] + 1) - T.row[q]) : 0;
    }
    if (B.n > kStateInL2) return;
#pragma unroll
    for (int q = 0; q < kU; ++q)
      if (T.v[q] >= 0 && ldcg(B.st + T.v[q]) == kAlive) T.len[q] = 0;      // (a label is no bound)
  }

  // Entry j of the round's list of actives (flag: see blk_flag).
  __device__ __forceinline__ void put_active(int64_t j, int64_t before, int32_t v, int32_t rank, int64_t row, int32_t len,
                                             uint8_t flag) {
    if (!CC_IN_BOUNDS(j, B.n, &C->err)) return;
    B.act_r[j] = rank;
    B.act_e[j] = before;
    B.act_d[j] = row;
    B.act_n[j] = len;
    if (algo != kAlgoC4) return;
    B.act_v[j] = v;
    B.blk_flag[j] = flag;
  }

  // Emits the entries of a tile that are numbered below `need`, the tile's first
  // alive entry being number `run` of the window; returns the tile's alive
  // count.  A vertex without neighbours, or without alive ones by its bound,
  // is a singleton center for which nothing is written (no pass can reach it,
  // and later windows start past it); the label pass reads an alive word of
  // degree 0 as its own cluster.  One scan and one
  // atomic on the packed list counter per tile (solo: none); the tile that
  // reaches need is scanned again without its rest.
  // kFused (select_attach): the rows of up to kLongAttach entries go to the
  // block's tile list, *cnt rows of *entries together, only longer ones to the
  // round's; *lost counts the new centers that another block had attached.
  template <bool kFused, bool kC4 = false, int kU>
  __device__ __forceinline__ int64_t sel_emit(const SelTile<kU>& T, int64_t run, int64_t need, bool solo,
                                              int32_t* cnt = nullptr, int32_t* entries = nullptr,
                                              int32_t* lost = nullptr) {
    const uint32_t tag = (uint32_t)P().tag;
    // alive << 48 | listed << 36 | entries of the listed rows
    constexpr int kA = 48, kL = 36;
    constexpr int64_t kEM = (int64_t(1) << kL) - 1;
    auto listed = [](int32_t len) { return len > 0 && (!kFused || len <= kLongAttach); };
    int64_t pk = 0;
#pragma unroll
    for (int q = 0; q < kU; ++q)
      if (T.v[q] >= 0) pk += (int64_t(1) << kA) + (listed(T.len[q]) ? (int64_t(1) << kL) + T.len[q] : 0);
    Scan sc = scan(pk);
    const int64_t alive = sc.tot >> kA;
    int64_t g = run + (sc.ex >> kA);
    bool want[kU];
    pk = 0;
#pragma unroll
    for (int q = 0; q < kU; ++q) {
      want[q] = T.v[q] >= 0 && g < need;
      if (want[q]) {
        if (g == 0) *(solo ? &S->sel_r0 : &C->r0) = (int32_t)(T.first + q);
        if (g == need - 1) *(solo ? &S->sel_cursor : &C->cursor_next) = T.first + q + 1;
        pk += listed(T.len[q]) ? (int64_t(1) << kL) + T.len[q] : 0;
      }
      g += T.v[q] >= 0 ? 1 : 0;
    }
    if (run + alive > need) sc = scan(pk);          // uniform
    const int64_t cnt_tot = (sc.tot >> kL) & 0xFFF, e_tot = sc.tot & kEM;
    if (threadIdx.x == 0) {
      // ClusterWild!: every one is a center; C4: so far those without neighbours
      const int64_t wanted = run + alive < need ? alive : need - run;
      // (other threads add to both below, for their long rows)
      atomicAdd(&S->tal[kTCenters], (unsigned long long)(algo == kAlgoCW ? wanted : wanted - cnt_tot));
      atomicAdd(&S->tal[kTEdges], (unsigned long long)(algo == kAlgoCW ? e_tot : 2 * e_tot));      // C4 reads them twice
    }
    if (kFused) {
      TileRows& R = S->u.rows;
      int32_t j = (int32_t)(sc.ex >> kL) & 0xFFF, ep = (int32_t)(sc.ex & kEM);
#pragma unroll
      for (int q = 0; q < kU; ++q) {
        if (!want[q] || T.len[q] == 0) continue;
        if (!is_alive(atomicExch(B.st + T.v[q], kActive))) *lost += 1;
        set_rtag(B.rtag, T.v[q], tag);
        if (listed(T.len[q])) {
          R.rank[j] = (int32_t)(T.first + q);
          R.pos[j] = ep;
          R.row[j] = T.row[q];
          R.len[j] = T.len[q];
          if (kC4) {
            R.v[j] = T.v[q];
            R.blocked[j] = 0;
          }
          ++j;
          ep += T.len[q];
          continue;
        }
        const unsigned long long at = atomicAdd(&C->act_pack, (1ull << kPackShift) | (unsigned long long)T.len[q]);
        put_active((int64_t)(at >> kPackShift), (int64_t)(at & kPackEdgeMask), T.v[q], (int32_t)(T.first + q),
                   T.row[q], T.len[q], 0);
        atomicAdd(&S->tal[kTEdges], (unsigned long long)T.len[q] * (kC4 ? 2 : 1));
        if (kC4) atomicAdd(&S->tal[kTCenters], ~0ull);      // not one yet
      }
      *cnt = (int32_t)cnt_tot;
      *entries = (int32_t)e_tot;
      return alive;
    }
    if (cnt_tot == 0) return alive;
    if (threadIdx.x == 0) {
      const unsigned long long add = ((unsigned long long)cnt_tot << kPackShift) | (unsigned long long)e_tot;
      unsigned long long old;
      if (solo) {
        old = S->sel_pack;
        S->sel_pack = old + add;
      } else {
        old = atomicAdd(&C->act_pack, add);
      }
      S->bcast[0] = (int64_t)(old >> kPackShift);
      S->bcast[1] = (int64_t)(old & kPackEdgeMask);
    }
#pragma unroll
    for (int q = 0; q < kU; ++q) {
      if (!want[q] || T.len[q] == 0) continue;
      set_rtag(B.rtag, T.v[q], tag);
      B.st[T.v[q]] = kActive;
      if (algo == kAlgoC4 && !fused()) B.arank[T.v[q]] = (int32_t)(T.first + q);
    }
    __syncthreads();
    int64_t j = S->bcast[0] + ((sc.ex >> kL) & 0xFFF), ep = S->bcast[1] + (sc.ex & kEM);
#pragma unroll
    for (int q = 0; q < kU; ++q) {
      if (!want[q] || T.len[q] == 0) continue;
      put_active(j, ep, T.v[q], (int32_t)(T.first + q), T.row[q], T.len[q], 0);
      ++j;
      ep += T.len[q];
    }
    return alive;
  }

  // Look-back over the team (one pass instead of count, barrier, emit):
  // block bid publishes its alive count in desc[bid * kDescStride] (one
  // 128-byte line per block, so that the pollers of different blocks'
  // counts meet in different L2 slices), tagged with the barrier
  // epoch; thread q of the block waits for the counts of predecessors q,
  // q + blockDim.x, ... and the block sums them (a single round of loads
  // while the team has at most blockDim.x blocks).  The last block also
  // stores the window's total in desc[G * kDescStride] for the coordinator.  A cleared
  // descriptor (flag 0) is never taken for a count, whatever the epoch.
  // Returns this block's exclusive prefix to every thread; every wait is
  // bounded.
  static constexpr unsigned long long kDescVal = (1ull << 38) - 1;
  __device__ __forceinline__ unsigned long long pack_desc(unsigned flag, long long v) const {
    return ((unsigned long long)(epoch & 0xFFFFFFu) << 40) | ((unsigned long long)flag << 38) |
           ((unsigned long long)v & kDescVal);
  }
  __device__ long long lookback(long long mine) {
    volatile unsigned long long* d = B.desc;
    if (threadIdx.x == 0) d[(int64_t)bid * kDescStride] = pack_desc(1, mine);
    const unsigned tag = epoch & 0xFFFFFFu;
    int32_t v = 0;
    const uint64_t t0 = globaltimer_ns();
    for (unsigned q = threadIdx.x; q < bid; q += blockDim.x) {
      unsigned long long x = d[(int64_t)q * kDescStride];
      unsigned spins = 0;
      while ((unsigned)(x >> 40) != tag || ((x >> 38) & 3u) == 0) {
        if ((++spins & 63) == 0 && (ld_volatile_int(&C->err) != kOk || globaltimer_ns() - t0 > kBarrierLimitNs)) {
          fail(kErrTimeout);
          x = 0;
          break;
        }
        x = d[(int64_t)q * kDescStride];
      }
      v += (int32_t)(x & kDescVal);          // counts of one window: below 2^31 together
    }
    const long long excl = sum_i32(v);
    if (threadIdx.x == 0 && bid == G - 1) d[(int64_t)G * kDescStride] = pack_desc(2, excl + mine);
    return excl;
  }

  // This thread's share of the window's alive entries in [s, e).
  __device__ __forceinline__ int32_t count_window(int64_t s, int64_t e) const {
    const int64_t step = 2 * (int64_t)blockDim.x * kSelU;
    int32_t cnt = 0;
    for (int64_t b = s; b < e; b += step) {
      int32_t v[2 * kSelU];
#pragma unroll
      for (int q = 0; q < 2 * kSelU; ++q) {
        const int64_t i = b + (int64_t)q * blockDim.x + threadIdx.x;
        v[q] = i < e ? ldcg(B.order + i) : -1;
      }
#pragma unroll
      for (int q = 0; q < 2 * kSelU; ++q) cnt += v[q] >= 0 && was_alive(v[q]) ? 1 : 0;
    }
    return cnt;
  }

  // This block's share of the window; solo: the coordinator block takes all of
  // it, inside a barrier.
  __device__ __noinline__ void select_window(bool solo) {
    int64_t s, e;
    if (solo) {
      s = P().win_lo;
      e = s + P().win_len;
    } else {
      slice(P().win_lo, P().win_len, &s, &e);
    }
    // Centers keep their active marker for good: an active of this round is
    // told from an earlier round's center by its rank (C4), which is >= r0,
    // the round's first active rank.
    // Count this block's alive entries; the first tile stays in registers and
    // its rows are asked for while the block waits for the others' counts.
    const int64_t tile = (int64_t)blockDim.x * kSelU, need = P().need;
    int64_t base = s, run = 0;
    do {
      SelTile<kSelU> T;
      sel_vertices(T, base, e);
      sel_rows(T);
      if (base == s && !solo) {
        int32_t cnt = 0;
#pragma unroll
        for (int q = 0; q < kSelU; ++q) cnt += T.v[q] >= 0 ? 1 : 0;
        run = lookback(sum_i32(cnt + count_window(s + tile, e)));       // this block's first alive entry is number `run` of the window
      }
      // emit the alive entries of the window numbered below `need`
      if (run < need) run += sel_emit<false>(T, run, need, solo);
      base += tile;
    } while (base < e && run < need);       // uniform across the block
    if (solo && threadIdx.x == 0) S->sel_total = run;
  }

  // Coordinator: the round's active set is complete, or the next window follows.
  __device__ __noinline__ void select_decide(bool solo) {
    if (!solo && threadIdx.x < 4) {
      const int i = threadIdx.x;            // side by side
      const int64_t x = i == 0 ? (int64_t)(ldcg(B.desc + (int64_t)G * kDescStride) & kDescVal)
                               : i == 1 ? (int64_t)vload(&C->r0)
                               : i == 2 ? vload(&C->cursor_next) : (int64_t)vload(&C->act_pack);
      if (i == 0) S->sel_total = x;
      else if (i == 1) S->sel_r0 = (int32_t)x;
      else if (i == 2) S->sel_cursor = x;
      else S->sel_pack = (unsigned long long)x;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      Coord& c = co();
      Plan& p = S->plan;
      const int64_t total = S->sel_total;
      p.take = total < c.need ? total : c.need;
      if (c.est) { c.k = total; p.k = total; }   // Sec. 5: all of the window
      if (p.r0 < 0) p.r0 = S->sel_r0;
      const int64_t left = c.est ? 0 : c.need - p.take;
      c.need = left;
      p.need = left;
      if (left == 0) {
        c.cursor = c.est ? c.batch_end : S->sel_cursor;
        p.act_n = (int64_t)(S->sel_pack >> kPackShift);
        p.act_E = (int64_t)(S->sel_pack & kPackEdgeMask);
        p.state = kRun;
      } else {
        const int64_t lo2 = c.win_lo + c.win_len;
        const int64_t avail = c.al_len - lo2;
        const int64_t alive_left = c.n_alive - (c.k - left);
        if (avail <= 0 || alive_left <= 0) {
          fail(kErrInternal);
          p.state = kAbort;
        } else {
          const int64_t est = (int64_t)((float)left * ((float)avail / (float)alive_left) * 1.1f) + 1024;
          c.win_lo = lo2;
          c.win_len = est < avail ? est : avail;
          p.win_lo = c.win_lo;
          p.win_len = c.win_len;
          if (solo) C->act_pack = S->sel_pack;   // a longer window goes on from here
          p.state = kSelect;
        }
      }
    }
    __syncthreads();
  }

  // Inside the barrier select a team of one block, which has nobody to share a
  // window with, and short windows that cannot be attached in the same pass.
  __device__ __noinline__ void select_here() {
    while (S->plan.state == kSelect && (G == 1 || (!fused() && P().win_len <= kInlineWindow))) {
      select_window(true);
      __syncthreads();
      select_decide(true);
    }
  }

  // ---------------- createCluster: push a center's rank to its neighbours ----
  // The arrays that the adjacency passes read and write, in registers: a pass
  // is a function of its own (its own register allocation), and a field of B
  // read inside its loops would be loaded again after every atomic.
  struct Words {
    uint32_t* st;
    uint32_t* rtag;
    uint32_t tag;
  };
  __device__ __forceinline__ Words words() const { return Words{B.st, B.rtag, (uint32_t)P().tag}; }

  // Tries to attach u (state word x, read earlier; 0: cannot be) to the center
  // of rank r; true when u was alive.
  static __device__ __forceinline__ bool attach_one(const Words& W, int32_t u, int32_t r, uint32_t x) {
    const uint32_t nv = kLab + (uint32_t)r;
    if (x > nv && is_alive(atomicMin(W.st + u, nv))) {
      set_rtag(W.rtag, u, W.tag);
      return true;
    }
    return false;
  }

  // One batch of a walk over centers' rows (payload: the center's rank, -1: not
  // a center); returns the vertices attached.
  template <class Batch>
  __device__ __forceinline__ int32_t attach_batch(const Words& W, const Batch& X) const {
    int32_t n = 0;
    constexpr int kB = sizeof(X.w) / sizeof(int32_t);
    uint32_t x[kB];
    // alive (tag 0): try the atomicMin directly; tagged this round (or 15k
    // rounds ago): the state word decides; removed earlier: nothing to do
#pragma unroll
    for (int q = 0; q < kB; ++q) {
      const bool push = X.w[q] >= 0 && X.aux[q] >= 0 && CC_IN_BOUNDS(X.w[q], B.n, &C->err);
      x[q] = push ? rtag_of(W.rtag, X.w[q]) : 16u;
    }
#pragma unroll
    for (int q = 0; q < kB; ++q) x[q] = x[q] == 0 ? 0xFFFFFFFFu : (x[q] == W.tag ? ldcg(W.st + X.w[q]) : 0u);
#pragma unroll
    for (int q = 0; q < kB; ++q) n += attach_one(W, X.w[q], X.aux[q], x[q]) ? 1 : 0;
    return n;
  }

  // The entries of the active rows; aux(j) = payload of active j.
  template <class Aux, class F>
  __device__ __forceinline__ void walk_actives(const Aux& aux, F&& f) {
    const int64_t* const pos = B.act_e;
    const int64_t* const row = B.act_d;
    const int32_t* const len = B.act_n;
    walk(P().act_n, P().act_E, [&](int32_t j) { return ldcg(pos + j); },
         [&](int32_t j) { return RowItem{ldcg(pos + j), ldcg(row + j), ldcg(len + j), aux(j)}; }, f);
  }

  __device__ __noinline__ void attach_from_actives(bool skip_blocked) {
    const Words W = words();
    const int32_t* const rank = B.act_r;
    const uint8_t* const blocked = B.blk_flag;
    int32_t attached = 0;
    // payload: the center's rank, -1 for a blocked active
    walk_actives([&](int32_t j) { return skip_blocked && ldcg(blocked + j) ? -1 : ldcg(rank + j); },
                 [&](const auto& X) {
      attached += attach_batch(W, X);
    });
    tally(kTAttached, attached);
  }

  // Selection and attachment of a window in one pass.  ClusterWild!: every alive
  // vertex of the window below the k-th is a center whatever the others do.  C4:
  // it is one unless a neighbour of lower rank was alive when the round began
  // (all of those are active too), which the ranks of pi tell without waiting
  // for the other blocks' actives; the others are blocked and listed for the
  // next phase.  So a block attaches its own centers' neighbours as soon as the
  // look-back tells it their numbers, without barriers and without the list of
  // actives in between.  A vertex that another block's center reaches before its
  // own block makes it active is taken back (sel_emit); one that is active
  // already has the smaller word.  Rows of more than kLongAttach entries, which
  // one block would walk alone, are left to the passes over that list.
  // kU entries per thread and tile: one for small graphs, whose windows are short
  // (planted 10^6 5.71 -> 5.47 ms, R-MAT 20 3.31 -> 3.19), two for large ones (R-MAT
  // 26: 17.6 ms against 17.9).
  template <bool kC4, int kU>
  __device__ __noinline__ void select_attach() {
    int64_t s, e;
    slice(P().win_lo, P().win_len, &s, &e);
    const Words W = words();
    TileRows& R = S->u.rows;
    const int32_t* const arank = B.arank;
    const int32_t r_lo = P().th;
    const int64_t tile = (int64_t)blockDim.x * kU, need = P().need;
    const WalkShape shape{B.tune.walk_batches, B.tune.prefetch_ahead};
    const int warp = (int)(threadIdx.x >> 5), nwarps = kThreads / 32;
    int64_t base = s, run = 0;
    int32_t attached = 0;
    do {
      SelTile<kU> T;
      sel_vertices(T, base, e);
      sel_rows(T);
#pragma unroll
      for (int q = 0; q < kU; ++q)
        if (T.len[q] > 0) prefetch_l2(B.col + T.row[q]);
      if (base == s) {
        int32_t cnt = 0;
#pragma unroll
        for (int q = 0; q < kU; ++q) cnt += T.v[q] >= 0 ? 1 : 0;
        run = lookback(sum_i32(cnt + count_window(s + tile, e)));
      }
      if (run < need) {
        int32_t cnt, E, lost = 0;
        run += sel_emit<true, kC4>(T, run, need, false, &cnt, &E, &lost);
        attached -= lost;
        __syncthreads();
        for (int pass = kC4 ? 0 : 1; pass < 2; ++pass) {
          auto at = [&](int32_t j) { return (int64_t)R.pos[j]; };
          auto load = [&](int32_t j) {
            return RowItem{(int64_t)R.pos[j], R.row[j], R.len[j], kC4 && pass == 1 && R.blocked[j] ? -1 : R.rank[j]};
          };
          auto f = [&](const auto& X) {
            if (!kC4 || pass == 1) {
              attached += attach_batch(W, X);
              return;
            }
            constexpr int kB = sizeof(X.w) / sizeof(int32_t);
            uint32_t tg[kB];
            int32_t ru[kB];
#pragma unroll
            for (int q = 0; q < kB; ++q) tg[q] = X.w[q] >= 0 ? rtag_of(W.rtag, X.w[q]) : 16u;
#pragma unroll
            for (int q = 0; q < kB; ++q) ru[q] = tg[q] == 0 || tg[q] == W.tag ? ldcg(arank + X.w[q]) : -1;
#pragma unroll
            for (int q = 0; q < kB; ++q) {
              if (ru[q] < r_lo || ru[q] >= X.aux[q]) continue;
              const uint32_t x = tg[q] == 0 ? 0u : ldcg(W.st + X.w[q]);
              // active in this round, or attached in it
              if (is_active(x) || x >= kLab + (uint32_t)r_lo) R.blocked[X.item[q]] = 1;
            }
          };
          if (E <= 64 * nwarps) row_walk<1>(warp, nwarps, cnt, E, B.col, shape, at, load, f);
          else row_walk<kRowB>(warp, nwarps, cnt, E, B.col, shape, at, load, f);
          if (kC4 && pass == 0) {
            __syncthreads();
            tile_classify(cnt);
          }
        }
      }
      base += tile;
    } while (base < e && run < need);       // uniform across the block
    tally(kTAttached, attached);
  }

  // C4: the actives of the block's tile are centers or go to the blocked list
  // (and, for the passes that read it, to the list of actives with flag 2).
  __device__ __forceinline__ void tile_classify(int32_t cnt) {
    const TileRows& R = S->u.rows;
    const int lane = threadIdx.x & 31;
    int32_t centers = 0, nblocked = 0;
    for (int32_t base = (int32_t)threadIdx.x - lane; base < cnt; base += kThreads) {
      const int32_t j = base + lane;
      const bool blocked = j < cnt && R.blocked[j];
      const int32_t len = blocked ? R.len[j] : 0;
      if (j < cnt && !blocked) {
        B.st[R.v[j]] = kActCenter;
        centers += 1;
      }
      if (!__any_sync(FULL, blocked)) continue;
      const int64_t pk = blocked ? (int64_t(1) << kPackShift) | len : 0, inc = warp_inclusive_sum<int64_t>(pk);
      unsigned long long old = 0;
      if (lane == 31) old = atomicAdd(&C->act_pack, (unsigned long long)inc);
      const int64_t at = (int64_t)__shfl_sync(FULL, old, 31) + inc - pk, i = at >> kPackShift;
      if (blocked) {
        put_active(i, at & (int64_t)kPackEdgeMask, R.v[j], R.rank[j], R.row[j], len, 2);
        nblocked += 1;
      }
      warp_append_rows(blocked, (int32_t)i, blocked ? R.row[j] : 0, len, 0x7FFFFFFF, blk_list());
      const int32_t ml = __reduce_max_sync(FULL, len);
      if (lane == 0) atomicMax(&C->blk_maxlen, (unsigned long long)ml);
    }
    tally(kTCenters, centers);
    tally(kTBlocked, nblocked);
  }

  // ---------------- C4: blocked detection ------------------------------------
  __device__ __noinline__ void c4_detect() {
    const Words W = words();
    const int32_t* const rank = B.act_r;
    const int32_t* const arank = B.arank;
    uint8_t* const blocked = B.blk_flag;
    const int32_t r0 = P().r0;
    // payload: the active's rank, -1 when it is known to be blocked
    walk_actives([&](int32_t j) { return ldcg(blocked + j) ? -1 : ldcg(rank + j); }, [&](const auto& X) {
      constexpr int kB = sizeof(X.w) / sizeof(int32_t);
      uint32_t tg[kB];
#pragma unroll
      for (int q = 0; q < kB; ++q) tg[q] = X.w[q] >= 0 ? rtag_of(W.rtag, X.w[q]) : 16u;
#pragma unroll
      for (int q = 0; q < kB; ++q) {
        // an earlier active neighbour: v must wait (isCenter); actives carry
        // this round's tag
        if (tg[q] != W.tag) continue;
        if (is_active(ldcg(W.st + X.w[q]))) {
          const int32_t ru = ldcg(arank + X.w[q]);
          if (ru >= r0 && ru < X.aux[q]) blocked[X.item[q]] = 1;
        }
      }
    });
  }

  // C4: unblocked actives become centers; blocked ones go to the blocked list.
  __device__ __noinline__ void c4_classify() {
    const int64_t an = P().act_n;
    int32_t centers = 0, nblocked = 0;
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)bid * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)G * blockDim.x) >> 5;
    for (int64_t base = gw * 32; base < an; base += nw * 32) {
      const int64_t j = base + lane;
      bool blocked = false;
      int64_t len = 0, row = 0;
      if (j < an) {
        const int32_t v = ldcg(B.act_v + j);
        const uint8_t flag = ldcg(B.blk_flag + j);      // 1: blocked; 2: the same, and listed already
        if (flag == 2) {
        } else if (flag) {
          blocked = true;
          row = ldcg(B.act_d + j);
          len = ldcg(B.act_n + j);
          nblocked += 1;
        } else {
          B.st[v] = kActCenter;
          centers += 1;
        }
      }
      if (!__any_sync(FULL, blocked)) continue;
      warp_append_rows(blocked, (int32_t)j, row, len, 0x7FFFFFFF, blk_list());
      const int64_t ml = warp_max<int64_t>(len);
      if (lane == 0) atomicMax(&C->blk_maxlen, (unsigned long long)ml);
    }
    tally(kTCenters, centers);
    tally(kTBlocked, nblocked);
  }

  // C4, a round's blocked actives one warp each (every one has a warp of its
  // own and no row is longer than warp_resolve_row): the warp waits until each
  // earlier-ranked active neighbour of its vertex is decided; the vertex is a
  // center iff none of them is a center (isCenter), otherwise it joins the
  // lowest-ranked one (every earlier center is known by then, so the label is
  // final at once).  A center then pushes its rank to its alive neighbours
  // (createCluster).  Waits go only to strictly earlier ranks and every vertex
  // has a resident warp, so the earliest undecided vertex always progresses:
  // the same decisions as the fixpoint, in one grid phase.  Every wait is
  // bounded.
  __device__ __noinline__ void c4_resolve_by_warp() {
    const Words W = words();
    const int64_t bn = P().b_n;
    const int lane = threadIdx.x & 31;
    const int64_t gw = (int64_t)(threadIdx.x >> 5) * G + bid;     // warps numbered across the blocks first
    const int32_t r0 = P().r0;
    int32_t v = 0, rv = 0;
    int64_t row = 0, len = 0;
    if (gw < bn) {                                                 // warp-uniform
      const int32_t j = ldcg(B.b_j + gw);
      v = ldcg(B.act_v + j);
      rv = ldcg(B.act_r + j);
      row = ldcg(B.b_e + gw) + ldcg(B.b_d + gw);
      len = ldcg(B.act_n + j);
    }
    int32_t minc = 0x7FFFFFFF;
    bool late = false;
    const uint64_t t0 = globaltimer_ns();
    for (int64_t base = 0; base < len; base += 32) {
      const int64_t e = base + lane;
      if (e >= len || late) continue;
      const int32_t u = __ldg(B.col + row + e);
      if (rtag_of(B.rtag, u) != W.tag) continue;                     // not an active of this round
      uint32_t x = ldcg(B.st + u);
      if (!is_active(x)) continue;                                 // a decided non-center, or attached
      const int32_t ru = ldcg(B.arank + u);
      if (ru < r0 || ru >= rv) continue;                           // not earlier in this round
      unsigned spins = 0;
      while (x == kActive) {
        if ((++spins & 63) == 0 && (globaltimer_ns() - t0 > kBarrierLimitNs || ld_volatile_int(&C->err) != kOk)) {
          late = true;
          break;
        }
        x = ld_relaxed_u32(B.st + u);
      }
      if (x == kActCenter) minc = ru < minc ? ru : minc;
    }
    if (__any_sync(FULL, late)) {
      if (lane == 0) fail(kErrTimeout);
      return;
    }
    minc = warp_min_i32(minc);
    const bool center = gw < bn && minc == 0x7FFFFFFF;
    if (gw < bn && lane == 0) atomicExch(B.st + v, center ? kActCenter : kLab + (uint32_t)minc);
    tally(kTCenters, center && lane == 0 ? 1 : 0);
    tally(kTNonCenter, gw < bn && !center && lane == 0 ? 1 : 0);
    if (!center) return;
    int32_t attached = 0;
    for (int64_t base = 0; base < len; base += 32) {
      const int64_t e = base + lane;
      const bool in = e < len;
      const int32_t u = in ? __ldg(B.col + row + e) : 0;
      const uint32_t tg = in ? rtag_of(B.rtag, u) : 16u;
      const uint32_t x = tg == 0 ? 0xFFFFFFFFu : (tg == W.tag ? ldcg(B.st + u) : 0u);
      attached += attach_one(W, u, rv, x) ? 1 : 0;
    }
    tally(kTAttached, attached);
  }

  // The entries of the blocked rows; aux = payload(j, v) of active j, vertex v.
  template <class Aux, class F>
  __device__ __forceinline__ void walk_blocked(const Aux& aux, F&& f) {
    walk(P().b_n, P().b_E, [&](int32_t q) { return ldcg(B.b_e + q); },
         [&](int32_t q) {
           const int32_t j = ldcg(B.b_j + q);
           const int64_t e = ldcg(B.b_e + q);
           return RowItem{e, e + ldcg(B.b_d + q), ldcg(B.act_n + j), aux(j, ldcg(B.act_v + j))};
         }, f);
  }

  // C4 fixpoint, step 1: look at the earlier active neighbours of every
  // undecided blocked vertex (payload: its rank, -1 when decided).
  __device__ __noinline__ void c4_fix_scan() {
    const uint32_t tag = (uint32_t)P().tag;
    const int32_t r0 = P().r0;
    walk_blocked([&](int32_t j, int32_t v) { return ldcg(B.st + v) == kActive ? ldcg(B.act_r + j) : -1; },
                 [&](const auto& X) {
      constexpr int kB = sizeof(X.w) / sizeof(int32_t);
#pragma unroll
      for (int i = 0; i < kB; ++i) {
        const int32_t u = X.w[i];
        if (u < 0 || X.aux[i] < 0) continue;
        if (rtag_of(B.rtag, u) != tag) continue;     // not an active of this round
        const uint32_t x = ldcg(B.st + u);
        const int32_t ru = is_active(x) ? ldcg(B.arank + u) : -1;
        if (ru >= r0 && ru < X.aux[i]) {
          if (x == kActCenter) B.hit_c[X.item[i]] = 1;
          else if (x == kActive) B.hit_p[X.item[i]] = 1;
        }
      }
    });
  }

  // C4 fixpoint, step 2: decide (isCenter without waiting) for blocked items
  // q = first, first + stride, ...  The hit flags go back to zero, so they
  // are zero whenever a fixpoint starts.
  __device__ long long c4_fix_decide(int64_t first, int64_t stride) {
    const int64_t bn = P().b_n;
    long long left = 0;
    int32_t centers = 0;
    for (int64_t q = first; q < bn; q += stride) {
      const int32_t j = ldcg(B.b_j + q);
      const int32_t v = ldcg(B.act_v + j), r = ldcg(B.act_r + j);
      (void)r;
      if (ldcg(B.st + v) != kActive) continue;
      if (ldcg(B.hit_c + q)) B.st[v] = kActNon;
      else if (!ldcg(B.hit_p + q)) { B.st[v] = kActCenter; centers += 1; }
      else left += 1;
      B.hit_c[q] = 0;
      B.hit_p[q] = 0;
    }
    tally(kTCenters, centers);
    return left;
  }

  // C4 after the fixpoint: blocked centers push, blocked non-centers pull the
  // lowest center rank among their neighbours (payload: a center's rank, -1
  // for a non-center).
  __device__ __noinline__ void c4_blocked_attach() {
    const Words W = words();
    const int32_t r0 = P().r0;
    int32_t attached = 0;
    walk_blocked([&](int32_t j, int32_t v) { return ldcg(B.st + v) == kActCenter ? ldcg(B.act_r + j) : -1; },
                 [&](const auto& X) {
      constexpr int kB = sizeof(X.w) / sizeof(int32_t);
#pragma unroll
      for (int i = 0; i < kB; ++i) {
        const int32_t u = X.w[i];
        if (u < 0) continue;
        const uint32_t x = ldcg(B.st + u);
        if (X.aux[i] >= 0) {
          attached += attach_one(W, u, X.aux[i], x) ? 1 : 0;
        } else if (x == kActCenter) {
          const int32_t ru = ldcg(B.arank + u);
          if (ru >= r0) atomicMin(B.pull + X.item[i], ru);   // a center of this round
        }
      }
    });
    tally(kTAttached, attached);
  }

  // C4: a non-center active takes its pulled label.
  __device__ __noinline__ void c4_pull_finalize() {
    const int64_t bn = P().b_n;
    int32_t noncenter = 0;
    for (int64_t q = (int64_t)bid * blockDim.x + threadIdx.x; q < bn; q += (int64_t)G * blockDim.x) {
      const int32_t v = ldcg(B.act_v + ldcg(B.b_j + q));
      if (ldcg(B.st + v) != kActNon) continue;
      const int32_t lab = ldcg(B.pull + q);
      if (lab == 0x7FFFFFFF) fail(kErrInternal);   // a non-center always has a center neighbour
      B.st[v] = kLab + (uint32_t)lab;
      noncenter += 1;
    }
    tally(kTNonCenter, noncenter);
  }

  // ---------------- objective: edges inside clusters --------------------------
  // This thread's share of the member-member edges inside clusters (batched
  // jobs; k_intra is the same as a kernel).
  __device__ __noinline__ int64_t intra_edges() {
    int64_t cnt = 0;
    walk(B.up.n, B.up.edges, [&](int32_t j) { return (int64_t)__ldg(B.up.epos + j); },
         [&](int32_t j) {
           return RowItem{(int64_t)__ldg(B.up.epos + j), __ldg(B.up.row + j), __ldg(B.up.len + j),
                          (int32_t)member_id(ldcg(B.st + __ldg(B.up.v + j)))};
         },
         [&](const auto& X) {
      constexpr int kB = sizeof(X.w) / sizeof(int32_t);
      uint32_t x[kB];
#pragma unroll
      for (int q = 0; q < kB; ++q) x[q] = X.w[q] >= 0 ? ldcg(B.st + X.w[q]) : 0;
#pragma unroll
      for (int q = 0; q < kB; ++q) cnt += X.w[q] >= 0 && x[q] == (uint32_t)X.aux[q] ? 1 : 0;
    });
    return cnt;
  }

  // Reduce the round tallies of this block into the control block.
  __device__ void flush_round_tallies() {
    __syncthreads();
    if (threadIdx.x < kTallies) {
      unsigned long long* dst[kTallies] = {reinterpret_cast<unsigned long long*>(&C->r_centers),
                                           reinterpret_cast<unsigned long long*>(&C->r_attached),
                                           reinterpret_cast<unsigned long long*>(&C->r_noncenter),
                                           reinterpret_cast<unsigned long long*>(&C->r_blocked),
                                           reinterpret_cast<unsigned long long*>(&C->r_edges)};
      const unsigned long long x = S->tal[threadIdx.x];
      if (x) { atomicAdd(dst[threadIdx.x], x); S->tal[threadIdx.x] = 0; }
    }
  }
};

// All rounds of one clustering job, run by the team of blocks in k.  The
// state words, the control block and the lists in k.B belong to this job.
template <int kPerSM>
__device__ void run_job(K<kPerSM>& k, int algo) {
  Shared& S = *k.S;
  Ctl* C = k.C;
  const bool est = algo >= 3;           // the Sec. 5 schedule: same rounds, C4 or ClusterWild!
  if (est) algo -= 2;
  if (k.bid == 0 && threadIdx.x == 0) {
    for (int i = 0; i < 8; ++i) S.co.ph_ns[i] = 0;
    S.co.t0 = globaltimer_ns();
    S.co.round_t0 = S.co.t0;
  }
  if (threadIdx.x == 0) {
    S.nz_cnt = -1;
    S.drawn = -1;
    k.algo = algo;
    k.est = est;
  }
  __syncthreads();
  if (!k.sync(7, [&] { k.co_init(); })) goto out;

  for (;;) {
    if (S.plan.state == kDone) break;
    if (S.plan.state == kRebuildOrder) {
      if (!k.rebuild_from_order()) goto out;
      continue;
    }
    if (S.plan.state == kRebuildAlive) {
      if (!k.rebuild_from_alive()) goto out;
      continue;
    }
    if (S.plan.state == kRecount) {
      if (!k.recount_phase()) goto out;
      continue;
    }
    if (S.plan.state == kRecountLong) {
      if (!k.recount_long()) goto out;
      continue;
    }
    if (k.est && S.plan.drop != S.drawn) {
      k.draw_batch();
      if (S.plan.state == kDrawBatch) {
        if (!k.sync(2, [&] {
              if (threadIdx.x == 0) {
                S.co.ahead = 0;
                k.batch_drawn((int64_t)vload(&C->drawn));
              }
              __syncthreads();
              k.plan_selection(S.co.delta);
            }))
          goto out;
        continue;
      }
    }
    if (S.plan.state == kSelect) {
      // (a round that has begun to attach goes on that way: only select_attach
      // takes back what its centers have reached)
      if (k.G > 1 && k.fused() && (S.plan.win_len <= kFuseWindow * (int64_t)k.G || S.plan.win_lo != (int64_t)S.plan.th)) {
        if (algo == kAlgoC4) k.template select_attach<true, kPerSM>();
        else k.template select_attach<false, kPerSM>();
        k.flush_round_tallies();
        if (!k.sync(4, [&] {
              k.select_decide(false);
              // the round goes on with what was left out
              if (S.plan.state != kRun) return;
              if (algo == kAlgoCW) {
                if (S.plan.act_n == 0) k.co_end_round();
              } else if (S.plan.act_n == (int64_t)(vload(&C->blk_pack) >> kPackShift)) {
                k.co_blocked();
              }
            }))
          goto out;
        continue;
      }
      k.select_window(false);
      if (!k.sync(3, [&] {
            k.select_decide(false);
            k.select_here();
          }))
        goto out;
      continue;
    }
    if (S.plan.state == kRun) {
      if (algo == kAlgoCW) {
        k.attach_from_actives(false);
        k.flush_round_tallies();
        if (!k.sync(4, [&] { k.co_end_round(); })) goto out;
      } else {
        k.c4_detect();
        if (!k.sync(4)) goto out;
        k.c4_classify();
        k.attach_from_actives(true);
        k.flush_round_tallies();
        if (!k.sync(4, [&] { k.co_blocked(); })) goto out;
      }
      continue;
    }
    // kResolve: C4's blocked actives
    if (S.plan.by_warp == 1) {
      k.c4_resolve_by_warp();
      k.flush_round_tallies();
      if (!k.sync(5, [&] { k.co_end_round(); })) goto out;
    } else {
      // the pull slots were set when the list was built; the hit flags are zero
      auto after_decide = [&](long long left) {
        if (threadIdx.x == 0) {
          S.plan.undecided = left;
          S.co.fix_iter += 1;
          if (S.co.fix_iter > 1) S.co.r_edges += S.plan.b_E;
          if (S.co.fix_iter > S.plan.b_n + 1) { k.fail(kErrInternal); S.plan.undecided = 0; }
        }
      };
      while (S.plan.undecided > 0) {
        k.c4_fix_scan();
        if (S.plan.b_n <= k.B.tune.inline_decide) {
          // a short blocked list: the coordinator decides inside the barrier
          if (!k.sync(5, [&] {
                const long long left = block_sum<int64_t>(k.c4_fix_decide(threadIdx.x, blockDim.x), S.scr);
                after_decide(left);
              }))
            goto out;
        } else {
          if (!k.sync(5, [&] { if (threadIdx.x == 0) C->undecided = 0; })) goto out;
          const long long left = block_sum<int64_t>(
              k.c4_fix_decide((int64_t)k.bid * blockDim.x + threadIdx.x, (int64_t)k.G * blockDim.x), S.scr);
          if (threadIdx.x == 0 && left)
            atomicAdd(reinterpret_cast<unsigned long long*>(&C->undecided), (unsigned long long)left);
          if (!k.sync(5, [&] { after_decide((long long)vload(&C->undecided)); })) goto out;
        }
      }
      k.c4_blocked_attach();
      if (!k.sync(5)) goto out;
      k.c4_pull_finalize();
      k.flush_round_tallies();
      if (!k.sync(5, [&] { k.co_end_round(); })) goto out;
    }
  }
out:
  // coordinator: results for the host
  if (k.bid == 0 && threadIdx.x == 0) {
    C->round = S.co.round;
    C->n_alive = S.co.n_alive;
    C->done = S.plan.state == kDone ? 1 : 0;
    for (int i = 0; i < 8; ++i) C->ph_ns[i] = S.co.ph_ns[i];
  }
}

template <int kPerSM>
__global__ void __launch_bounds__(kThreads, kPerSM) k_rounds(const __grid_constant__ RoundBuffers B) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Shared& S = *reinterpret_cast<Shared*>(smem_raw);
  __shared__ K<kPerSM> k;
  if (threadIdx.x == 0) {
    k.B = B;
    k.C = B.ctl;
    k.S = &S;
    k.G = gridDim.x;
    k.bid = blockIdx.x;
    k.epoch = 0;
    S.failed = 0;
  }
  if (threadIdx.x < kTallies) S.tal[threadIdx.x] = 0;
  // look-back descriptors of an earlier launch could carry the same epochs:
  // clear this block's before the first barrier
  if (threadIdx.x == 0) B.desc[(int64_t)blockIdx.x * kDescStride] = 0;
  __syncthreads();
  run_job(k, vload(&B.ctl->algo));
}


// Labels (center vertex id = order[center rank]) of the vertices first +
// threadIdx.x + i * stride, by a block; with kObjective also this thread's share
// of sum_c C(s_c, 2): the pairs that each member makes with its center and the
// members counted before it (one add per cluster and warp, see k_sizes_pairs).
// A center still carries its active word (an isolated vertex its alive word):
// it is its own cluster.  *members: the members counted, which are also the
// member-center edges (every member is adjacent to its center).  sig: the
// signatures of the state words go there (eight per word).
template <bool kObjective>
__device__ __forceinline__ int64_t finish_vertices(const RoundBuffers& B, int32_t* labels, uint32_t* sig,
                                                   int64_t first, int64_t stride, int64_t* members) {
  const int lane = threadIdx.x & 31;
  const int64_t n = B.n;
  int64_t pairs = 0, mem = 0;
  for (int64_t b = first + threadIdx.x - lane; b < n; b += stride) {
    const int64_t v = b + lane;
    const uint32_t x = v < n ? ldcg(B.st + v) : kAlive;
    int32_t c = -1;                        // rank of the cluster that v joined as a member
    if (v < n) {
      int32_t lab = (int32_t)v;
      if (!is_active(x) && x != kAlive) {
        c = (int32_t)(x - kLab);
        if (is_alive(x) || c < 0 || c >= n) {
          atomicCAS(&B.ctl->err, kOk, kErrInternal);
          c = lab = -1;
        } else {
          lab = ldcg(B.order + c);
        }
      }
      if (labels) labels[v] = lab;
    }
    if (!kObjective) continue;
    const unsigned same = __match_any_sync(FULL, c >= 0 ? c : ~lane);
    if (c >= 0) {
      mem += 1;
      if (lane == __ffs(same) - 1) {
        const int64_t k = __popc(same);
        const int64_t old = atomicAdd(B.size + c, (int32_t)k);
        pairs += k * old + k * (k + 1) / 2;
      }
    }
    if (sig) {
      const uint32_t w = pack_sig8(cluster_sig(x));
      if (v < n && (lane & 7) == 0) sig[v >> 3] = w;
    }
  }
  *members = mem;
  return pairs;
}

// ---------------------------------------------------------------------------
// Batched engine: many (graph, permutation) jobs in one persistent launch.
// The grid is cut into teams (BatchPlan), and a team takes its next job from
// its class's queue, then from those of smaller jobs.  A job is the whole
// pipeline: permutation, state set-up, all rounds, objective.  Each team owns
// one scratch slot, reused job after job.
// ---------------------------------------------------------------------------

// pi for the job in k.B, computed by the team: bucket by the top key bits
// (histogram, exclusive scan, scatter), then a counting sort on the next
// kPermSubBits bits plus an insertion sort inside each bucket.  Also writes
// the initial state words.
template <int kPerSM>
__device__ bool team_permutation(K<kPerSM>& k, uint64_t seed, bool ranks) {
  const RoundBuffers& B = k.B;
  Shared& S = *k.S;
  const int64_t n = B.n;
  int bits = 0;
  while (bits < 12 && (n >> bits) > 768) ++bits;
  const int nb = 1 << bits;
  int64_t* cursor = B.pcnt;            // nb counts, then cursors
  int64_t* start = B.pcnt + nb + 1;    // nb + 1 bucket starts
  const int64_t tid = (int64_t)k.bid * blockDim.x + threadIdx.x, nthr = (int64_t)k.G * blockDim.x;
  // 1: histogram (shared memory, then one global add per non-empty bucket) and state words
  for (int i = threadIdx.x; i < nb; i += blockDim.x) S.u.perm.hist[i] = 0;
  __syncthreads();
  for (int64_t v = tid; v < n; v += nthr) {
    const uint64_t key = perm_key(seed, (uint64_t)v);
    atomicAdd(&S.u.perm.hist[bits == 0 ? 0 : (int)(key >> (64 - bits))], 1);
    const int64_t d = __ldg(B.off + v + 1) - __ldg(B.off + v);
    B.st[v] = kAlive | (uint32_t)d;
    B.size[v] = 0;
    B.hit_c[v] = 0;
    B.hit_p[v] = 0;
  }
  for (int64_t i = tid; i < rtag_words(n); i += nthr) B.rtag[i] = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < nb; i += blockDim.x) {
    const int h = S.u.perm.hist[i];
    if (h) atomicAdd(reinterpret_cast<unsigned long long*>(cursor + i), (unsigned long long)h);
  }
  if (!k.sync(7, [&] {
        int64_t run = 0;
        for (int base = 0; base < nb; base += blockDim.x) {
          const int b = base + threadIdx.x;
          const int64_t c = b < nb ? ldcg(cursor + b) : 0;
          int64_t tot;
          const int64_t ex = block_exclusive_sum<int64_t>(c, S.scr, &tot);
          if (b < nb) { start[b] = run + ex; cursor[b] = run + ex; }
          run += tot;
        }
        if (threadIdx.x == 0) start[nb] = run;
      }))
    return false;
  // 2: scatter
  for (int64_t v = tid; v < n; v += nthr) {
    const uint64_t key = perm_key(seed, (uint64_t)v);
    const int b = bits == 0 ? 0 : (int)(key >> (64 - bits));
    const int64_t pos = (int64_t)atomicAdd(reinterpret_cast<unsigned long long*>(cursor + b), 1ull);
    B.ptmp[pos] = (int32_t)v;
  }
  if (!k.sync(7)) return false;
  // 3: sort each bucket by (key, v)
  PermSmem& P = S.u.perm;
  const int shift = 64 - bits - kPermSubBits;
  for (int b = (int)k.bid; b < nb; b += (int)k.G) {
    const int64_t s0 = ldcg(start + b), len = ldcg(start + b + 1) - s0;
    if (len <= 0) continue;
    if (len > kPermCap) {
      // rare: rank by counting (exact, quadratic)
      for (int64_t i = threadIdx.x; i < len; i += blockDim.x) {
        const int32_t vi = ldcg(B.ptmp + s0 + i);
        const uint64_t ki = perm_key(seed, (uint64_t)vi);
        int64_t r = 0;
        for (int64_t j = 0; j < len; ++j) {
          const int32_t vj = ldcg(B.ptmp + s0 + j);
          const uint64_t kj = perm_key(seed, (uint64_t)vj);
          r += (kj < ki || (kj == ki && vj < vi)) ? 1 : 0;
        }
        B.order_w[s0 + r] = vi;
        if (ranks) B.arank[vi] = (int32_t)(s0 + r);
      }
      __syncthreads();
      continue;
    }
    for (int i = threadIdx.x; i < kPermSub; i += blockDim.x) P.cnt[i] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < len; i += blockDim.x) {
      const int32_t v = ldcg(B.ptmp + s0 + i);
      const uint64_t key = perm_key(seed, (uint64_t)v);
      P.sv[i] = v;
      P.sk[i] = key;
      atomicAdd(&P.cnt[(int)((key >> shift) & (kPermSub - 1))], 1);
    }
    __syncthreads();
    {
      const int i0 = threadIdx.x * 2;
      const int c0 = i0 < kPermSub ? P.cnt[i0] : 0, c1 = i0 + 1 < kPermSub ? P.cnt[i0 + 1] : 0;
      int64_t tot;
      const int64_t ex = block_exclusive_sum<int64_t>(c0 + c1, S.scr, &tot);
      if (i0 < kPermSub) P.cnt[i0] = (int)ex;
      if (i0 + 1 < kPermSub) P.cnt[i0 + 1] = (int)ex + c0;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < len; i += blockDim.x) {
      const uint64_t key = P.sk[i];
      const int pos = atomicAdd(&P.cnt[(int)((key >> shift) & (kPermSub - 1))], 1);
      P.ok[pos] = key;
      P.ov[pos] = P.sv[i];
    }
    __syncthreads();
    for (int q = threadIdx.x; q < kPermSub; q += blockDim.x) {
      const int lo = q == 0 ? 0 : P.cnt[q - 1], hi = P.cnt[q];
      for (int i = lo + 1; i < hi; ++i) {
        const uint64_t key = P.ok[i];
        const int32_t v = P.ov[i];
        int j = i - 1;
        while (j >= lo && (key < P.ok[j] || (key == P.ok[j] && v < P.ov[j]))) {
          P.ok[j + 1] = P.ok[j];
          P.ov[j + 1] = P.ov[j];
          --j;
        }
        P.ok[j + 1] = key;
        P.ov[j + 1] = v;
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < len; i += blockDim.x) {
      B.order_w[s0 + i] = P.ov[i];
      if (ranks) B.arank[P.ov[i]] = (int32_t)(s0 + i);
    }
    __syncthreads();
  }
  return k.sync(7);
}

template <int kPerSM>
__global__ void __launch_bounds__(kThreads, kPerSM)
k_batch(BatchJob* __restrict__ jobs, const RoundBuffers* __restrict__ slots, const __grid_constant__ BatchPlan plan,
        int algo, int64_t eps_ppm) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Shared& S = *reinterpret_cast<Shared*>(smem_raw);
  __shared__ K<kPerSM> k;
  RoundBuffers& rb = k.B;
  int cls = 0;
  while (cls + 1 < plan.n && (int)blockIdx.x >= plan.block0[cls + 1]) ++cls;
  const unsigned G = (unsigned)plan.team[cls], rel = blockIdx.x - (unsigned)plan.block0[cls];
  const RoundBuffers& slot = slots[plan.slot0[cls] + (int)(rel / G)];
  Ctl* const C = slot.ctl;
  if (threadIdx.x == 0) {
    k.C = C;
    k.S = &S;
    k.G = G;
    k.bid = rel % G;
    k.epoch = 0;
    S.failed = 0;
    S.plan.state = kDone;
  }
  // the team's next job (-1: none left), published with the plan
  auto take_job = [&] {
    S.plan.k = -1;
    for (int q = cls; q < plan.n && S.plan.k < 0; ++q) {
      const int j = plan.job0[q] + atomicAdd(&slots[0].ctl->queue[q], 1);
      if (j < plan.job0[q + 1]) S.plan.k = j;
    }
  };
  __syncthreads();
  if (!k.sync(7, [&] { if (threadIdx.x == 0) take_job(); })) return;
  for (int j; (j = (int)S.plan.k) >= 0;) {
    if (threadIdx.x == 0) {
      rb = slot;
      const BatchJob& jb = jobs[j];
      rb.n = jb.n;
      rb.nnz = jb.nnz;
      rb.max_deg = jb.max_deg;
      rb.off = jb.off;
      rb.col = jb.col;
      rb.dsort = jb.dsort;
      rb.dge = jb.dge;
      rb.up = jb.up;
      rb.nz_static = jb.nz;
      rb.nz_n = jb.nz_n;
      rb.order = rb.order_w;
      rb.stats = nullptr;
      rb.stats_cap = 0;
      if (k.bid == 0) jobs[j].t0 = (int64_t)globaltimer_ns();   // device clock at the job's start
    }
    __syncthreads();
    // zero the permutation counters, reset the control block (not the barrier counters)
    const int64_t zn = 2 * (int64_t)kPermMaxBuckets + 2;
    for (int64_t i = (int64_t)k.bid * blockDim.x + threadIdx.x; i < zn; i += (int64_t)G * blockDim.x) rb.pcnt[i] = 0;
    if (threadIdx.x == 0) rb.desc[(int64_t)k.bid * kDescStride] = 0;   // look-back descriptors of an earlier launch
    if (!k.sync(7, [&] {
          if (threadIdx.x == 0) {
            C->err = 0;
            S.failed = 0;
            C->algo = algo;
            C->eps_ppm = eps_ppm;
            C->seed = jobs[j].seed;
            C->intra = 0; C->pairs = 0;
            C->undecided = 0; C->h_pack = 0;
            S.plan.state = kRun;
          }
        }))
      break;
    if (!team_permutation(k, jobs[j].seed, algo == kAlgoC4 || algo == kAlgoC4 + 2)) break;
    if (threadIdx.x < kTallies) S.tal[threadIdx.x] = 0;
    __syncthreads();
    run_job(k, algo);
    if (S.plan.state == kAbort) {
      if (k.bid == 0 && threadIdx.x == 0) jobs[j].err = ld_volatile_int(&C->err) ? ld_volatile_int(&C->err) : kErrInternal;
      break;
    }
    // labels and the objective (see k_finalize_labels; k_intra)
    int64_t members;
    const int64_t pairs = block_sum<int64_t>(
        finish_vertices<true>(rb, jobs[j].labels, nullptr, (int64_t)k.bid * blockDim.x, (int64_t)G * blockDim.x,
                              &members), S.scr);
    const int64_t inside = block_sum<int64_t>(members + k.intra_edges(), S.scr);
    if (threadIdx.x == 0) {
      if (pairs) atomicAdd(&C->pairs, (unsigned long long)pairs);
      if (inside) atomicAdd(&C->intra, (unsigned long long)inside);
    }
    if (!k.sync(6, [&] {
          if (threadIdx.x == 0) {
            BatchJob& jb = jobs[j];
            const int done = S.plan.state == kDone && S.co.n_alive == 0;
            jb.rounds = S.co.round;
            jb.D = jb.nnz / 2 - 2 * (int64_t)vload(&C->intra) + (int64_t)vload(&C->pairs);
            jb.err = done && vload(&C->err) == kOk ? 0 : kErrInternal;
            jb.t1 = (int64_t)globaltimer_ns();
            S.plan.state = kDone;
            take_job();
          }
        }))
      break;
  }
}

__global__ void k_init_state(RoundBuffers B, int algo, int64_t eps_ppm, uint64_t seed, int32_t withhold) {
  const int64_t n = B.n;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int64_t d = __ldg(B.off + v + 1) - __ldg(B.off + v);
    B.st[v] = kAlive | (uint32_t)d;
    B.size[v] = 0;                     // members per center rank
    B.hit_c[v] = 0;                    // C4 fixpoint flags start (and stay) zero
    B.hit_p[v] = 0;
    if ((algo == kAlgoC4 || algo == kAlgoC4 + 2) && n <= kStateInL2) B.arank[__ldg(B.order + v)] = (int32_t)v;
  }
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rtag_words(n); i += (int64_t)gridDim.x * blockDim.x)
    B.rtag[i] = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    Ctl* C = B.ctl;
    C->algo = algo;
    C->eps_ppm = eps_ppm;
    C->seed = seed;
    C->withhold = withhold;
    C->n_alive = n;
    C->done = n > 0 ? 0 : 1;
  }
}

__global__ void k_finalize_labels(RoundBuffers B, int32_t* __restrict__ labels, bool objective, bool sig) {
  __shared__ int64_t scr[33];
  const int64_t first = (int64_t)blockIdx.x * blockDim.x, stride = (int64_t)gridDim.x * blockDim.x;
  if (!objective) {
    int64_t members;
    finish_vertices<false>(B, labels, nullptr, first, stride, &members);
    return;
  }
  int64_t members;
  const int64_t pairs =
      block_sum<int64_t>(finish_vertices<true>(B, labels, sig ? B.rtag : nullptr, first, stride, &members), scr);
  members = block_sum<int64_t>(members, scr);
  if (threadIdx.x == 0) {
    if (pairs) atomicAdd(&B.ctl->pairs, (unsigned long long)pairs);
    if (members) atomicAdd(&B.ctl->intra, (unsigned long long)members);
  }
}

}  // namespace

Tuning default_tuning() {
  return Tuning{kLbsBatches, kLbsPfAhead, kInlineH, kInlineDecide, kInlineRebuild, kHeavyShift, kWarpResolveRow};
}

size_t rounds_workspace_bytes(int64_t n, int32_t max_deg, int grid) {
  const size_t nn = (size_t)(n > 0 ? n : 1);
  size_t b = 0;
  b += align_up(sizeof(Ctl));
  b += align_up(4 * nn);                 // st
  b += align_up(4 * ((nn >> 3) + 1));    // rtag
  b += align_up(4 * nn);                 // arank
  b += 2 * align_up(4 * nn) + 2 * align_up(8 * nn);   // act_v, act_r, act_e, act_d
  b += align_up(4 * nn) + align_up(4 * kHList);       // act_n, h_acc
  b += align_up(4 * nn);                 // size
  b += 3 * align_up(4 * nn);             // hv, hv2, nz0
  b += 3 * align_up(nn);                 // blk_flag, hit_c, hit_p
  b += align_up(4 * nn);                 // pull
  b += align_up(4 * nn) + 2 * align_up(8 * nn);       // b_j, b_e, b_d
  b += align_up(8 * kDescStride * ((size_t)grid + 1)); // desc
  return b;
}

void rounds_carve(void* ws, int64_t n, int32_t max_deg, int grid, RoundBuffers* B) {
  const size_t nn = (size_t)(n > 0 ? n : 1);
  B->tune = default_tuning();
  char* p = static_cast<char*>(ws);
  auto take = [&](size_t bytes) { char* q = p; p += align_up(bytes); return q; };
  B->ctl = reinterpret_cast<Ctl*>(take(sizeof(Ctl)));
  B->st = reinterpret_cast<uint32_t*>(take(4 * nn));
  B->rtag = reinterpret_cast<uint32_t*>(take(4 * ((nn >> 3) + 1)));
  B->arank = reinterpret_cast<int32_t*>(take(4 * nn));
  B->act_v = reinterpret_cast<int32_t*>(take(4 * nn));
  B->act_r = reinterpret_cast<int32_t*>(take(4 * nn));
  B->act_e = reinterpret_cast<int64_t*>(take(8 * nn));
  B->act_d = reinterpret_cast<int64_t*>(take(8 * nn));
  B->act_n = reinterpret_cast<int32_t*>(take(4 * nn));
  B->h_acc = reinterpret_cast<unsigned*>(take(4 * kHList));
  B->size = reinterpret_cast<int32_t*>(take(4 * nn));
  B->hv = reinterpret_cast<int32_t*>(take(4 * nn));
  B->hv2 = reinterpret_cast<int32_t*>(take(4 * nn));
  B->nz0 = reinterpret_cast<int32_t*>(take(4 * nn));
  B->blk_flag = reinterpret_cast<uint8_t*>(take(nn));
  B->hit_c = reinterpret_cast<uint8_t*>(take(nn));
  B->hit_p = reinterpret_cast<uint8_t*>(take(nn));
  B->pull = reinterpret_cast<int32_t*>(take(4 * nn));
  B->b_j = reinterpret_cast<int32_t*>(take(4 * nn));
  B->b_e = reinterpret_cast<int64_t*>(take(8 * nn));
  B->b_d = reinterpret_cast<int64_t*>(take(8 * nn));
  B->desc = reinterpret_cast<unsigned long long*>(take(8 * kDescStride * ((size_t)grid + 1)));
}

// Blocks of k_rounds per SM.  Rounds of few entries are a chain of barriers and
// dependent reads: one block per SM, whose barrier has half the arrivals and
// whose 128 registers spill nothing, is faster; longer walks want the entries in
// flight of twice as many warps.  The rounds of a run grow with log Delta, so the
// measure is entries / log2 of the largest degree (one / two blocks per SM, ms):
//   planted 2M  68M / 6    C4  2.50 / 2.57        R-MAT 21   64M / 16  C4  4.78 / 5.44
//   planted 3M 103M / 6    CW  2.22 / 2.14        R-MAT 23  260M / 17  CW  5.88 / 6.15
//   planted 4M 137M / 6    C4  3.77 / 3.43        R-MAT 24  520M / 18  C4 11.83 / 11.65
//   planted 8M 275M / 6    CW  4.48 / 3.56        R-MAT 24             CW  8.61 / 8.63
constexpr int64_t kTwoPerSM = int64_t(1) << 24;
inline int blocks_per_sm(int64_t nnz, int32_t max_deg) {
  int log = 1;
  while (log < 31 && (max_deg >> (log + 1)) != 0) ++log;
  return nnz / log < kTwoPerSM ? 1 : 2;
}

int rounds_grid_size(int device, int64_t nnz, int32_t max_deg) {
  int sms = 0, per = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  if (blocks_per_sm(nnz, max_deg) == 1) return sms;
  cudaFuncSetAttribute(k_rounds<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Shared));
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_rounds<2>, kThreads, sizeof(Shared));
  if (per < 1) per = 1;
  if (per > 2) per = 2;
  return sms * per;
}

cudaError_t launch_rounds(const RoundBuffers& b, int algo, int64_t eps_ppm, uint64_t seed, int grid,
                          cudaStream_t stream, int32_t withhold) {
  cudaError_t e = cudaMemsetAsync(b.ctl, 0, sizeof(Ctl), stream);
  if (e != cudaSuccess) return e;
  k_init_state<<<grid, 256, 0, stream>>>(b, algo, eps_ppm, seed, withhold);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (b.n <= 0) return cudaSuccess;
  RoundBuffers arg = b;
  void* args[] = {&arg};
  const void* const f = blocks_per_sm(b.nnz, b.max_deg) == 1 ? (const void*)k_rounds<1> : (const void*)k_rounds<2>;
  e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Shared));
  if (e != cudaSuccess) return e;
  return cudaLaunchCooperativeKernel(f, dim3(grid), dim3(kThreads), args, sizeof(Shared),
                                     stream);
}

cudaError_t launch_finalize_labels(const RoundBuffers& b, const FullRows& all, int32_t* labels_out, bool objective,
                                   int num_sms, cudaStream_t stream) {
  if (b.n <= 0) return cudaSuccess;
  const int64_t want = (b.n + 255) / 256;
  const int grid = (int)(want < 2048 ? want : 2048);
  const bool sig = intra_wants_signatures(b.n, b.up);
  k_finalize_labels<<<grid, 256, 0, stream>>>(b, labels_out, objective, sig);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || !objective) return e;
  return launch_intra(b.col, b.up, all, b.st, sig ? b.rtag : nullptr, kLab, kAlive, &b.ctl->intra, num_sms, stream);
}

int batch_grid_size(int device) {
  int sms = 0, per = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  cudaFuncSetAttribute(k_batch<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Shared));
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch<2>, kThreads, sizeof(Shared));
  if (per < 1) per = 1;
  if (per > 2) per = 2;
  return sms * per;
}

size_t batch_slot_bytes(int64_t n_max, int team_size) {
  const size_t nn = (size_t)(n_max > 0 ? n_max : 1);
  return rounds_workspace_bytes(n_max, 0, team_size) + 2 * align_up(4 * nn) +
         align_up(8 * (2 * (size_t)kPermMaxBuckets + 2));
}

void batch_slot_carve(void* ws, int64_t n_max, int team_size, RoundBuffers* B) {
  const size_t nn = (size_t)(n_max > 0 ? n_max : 1);
  rounds_carve(ws, n_max, 0, team_size, B);
  char* p = static_cast<char*>(ws) + rounds_workspace_bytes(n_max, 0, team_size);
  B->order_w = reinterpret_cast<int32_t*>(p); p += align_up(4 * nn);
  B->ptmp = reinterpret_cast<int32_t*>(p); p += align_up(4 * nn);
  B->pcnt = reinterpret_cast<int64_t*>(p);
  B->order = B->order_w;
}

cudaError_t launch_batch(const BatchJob* jobs_dev, const RoundBuffers* slots_dev, const BatchPlan& plan, int algo,
                         int64_t eps_ppm, cudaStream_t stream) {
  const void* const f = (const void*)k_batch<2>;
  const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Shared));
  if (e != cudaSuccess) return e;
  BatchJob* jobs = const_cast<BatchJob*>(jobs_dev);
  BatchPlan p = plan;
  void* args[] = {&jobs, &slots_dev, &p, &algo, &eps_ppm};
  const dim3 grid((unsigned)p.block0[p.n]);
  // teams of one block wait for no other block: an ordinary launch suffices,
  // and several batches can share the GPU
  bool alone = true;
  for (int c = 0; c < p.n; ++c) alone = alone && p.team[c] == 1;
  return alone ? cudaLaunchKernel(f, grid, dim3(kThreads), args, sizeof(Shared), stream)
               : cudaLaunchCooperativeKernel(f, grid, dim3(kThreads), args, sizeof(Shared), stream);
}

}  // namespace ccg
