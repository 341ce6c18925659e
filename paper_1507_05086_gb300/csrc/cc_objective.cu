// cc_objective.cu -- the disagreement objective (Sec. 2) of an arbitrary
// labelling, CSR validation and small graph utilities.
//
// Disagreements: with m positive edges, intra = positive edges inside a
// cluster and s_c the cluster sizes,
//     D = (m - intra) + (sum_c C(s_c, 2) - intra) = m - 2 intra + sum_c C(s_c, 2).
// One pass over the vertices adds up the sizes and the pairs, one
// edge-balanced pass over the upper parts of the rows (every edge once)
// counts intra.
#include <cstdint>

#include "cc_device.cuh"
#include "cc_internal.h"

namespace ccg {
namespace {

constexpr int kObjThreads = 512;
constexpr int kObjBlocks = 2;          // blocks of k_intra per SM
// Graphs above this many vertices read 4-bit signatures before ids: up to it
// the ids (64 MB) fit the 129 MB L2 themselves.
constexpr int64_t kSigMin = int64_t(1) << 24;

// sum_c C(s_c, 2) = sum over the vertices of the number of members that their
// cluster had before them, so the add that counts a member also gives its
// pairs (no second pass over the sizes).  Lanes of a warp with the same label
// share one add: the adds of a cluster queue on one word, which bound the
// whole call on a planted partition (2M vertices, the largest cluster 0.77M
// members: 915 us with one add per vertex and both ends of every edge read,
// 310 us so).
__global__ void k_sizes_pairs(int64_t n, const int32_t* __restrict__ labels, int32_t* __restrict__ size,
                              unsigned long long* out) {
  __shared__ int64_t scr[33];
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t pairs = 0;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; b < n; b += stride) {
    const int64_t v = b + lane;
    int32_t c = v < n ? __ldg(labels + v) : -1;
    if (v < n && (c < 0 || c >= n)) { atomicExch(out + 2, 1ull); c = -1; }
    const unsigned same = __match_any_sync(FULL, c);
    if (c < 0 || lane != __ffs(same) - 1) continue;
    const int64_t k = __popc(same);
    const int64_t old = atomicAdd(size + c, (int32_t)k);
    pairs += k * old + k * (k - 1) / 2;
  }
  pairs = block_sum<int64_t>(pairs, scr);
  if (threadIdx.x == 0 && pairs) atomicAdd(out + 1, (unsigned long long)pairs);
}

// Edges (u, w) with id[u] == id[w] in [lo, hi), every edge read from its lower
// end only (half of the CSR's entries).  Bound by the random id reads in L2: at R-MAT 24
// (260M edges, 1.04 ms, 250e9 edges/s) L2 runs at 66 % and L1 at 69 % of their
// throughput, above the 236e9 reads/s of a library gather from a 32 MiB table.
// With sig, a 4-bit signature per vertex decides first, so that ids are read
// only where the signatures agree.  Whole objective of a ClusterWild! labelling
// of R-MAT 22 / 24 / 26: both ends of every edge 0.59 / 2.43 / 12.5 ms, upper
// ends over 128-edge batches (lbs_for_each) 0.40 / 1.52 / 7.6 ms, by units of 32
// entries 0.32 / 1.22 / 5.8 ms.  Three blocks per SM at 40 registers spill: 0.49 /
// 1.90 / 7.4; four units per batch at three blocks: 0.37 / 1.41 / 5.7.  By rows
// (row_walk) 0.37 ms at R-MAT 22 but 5.3 at R-MAT 26, where the ids come from
// DRAM: with sig the walk is by rows, else by units.
template <bool kSig>
__global__ void __launch_bounds__(kObjThreads, kObjBlocks) k_intra(UpperRows up, const int32_t* __restrict__ col,
                                                      uint32_t lo, uint32_t hi,
                                                      const uint32_t* __restrict__ id,
                                                      const uint32_t* __restrict__ sig, unsigned long long* out) {
  __shared__ int64_t scr[33];
  int64_t cnt = 0;
  auto center = [&](int64_t j) {
    const uint32_t x = __ldg(id + __ldg(up.v + j));
    return (int32_t)(x >= lo && x < hi ? x : 0xFFFFFFFFu);
  };
  auto count = [&](const auto& X) {
    constexpr int kB = sizeof(X.w) / sizeof(int32_t);
    uint32_t x[kB];
    if (kSig) {
#pragma unroll
      for (int q = 0; q < kB; ++q) x[q] = X.w[q] >= 0 ? __ldg(sig + (X.w[q] >> 3)) >> ((X.w[q] & 7) * 4) : 0;
#pragma unroll
      for (int q = 0; q < kB; ++q)
        if (X.w[q] >= 0 && ((x[q] ^ cluster_sig((uint32_t)X.aux[q])) & 15u) == 0)
          cnt += __ldg(id + X.w[q]) == (uint32_t)X.aux[q] ? 1 : 0;
    } else {
#pragma unroll
      for (int q = 0; q < kB; ++q) x[q] = X.w[q] >= 0 ? __ldg(id + X.w[q]) : 0;
#pragma unroll
      for (int q = 0; q < kB; ++q) cnt += X.w[q] >= 0 && x[q] == (uint32_t)X.aux[q] ? 1 : 0;
    }
  };
  const int gwarp = (int)(threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x;
  const int nwarps = (int)((gridDim.x * blockDim.x) >> 5);
  if (kSig) {
    row_walk<kUnitB>(gwarp, nwarps, (int32_t)up.n, up.edges, col, WalkShape{},
                     [&](int32_t j) { return (int64_t)__ldg(up.epos + j); },
                     [&](int32_t j) {
                       return RowItem{(int64_t)__ldg(up.epos + j), __ldg(up.row + j), __ldg(up.len + j), center(j)};
                     },
                     count);
  } else {
    unit_walk(gwarp, nwarps, up.n, up.units, col, WalkShape{}, [&](int64_t j) { return __ldg(up.pos + j); },
              [&](int64_t j) { return UnitItem{__ldg(up.pos + j), __ldg(up.len + j), __ldg(up.row + j), center(j)}; },
              count);
  }
  cnt = block_sum<int64_t>(cnt, scr);
  if (threadIdx.x == 0 && cnt) atomicAdd(out, (unsigned long long)cnt);
}

// The same over all entries of graphs with short rows, every edge at its lower
// end.  A row of two or three upper entries leaves most of its unit empty, and a
// window of row_walk is then only a few lines of the column array; lbs_for_each
// puts up to 128 rows into a batch.  Whole objective of a ClusterWild! labelling
// (by units, above 2^24 vertices by rows / by this kernel): ring of 4M vertices
// 0.26 / 0.13 ms, of 20M 0.77 / 0.52, grid of 9M 0.69 / 0.29, Erdos-Renyi of 1M and
// mean degree 3 0.10 / 0.06, random tree of 2M 0.14 / 0.08.
__global__ void __launch_bounds__(kObjThreads) k_intra_short(FullRows all, const int32_t* __restrict__ col,
                                                            uint32_t lo, uint32_t hi,
                                                            const uint32_t* __restrict__ id, unsigned long long* out) {
  __shared__ LbsWarp lbs[kObjThreads / 32];
  __shared__ int64_t scr[33];
  int64_t cnt = 0;
  lbs_for_each(all.pos, all.n, all.nnz, &lbs[threadIdx.x >> 5], [&](const Lbs& L) {
    uint32_t x[kLbsK];
    int32_t w[kLbsK];
#pragma unroll
    for (int t = 0; t < kLbsK; ++t) {
      const int32_t u = L.ok(t) ? __ldg(all.v + L.item(t)) : 0;
      w[t] = L.ok(t) ? __ldg(col + L.edge(t)) : -1;
      x[t] = L.ok(t) ? __ldg(id + u) : 0;
      if (w[t] <= u) w[t] = -1;
    }
#pragma unroll
    for (int t = 0; t < kLbsK; ++t)
      if (w[t] >= 0 && x[t] >= lo && x[t] < hi) cnt += __ldg(id + w[t]) == x[t] ? 1 : 0;
  }, nullptr, nullptr, 0, col);
  cnt = block_sum<int64_t>(cnt, scr);
  if (threadIdx.x == 0 && cnt) atomicAdd(out, (unsigned long long)cnt);
}

// Short rows: fewer than kShortFill upper entries per unit.  Erdos-Renyi graphs of
// 4M vertices and mean degree 8 / 12, 4.1 and 6.1 entries per unit, take 0.32 /
// 0.33 ms by units and 0.24 / 0.33 by k_intra_short.
constexpr int kShortFill = 6;
inline bool short_rows(const UpperRows& up) { return up.edges < kShortFill * up.units; }

// sig word i: the signatures of the ids of vertices 8 i .. 8 i + 7.
__global__ void k_signatures(int64_t n, const uint32_t* __restrict__ id, uint32_t* __restrict__ sig) {
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; b < n; b += stride) {
    const int64_t v = b + lane;
    const uint32_t s = pack_sig8(v < n ? cluster_sig(__ldg(id + v)) : 0u);
    if (v < n && (lane & 7) == 0) sig[v >> 3] = s;
  }
}

// ---- validation ---------------------------------------------------------------
// Error codes written to flags[0] (first one wins).
constexpr int kBadOffsets = 1, kBadColumn = 2, kSelfLoop = 3, kUnsorted = 4, kAsymmetric = 5;

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 33)) * 0xFF51AFD7ED558CCDull;
  z = (z ^ (z >> 33)) * 0xC4CEB9FE1A85EC53ull;
  return z ^ (z >> 33);
}

// Offsets: monotone, inside [0, nnz]; largest degree.
__global__ void k_validate_offsets(int64_t n, int64_t nnz, const int64_t* __restrict__ off, int* flags) {
  int dmax = 0;
  for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
    const int64_t a = off[u], b = off[u + 1];
    if (a < 0 || b < a || b > nnz) { atomicCAS(flags, 0, kBadOffsets); continue; }
    const int64_t d = b - a;
    dmax = max(dmax, d > 0x7FFFFFFF ? 0x7FFFFFFF : (int)d);
  }
  dmax = warp_max(dmax);
  if ((threadIdx.x & 31) == 0 && dmax > 0) atomicMax(flags + 1, dmax);
}

// Entries, edge-balanced over the non-empty rows: range, order, self loops;
// symmetry by comparing two hash sums of the pairs (min, max) seen from the
// lower and from the upper endpoint (equal multisets give equal sums).
constexpr int kValThreads = 512;

__global__ void __launch_bounds__(kValThreads) k_validate_edges(int64_t n, int64_t e0, int64_t e1, int64_t nz_n,
                                                               const int32_t* __restrict__ nz_row,
                                                               const int64_t* __restrict__ nz_pos,
                                                               const int32_t* __restrict__ col,
                                                               int64_t* __restrict__ up_at, int* flags,
                                                               unsigned long long* sums) {
  __shared__ LbsWarp lbs[kValThreads / 32];
  unsigned long long lo1 = 0, lo2 = 0, up1 = 0, up2 = 0;
  long long nlo = 0, nup = 0;
  int bad = 0;
  lbs_for_each(nz_pos, nz_n, e1, &lbs[threadIdx.x >> 5], [&](const Lbs& L) {
#pragma unroll
    for (int t = 0; t < kLbsK; ++t) {
      if (!L.ok(t)) continue;
      const int64_t e = L.edge(t);
      const int32_t u = __ldg(nz_row + L.item(t));
      const int32_t w = __ldg(col + e);
      if (w < 0 || w >= n) { bad = bad ? bad : kBadColumn; continue; }
      if (w == u) { bad = bad ? bad : kSelfLoop; continue; }
      const int32_t prev = L.in_row(t) > 0 ? __ldg(col + e - 1) : -1;
      if (prev >= w) bad = bad ? bad : kUnsorted;
      if (w > u && prev < u) up_at[L.item(t)] = e;      // the row's upper part starts here
      const uint64_t key = u < w ? (((uint64_t)u << 32) | (uint32_t)w) : (((uint64_t)w << 32) | (uint32_t)u);
      const uint64_t h1 = mix64(key ^ 0x9E3779B97F4A7C15ull), h2 = mix64(key + 0x632BE59BD9B4E019ull);
      if (u < w) { lo1 += h1; lo2 += h2; ++nlo; } else { up1 += h1; up2 += h2; ++nup; }
    }
  }, nullptr, nullptr, e0, col);
  if (bad) atomicCAS(flags, 0, bad);
  lo1 = warp_sum(lo1); lo2 = warp_sum(lo2); up1 = warp_sum(up1); up2 = warp_sum(up2);
  nlo = warp_sum(nlo); nup = warp_sum(nup);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(sums + 0, lo1); atomicAdd(sums + 1, lo2);
    atomicAdd(sums + 2, up1); atomicAdd(sums + 3, up2);
    atomicAdd(sums + 4, (unsigned long long)nlo); atomicAdd(sums + 5, (unsigned long long)nup);
  }
}

// Exact symmetry (opt-in): every entry (u, w) with u < w must have u in row w,
// found by binary search in that sorted row.  Together with the equal counts
// of lower and upper entries (k_validate_symmetry) this makes the entries
// seen from the two ends the same set of pairs.
__global__ void __launch_bounds__(kValThreads) k_validate_reverse(int64_t nz_n, const int32_t* __restrict__ nz_row,
                                                                 const int64_t* __restrict__ nz_pos, int64_t nnz,
                                                                 const int64_t* __restrict__ off,
                                                                 const int32_t* __restrict__ col, int* flags) {
  __shared__ LbsWarp lbs[kValThreads / 32];
  int bad = 0;
  lbs_for_each(nz_pos, nz_n, nnz, &lbs[threadIdx.x >> 5], [&](const Lbs& L) {
#pragma unroll
    for (int t = 0; t < kLbsK; ++t) {
      if (!L.ok(t)) continue;
      const int32_t u = __ldg(nz_row + L.item(t));
      const int32_t w = __ldg(col + L.edge(t));
      if (w <= u) continue;
      int64_t lo = __ldg(off + w), hi = __ldg(off + w + 1);
      while (lo < hi) {
        const int64_t mid = lo + ((hi - lo) >> 1);
        if (__ldg(col + mid) < u) lo = mid + 1;
        else hi = mid;
      }
      if (lo >= __ldg(off + w + 1) || __ldg(col + lo) != u) bad = kAsymmetric;
    }
  }, nullptr, nullptr, 0, col);
  if (bad) atomicCAS(flags, 0, bad);
}

__global__ void k_validate_finish(int64_t n, const int64_t* __restrict__ off, int64_t nnz, int* flags,
                                  const unsigned long long* sums) {
  (void)sums;
  if (off[0] != 0 || off[n] != nnz) atomicCAS(flags, 0, kBadOffsets);
}

__global__ void k_validate_symmetry(int* flags, const unsigned long long* sums) {
  if (sums[0] != sums[2] || sums[1] != sums[3] || sums[4] != sums[5]) atomicCAS(flags, 0, kAsymmetric);
}

__global__ void k_off32_to_64(int64_t n, const int32_t* __restrict__ in, int64_t* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = in[i];
}

// Non-empty rows: per-block counts, a single-block scan, then the write.
constexpr int kNzTile = 1024;

__global__ void k_nz_count(int64_t n, const int64_t* __restrict__ off, int64_t* __restrict__ tile_cnt) {
  __shared__ int64_t scr[33];
  const int64_t ntiles = (n + kNzTile - 1) / kNzTile;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int64_t v = t * kNzTile + threadIdx.x;
    int64_t c = (v < n && off[v + 1] > off[v]) ? 1 : 0;
    c = block_sum<int64_t>(c, scr);
    if (threadIdx.x == 0) tile_cnt[t] = c;
  }
}

// Block b scans the counts at tile_cnt + b * stride, its sum goes to total[b].
__global__ void k_nz_scan(int64_t ntiles, int64_t* __restrict__ tile_cnt, int64_t stride,
                          int64_t* __restrict__ total) {
  tile_cnt += blockIdx.x * stride;
  __shared__ int64_t scr[33];
  int64_t run = 0;
  for (int64_t base = 0; base < ntiles; base += blockDim.x) {
    const int64_t t = base + threadIdx.x;
    const int64_t x = t < ntiles ? tile_cnt[t] : 0;
    int64_t tot;
    const int64_t ex = block_exclusive_sum<int64_t>(x, scr, &tot);
    if (t < ntiles) tile_cnt[t] = run + ex;
    run += tot;
  }
  if (threadIdx.x == 0) total[blockIdx.x] = run;
}

__global__ void k_nz_write(int64_t n, const int64_t* __restrict__ off, const int64_t* __restrict__ tile_off,
                           int32_t* __restrict__ nz_row, int64_t* __restrict__ nz_pos, int64_t* __restrict__ up_at) {
  __shared__ int64_t scr[33];
  const int64_t ntiles = (n + kNzTile - 1) / kNzTile;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int64_t v = t * kNzTile + threadIdx.x;
    const int64_t c = (v < n && off[v + 1] > off[v]) ? 1 : 0;
    int64_t tot;
    const int64_t ex = block_exclusive_sum<int64_t>(c, scr, &tot);
    if (c) {
      nz_row[tile_off[t] + ex] = (int32_t)v;
      nz_pos[tile_off[t] + ex] = off[v];
      up_at[tile_off[t] + ex] = off[v + 1];
    }
  }
}

// Rows with a non-empty upper part, by the same three steps; counts are
// packed (rows << kPackShift | units); the entries are counted beside them.
__device__ __forceinline__ int64_t upper_len(int64_t j, int64_t nz_n, int64_t nnz, const int64_t* nz_pos,
                                             const int64_t* up_at) {
  return j < nz_n ? (j + 1 < nz_n ? nz_pos[j + 1] : nnz) - up_at[j] : 0;
}

__global__ void k_up_count(int64_t nz_n, int64_t nnz, const int64_t* __restrict__ nz_pos,
                           const int64_t* __restrict__ up_at, int64_t* __restrict__ tile_cnt,
                           int64_t* __restrict__ tile_len) {
  __shared__ int64_t scr[33];
  const int64_t ntiles = (nz_n + kNzTile - 1) / kNzTile;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int64_t len = upper_len(t * kNzTile + threadIdx.x, nz_n, nnz, nz_pos, up_at);
    const int64_t c = block_sum<int64_t>(len > 0 ? (int64_t(1) << kPackShift) | units_of(len) : 0, scr);
    const int64_t e = block_sum<int64_t>(len, scr);
    if (threadIdx.x == 0) { tile_cnt[t] = c; tile_len[t] = e; }
  }
}

__global__ void k_up_write(int64_t nz_n, int64_t nnz, const int32_t* __restrict__ nz_row,
                           const int64_t* __restrict__ nz_pos, const int64_t* __restrict__ up_at,
                           const int64_t* __restrict__ tile_off, const int64_t* __restrict__ tile_len_off,
                           int32_t* __restrict__ v, int64_t* __restrict__ row, int32_t* __restrict__ len,
                           uint32_t* __restrict__ pos, uint32_t* __restrict__ epos) {
  __shared__ int64_t scr[33];
  const int64_t ntiles = (nz_n + kNzTile - 1) / kNzTile;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int64_t j = t * kNzTile + threadIdx.x;
    const int64_t l = upper_len(j, nz_n, nnz, nz_pos, up_at);
    int64_t tot;
    const int64_t ex = block_exclusive_sum<int64_t>(l > 0 ? (int64_t(1) << kPackShift) | units_of(l) : 0, scr, &tot);
    const int64_t ee = block_exclusive_sum<int64_t>(l, scr, &tot);
    if (l > 0) {
      const uint64_t at = (uint64_t)(tile_off[t] + ex);
      const int64_t o = (int64_t)(at >> kPackShift);
      v[o] = nz_row[j];
      row[o] = up_at[j];
      len[o] = (int32_t)l;
      pos[o] = (uint32_t)(at & kPackEdgeMask);
      epos[o] = (uint32_t)(tile_len_off[t] + ee);
    }
  }
}

// ---- the non-isolated vertices ordered by degree --------------------------
// dsort lists the non-isolated vertices, largest degree first (ties in any
// order), and dge[t] (t = 0 .. max_deg + 1) counts the vertices of degree
// >= t, so dsort[0 .. dge[t]) are exactly the vertices of degree >= t.  The
// round kernel's Delta rebuild reads such a prefix.  Degrees below kDegSmall
// are counted and placed through shared-memory bins (one global atomic per
// block and bin), larger ones (few vertices) directly.
constexpr int kDegSmall = 2048;
constexpr int kDegThreads = 1024;
constexpr int kDegPer = 4;

__global__ void __launch_bounds__(kDegThreads) k_deg_hist(int64_t nz_n, const int32_t* __restrict__ nz_row,
                                                         const int64_t* __restrict__ off,
                                                         unsigned long long* __restrict__ cnt) {
  __shared__ int bin[kDegSmall];
  for (int b = threadIdx.x; b < kDegSmall; b += blockDim.x) bin[b] = 0;
  __syncthreads();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nz_n; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t v = nz_row[i];
    const int64_t d = off[v + 1] - off[v];
    if (d < kDegSmall) atomicAdd(&bin[d], 1);
    else atomicAdd(cnt + d, 1ull);
  }
  __syncthreads();
  for (int b = threadIdx.x; b < kDegSmall; b += blockDim.x)
    if (bin[b]) atomicAdd(cnt + b, (unsigned long long)bin[b]);
}

// dge[t] = sum of cnt[d] over d >= t (suffix sums), in three steps over tiles
// of kDegThreads entries: each tile's own suffix sums and total, a suffix
// scan of the tile totals by one block, then each entry adds the totals of
// the tiles after its own.  cnt[d] then becomes the first position of degree
// d in dsort, dge[d + 1] = dge[d] - cnt[d].
__global__ void __launch_bounds__(kDegThreads) k_deg_suffix_tiles(int64_t len, const unsigned long long* __restrict__ cnt,
                                                                 int64_t* __restrict__ dge, int64_t* __restrict__ tile_tot) {
  __shared__ int64_t scr[33];
  // tile t covers indices [len - (t + 1) * kDegThreads, len - t * kDegThreads), read top down
  const int64_t idx = len - 1 - ((int64_t)blockIdx.x * kDegThreads + threadIdx.x);
  const int64_t x = idx >= 0 ? (int64_t)cnt[idx] : 0;
  int64_t tot;
  const int64_t ex = block_exclusive_sum<int64_t>(x, scr, &tot);
  if (idx >= 0) dge[idx] = ex + x;
  if (threadIdx.x == 0) tile_tot[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(kDegThreads) k_deg_suffix_totals(int64_t ntiles, int64_t* __restrict__ tile_tot) {
  __shared__ int64_t scr[33];
  int64_t run = 0;
  for (int64_t base = 0; base < ntiles; base += blockDim.x) {
    const int64_t t = base + threadIdx.x;
    const int64_t x = t < ntiles ? tile_tot[t] : 0;
    int64_t tot;
    const int64_t ex = block_exclusive_sum<int64_t>(x, scr, &tot);
    if (t < ntiles) tile_tot[t] = run + ex;     // the totals of the tiles above tile t
    run += tot;
  }
}

__global__ void __launch_bounds__(kDegThreads) k_deg_suffix_add(int64_t len, unsigned long long* __restrict__ cnt,
                                                               int64_t* __restrict__ dge,
                                                               const int64_t* __restrict__ tile_tot) {
  const int64_t idx = len - 1 - ((int64_t)blockIdx.x * kDegThreads + threadIdx.x);
  if (idx < 0) return;
  const int64_t d = dge[idx] + tile_tot[blockIdx.x];
  dge[idx] = d;
  if (idx < len - 1) cnt[idx] = (unsigned long long)(d - (int64_t)cnt[idx]);
}

__global__ void __launch_bounds__(kDegThreads) k_deg_scatter(int64_t nz_n, const int32_t* __restrict__ nz_row,
                                                            const int64_t* __restrict__ off,
                                                            unsigned long long* __restrict__ cur,
                                                            int32_t* __restrict__ dsort) {
  __shared__ int bin[kDegSmall];
  __shared__ unsigned long long base[kDegSmall];
  const int64_t tile = (int64_t)kDegThreads * kDegPer;
  for (int64_t t0 = blockIdx.x * tile; t0 < nz_n; t0 += (int64_t)gridDim.x * tile) {
    for (int b = threadIdx.x; b < kDegSmall; b += blockDim.x) bin[b] = 0;
    __syncthreads();
    int32_t v[kDegPer];
    int32_t d[kDegPer];
    int r[kDegPer];
#pragma unroll
    for (int q = 0; q < kDegPer; ++q) {
      const int64_t i = t0 + (int64_t)q * blockDim.x + threadIdx.x;
      v[q] = i < nz_n ? nz_row[i] : -1;
      d[q] = v[q] >= 0 ? (int32_t)(off[v[q] + 1] - off[v[q]]) : 0;
      r[q] = 0;
      if (v[q] < 0) continue;
      if (d[q] < kDegSmall) r[q] = atomicAdd(&bin[d[q]], 1);
      else dsort[atomicAdd(cur + d[q], 1ull)] = v[q];
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kDegSmall; b += blockDim.x)
      if (bin[b]) base[b] = atomicAdd(cur + b, (unsigned long long)bin[b]);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kDegPer; ++q)
      if (v[q] >= 0 && d[q] < kDegSmall) dsort[base[d[q]] + r[q]] = v[q];
    __syncthreads();
  }
}

}  // namespace

size_t degree_order_workspace_bytes(int32_t max_deg) {
  const size_t len = (size_t)max_deg + 2;
  return align_up(8 * len) + align_up(8 * ((len + kDegThreads - 1) / kDegThreads));
}

cudaError_t launch_degree_order(int64_t nz_n, const int32_t* nz_row, const int64_t* off, int32_t max_deg,
                                int32_t* dsort, int64_t* dge, void* ws, int num_sms, cudaStream_t stream) {
  const int64_t len = (int64_t)max_deg + 2;             // degrees 0 .. max_deg + 1
  const int64_t ntiles = (len + kDegThreads - 1) / kDegThreads;
  unsigned long long* cnt = static_cast<unsigned long long*>(ws);
  int64_t* tile_tot = reinterpret_cast<int64_t*>(static_cast<char*>(ws) + align_up(8 * (size_t)len));
  cudaError_t e = cudaMemsetAsync(cnt, 0, 8 * (size_t)len, stream);
  if (e != cudaSuccess) return e;
  const int g = num_sms > 0 ? num_sms : 1;
  if (nz_n > 0) k_deg_hist<<<g, kDegThreads, 0, stream>>>(nz_n, nz_row, off, cnt);
  k_deg_suffix_tiles<<<(unsigned)ntiles, kDegThreads, 0, stream>>>(len, cnt, dge, tile_tot);
  k_deg_suffix_totals<<<1, kDegThreads, 0, stream>>>(ntiles, tile_tot);
  k_deg_suffix_add<<<(unsigned)ntiles, kDegThreads, 0, stream>>>(len, cnt, dge, tile_tot);
  if (nz_n > 0) k_deg_scatter<<<g, kDegThreads, 0, stream>>>(nz_n, nz_row, off, cnt, dsort);
  return cudaGetLastError();
}

bool intra_wants_signatures(int64_t n, const UpperRows& up) { return n > kSigMin && !short_rows(up); }

size_t objective_workspace_bytes(int64_t n) {
  const size_t nn = (size_t)(n > 0 ? n : 1);
  return align_up(4 * nn) + (n > kSigMin ? align_up(4 * ((nn >> 3) + 1)) : 0);
}

cudaError_t launch_intra(const int32_t* col, const UpperRows& up, const FullRows& all, const uint32_t* id,
                         const uint32_t* sig, uint32_t lo, uint32_t hi, unsigned long long* out, int num_sms,
                         cudaStream_t stream) {
  if (up.units <= 0) return cudaGetLastError();
  if (short_rows(up)) {
    k_intra_short<<<num_sms * kObjBlocks, kObjThreads, 0, stream>>>(all, col, lo, hi, id, out);
    return cudaGetLastError();
  }
  const int64_t per = kObjThreads / 32 * kUnitB;
  const int64_t want = (up.units + per - 1) / per;
  const int g = (int)(want < (int64_t)num_sms * kObjBlocks ? want : (int64_t)num_sms * kObjBlocks);
  if (sig) k_intra<true><<<g, kObjThreads, 0, stream>>>(up, col, lo, hi, id, sig, out);
  else k_intra<false><<<g, kObjThreads, 0, stream>>>(up, col, lo, hi, id, nullptr, out);
  return cudaGetLastError();
}

cudaError_t launch_disagreements(int64_t n, const int32_t* col, const UpperRows& up, const FullRows& all,
                                 const int32_t* labels, void* ws, unsigned long long* out, int num_sms,
                                 cudaStream_t stream) {
  int32_t* size = static_cast<int32_t*>(ws);
  cudaError_t e = cudaMemsetAsync(size, 0, 4 * (size_t)(n > 0 ? n : 1), stream);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(out, 0, 3 * sizeof(unsigned long long), stream);
  if (e != cudaSuccess) return e;
  if (n <= 0) return cudaSuccess;
  const int64_t want = (n + 255) / 256;
  const int g = (int)(want < (int64_t)num_sms * 8 ? want : (int64_t)num_sms * 8);
  k_sizes_pairs<<<g, 256, 0, stream>>>(n, labels, size, out);
  const uint32_t* id = reinterpret_cast<const uint32_t*>(labels);
  uint32_t* sig = nullptr;
  if (intra_wants_signatures(n, up)) {
    sig = reinterpret_cast<uint32_t*>(static_cast<char*>(ws) + align_up(4 * (size_t)n));
    k_signatures<<<g, 256, 0, stream>>>(n, id, sig);
  }
  return launch_intra(col, up, all, id, sig, 0u, 0xFFFFFFFFu, out, num_sms, stream);
}

size_t validate_workspace_bytes() { return align_up(8 * sizeof(unsigned long long)) + align_up(2 * sizeof(int)); }

cudaError_t launch_validate_offsets(int64_t n, int64_t nnz, const int64_t* off, void* ws, int num_sms,
                                    cudaStream_t stream) {
  int* flags = reinterpret_cast<int*>(static_cast<char*>(ws) + align_up(8 * sizeof(unsigned long long)));
  cudaError_t e = cudaMemsetAsync(ws, 0, validate_workspace_bytes(), stream);
  if (e != cudaSuccess) return e;
  if (n > 0) k_validate_offsets<<<num_sms * 8, 256, 0, stream>>>(n, nnz, off, flags);
  k_validate_finish<<<1, 1, 0, stream>>>(n, off, nnz, flags, nullptr);
  return cudaGetLastError();
}

cudaError_t launch_validate_edges(int64_t n, int64_t e0, int64_t e1, bool last, const int32_t* nz_row,
                                  const int64_t* nz_pos, int64_t nz_n, const int32_t* col, int64_t* up_at, void* ws,
                                  int num_sms, cudaStream_t stream) {
  unsigned long long* sums = static_cast<unsigned long long*>(ws);
  int* flags = reinterpret_cast<int*>(static_cast<char*>(ws) + align_up(8 * sizeof(unsigned long long)));
  if (e1 > e0)
    k_validate_edges<<<num_sms * 2, kValThreads, 0, stream>>>(n, e0, e1, nz_n, nz_row, nz_pos, col, up_at, flags,
                                                              sums);
  if (last) k_validate_symmetry<<<1, 1, 0, stream>>>(flags, sums);
  return cudaGetLastError();
}

cudaError_t launch_validate_reverse(int64_t nnz, const int64_t* off, const int32_t* nz_row, const int64_t* nz_pos,
                                    int64_t nz_n, const int32_t* col, void* ws, int num_sms, cudaStream_t stream) {
  int* flags = reinterpret_cast<int*>(static_cast<char*>(ws) + align_up(8 * sizeof(unsigned long long)));
  if (nnz > 0) k_validate_reverse<<<num_sms * 2, kValThreads, 0, stream>>>(nz_n, nz_row, nz_pos, nnz, off, col, flags);
  return cudaGetLastError();
}

cudaError_t launch_offsets_i32_to_i64(int64_t n, const int32_t* in, int64_t* out, cudaStream_t stream) {
  const int64_t want = (n + 256) / 256;
  k_off32_to_64<<<(int)(want < 4096 ? want : 4096), 256, 0, stream>>>(n, in, out);
  return cudaGetLastError();
}

size_t nonempty_workspace_bytes(int64_t n) {
  const int64_t ntiles = (n + kNzTile - 1) / kNzTile;
  return 2 * align_up(8 * (size_t)(ntiles + 1)) + align_up(8);
}

// nz_row/nz_pos get the non-empty rows and their first CSR positions; the
// count is written to *count_dev (device int64).
cudaError_t launch_nonempty_rows(int64_t n, const int64_t* off, int32_t* nz_row, int64_t* nz_pos, int64_t* up_at,
                                 void* ws, int64_t* count_dev, int num_sms, cudaStream_t stream) {
  if (n <= 0) return cudaMemsetAsync(count_dev, 0, sizeof(int64_t), stream);
  const int64_t ntiles = (n + kNzTile - 1) / kNzTile;
  int64_t* tile = static_cast<int64_t*>(ws);
  const int g = (int)(ntiles < (int64_t)num_sms * 4 ? ntiles : (int64_t)num_sms * 4);
  k_nz_count<<<g, kNzTile, 0, stream>>>(n, off, tile);
  k_nz_scan<<<1, 1024, 0, stream>>>(ntiles, tile, 0, count_dev);
  k_nz_write<<<g, kNzTile, 0, stream>>>(n, off, tile, nz_row, nz_pos, up_at);
  return cudaGetLastError();
}

cudaError_t launch_upper_rows(int64_t nz_n, int64_t nnz, const int32_t* nz_row, const int64_t* nz_pos,
                              const int64_t* up_at, int32_t* v, int64_t* row, int32_t* len, uint32_t* pos,
                              uint32_t* epos, void* ws, unsigned long long* count_dev, int num_sms,
                              cudaStream_t stream) {
  if (nz_n <= 0) return cudaMemsetAsync(count_dev, 0, 2 * sizeof(unsigned long long), stream);
  const int64_t ntiles = (nz_n + kNzTile - 1) / kNzTile;
  int64_t* tile = static_cast<int64_t*>(ws);
  const int64_t stride = (int64_t)(align_up(8 * (size_t)(ntiles + 1)) / 8);
  int64_t* tile_len = tile + stride;
  const int g = (int)(ntiles < (int64_t)num_sms * 4 ? ntiles : (int64_t)num_sms * 4);
  k_up_count<<<g, kNzTile, 0, stream>>>(nz_n, nnz, nz_pos, up_at, tile, tile_len);
  k_nz_scan<<<2, 1024, 0, stream>>>(ntiles, tile, stride, reinterpret_cast<int64_t*>(count_dev));
  k_up_write<<<g, kNzTile, 0, stream>>>(nz_n, nnz, nz_row, nz_pos, up_at, tile, tile_len, v, row, len, pos, epos);
  return cudaGetLastError();
}

}  // namespace ccg
