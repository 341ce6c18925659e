// cc_perm.cu -- the random order pi of Alg. 1 / Alg. 2 on the device.
//
// pi lists the vertices by ascending (splitmix64(seed ^ v), v).  The keys are
// uniform 64-bit values, so a two-level sort suffices:
//   1. k_bucket_scatter puts the vertices into buckets by the top b key bits (b
//      chosen so that a bucket holds 2048-4096 vertices).  A bucket has a fixed
//      place for its expected number and twelve standard deviations more, so
//      nothing is counted beforehand; what does not fit goes to a spill list.
//      Above kOneLevelBits bits it runs twice, by the top kCoarseBits bits first.
//   2. k_bucket_starts: exclusive scan of the buckets' sizes.
//   3. k_bucket_sort sorts each bucket in shared memory by the full (key, v): a
//      counting sort on the next 12 key bits, then an insertion sort per
//      sub-bucket of about one element, and writes its slice of order[].
// Keys are recomputed from v wherever needed instead of being stored, so the
// only global traffic is 4 bytes per vertex scattered (twice, and read once, in
// two levels) and 4+4+4 bytes per vertex read and written by the bucket sort.
// Bound by the shared-memory atomics of the two sorts; 10K / 1M / 4.2M / 16.8M /
// 67M vertices take 20 / 35 / 87 / 290 / 1255 us (36 / 130 / 280 / 730 / 2430 when
// buckets of 512 were counted and filled by one global atomic per vertex each).
#include <cstdint>

#include "cc_device.cuh"
#include "cc_internal.h"

namespace ccg {
namespace {

constexpr int kMeanMax = 4096;         // expected vertices per bucket, at most
constexpr int kBucketCap = 4928;       // at least bucket_cap(4096)
constexpr int kScatterThreads = 512;
constexpr int kSortThreads = 512;
constexpr int kSpillCap = 1 << 16;     // vertices that found their bucket full
// Up to 2^12 buckets (16M vertices) one scatter; above, a chunk holds too few
// vertices per bucket for neighbouring writes (16M vertices in one level 0.29 ms,
// in two 0.34; 67M into 2^14 buckets at once 2.4, in two levels 1.26).
constexpr int kOneLevelBits = 12;
constexpr int kCoarseBits = 9;
constexpr int kChunk = 16384;          // vertices per block and scatter, at most
constexpr int kBitsMax = 19;           // buckets of 2^31 - 1 vertices (bucket_bits)

__device__ __forceinline__ uint32_t bucket_of(uint64_t key, int bits) {
  return bits == 0 ? 0u : (uint32_t)(key >> (64 - bits));
}

// Places of a bucket of `mean` expected vertices.
int64_t bucket_cap(int64_t mean) {
  int64_t root = 0;
  while (root * root < mean) ++root;
  return (mean + 12 * root + 63) & ~int64_t(31);
}

__device__ __forceinline__ void spill_one(int32_t v, uint32_t* spill) {
  const uint32_t q = atomicAdd(spill, 1u);
  if (q < (uint32_t)kSpillCap) spill[1 + q] = (uint32_t)v;
}

// A block's share of a scatter: the vertices source(0 .. len) go to the `nb`
// buckets from `first` on.  They are counted by bucket in shared memory and
// brought into bucket order there; one atomic takes the places of all of a
// bucket's vertices, and neighbouring threads write neighbouring places.  (One
// atomic per vertex, after as many to count the buckets, took 187 of the 280 us
// of 4.2M vertices: the counters of 8192 buckets lie in 256 lines.  Written
// straight to their places the vertices of a warp go to 32 pages of memory: 67M
// into 512 buckets 0.58 ms.)  spilled(v) gets the vertices that found no place.
struct ScatterSmem {
  uint32_t* next;                        // [nb] count, then next place in buf
  uint32_t* delta;                       // [nb] place in the bucket, less the one in buf
  int32_t* buf;                          // [chunk]
  __device__ ScatterSmem(uint32_t* raw, int nb)
      : next(raw), delta(raw + nb), buf(reinterpret_cast<int32_t*>(raw + 2 * nb)) {}
};
constexpr size_t scatter_smem(int nb, int64_t chunk) { return sizeof(uint32_t) * (2 * (size_t)nb + (size_t)chunk); }

template <class Source, class Spilled>
__device__ __forceinline__ void scatter_chunk(int len, uint64_t seed, int bits, uint32_t first, int nb, int64_t cap,
                                              const ScatterSmem& M, uint32_t* __restrict__ count,
                                              int32_t* __restrict__ tmp, const Source& source,
                                              const Spilled& spilled) {
  __shared__ int32_t scr[33];
  auto bucket = [&](int32_t v) { return bucket_of(perm_key(seed, (uint64_t)v), bits) - first; };
  for (int b = threadIdx.x; b < nb; b += kScatterThreads) M.next[b] = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < len; i += kScatterThreads) atomicAdd(&M.next[bucket(source(i))], 1u);
  __syncthreads();
  int32_t run = 0;
  for (int b0 = 0; b0 < nb; b0 += kScatterThreads) {
    const int b = b0 + threadIdx.x;
    const int32_t k = b < nb ? (int32_t)M.next[b] : 0;
    int32_t tot;
    const int32_t at = run + block_exclusive_sum<int32_t>(k, scr, &tot);
    run += tot;
    if (b >= nb) continue;
    M.next[b] = (uint32_t)at;
    if (k) M.delta[b] = atomicAdd(count + first + b, (uint32_t)k) - (uint32_t)at;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < len; i += kScatterThreads) {
    const int32_t v = source(i);
    M.buf[atomicAdd(&M.next[bucket(v)], 1u)] = v;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < len; i += kScatterThreads) {
    const int32_t v = M.buf[i];
    const uint32_t b = bucket(v), at = M.delta[b] + (uint32_t)i;
    if (at < (uint32_t)cap) tmp[(int64_t)(first + b) * cap + at] = v;
    else spilled(v);
  }
}

// All vertices, a chunk per block, into the 2^bits buckets of cap places.
__global__ void __launch_bounds__(kScatterThreads)
k_bucket_scatter(int64_t n, uint64_t seed, int bits, int cap, int64_t chunk, uint32_t* __restrict__ count,
                 int32_t* __restrict__ tmp, uint32_t* __restrict__ spill) {
  extern __shared__ uint32_t sm[];
  const int64_t c0 = (int64_t)blockIdx.x * chunk;
  scatter_chunk((int)(n - c0 < chunk ? n - c0 : chunk), seed, bits, 0u, 1 << bits, cap, ScatterSmem(sm, 1 << bits), count,
                tmp,
                [&](int i) { return (int32_t)(c0 + i); }, [&](int32_t v) { spill_one(v, spill); });
}

// The same into the coarse buckets; what finds no place there goes to its
// bucket of 2^bits directly.
__global__ void __launch_bounds__(kScatterThreads)
k_bucket_coarse(int64_t n, uint64_t seed, int64_t coarse_cap, int64_t chunk, uint32_t* __restrict__ coarse_count,
                int32_t* __restrict__ coarse, int bits, int cap, uint32_t* __restrict__ count,
                int32_t* __restrict__ tmp, uint32_t* __restrict__ spill) {
  extern __shared__ uint32_t sm[];
  const int64_t c0 = (int64_t)blockIdx.x * chunk;
  scatter_chunk((int)(n - c0 < chunk ? n - c0 : chunk), seed, kCoarseBits, 0u, 1 << kCoarseBits, coarse_cap,
                ScatterSmem(sm, 1 << kCoarseBits), coarse_count, coarse, [&](int i) { return (int32_t)(c0 + i); }, [&](int32_t v) {
                  const uint32_t b = bucket_of(perm_key(seed, (uint64_t)v), bits), at = atomicAdd(count + b, 1u);
                  if (at < (uint32_t)cap) tmp[(int64_t)b * cap + at] = v;
                  else spill_one(v, spill);
                });
}

// Chunk blockIdx.x of coarse bucket blockIdx.y into its part of the 2^bits buckets.
__global__ void __launch_bounds__(kScatterThreads)
k_bucket_fine(uint64_t seed, int64_t coarse_cap, const uint32_t* __restrict__ coarse_count,
              const int32_t* __restrict__ coarse, int bits, int cap, uint32_t* __restrict__ count,
              int32_t* __restrict__ tmp, uint32_t* __restrict__ spill) {
  extern __shared__ uint32_t sm[];
  const int64_t have = coarse_count[blockIdx.y], size = have < coarse_cap ? have : coarse_cap;
  const int64_t c0 = (int64_t)blockIdx.x * kChunk;
  if (c0 >= size) return;
  const int32_t* const from = coarse + (int64_t)blockIdx.y * coarse_cap + c0;
  const int nb = 1 << (bits - kCoarseBits);
  scatter_chunk((int)(size - c0 < kChunk ? size - c0 : kChunk), seed, bits, blockIdx.y * (uint32_t)nb, nb, cap,
                ScatterSmem(sm, nb), count, tmp, [&](int i) { return __ldg(from + i); }, [&](int32_t v) { spill_one(v, spill); });
}

// start[0..nb] = exclusive scan of the buckets' sizes.
__global__ void __launch_bounds__(1024) k_bucket_starts(int nb, const uint32_t* __restrict__ count,
                                                        int64_t* __restrict__ start) {
  __shared__ int64_t scr[33];
  const int per = (nb + 1023) / 1024, b0 = (int)threadIdx.x * per;
  int64_t sum = 0;
  for (int q = 0; q < per; ++q) sum += b0 + q < nb ? (int64_t)count[b0 + q] : 0;
  int64_t tot;
  int64_t run = block_exclusive_sum<int64_t>(sum, scr, &tot);
  for (int q = 0; q < per && b0 + q < nb; ++q) {
    start[b0 + q] = run;
    run += (int64_t)count[b0 + q];
  }
  if (threadIdx.x == 0) start[nb] = tot;
}

__device__ __forceinline__ bool kv_less(uint64_t ka, int32_t va, uint64_t kb, int32_t vb) {
  return ka < kb || (ka == kb && va < vb);
}

// One block per bucket (grid-stride).  Inside a bucket the keys share their
// top `bits` bits and the next kSubBits bits are still uniform, so a counting
// sort on those bits spreads the bucket over kSub sub-buckets of about one
// element each; one thread then finishes each sub-bucket with an insertion
// sort on the 32 key bits below, which stand beside the vertex in shared memory
// (equal ones: on the full key and the vertex).  The bucket is read twice, for
// the counts and for the places: a copy of it in shared memory would halve the
// blocks per SM.
constexpr int kSubBits = 12;
constexpr int kSub = 1 << kSubBits;
static_assert(kSub % kSortThreads == 0, "every thread scans the same number of sub-buckets");

struct SortSmem {
  uint32_t k[kBucketCap];
  int32_t v[kBucketCap];
  int32_t cnt[kSub];
  int32_t scr[33];
};

__device__ __forceinline__ bool sub_less(uint64_t seed, uint32_t ka, int32_t va, uint32_t kb, int32_t vb) {
  return ka != kb ? ka < kb : kv_less(perm_key(seed, (uint64_t)va), va, perm_key(seed, (uint64_t)vb), vb);
}

__global__ void __launch_bounds__(kSortThreads)
k_bucket_sort(uint64_t seed, int bits, int nb, int cap, const int64_t* __restrict__ start,
              const int32_t* __restrict__ tmp, int32_t* __restrict__ order, const uint32_t* __restrict__ spill,
              int* __restrict__ err) {
  extern __shared__ __align__(16) unsigned char raw[];
  SortSmem& S = *reinterpret_cast<SortSmem*>(raw);
  constexpr int kPer = kSub / kSortThreads;
  const uint32_t spilled = *spill;
  if (spilled > (uint32_t)kSpillCap) {
    // reported; the kernels that follow find vertices in order all the same
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicCAS(err, kOk, kErrInternal);
    const int64_t n = start[nb];
    for (int64_t i = blockIdx.x * (int64_t)kSortThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kSortThreads)
      order[i] = (int32_t)i;
    return;
  }
  for (int b = blockIdx.x; b < nb; b += gridDim.x) {
    const int64_t s0 = start[b];
    const int len = (int)(start[b + 1] - s0);
    const int32_t* const in = tmp + (int64_t)b * cap;
    if (len > cap) {
      // a bucket with spilled vertices (next to impossible for a hash): each
      // one's position is the number of smaller ones, by counting
      auto member = [&](int i) -> int32_t { return i < cap ? in[i] : (int32_t)spill[1 + i - cap]; };
      const int all = cap + (int)spilled;
      for (int i = threadIdx.x; i < all; i += kSortThreads) {
        const int32_t vi = member(i);
        const uint64_t ki = perm_key(seed, (uint64_t)vi);
        if ((int)bucket_of(ki, bits) != b) continue;
        int64_t r = 0;
        for (int j = 0; j < all; ++j) {
          const int32_t vj = member(j);
          const uint64_t kj = perm_key(seed, (uint64_t)vj);
          r += (int)bucket_of(kj, bits) == b && kv_less(kj, vj, ki, vi) ? 1 : 0;
        }
        order[s0 + r] = vi;
      }
      continue;
    }
    auto sub_of = [&](uint64_t key) { return (int)((key << bits) >> (64 - kSubBits)); };
#pragma unroll
    for (int q = 0; q < kPer; ++q) S.cnt[threadIdx.x + q * kSortThreads] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < len; i += kSortThreads) atomicAdd(&S.cnt[sub_of(perm_key(seed, (uint64_t)in[i]))], 1);
    __syncthreads();
    // exclusive scan of the sub-bucket counts
    {
      int32_t c[kPer], sum = 0, tot;
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        c[q] = S.cnt[threadIdx.x * kPer + q];
        sum += c[q];
      }
      int32_t run = block_exclusive_sum<int32_t>(sum, S.scr, &tot);
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        S.cnt[threadIdx.x * kPer + q] = run;
        run += c[q];
      }
    }
    __syncthreads();
    // scatter into sub-buckets (arbitrary order inside a sub-bucket); the
    // counters end at the next sub-bucket's start
    for (int i = threadIdx.x; i < len; i += kSortThreads) {
      const int32_t v = in[i];
      const uint64_t key = perm_key(seed, (uint64_t)v);
      const int pos = atomicAdd(&S.cnt[sub_of(key)], 1);
      S.k[pos] = (uint32_t)((key << (bits + kSubBits)) >> 32);
      S.v[pos] = v;
    }
    __syncthreads();
    // sub-bucket q now spans [q == 0 ? 0 : cnt[q-1], cnt[q]): insertion sort
    for (int q = threadIdx.x; q < kSub; q += kSortThreads) {
      const int lo = q == 0 ? 0 : S.cnt[q - 1], hi = S.cnt[q];
      for (int i = lo + 1; i < hi; ++i) {
        const uint32_t k = S.k[i];
        const int32_t v = S.v[i];
        int j = i - 1;
        while (j >= lo && sub_less(seed, k, v, S.k[j], S.v[j])) {
          S.k[j + 1] = S.k[j];
          S.v[j + 1] = S.v[j];
          --j;
        }
        S.k[j + 1] = k;
        S.v[j + 1] = v;
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < len; i += kSortThreads) order[s0 + i] = S.v[i];
    __syncthreads();
  }
}

// Bucket sizes: 2048 to 4096 expected vertices, fewer (512 at least) while there
// are not two buckets per SM.
int bucket_bits(int64_t n) {
  int bits = 0;
  while ((n >> bits) > kMeanMax) ++bits;
  while ((1 << bits) < 304 && (n >> (bits + 1)) >= 512) ++bits;
  return bits;
}

// One launch, checked at once: a later success of cudaFuncSetAttribute clears
// the error of a refused launch.  The limit of a kernel's dynamic shared memory
// belongs to the kernel, not to the call, and other threads launch it for graphs
// of other sizes: every call sets the kernel's own largest need, `most`.
template <class... P, class... A>
cudaError_t launch(void (*kernel)(P...), dim3 grid, int threads, size_t smem, size_t most, cudaStream_t stream,
                   A... args) {
  if (most > 0) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (e != cudaSuccess) return e;
  }
  kernel<<<grid, threads, smem, stream>>>(args...);
  return cudaGetLastError();
}

}  // namespace

size_t perm_workspace_bytes(int64_t n) {
  const int bits = bucket_bits(n);
  const int64_t nb = int64_t(1) << bits;
  const int64_t nc = bits > kOneLevelBits ? int64_t(1) << kCoarseBits : 0;
  return align_up(sizeof(uint32_t) * (nc + nb + 1 + kSpillCap)) + align_up(sizeof(int64_t) * (nb + 1)) +
         align_up(sizeof(int32_t) * nb * bucket_cap((n >> bits) + 1)) +
         align_up(sizeof(int32_t) * nc * bucket_cap((n >> kCoarseBits) + 1));
}

// order[0..n) = pi for `seed`.  ws must hold perm_workspace_bytes(n).  A
// failed device-side check is reported through *err.
cudaError_t launch_permutation(int64_t n, uint64_t seed, int32_t* order, void* ws, int num_sms,
                               int* err, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const int bits = bucket_bits(n), nb = 1 << bits, cap = (int)bucket_cap((n >> bits) + 1);
  const int nc = bits > kOneLevelBits ? 1 << kCoarseBits : 0;
  char* p = static_cast<char*>(ws);
  uint32_t* coarse_count = reinterpret_cast<uint32_t*>(p);
  uint32_t* count = coarse_count + nc;
  uint32_t* spill = count + nb;                              // their number, then the vertices
  p += align_up(sizeof(uint32_t) * ((size_t)nc + nb + 1 + kSpillCap));
  int64_t* start = reinterpret_cast<int64_t*>(p);
  p += align_up(sizeof(int64_t) * ((size_t)nb + 1));
  int32_t* tmp = reinterpret_cast<int32_t*>(p);
  p += align_up(sizeof(int32_t) * (size_t)nb * cap);
  int32_t* coarse = reinterpret_cast<int32_t*>(p);
  cudaError_t e = cudaMemsetAsync(coarse_count, 0, sizeof(uint32_t) * ((size_t)nc + nb + 1), stream);
  if (e != cudaSuccess) return e;
  // chunks: two per SM at least
  const int64_t share = (n + (int64_t)num_sms * 2 - 1) / ((int64_t)num_sms * 2);
  const int64_t chunk = share < 2048 ? 2048 : (share < kChunk ? share : kChunk);
  const unsigned grid = (unsigned)((n + chunk - 1) / chunk);
  if (nc == 0) {
    e = launch(k_bucket_scatter, grid, kScatterThreads, scatter_smem(nb, chunk),
               scatter_smem(1 << kOneLevelBits, kChunk), stream, n, seed, bits, cap, chunk, count, tmp, spill);
    if (e != cudaSuccess) return e;
  } else {
    const int64_t coarse_cap = bucket_cap((n >> kCoarseBits) + 1);
    e = launch(k_bucket_coarse, grid, kScatterThreads, scatter_smem(nc, chunk), scatter_smem(1 << kCoarseBits, kChunk),
               stream, n, seed, coarse_cap, chunk, coarse_count, coarse, bits, cap, count, tmp, spill);
    if (e != cudaSuccess) return e;
    const dim3 fine((unsigned)((coarse_cap + kChunk - 1) / kChunk), (unsigned)nc);
    e = launch(k_bucket_fine, fine, kScatterThreads, scatter_smem(nb / nc, kChunk),
               scatter_smem(1 << (kBitsMax - kCoarseBits), kChunk), stream, seed, coarse_cap, coarse_count, coarse,
               bits, cap, count, tmp, spill);
    if (e != cudaSuccess) return e;
  }
  e = launch(k_bucket_starts, 1, 1024, 0, 0, stream, nb, count, start);
  if (e != cudaSuccess) return e;
  return launch(k_bucket_sort, nb < num_sms * 4 ? nb : num_sms * 4, kSortThreads, sizeof(SortSmem), sizeof(SortSmem),
                stream, seed, bits, nb, cap, start, tmp, order, spill, err);
}

}  // namespace ccg
