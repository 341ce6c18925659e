// One warp on the host: 32 threads that meet at every collective, so that the
// warp-wide index arithmetic of the device headers runs on a CPU.  Reads of the
// column array do not touch memory: they yield the position that was asked for.
#pragma once

#include <barrier>
#include <cstdint>
#include <cstring>

#define __device__
#define __host__
#define __forceinline__ inline

struct Index {
  unsigned x = 0, y = 0, z = 0;
};
inline thread_local Index threadIdx;
inline Index blockIdx, blockDim, gridDim;

namespace host_warp {
inline std::barrier<> meet(32);
inline uint64_t slot[32];
template <class T>
void put(T v) {
  static_assert(sizeof(T) <= 8);
  uint64_t w = 0;
  std::memcpy(&w, &v, sizeof(T));
  slot[threadIdx.x] = w;
  meet.arrive_and_wait();
}
template <class T>
T get(unsigned lane) {
  T v;
  std::memcpy(&v, &slot[lane & 31], sizeof(T));
  return v;
}
inline const int32_t* const columns = reinterpret_cast<const int32_t*>(uintptr_t(1) << 44);
}  // namespace host_warp

template <class T>
T __shfl_sync(unsigned, T v, int lane) {
  host_warp::put(v);
  const T r = host_warp::get<T>((unsigned)lane);
  host_warp::meet.arrive_and_wait();
  return r;
}
template <class T>
T __shfl_up_sync(unsigned m, T v, int o) {
  return __shfl_sync(m, v, (int)threadIdx.x >= o ? (int)threadIdx.x - o : (int)threadIdx.x);
}
template <class T>
T __shfl_xor_sync(unsigned m, T v, int o) {
  return __shfl_sync(m, v, (int)threadIdx.x ^ o);
}
inline unsigned __ballot_sync(unsigned, int p) {
  host_warp::put<int>(p != 0);
  unsigned r = 0;
  for (unsigned i = 0; i < 32; ++i) r |= (unsigned)host_warp::get<int>(i) << i;
  host_warp::meet.arrive_and_wait();
  return r;
}
inline int __any_sync(unsigned m, int p) { return __ballot_sync(m, p) != 0; }
inline int __all_sync(unsigned m, int p) { return __ballot_sync(m, p) == 0xFFFFFFFFu; }
inline int __reduce_max_sync(unsigned m, int v) {
  for (int o = 16; o > 0; o >>= 1) {
    const int y = __shfl_xor_sync(m, v, o);
    v = y > v ? y : v;
  }
  return v;
}
inline int __reduce_add_sync(unsigned m, int v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(m, v, o);
  return v;
}
inline void __syncwarp() { host_warp::meet.arrive_and_wait(); }
inline void __syncthreads() { host_warp::meet.arrive_and_wait(); }
inline int __popc(unsigned x) { return __builtin_popcount(x); }
inline int __ffs(unsigned x) { return __builtin_ffs((int)x); }
inline int32_t __ldg(const int32_t* p) { return (int32_t)((p - host_warp::columns) & 0x7FFFFFFF); }
template <class T>
T __ldcg(const T* p) {
  return *p;
}
inline int atomicCAS(int*, int, int) { return 0; }
inline unsigned long long atomicAdd(unsigned long long* p, unsigned long long v) {
  const unsigned long long old = *p;
  *p += v;
  return old;
}

// statements in the GPU's own assembly have no counterpart here
#define asm if (0) asm
