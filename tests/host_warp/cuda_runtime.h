// Host stand-in for the CUDA names that csrc/common.cuh uses, so that its warp
// functions run on the CPU: a warp is 32 threads that meet at every warp
// operation.  Read-only loads (__ldg) go to hooks of the including program,
// which sees the address of every access before it is made.
#pragma once
#include <stdint.h>

#include <algorithm>
#include <barrier>
#include <cmath>
#include <cstring>
#include <thread>
#include <vector>

#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __launch_bounds__(...)
#define __shared__ static
#define __align__(n) alignas(n)
using std::max;
using std::min;

struct WarpDim {
  int x, y, z;
};
inline thread_local WarpDim threadIdx{0, 0, 0};
inline WarpDim blockIdx{0, 0, 0}, blockDim{32, 1, 1}, gridDim{1, 1, 1};

inline std::barrier<> warp_meet(32);
inline void __syncwarp() { warp_meet.arrive_and_wait(); }
inline void __syncthreads() { __syncwarp(); }
inline void __threadfence() {}
inline void __nanosleep(unsigned) {}
template <typename T>
inline T warp_from(T v, int lane) {
  static T all[32];
  all[threadIdx.x] = v;
  __syncwarp();
  const T r = all[lane & 31];
  __syncwarp();
  return r;
}
template <typename T>
inline T __shfl_sync(unsigned, T v, int lane) { return warp_from(v, lane); }
template <typename T>
inline T __shfl_xor_sync(unsigned, T v, int w) { return warp_from(v, threadIdx.x ^ w); }
inline unsigned __ballot_sync(unsigned, bool p) {
  unsigned r = 0;
  for (int l = 0; l < 32; ++l) r |= (unsigned)warp_from<int>(p, l) << l;
  return r;
}
inline unsigned __reduce_max_sync(unsigned, unsigned v) {
  unsigned r = 0;
  for (int l = 0; l < 32; ++l) r = max(r, warp_from(v, l));
  return r;
}
inline int __popc(unsigned v) { return __builtin_popcount(v); }
inline int __ffs(unsigned v) { return __builtin_ffs((int)v); }

template <typename To, typename From>
inline To warp_bits(From v) {
  static_assert(sizeof(To) == sizeof(From), "same size");
  To r;
  memcpy(&r, &v, sizeof(r));
  return r;
}
inline int __double2hiint(double v) { return (int)(warp_bits<uint64_t>(v) >> 32); }
inline int __double2loint(double v) { return (int)warp_bits<uint64_t>(v); }
inline double __hiloint2double(int h, int l) { return warp_bits<double>((uint64_t)(unsigned)h << 32 | (unsigned)l); }
inline unsigned __float_as_uint(float v) { return warp_bits<unsigned>(v); }
inline double __dmul_rn(double a, double b) { return a * b; }
inline double rsqrt(double v) { return (double)(1.0L / sqrtl((long double)v)); }
inline int rsqrtf_off = 0;  // CUDA's rsqrtf is within 2 units in the last place: the error to take, in units
inline float rsqrtf(float v) {
  float r = (float)(1.0 / std::sqrt((double)v));
  for (int k = 0; k < std::abs(rsqrtf_off); ++k) r = std::nextafter(r, rsqrtf_off < 0 ? 0.0f : 4e38f);
  return r;
}
inline size_t __cvta_generic_to_shared(const void *p) { return (size_t)p; }
inline unsigned atomicAdd(unsigned *p, unsigned v) { return __atomic_fetch_add(p, v, __ATOMIC_SEQ_CST); }
inline unsigned atomicExch(unsigned *p, unsigned v) { return __atomic_exchange_n(p, v, __ATOMIC_SEQ_CST); }
template <typename T>
inline T __ldcg(const T *p) { return *p; }

int load_hook(const int *p);
double load_hook(const double *p);
float load_hook(const float *p);
template <typename T>
inline T __ldg(const T *p) { return load_hook(p); }

// Runs f() as the 32 lanes of one warp.
template <typename F>
inline void run_warp(F f) {
  std::vector<std::thread> lanes;
  for (int l = 0; l < 32; ++l)
    lanes.emplace_back([&f, l] {
      threadIdx.x = l;
      f();
    });
  for (auto &t : lanes) t.join();
}
