// A block's threads on the CPU, for ThreadSanitizer: fibers that run one after
// the other between collectives.  Votes and shuffles make the lanes
// of their mask meet and exchange values, but order no memory, as the CUDA
// programming model has it; __syncwarp also orders memory among the lanes of
// its mask, __syncthreads among the threads of the block.  What one lane writes
// and another reads or writes without either in between is then a data race
// that ThreadSanitizer reports, whatever order the lanes happen to run in.
#pragma once
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <functional>

#include <cuda_runtime.h>

#undef __device__
#undef __host__
#undef __forceinline__
#undef __noinline__
#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
#undef __global__
#undef __shared__
#undef __launch_bounds__
#define __global__
#define __shared__ static
#define __launch_bounds__(...)

namespace warp {
struct Index {
  int x;
};
Index thread_idx();
inline int lane() { return thread_idx().x & 31; }
// val of every lane of the warp's mask, at the call site `line` of all of them
void meet(unsigned mask, uint64_t val, uint64_t out[32], int line, bool orders_memory);
void block_barrier(int line);
// runs f(thread) on a block of n threads, from thread 0 up or from the last one
// down; false if they never meet at some collective
bool run(const std::function<void(int)>& f, int n, bool downwards);

template <class T>
T shfl(unsigned mask, T v, int src, int line) {
  uint64_t u = 0, out[32];
  std::memcpy(&u, &v, sizeof v);
  meet(mask, u, out, line, false);
  T r;
  std::memcpy(&r, &out[src & 31], sizeof r);
  return r;
}
template <class T>
T shfl_in(int line, unsigned mask, T v, int src, int width = 32) {
  return shfl(mask, v, width == 32 ? src : ((lane() & ~(width - 1)) | src), line);
}
template <class T>
T shfl_up(int line, unsigned mask, T v, int o, int width = 32) {
  const int l = lane();
  return shfl(mask, v, (l & (width - 1)) >= o ? l - o : l, line);
}
template <class T>
T shfl_down(int line, unsigned mask, T v, int o) {
  const int l = lane();
  return shfl(mask, v, l + o < 32 ? l + o : l, line);
}
template <class T, class Op>
T reduce(unsigned mask, T v, int line, Op op) {
  uint64_t u = 0, out[32];
  std::memcpy(&u, &v, sizeof v);
  meet(mask, u, out, line, false);
  bool any = false;
  T r{};
  for (int i = 0; i < 32; ++i) {
    if (!(mask >> i & 1)) continue;
    T w;
    std::memcpy(&w, &out[i], sizeof w);
    r = any ? op(r, w) : w;
    any = true;
  }
  return r;
}
inline unsigned ballot(unsigned mask, bool p, int line) {
  uint64_t out[32];
  meet(mask, p, out, line, false);
  unsigned r = 0;
  for (int i = 0; i < 32; ++i) r |= (mask >> i & 1) && out[i] ? 1u << i : 0u;
  return r;
}
inline void sync(int line, unsigned mask = 0xffffffffu) {
  uint64_t out[32];
  meet(mask, 0, out, line, true);
}
template <class To, class From>
To bits(From v) {
  To r;
  std::memcpy(&r, &v, sizeof r);
  return r;
}
}  // namespace warp

#define threadIdx warp::thread_idx()
#define __shfl_sync(...) warp::shfl_in(__LINE__, __VA_ARGS__)
#define __shfl_up_sync(...) warp::shfl_up(__LINE__, __VA_ARGS__)
#define __shfl_down_sync(...) warp::shfl_down(__LINE__, __VA_ARGS__)
#define __shfl_xor_sync(m, v, o) warp::shfl(m, v, warp::lane() ^ (o), __LINE__)
#define __reduce_min_sync(m, v) warp::reduce(m, v, __LINE__, [](auto a, auto b) { return b < a ? b : a; })
#define __reduce_max_sync(m, v) warp::reduce(m, v, __LINE__, [](auto a, auto b) { return a < b ? b : a; })
#define __reduce_add_sync(m, v) warp::reduce(m, v, __LINE__, [](auto a, auto b) { return a + b; })
#define __ballot_sync(m, p) warp::ballot(m, p, __LINE__)
#define __any_sync(m, p) (warp::ballot(m, p, __LINE__) != 0u)
#define __all_sync(m, p) (warp::ballot(m, p, __LINE__) == (m))
#define __syncwarp(...) warp::sync(__LINE__ __VA_OPT__(, ) __VA_ARGS__)
#define __syncthreads() warp::block_barrier(__LINE__)

using std::max;
using std::min;
inline int __popc(unsigned v) { return __builtin_popcount(v); }
inline int __ffs(int v) { return __builtin_ffs(v); }
inline int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
inline uint64_t __umul64hi(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
inline long long __double_as_longlong(double v) { return warp::bits<long long>(v); }
inline double __longlong_as_double(long long v) { return warp::bits<double>(v); }
inline int __double2hiint(double v) { return (int)(warp::bits<long long>(v) >> 32); }
inline int __float_as_int(float v) { return warp::bits<int>(v); }
inline float __int_as_float(int v) { return warp::bits<float>(v); }
inline unsigned __float_as_uint(float v) { return warp::bits<unsigned>(v); }
inline float __uint_as_float(unsigned v) { return warp::bits<float>(v); }
inline float __ull2float_rz(unsigned long long v) {
  const float f = (float)v;
  return (double)f > (double)v ? std::nextafter(f, 0.0f) : f;
}
template <class T>
T __ldcg(const T* p) { return *p; }
inline int atomicAdd(int* p, int v) { return __atomic_fetch_add(p, v, __ATOMIC_RELAXED); }
inline int atomicOr(int* p, int v) { return __atomic_fetch_or(p, v, __ATOMIC_RELAXED); }
inline int atomicCAS(int* p, int c, int v) {
  __atomic_compare_exchange_n(p, &c, v, false, __ATOMIC_RELAXED, __ATOMIC_RELAXED);
  return c;
}
