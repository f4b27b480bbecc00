// Host stand-in for the CUDA headers: enough to compile the sweep kernels'
// device code with a host compiler and run a CTA as one thread per CUDA
// thread (barriers for __syncthreads, a per-warp exchange for shuffles).
#pragma once
#include <atomic>
#include <barrier>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <memory>
#include <mutex>
#include <vector>

#define __device__
#define __host__
#define __global__
#define __constant__
#define __shared__
#define __forceinline__ inline
#define __noinline__
#define __restrict__
#define __align__(n)
#define __launch_bounds__(...)

struct float2 { float x, y; };
struct float4 { float x, y, z, w; };
struct int2 { int x, y; };
struct dim3 { unsigned x = 1, y = 1, z = 1; };
inline float2 make_float2(float a, float b) { return {a, b}; }
inline float4 make_float4(float a, float b, float c, float d) { return {a, b, c, d}; }
inline float2 __ffma2_rn(float2 a, float2 b, float2 c) { return {fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)}; }
inline float2 __fmul2_rn(float2 a, float2 b) { return {a.x * b.x, a.y * b.y}; }
inline uint32_t __float_as_uint(float f) { uint32_t u; memcpy(&u, &f, 4); return u; }
inline float __uint_as_float(uint32_t u) { float f; memcpy(&f, &u, 4); return f; }
inline int __popc(uint32_t v) { return __builtin_popcount(v); }
inline int64_t min(int64_t a, int64_t b) { return a < b ? a : b; }
using std::isfinite;

struct Cta {
  unsigned threads;
  std::barrier<> all;
  std::vector<std::unique_ptr<std::barrier<>>> warp;
  std::vector<double> slot;
  explicit Cta(unsigned n) : threads(n), all(n), slot(n) {
    for (unsigned w = 0; w < n / 32; w++) warp.emplace_back(new std::barrier<>(32));
  }
};
inline thread_local dim3 threadIdx, blockIdx, blockDim, gridDim;
inline thread_local Cta* cta;
inline std::mutex atomic_mu;

inline void __syncthreads() { cta->all.arrive_and_wait(); }
template <class T>
T __shfl_xor_sync(unsigned, T v, int o) {
  const unsigned t = threadIdx.x;
  std::barrier<>& b = *cta->warp[t / 32];
  cta->slot[t] = (double)v;
  b.arrive_and_wait();
  const T r = (T)cta->slot[t ^ (unsigned)o];
  b.arrive_and_wait();
  return r;
}
inline uint32_t __ballot_sync(unsigned, bool v) {
  uint32_t r = v ? 1u << (threadIdx.x & 31) : 0u;
  for (int o = 16; o > 0; o >>= 1) r |= __shfl_xor_sync(0u, r, o);
  return r;
}
template <class T, class U>
T atomicAdd(T* p, U v) {
  std::lock_guard<std::mutex> l(atomic_mu);
  const T old = *p;
  *p = (T)(old + v);
  return old;
}
inline int atomicOr(int* p, int v) {
  std::lock_guard<std::mutex> l(atomic_mu);
  const int old = *p;
  *p |= v;
  return old;
}
