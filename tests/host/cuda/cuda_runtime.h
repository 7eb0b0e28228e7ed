// Host stand-in for the CUDA names that the device headers use: one block of one thread, so that the
// CTA-level transforms can be run and compared on the CPU.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#define __host__
#define __device__
#define __global__
#define __constant__
#define __shared__
#define __forceinline__ inline
#define __align__(n)
#define __launch_bounds__(...)
struct Idx3 {
  unsigned x, y, z;
};
static Idx3 threadIdx{0, 0, 0}, blockIdx{0, 0, 0}, blockDim{1, 1, 1}, gridDim{1, 1, 1};
struct float2 {
  float x, y;
};
struct double2 {
  double x, y;
};
using std::max;
using std::min;
inline float2 make_float2(float a, float b) { return {a, b}; }
inline double2 make_double2(double a, double b) { return {a, b}; }
inline float2 __fadd2_rn(float2 a, float2 b) { return {a.x + b.x, a.y + b.y}; }
inline float2 __ffma2_rn(float2 a, float2 b, float2 c) { return {std::fma(a.x, b.x, c.x), std::fma(a.y, b.y, c.y)}; }
template <typename T> T __ldg(const T* p) { return *p; }
template <typename T> T __ldcg(const T* p) { return *p; }
inline uint64_t bits_of(double v) {
  uint64_t u;
  std::memcpy(&u, &v, 8);
  return u;
}
inline int __double2hiint(double v) { return (int)(bits_of(v) >> 32); }
inline int __double2loint(double v) { return (int)bits_of(v); }
inline double __hiloint2double(int h, int l) {
  const uint64_t u = (uint64_t)(uint32_t)h << 32 | (uint32_t)l;
  double v;
  std::memcpy(&v, &u, 8);
  return v;
}
inline int __popc(unsigned v) { return __builtin_popcount(v); }
inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
inline float __double2float_ru(double v) {
  const float f = (float)v;
  return (double)f < v ? std::nextafterf(f, INFINITY) : f;
}
// (sums and products of two floats are exact, or rounded once below float's half unit, in double)
inline float __fadd_ru(float a, float b) { return __double2float_ru((double)a + b); }
inline float __fmul_ru(float a, float b) { return __double2float_ru((double)a * b); }
inline float __fmaf_ru(float a, float b, float c) { return __double2float_ru((double)a * b + c); }
inline float __int_as_float(int i) {
  float f;
  std::memcpy(&f, &i, 4);
  return f;
}
inline void __syncthreads() {}
inline void __threadfence() {}
inline void sincospi(double x, double* s, double* c) {
  *s = std::sin(M_PI * x);
  *c = std::cos(M_PI * x);
}
// the other lanes of the one-thread warp hold nothing: neutral for the sums and maxima of moduli
template <typename T> T __shfl_xor_sync(unsigned, T, int) { return T(0); }
inline int __reduce_max_sync(unsigned, int v) { return v; }
template <typename T> T atomicAdd(T* p, T v) {
  const T old = *p;
  *p += v;
  return old;
}
