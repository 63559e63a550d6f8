// What csrc/qcd.cuh and the headers it includes take from CUDA, for a host
// compiler: the device functions then run on the CPU, one thread at a time.
#pragma once
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cstring>
#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
#define __align__(x)
#define __shared__
struct float4 {
  float x, y, z, w;
};
struct double2 {
  double x, y;
};
struct Dim {
  unsigned x, y, z;
};
static Dim threadIdx, blockDim;
template <class T, class U>
inline T bits_as(U x) {
  T y;
  static_assert(sizeof x == sizeof y, "same size");
  std::memcpy(&y, &x, sizeof y);
  return y;
}
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fdiv_rn(float a, float b) { return a / b; }
inline float __fdividef(float a, float b) { return a / b; }
inline float __fsqrt_rn(float a) { return std::sqrt(a); }
inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
inline double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
inline double rsqrt(double x) { return 1.0 / std::sqrt(x); }
inline float rsqrtf(float x) { return 1.0f / std::sqrt(x); }
inline unsigned __float_as_uint(float x) { return bits_as<unsigned>(x); }
inline float __uint_as_float(unsigned x) { return bits_as<float>(x); }
inline float __int_as_float(int x) { return bits_as<float>(x); }
inline long long __double_as_longlong(double x) { return bits_as<long long>(x); }
inline int __double2hiint(double x) { return (int)(bits_as<long long>(x) >> 32); }
inline size_t __cvta_generic_to_shared(const void* p) { return reinterpret_cast<size_t>(p); }
