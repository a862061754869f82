// Host stand-ins of the CUDA declarations and builtins that the device headers
// (csrc/mhd_int53.cuh, mhd_df.cuh, mhd_device.cuh, mhd_adjoint.cuh) use, so that
// their arithmetic compiles with g++ and runs on the CPU, one lane at a time.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>

using std::fabs;
using std::fmax;
using std::fmin;
using std::sqrt;

#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __noinline__
#define __align__(n) alignas(n)
#define __launch_bounds__(...)

struct CUstream_st;
typedef CUstream_st* cudaStream_t;
struct float2 {
  float x, y;
};

template <class A, class B> inline A word_cast(B b) {
  static_assert(sizeof(A) == sizeof(B), "");
  A a;
  memcpy(&a, &b, sizeof a);
  return a;
}
inline long long __double_as_longlong(double x) { return word_cast<long long>(x); }
inline double __longlong_as_double(long long x) { return word_cast<double>(x); }
inline int __double2hiint(double x) { return (int)(word_cast<uint64_t>(x) >> 32); }
inline int __double2loint(double x) { return (int)word_cast<uint64_t>(x); }
inline double __hiloint2double(int h, int l) { return word_cast<double>(((uint64_t)(uint32_t)h << 32) | (uint32_t)l); }
inline float __uint_as_float(unsigned u) { return word_cast<float>(u); }
inline unsigned __float_as_uint(float f) { return word_cast<unsigned>(f); }
inline int __float_as_int(float f) { return word_cast<int>(f); }
inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
  return (unsigned)(((((uint64_t)hi << 32) | lo) << s) >> 32);
}
inline unsigned __funnelshift_r(unsigned lo, unsigned hi, unsigned s) {
  return (unsigned)((((uint64_t)hi << 32) | lo) >> s);
}
inline int __any_sync(unsigned, int p) { return p != 0; }
inline unsigned __activemask() { return 1; }

// (volatile: never contracted into a multiply-add by the host compiler)
inline float __fadd_rn(float a, float b) {
  volatile float r = a + b;
  return r;
}
inline float __fsub_rn(float a, float b) {
  volatile float r = a - b;
  return r;
}
inline float __fmul_rn(float a, float b) {
  volatile float r = a * b;
  return r;
}
inline float __frcp_rn(float x) { return 1.0f / x; }
inline float rsqrtf(float x) { return (float)(1.0 / std::sqrt((double)x)); }
inline double __drcp_rn(double x) { return 1.0 / x; }
inline double __dsqrt_rn(double x) { return std::sqrt(x); }
inline double rsqrt(double x) { return (double)(1.0L / sqrtl((long double)x)); }
