// mhd_int53.cuh -- reciprocal, square root, reciprocal square root and product
// of doubles on the integer and FP32 pipes.
//
// GB300 issues one FP64 warp instruction per SM every 16 clocks against four
// of any other kind per clock, so an FP64 instruction costs 64 issue slots
// and the FP64 step leaves over 90 % of the issue slots idle.  These
// functions use none: a float seed from the special-function unit (relative
// error below 2^-22, PTX rcp.approx / rsqrt.approx), one cubically convergent
// Newton-type step on 64-bit fixed-point significands (the truncated series
// 1/(1-e) = 1 + e + e^2, (1-e)^(-1/2) = 1 + e/2 + 3 e^2/8 with |e| < 2^-20.5,
// so the neglected term is below 2^-61), and for the reciprocal and the
// square root an exact integer remainder that settles the rounding: those two
// are correctly rounded, the same values as IEEE division and square root.
// The reciprocal square root is rounded from its 2^-60.5 approximation, within
// 0.51 ulp.  Plain integer C++, so host code can check it with any seed
// inside the error bound.
//
// Measured: the library's __drcp_rn, rsqrt and sqrt run at 0.35, 0.33 and 0.21
// per clock and SM (5.4, 5.7 and 9 times an FP64 multiply-add); with these
// functions the FP64 PLMC step at 256^3 went from 87.5 to 72.1 ms.
#pragma once

#include <stdint.h>
#include <string.h>

#include <cmath>

#if defined(__CUDACC__)
#define MHD_INT_HD __host__ __device__ __forceinline__
#else
#define MHD_INT_HD inline
#endif

namespace mhd {

MHD_INT_HD uint64_t mulhi_u64(uint64_t a, uint64_t b) {
#if defined(__CUDA_ARCH__)
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
MHD_INT_HD int32_t mulhi_s32(int32_t a, int32_t b) { return (int32_t)(((int64_t)a * b) >> 32); }
MHD_INT_HD uint32_t float_word(float x) {
#if defined(__CUDA_ARCH__)
  return __float_as_uint(x);
#else
  uint32_t u;
  memcpy(&u, &x, 4);
  return u;
#endif
}

// 24-bit significand of a seed clamped to [0.5, 1): the seed is R0 / 2^24
MHD_INT_HD uint32_t seed24(float seed) {
  const float r = fminf(fmaxf(seed, 0.5f), 0.99999994f);
  return (float_word(r) & 0x7fffffu) | 0x800000u;
}
// R0 (1 + d): R0 / 2^24 the seed, d / 2^62 the correction; scale 2^62
MHD_INT_HD uint64_t corrected(uint32_t R0, int64_t d) {
  const uint64_t lo = (uint64_t)R0 * (uint32_t)d;
  const int64_t hi = (int64_t)(int32_t)R0 * (int32_t)(d >> 32) + (int64_t)(lo >> 32);
  return ((uint64_t)R0 << 38) + (((uint64_t)hi << 8) | ((uint32_t)lo >> 24));
}

// 1 / m for m = M / 2^52 in [1, 2): the 53-bit significand q in [2^52, 2^53]
// of the correctly rounded value q / 2^53.  seed ~ 1/m.
MHD_INT_HD uint64_t rcp_sig(uint64_t M, float seed) {
  const uint32_t R0 = seed24(seed), R = R0 << 7;
  const uint64_t X = M << 11;  // m 2^63
  const uint64_t p = (uint64_t)(uint32_t)(X >> 32) * R + (((uint64_t)(uint32_t)X * R) >> 32);
  const int64_t e = (int64_t)((1ull << 62) - p);  // (1 - m r) 2^62
  const int32_t t = (int32_t)(e >> 12);
  const uint64_t y = corrected(R0, e + (mulhi_s32(t, t) >> 6));
  const uint64_t q = (y + 256) >> 9;
  const int64_t rem = (int64_t)(0 - M * q);  // 2^105 - M q, |rem| < M
  return q + (2 * rem > (int64_t)M) - (-2 * rem > (int64_t)M);
}

// 1 / sqrt(m) for m = X / 2^62 in [1, 4): scale 2^62, in [2^61, 2^62].
MHD_INT_HD uint64_t rsqrt_fix(uint64_t X, float seed) {
  const uint32_t R0 = seed24(seed);
  const uint64_t p = mulhi_u64(X, ((uint64_t)R0 * R0) << 16);
  const int64_t e = (int64_t)((1ull << 62) - p);  // (1 - m r^2) 2^62
  const int32_t t = (int32_t)(e >> 12);
  return corrected(R0, (e >> 1) + ((3 * mulhi_s32(t, t)) >> 9));
}
// nearest 53-bit significand q in [2^52, 2^53] of 1/sqrt(m) = q / 2^53
MHD_INT_HD uint64_t rsqrt_sig(uint64_t M, int odd, float seed) { return (rsqrt_fix(M << (10 + odd), seed) + 256) >> 9; }
// significand q in [2^52, 2^53] of the correctly rounded sqrt(m) = q / 2^52,
// m = M 2^odd / 2^52
MHD_INT_HD uint64_t sqrt_sig(uint64_t M, int odd, float seed) {
  const uint64_t X = M << (10 + odd);
  const uint64_t q = (mulhi_u64(X, rsqrt_fix(X, seed)) + 128) >> 8;
  const int64_t rem = (int64_t)((M << (52 + odd)) - q * q);  // m 2^104 - q^2 (mod 2^64: |rem| < 2^54)
  return q + (rem > (int64_t)q) - (rem <= -(int64_t)q);
}

// Product of two 53-bit significands a, b in [2^52, 2^53): the 53-bit
// significand q in [2^52, 2^53] of the product rounded to nearest even; big:
// the product of the two values in [1, 2) is 2 or more.
MHD_INT_HD uint64_t mul_sig(uint64_t a, uint64_t b, int& big) {
  const uint64_t A = a << 10, B = b << 11;  // A B in [2^125, 2^127)
  const uint32_t al = (uint32_t)A, ah = (uint32_t)(A >> 32), bl = (uint32_t)B, bh = (uint32_t)(B >> 32);
  const uint64_t p0 = (uint64_t)al * bl;
  const uint64_t p1 = (uint64_t)al * bh + (uint32_t)(p0 >> 32);
  const uint64_t p2 = (uint64_t)ah * bl + (uint32_t)p1;
  uint64_t hi = (uint64_t)ah * bh + (p1 >> 32) + (p2 >> 32);
  hi |= ((uint32_t)p2 | (uint32_t)p0) != 0;  // sticky
  big = (int)(hi >> 62);
  const int sh = 9 + big;
  return (hi + (((1ull << sh) >> 1) - 1 + ((hi >> sh) & 1))) >> sh;
}

// (MHD_HOST_CHECK: compiled for the host against stand-ins of the builtins)
#if defined(__CUDACC__) || defined(MHD_HOST_CHECK)

__device__ __forceinline__ float rcp_seed(float x) {
#if defined(MHD_HOST_CHECK)
  return 1.0f / x;
#else
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#endif
}
__device__ __forceinline__ float rsqrt_seed(float x) {
#if defined(MHD_HOST_CHECK)
  return 1.0f / std::sqrt(x);
#else
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#endif
}

__device__ __forceinline__ uint64_t sig53(int hi, int lo) {
  return ((uint64_t)(uint32_t)((hi & 0xfffff) | 0x100000) << 32) | (uint32_t)lo;
}
// top 23 fraction bits, for the float seed operand
__device__ __forceinline__ uint32_t frac23(int hi, int lo) {
  return __funnelshift_l((uint32_t)lo, (uint32_t)hi, 3) & 0x7fffffu;
}

// The functions on doubles.  bad is set where an operand or the result is
// outside the range they cover (subnormal, infinite, NaN, negative under a
// root, zero under a reciprocal): the value returned there means nothing.
__device__ __forceinline__ double rcp_try(double x, bool& bad) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int ex = (hi >> 20) & 0x7ff;
  bad |= (unsigned)(ex - 1) >= 2044u;
  const uint64_t q = rcp_sig(sig53(hi, lo), rcp_seed(__uint_as_float(0x3f800000u | frac23(hi, lo))));
  const int rh = (int)(uint32_t)(q >> 32) + ((2044 - ex) << 20);
  return __hiloint2double(rh | (hi & (int)0x80000000), (int)(uint32_t)q);
}
__device__ __forceinline__ double rsqrt_try(double x, bool& bad) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  bad |= (unsigned)(hi - 0x00100000) >= 0x7fe00000u;  // not positive and normal
  const int ex = hi >> 20, odd = (ex & 1) ^ 1, k = (ex - 1023 - odd) >> 1;
  const float seed = rsqrt_seed(__uint_as_float((0x3f800000u + ((unsigned)odd << 23)) | frac23(hi, lo)));
  const uint64_t q = rsqrt_sig(sig53(hi, lo), odd, seed);
  return __hiloint2double((int)(uint32_t)(q >> 32) + ((1021 - k) << 20), (int)(uint32_t)q);
}
__device__ __forceinline__ double sqrt_try(double x, bool& bad) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const bool zero = ((hi & 0x7fffffff) | lo) == 0;
  bad |= !zero & ((unsigned)(hi - 0x00100000) >= 0x7fe00000u);
  const int ex = hi >> 20, odd = (ex & 1) ^ 1, k = (ex - 1023 - odd) >> 1;
  const float seed = rsqrt_seed(__uint_as_float((0x3f800000u + ((unsigned)odd << 23)) | frac23(hi, lo)));
  const uint64_t q = sqrt_sig(sig53(hi, lo), odd, seed);
  const double r = __hiloint2double((int)(uint32_t)(q >> 32) + ((1022 + k) << 20), (int)(uint32_t)q);
  return zero ? x : r;
}
// a b (the IEEE product)
__device__ __forceinline__ double mul_try(double a, double b, bool& bad) {
  const int ha = __double2hiint(a), la = __double2loint(a), hb = __double2hiint(b), lb = __double2loint(b);
  const int ea = (ha >> 20) & 0x7ff, eb = (hb >> 20) & 0x7ff;
  int big;
  const uint64_t q = mul_sig(sig53(ha, la), sig53(hb, lb), big);
  const int e = ea + eb - 1023 + big;
  const bool zero = (((ha << 1) | la) == 0) | (((hb << 1) | lb) == 0);
  bad |= ((unsigned)(ea - 1) >= 2046u) | ((unsigned)(eb - 1) >= 2046u) | ((unsigned)(e - 1) >= 2045u) ? !(zero & (ea < 2047) & (eb < 2047)) : false;
  const int s = (ha ^ hb) & (int)0x80000000;
  const int rh = (int)(uint32_t)(q >> 32) + ((e - 1) << 20);
  return __hiloint2double((zero ? 0 : rh) | s, zero ? 0 : (int)(uint32_t)q);
}

// For every operand: outside that range the library function, called only in
// warps where a lane needs it.
static __device__ __noinline__ double rcp_other(double x) { return __drcp_rn(x); }
static __device__ __noinline__ double sqrt_other(double x) { return __dsqrt_rn(x); }
static __device__ __noinline__ double rsqrt_other(double x) { return rsqrt(x); }
static __device__ __noinline__ double mul_other(double a, double b) { return a * b; }
__device__ __forceinline__ double rcp_int(double x) {
  bool bad = false;
  double r = rcp_try(x, bad);
  if (__any_sync(__activemask(), bad)) {
    if (bad) r = rcp_other(x);
  }
  return r;
}
__device__ __forceinline__ double rsqrt_int(double x) {
  bool bad = false;
  double r = rsqrt_try(x, bad);
  if (__any_sync(__activemask(), bad)) {
    if (bad) r = rsqrt_other(x);
  }
  return r;
}
__device__ __forceinline__ double sqrt_int(double x) {
  bool bad = false;
  double r = sqrt_try(x, bad);
  if (__any_sync(__activemask(), bad)) {
    if (bad) r = sqrt_other(x);
  }
  return r;
}

#endif  // __CUDACC__ || MHD_HOST_CHECK

}  // namespace mhd
