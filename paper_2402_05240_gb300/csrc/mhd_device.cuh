// mhd_device.cuh -- device arithmetic of the VL+CT ideal-MHD step (sm_103a).
//
// Templated on the compute type T (double for the FP64 step, float for the
// FP32-bulk step).  Pressure recovery from the conserved state is always done
// in double (the cancellation E - KE - B^2/2 sets the pressure floor).
//
// Method: Caddy & Schneider (arXiv:2402.05240) Sec. 2.1-2.2; HLLD of Miyoshi
// & Kusano (2005); primitive eigenvectors in the normalisation of Stone et
// al. (2008, App. A) with the left eigenvectors in closed form; PPM limiters
// of Colella & Sekora (2008) and McCorquodale & Colella (2011) applied in the
// characteristic variables (Felker & Stone 2018).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <type_traits>

#include "mhd_df.cuh"
#include "mhd_int53.cuh"
#include "mhd_launch.h"

namespace mhd {

// ------------------------------------------------------------ grid helpers --
__device__ __forceinline__ int wrapi(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

__device__ __forceinline__ long long cidx(const Grid& g, int i, int j, int k) {
  return ((long long)k * g.n[1] + j) * g.n[0] + i;
}

// index of cell (i,j,k) + s e_a, |s| < n[a]
template <int A>
__device__ __forceinline__ long long nb(const Grid& g, int i, int j, int k, int s) {
  if (A == 0) return cidx(g, wrapi(i + s, g.n[0]), j, k);
  if (A == 1) return cidx(g, i, wrapi(j + s, g.n[1]), k);
  return cidx(g, i, j, wrapi(k + s, g.n[2]));
}

template <class T> __device__ __forceinline__ T tsqrt(T x);
template <> __device__ __forceinline__ double tsqrt<double>(double x) { return sqrt_int(x); }
template <> __device__ __forceinline__ float tsqrt<float>(float x) { return sqrtf(x); }

// correctly rounded reciprocal (cheaper than a general division) and
// reciprocal square root; double: on the integer pipes (mhd_int53.cuh)
template <class T> __device__ __forceinline__ T trcp(T x);
template <> __device__ __forceinline__ double trcp<double>(double x) { return rcp_int(x); }
template <> __device__ __forceinline__ float trcp<float>(float x) { return __frcp_rn(x); }
template <class T> __device__ __forceinline__ T trsqrt(T x);
template <> __device__ __forceinline__ double trsqrt<double>(double x) { return rsqrt_int(x); }
template <> __device__ __forceinline__ float trsqrt<float>(float x) { return rsqrtf(x); }

template <> __device__ __forceinline__ df tsqrt<df>(df x) { return df_sqrt(x); }
template <> __device__ __forceinline__ df trcp<df>(df x) { return df(1.0f, 0.0f) / x; }
template <> __device__ __forceinline__ df trsqrt<df>(df x) { return df_rsqrt(x); }

// Comparisons of the step's branch decisions.  The generic forms use
// floating-point compares; for double they test the bit pattern on the
// integer pipes (the FP64 pipe bounds the FP64 step), with the same result
// for every non-NaN operand.  Positive doubles order like their bit
// patterns as signed 64-bit integers; -0 is the most negative pattern.
constexpr long long kAbsBits = 0x7fffffffffffffffLL;
constexpr long long kNegZero = (long long)0x8000000000000000ULL;
__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }
template <class T> __device__ __forceinline__ bool ge0(T x) { return x >= T(0); }
template <class T> __device__ __forceinline__ bool gt0(T x) { return x > T(0); }
template <class T> __device__ __forceinline__ bool lt0(T x) { return x < T(0); }
template <class T> __device__ __forceinline__ bool le0(T x) { return x <= T(0); }
template <class T> __device__ __forceinline__ bool is0(T x) { return x == T(0); }
// |x| < t for t >= 0
template <class T> __device__ __forceinline__ bool abs_lt(T x, T t) { return fabs(x) < t; }
// x < t for x, t >= 0
template <class T> __device__ __forceinline__ bool nonneg_lt(T x, T t) { return x < t; }
// x < t for t > 0 (x of any sign)
template <class T> __device__ __forceinline__ bool lt_pos(T x, T t) { return x < t; }
// max(x, t) for t > 0 (x of any sign)
template <class T> __device__ __forceinline__ T max_pos(T x, T t) { return fmax(x, t); }
// max(x, y) for x, y >= 0
template <class T> __device__ __forceinline__ T max_nonneg(T x, T y) { return fmax(x, y); }
// min and max of two values of any sign
template <class T> __device__ __forceinline__ T min_s(T x, T y) { return fmin(x, y); }
template <class T> __device__ __forceinline__ T max_s(T x, T y) { return fmax(x, y); }

// (a normalised pair has the sign of its leading float, and is zero with it)
template <> __device__ __forceinline__ bool ge0<df>(df x) { return x.hi >= 0.0f; }
template <> __device__ __forceinline__ bool gt0<df>(df x) { return x.hi > 0.0f; }
template <> __device__ __forceinline__ bool lt0<df>(df x) { return x.hi < 0.0f; }
template <> __device__ __forceinline__ bool le0<df>(df x) { return x.hi <= 0.0f; }
template <> __device__ __forceinline__ bool is0<df>(df x) { return x.hi == 0.0f; }
template <> __device__ __forceinline__ bool ge0<double>(double x) {
  const long long b = dbits(x);
  return (b >= 0) | (b == kNegZero);
}
template <> __device__ __forceinline__ bool gt0<double>(double x) { return dbits(x) > 0; }
template <> __device__ __forceinline__ bool lt0<double>(double x) {
  const long long b = dbits(x);
  return (b < 0) & (b != kNegZero);
}
template <> __device__ __forceinline__ bool le0<double>(double x) { return dbits(x) <= 0; }
template <> __device__ __forceinline__ bool is0<double>(double x) { return (dbits(x) & kAbsBits) == 0; }
template <> __device__ __forceinline__ bool abs_lt<double>(double x, double t) {
  return (dbits(x) & kAbsBits) < dbits(t);
}
template <> __device__ __forceinline__ bool nonneg_lt<double>(double x, double t) { return dbits(x) < dbits(t); }
template <> __device__ __forceinline__ bool lt_pos<double>(double x, double t) { return dbits(x) < dbits(t); }
template <> __device__ __forceinline__ double max_pos<double>(double x, double t) {
  return dbits(x) > dbits(t) ? x : t;
}
template <> __device__ __forceinline__ double max_nonneg<double>(double x, double y) {
  return dbits(x) >= dbits(y) ? x : y;
}
// x finite (not +-inf, not NaN), and x > 0 and not NaN, on the bit pattern
__device__ __forceinline__ bool finite_bits(double x) { return (dbits(x) & kAbsBits) < 0x7ff0000000000000LL; }
__device__ __forceinline__ bool pos_bits(double x) {
  const long long b = dbits(x);
  return b > 0 && b <= 0x7ff0000000000000LL;
}
// |x|; for double on the bit pattern
template <class T> __device__ __forceinline__ T absv(T x) { return fabs(x); }
template <> __device__ __forceinline__ double absv<double>(double x) {
  return __hiloint2double(__double2hiint(x) & 0x7fffffff, __double2loint(x));
}
// order key: sign-magnitude patterns mapped to a monotone signed integer
__device__ __forceinline__ long long dkey(double x) {
  const long long b = dbits(x);
  return b ^ ((b >> 63) & kAbsBits);
}
template <> __device__ __forceinline__ double min_s<double>(double x, double y) {
  return dkey(y) < dkey(x) ? y : x;
}
template <> __device__ __forceinline__ double max_s<double>(double x, double y) {
  return dkey(x) < dkey(y) ? y : x;
}

template <class T> __device__ __forceinline__ T neg(T x) { return -x; }
template <> __device__ __forceinline__ double neg<double>(double x) {
  return __hiloint2double(__double2hiint(x) ^ (int)0x80000000, __double2loint(x));
}
// (Sign operations on doubles work on the high word through the word
// intrinsics: written on the 64-bit pattern the compiler recognises them as
// negations and absolute values and, where they feed a selection, issues them
// as additions on the FP64 pipe.)
// Scalings by 2, 4 and 1/2.  Double: on the bit pattern.  twice() is the IEEE
// product for every operand (the reverse doubles cotangents, which may be
// infinite or NaN); half() and quarter() cut results below 2^-1022 to a
// multiple of the smallest subnormal and are exact otherwise; quad()
// falls back to the multiplication, executed only in warps where a lane needs
// it, where operand or result is not normal.
template <class T> __device__ __forceinline__ T twice(T x) { return T(2) * x; }
template <> __device__ __forceinline__ df twice<df>(df x) { return df(2.0f * x.hi, 2.0f * x.lo); }
template <> __device__ __forceinline__ double twice<double>(double v) {
  const int hi = __double2hiint(v), lo = __double2loint(v), m = hi & 0x7fffffff;
  const bool small = m < 0x00100000;  // zero or subnormal
  int rh = small ? (int)__funnelshift_l((unsigned)lo, (unsigned)m, 1) | (hi & (int)0x80000000) : hi + 0x00100000;
  int rl = small ? (int)((unsigned)lo << 1) : lo;
  if (m >= 0x7fe00000) {  // the result is an infinity, or v a NaN
    rh = m >= 0x7ff00000 ? hi : (hi | 0x7ff00000) & (int)0xfff00000;
    rl = m >= 0x7ff00000 ? lo : 0;
  }
  return __hiloint2double(rh, rl);
}
// twice_n: for the limiters' operands, zero or normal and without overflow.
// (256^3, FP64, with twice() in its place: PLMC reconstruction 18.56 -> 18.79 ms,
// PPMC 32.65 -> 32.86.)
template <class T> __device__ __forceinline__ T twice_n(T x) { return twice<T>(x); }
template <> __device__ __forceinline__ double twice_n<double>(double v) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  return __hiloint2double(((hi & 0x7fffffff) | lo) ? hi + 0x00100000 : hi, lo);
}
// (twice_f, half_f: scalings inside a sum -- a multiplication that the
// compiler fuses with the addition, except for float pairs)
template <class T> __device__ __forceinline__ T twice_f(T x) { return T(2) * x; }
template <> __device__ __forceinline__ df twice_f<df>(df x) { return twice<df>(x); }
// a - 2 b.  (Double: the compiler rewrites 2 b as b + b, two FP64-pipe
// instructions where one multiply-add does.)
template <class T> __device__ __forceinline__ T sub_twice(T a, T b) { return a - twice_f<T>(b); }
template <> __device__ __forceinline__ double sub_twice<double>(double a, double b) { return fma(-2.0, b, a); }
template <class T> __device__ __forceinline__ T half(T x) { return T(0.5) * x; }
template <> __device__ __forceinline__ df half<df>(df x) { return df(0.5f * x.hi, 0.5f * x.lo); }
template <class T> __device__ __forceinline__ T half_f(T x) { return T(0.5) * x; }
template <> __device__ __forceinline__ df half_f<df>(df x) { return half<df>(x); }
template <> __device__ __forceinline__ double half<double>(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x), m = hi & 0x7fffffff;
  const bool small = m < 0x00200000;  // operand or result not normal
  const int rl = small ? (int)__funnelshift_r((unsigned)lo, (unsigned)m, 1) : lo;
  const int rh = small ? (m >> 1) | (hi & (int)0x80000000) : hi - 0x00100000;
  return __hiloint2double(m >= 0x7ff00000 ? hi : rh, rl);
}
template <class T> __device__ __forceinline__ T quad(T x) { return T(4) * x; }
template <> __device__ __forceinline__ df quad<df>(df x) { return df(4.0f * x.hi, 4.0f * x.lo); }
template <> __device__ __forceinline__ double quad<double>(double x) {
  const int hi = __double2hiint(x);
  const bool fast = (unsigned)(hi & 0x7fffffff) - 0x00100000u < 0x7fd00000u - 0x00100000u;
  double r = __hiloint2double(hi + 0x00200000, __double2loint(x));
  if (__any_sync(__activemask(), !fast)) {
    if (!fast) r = 4.0 * x;
  }
  return r;
}
// c ? a : b.  Double: a selection the compiler cannot move past the arithmetic
// that consumes it (it turns (c ? a : b) - (c ? x : y) into a selection between
// two differences, twice the FP64-pipe work).
template <class T> __device__ __forceinline__ T pick(bool c, T a, T b) { return c ? a : b; }
#if defined(__CUDA_ARCH__)
template <> __device__ __forceinline__ double pick<double>(bool c, double a, double b) {
  double r;
  asm("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %1, 0;\n\tselp.f64 %0, %2, %3, p;\n\t}" : "=d"(r) : "r"((int)c), "d"(a), "d"(b));
  return r;
}
#endif
// x / 4; as half() (edge fields, and |B_cc|^2 of the FP32-bulk pressure)
template <class T> __device__ __forceinline__ T quarter(T x) { return T(0.25) * x; }
template <> __device__ __forceinline__ df quarter<df>(df x) { return df(0.25f * x.hi, 0.25f * x.lo); }
template <> __device__ __forceinline__ double quarter<double>(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x), m = hi & 0x7fffffff;
  const bool small = m < 0x00300000;  // operand or result not normal
  // (exponent field 2: down to 1, whose significand stands as a subnormal's does)
  const int low = m < 0x00200000 ? m : m - 0x00100000, sh = m < 0x00200000 ? 2 : 1;
  const int rl = small ? (int)__funnelshift_r((unsigned)lo, (unsigned)low, sh) : lo;
  const int rh = small ? (low >> sh) | (hi & (int)0x80000000) : hi - 0x00200000;
  return __hiloint2double(m >= 0x7ff00000 ? hi : rh, rl);
}
// s x for s = +-1 (a sign flip for double and float pairs)
template <class T> __device__ __forceinline__ T times_sign(T x, T s) { return x * s; }
template <> __device__ __forceinline__ df times_sign<df>(df x, df s) { return s.hi < 0.0f ? df(-x.hi, -x.lo) : x; }
template <> __device__ __forceinline__ double times_sign<double>(double x, double s) {
  return __hiloint2double(__double2hiint(x) ^ (__double2hiint(s) & (int)0x80000000), __double2loint(x));
}

// Conversions between the compute type and double without the conversion
// instructions, which issue at the FP64 rate on this GPU (mhd_df.cuh).
template <class T> __device__ __forceinline__ double to_d(T x);
template <> __device__ __forceinline__ double to_d<double>(double x) { return x; }
template <> __device__ __forceinline__ double to_d<float>(float x) { return f2d_bits(x); }
template <> __device__ __forceinline__ double to_d<df>(df x) { return (double)x; }
// the nearest float (float pairs: the leading one)
template <class T> __device__ __forceinline__ float to_f(T x);
template <> __device__ __forceinline__ float to_f<double>(double x) { return d2f_bits(x); }
template <> __device__ __forceinline__ float to_f<df>(df x) { return x.hi; }
template <class T> __device__ __forceinline__ T from_d(double x);
template <> __device__ __forceinline__ double from_d<double>(double x) { return x; }
template <> __device__ __forceinline__ float from_d<float>(double x) { return d2f_bits(x); }
template <> __device__ __forceinline__ df from_d<df>(double x) { return df(x); }
// (float pairs: with the longer low part)
template <class T> __device__ __forceinline__ T nearest(double x) { return from_d<T>(x); }
template <> __device__ __forceinline__ df nearest<df>(double x) { return df_nearest(x); }

// Exact<T>: the full update widens each flux and edge value to double before
// differencing (a difference of two floats is exact in double).  df values
// already carry ~48 bits, so their differences and increments are formed in
// df and added to the double state once.
template <class T> struct Exact { static constexpr bool full = true; };
template <> struct Exact<df> { static constexpr bool full = false; };

template <class T> struct Eps;
template <> struct Eps<double> { static constexpr double hlld = 1e-8; };
template <> struct Eps<float> { static constexpr float hlld = 1e-4f; };
template <> struct Eps<df> { static constexpr float hlld = 1e-8f; };

// a / b for |a| <= |b|, b != 0
template <class T> __device__ __forceinline__ T ratio_le1(T a, T b) { return a / b; }
static __device__ __noinline__ double div_call(double a, double b) { return a / b; }
template <> __device__ __forceinline__ double ratio_le1<double>(double a, double b) {
  // biased exponent >= 64: 1/b is finite and normal.  The division for
  // smaller b is a call made only in warps where some lane needs it (inlined,
  // the compiler evaluates it in every warp, on the FP64 pipe)
  const bool tiny = ((dbits(b) >> 52) & 0x7ff) < 64;
  double r = a * trcp<double>(b);
  if (__any_sync(__activemask(), tiny)) {
    if (tiny) r = div_call(a, b);
  }
  return r;
}

// A product that no sum takes up, as a call on the integer pipes (double; any
// operands) -- see Ops
static __device__ __noinline__ double mul_call(double a, double b) {
  bool bad = false;
  double r = mul_try(a, b, bad);
  if (__any_sync(__activemask(), bad)) {
    if (bad) r = mul_other(a, b);
  }
  return r;
}
// (float pairs: the unnormalised product, which a sum may take as it stands)
template <class T> __device__ __forceinline__ auto mulc(T a, T b) {
  if constexpr (std::is_same<T, double>::value) return mul_call(a, b);
  else return a * b;
}

// The operations of the reconstruction and the Riemann solver that have more
// than one form.  Ops: complete functions.  TryOps<double>: the integer-pipe
// functions alone; `bad` tells that an operand left their range, and the
// caller then evaluates the cell again with Ops, out of line (recon_cell,
// hlld): one test per cell in the place of one per function.  mul is for
// products that no sum takes up (a multiply-add is one FP64 instruction
// anyway): on the integer pipes a product costs about 38 issue slots against
// the 64 of an FP64 instruction, and the FP64 pipe has the less idle time.
// The product is a call, operands and result in registers: inlined, its copies
// spill registers and outgrow the instruction cache (PPMC with the projections'
// products 45.8 ms inlined, 33.2 ms as calls; Riemann kernels with 38 products
// 10.2 and 8.7 ms).  Measured at 256^3, FP64: Riemann kernels 10.9 -> 8.7 ms, PLMC
// reconstruction 23.9 -> 18.4 ms, PPMC 41.4 -> 32.5 ms.
template <class T> struct Ops {
  static constexpr bool bad = false;
  __device__ __forceinline__ T rcp(T x) { return trcp<T>(x); }
  __device__ __forceinline__ T sqrt(T x) { return tsqrt<T>(x); }
  __device__ __forceinline__ T rsqrt(T x) { return trsqrt<T>(x); }
  __device__ __forceinline__ T quad(T x) { return mhd::quad<T>(x); }
  __device__ __forceinline__ T twice(T x) { return mhd::twice<T>(x); }
  __device__ __forceinline__ auto mul(T a, T b) { return mulc<T>(a, b); }
};
struct TryValue {
  double v;
  int bad;
};
static __device__ __noinline__ TryValue mul_try_call(double a, double b) {
  bool bad = false;
  const double v = mul_try(a, b, bad);
  return TryValue{v, bad};
}
template <class T> struct TryOps : Ops<T> {};
template <> struct TryOps<double> {
  bool bad = false;
  __device__ __forceinline__ double rcp(double x) { return rcp_try(x, bad); }
  __device__ __forceinline__ double sqrt(double x) { return sqrt_try(x, bad); }
  __device__ __forceinline__ double rsqrt(double x) { return rsqrt_try(x, bad); }
  __device__ __forceinline__ double quad(double x) {  // x >= 0
    const long long b = dbits(x);
    bad |= (b != 0) & ((unsigned long long)(b - (1LL << 52)) >= (0x7fdULL << 52) - (1ULL << 52));
    return __longlong_as_double(b ? b + (2LL << 52) : b);
  }
  // (of a root or a product: below 2^1023, and not normal or zero only where
  // bad is set already)
  __device__ __forceinline__ double twice(double x) { return twice_n<double>(x); }
  __device__ __forceinline__ double mul(double a, double b) {
    const TryValue r = mul_try_call(a, b);
    bad |= r.bad != 0;
    return r.v;
  }
};

// ------------------------------------------------- primitives (Sec. 2.2.1) --
// Cell primitives: rho, v, P (pressure recovered in double) and B_cc, the mean
// of the two faces of each component.
struct PrimD {
  double rho, v[3], p, b[3];
};

// ----------------------------------------------------- fast speed (Eq. c_f) --
// c_f^2 = (a2 + b2 + sqrt((a2 - b2)^2 + 4 a2 bt2)) / 2 with a2 = gamma P / rho,
// b2 = |B|^2 / rho, bt2 = |B_t|^2 / rho: the printed discriminant
// (gamma P + B^2)^2 - 4 gamma P B_l^2 (over rho^2) as a sum of non-negative terms.
template <class T>
__device__ __forceinline__ T fast_speed_sq(T gamma, T rho, T p, T bl, T bt1, T bt2) {
  T ir = trcp<T>(rho);
  T a2 = gamma * p * ir;
  T t2 = (bt1 * bt1 + bt2 * bt2) * ir;
  T b2 = bl * bl * ir + t2;
  T dd = a2 - b2;
  return T(0.5) * (a2 + b2 + tsqrt<T>(dd * dd + T(4) * a2 * t2));
}
template <class T>
__device__ __forceinline__ T fast_speed(T gamma, T rho, T p, T bl, T bt1, T bt2) {
  return tsqrt<T>(fast_speed_sq<T>(gamma, rho, p, bl, bt1, bt2));
}

// ------------------------------------------------------------------- HLLD --
// Miyoshi & Kusano (2005) in the solver frame; w = (rho, u, v, w, P, By, Bz),
// bn = longitudinal face field.  Outer speeds S_L = min(u) - max(c_f),
// S_R = max(u) + max(c_f); degenerate star / double-star states below
// Eps<T>::hlld * p_T*; flux selection with ties to the left.  gm1i = 1/(gamma - 1).
//
// Double and float pairs (hlld_diff): every increment of F + S (U* - U) +
// S* (U** - U*) is formed from the differences that cause it.  With delta =
// S_M - u = (rho'(S' - u')(u_R - u_L) + p_L - p_R) / den (primes: the other
// side), t = B_n delta / D and q - 1 = rho (S - u) delta / D, the star
// increments are rho* - rho = rho delta / (S - S_M), v* - v = -B_t t, B* - B_t =
// B_t (q - 1), and the double-star ones share one velocity difference.  That
// takes 90 operations where no lane of the warp lies between the Alfven waves
// and 132 where one does, against 156 in the jump form; equal states give
// their physical flux exactly, and the degenerate limit is delta / D = 0.
// The other side's star state is formed for double-star faces alone.  Both
// types are bound by the arithmetic (FP64 pipe, issue slots): against the
// jump form the PLMC step went from 72.1 to 61.8 ms (FP64, 256^3) and from
// 116.4 to 104.7 ms (float pairs, 459^3).
// float (hlld_jump): kept in the jump form, whose rounding fixes the
// FP32-bulk mode's results.
template <class T>
__device__ __forceinline__ void hlld_jump(T gamma, T gm1i, const T* wl, const T* wr, T bn, T* f) {
  const T bn2 = bn * bn;
  // total pressures of both sides; the conserved energy is formed only for
  // the side whose states the flux is taken from
  const T btL = wl[5] * wl[5] + wl[6] * wl[6], btR = wr[5] * wr[5] + wr[6] * wr[6];
  const T bbL = bn2 + btL;
  const T bbR = bn2 + btR;
  const T ptL = wl[4] + T(0.5) * bbL;
  const T ptR = wr[4] + T(0.5) * bbR;
  auto energy = [&](const T* w, T bb) {
    return w[4] * gm1i + T(0.5) * w[0] * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]) + T(0.5) * bb;
  };
  // max(c_f,L, c_f,R) (Eq. c_f with the face B_n): rho c_f^2 =
  // (gamma P + B^2 + sqrt((gamma P - B^2)^2 + 4 gamma P B_t^2)) / 2 needs no
  // division, the larger c_f^2 = X / rho is chosen by cross-multiplication,
  // and only its side takes a reciprocal and a root
  auto rho_cf2 = [&](T p, T bb, T bt) {
    const T gp = gamma * p;
    const T dd = gp - bb;
    return T(0.5) * (gp + bb + tsqrt<T>(dd * dd + T(4) * gp * bt));
  };
  const T XL = rho_cf2(wl[4], bbL, btL), XR = rho_cf2(wr[4], bbR, btR);
  const bool lmax = !nonneg_lt<T>(XL * wr[0], XR * wl[0]);
  const T cmax = tsqrt<T>((lmax ? XL : XR) * trcp<T>(lmax ? wl[0] : wr[0]));
  const T SL = min_s<T>(wl[1], wr[1]) - cmax;
  const T SR = max_s<T>(wl[1], wr[1]) + cmax;

  auto phys = [&](const T* w, T e, T pt, T* F) {
    const T mu = w[0] * w[1];
    F[0] = mu;
    F[1] = mu * w[1] + pt - bn2;
    F[2] = mu * w[2] - bn * w[5];
    F[3] = mu * w[3] - bn * w[6];
    F[4] = (e + pt) * w[1] - bn * (w[1] * bn + w[2] * w[5] + w[3] * w[6]);
    F[5] = w[5] * w[1] - bn * w[2];
    F[6] = w[6] * w[1] - bn * w[3];
  };
  // Supersonic faces take the upwind side's physical flux; the others its
  // star or double-star flux.  One physical flux serves both cases, so a
  // warp mixing them evaluates it once.
  const bool sub = !ge0<T>(SL) && !le0<T>(SR);
  T dL = T(0), dR = T(0), rdL = T(0), rdR = T(0), SM = T(0), pts = T(0);
  if (sub) {
    dL = SL - wl[1];
    dR = SR - wr[1];
    rdL = wl[0] * dL;
    rdR = wr[0] * dR;
    const T iden = trcp<T>(rdR - rdL);
    SM = (rdR * wr[1] - rdL * wl[1] - ptR + ptL) * iden;
    pts = (rdR * ptL - rdL * ptR + rdL * rdR * (wr[1] - wl[1])) * iden;
  }
  // the side whose states the flux comes from (ties to the left)
  const bool left = sub ? ge0<T>(SM) : ge0<T>(SL);
  const T* w = left ? wl : wr;
  const T pt = left ? ptL : ptR;
  const T e = energy(w, left ? bbL : bbR);
  T F[7];
  phys(w, e, pt, F);
  if (!sub) {
#pragma unroll
    for (int q = 0; q < 7; ++q) f[q] = F[q];
    return;
  }

  // single-star states of one side: rho*, v*, w*, By*, Bz* (both sides feed
  // the double-star states)
  struct Star {
    T r, v, w, by, bz, sq, rsq, iSM;
  };
  auto star = [&](const T* ws, T S, T d, T rd) {
    Star st;
    st.iSM = trcp<T>(S - SM);
    st.r = rd * st.iSM;
    const T D = rd * (S - SM) - bn2;
    if (abs_lt<T>(D, Eps<T>::hlld * pts)) {
      st.v = ws[2];
      st.w = ws[3];
      st.by = ws[5];
      st.bz = ws[6];
    } else {
      const T iD = trcp<T>(D);
      const T t = bn * (SM - ws[1]) * iD;
      st.v = ws[2] - ws[5] * t;
      st.w = ws[3] - ws[6] * t;
      const T q = (rd * d - bn2) * iD;
      st.by = ws[5] * q;
      st.bz = ws[6] * q;
    }
    st.rsq = trsqrt<T>(st.r);
    st.sq = st.r * st.rsq;
    return st;
  };
  const Star sL = star(wl, SL, dL, rdL);
  const Star sR = star(wr, SR, dR, rdR);

  const Star& s = left ? sL : sR;
  const T S = left ? SL : SR;
  const T d = left ? dL : dR;
  // star energy E* of that side
  const T vb = w[1] * bn + w[2] * w[5] + w[3] * w[6];
  const T vbs = SM * bn + s.v * s.by + s.w * s.bz;
  const T es = (d * e - pt * w[1] + pts * SM + bn * (vb - vbs)) * s.iSM;

  // double-star (rotational) states
  T SsL = SM, SsR = SM;
  T vss, wss, byss, bzss, ess;
  const bool dbl = !nonneg_lt<T>(T(0.5) * bn2, Eps<T>::hlld * pts);
  if (dbl) {
    const T sg = gt0<T>(bn) ? T(1) : T(-1);
    const T abn = fabs(bn);
    SsL = SM - abn * sL.rsq;
    SsR = SM + abn * sR.rsq;
    const T inv = trcp<T>(sL.sq + sR.sq);
    vss = (sL.sq * sL.v + sR.sq * sR.v + (sR.by - sL.by) * sg) * inv;
    wss = (sL.sq * sL.w + sR.sq * sR.w + (sR.bz - sL.bz) * sg) * inv;
    byss = (sL.sq * sR.by + sR.sq * sL.by + sL.sq * sR.sq * (sR.v - sL.v) * sg) * inv;
    bzss = (sL.sq * sR.bz + sR.sq * sL.bz + sL.sq * sR.sq * (sR.w - sL.w) * sg) * inv;
    const T vbss = SM * bn + vss * byss + wss * bzss;
    // E** = E* -+ sqrt(rho*) (v*.B* - v**.B**) sgn(B_n), - on the left
    if (left)
      ess = es - s.sq * (SM * bn + s.v * s.by + s.w * s.bz - vbss) * sg;
    else
      ess = es + s.sq * (SM * bn + s.v * s.by + s.w * s.bz - vbss) * sg;
  }
  const T U0[7] = {w[0], w[0] * w[1], w[0] * w[2], w[0] * w[3], e, w[5], w[6]};
  const T Us[7] = {s.r, s.r * SM, s.r * s.v, s.r * s.w, es, s.by, s.bz};
  // F* = F + S (U* - U)
  for (int q = 0; q < 7; ++q) f[q] = F[q] + S * (Us[q] - U0[q]);
  const T Ss = left ? SsL : SsR;
  const bool inner = left ? lt0<T>(SsL) : ge0<T>(SsR);
  if (dbl && inner) {
    const T Uss[7] = {s.r, s.r * SM, s.r * vss, s.r * wss, ess, byss, bzss};
    for (int q = 0; q < 7; ++q) f[q] = f[q] + Ss * (Uss[q] - Us[q]);
  }
}

template <class T, class O>
__device__ __forceinline__ void hlld_diff(O& o, T gamma, T gm1i, const T* wl, const T* wr, T bn, T* f) {
  const T bn2 = o.mul(bn, bn);
  const T btL = o.mul(wl[5], wl[5]) + wl[6] * wl[6], btR = o.mul(wr[5], wr[5]) + wr[6] * wr[6];
  const T bbL = bn2 + btL, bbR = bn2 + btR;
  const T ptL = wl[4] + half<T>(bbL), ptR = wr[4] + half<T>(bbR);
  // 2 rho c_f^2 = gamma P + B^2 + sqrt((gamma P - B^2)^2 + 4 gamma P B_t^2):
  // no division; the larger c_f^2 is chosen by cross-multiplication, and only
  // its side takes a reciprocal and a root
  auto two_rho_cf2 = [&](T p, T bb, T bt) {
    const T gp = o.mul(gamma, p);
    const T dd = gp - bb;
    return gp + bb + o.sqrt(dd * dd + o.mul(o.quad(gp), bt));
  };
  const T XL = two_rho_cf2(wl[4], bbL, btL), XR = two_rho_cf2(wr[4], bbR, btR);
  const bool lmax = !nonneg_lt<T>(o.mul(XL, wr[0]), o.mul(XR, wl[0]));
  const T cmax = o.sqrt(o.mul(half<T>(lmax ? XL : XR), o.rcp(lmax ? wl[0] : wr[0])));
  const T SL = min_s<T>(wl[1], wr[1]) - cmax;
  const T SR = max_s<T>(wl[1], wr[1]) + cmax;
  const bool sub = !ge0<T>(SL) && !le0<T>(SR);
  T rdL = T(0), rdR = T(0), dlL = T(0), dlR = T(0), SM = T(0), pts = T(0);
  if (sub) {
    rdL = o.mul(wl[0], SL - wl[1]);
    rdR = o.mul(wr[0], SR - wr[1]);
    const T iden = o.rcp(rdR - rdL);
    const T du = wr[1] - wl[1], dp = ptL - ptR;
    dlL = o.mul(rdR * du + dp, iden);  // S_M - u of both sides
    dlR = o.mul(rdL * du + dp, iden);
    SM = wl[1] + dlL;
    pts = ptL + rdL * dlL;
  }
  // the side whose states the flux is taken from (ties to the left)
  const bool left = sub ? ge0<T>(SM) : ge0<T>(SL);
  const T* w = left ? wl : wr;
  const T r = w[0], u = w[1], v = w[2], vw = w[3], by = w[5], bz = w[6];
  const T pt = left ? ptL : ptR, bt = left ? btL : btR;
  const T e = w[4] * gm1i + (half<T>(r) * (o.mul(u, u) + v * v + vw * vw) + half<T>(left ? bbL : bbR));
  const T mu = o.mul(r, u);
  const T vby = o.mul(v, by) + vw * bz;
  // the increments S (U* - U) of the star region: zero for a supersonic face
  T m1 = T(0), sm1 = T(0), C = bn, A = u, dE = T(0);
  T rs = T(0), z = T(0), rd = T(0), Ss = T(0);
  bool inner = false;
  if (sub) {
    const T S = left ? SL : SR, dl = left ? dlL : dlR;
    rd = left ? rdL : rdR;
    const T Sd = S - SM;
    const T iSd = o.rcp(Sd);
    rs = o.mul(rd, iSd);
    const T D = rd * Sd - bn2;
    // (the degenerate limit keeps the transverse state: z = 0)
    z = abs_lt<T>(D, Eps<T>::hlld * pts) ? T(0) : dl * o.rcp(D);
    const T t = o.mul(bn, z), rz = o.mul(rd, z);  // v* = v - B_t t, B* = B_t (1 + rz)
    // (a density jump below the rounding of rho* is none: the mass flux then
    // keeps the sign of the resolved velocity, which the edge fields upwind by)
    m1 = rs == r ? T(0) : o.mul(S, o.mul(r, o.mul(dl, iSd)));
    sm1 = S * (rs * SM - mu);
    C = bn + o.mul(S, rs) * t;
    A = u + S * rz;
    const T ps = pt + rd * dl;
    const T bbt = o.mul(bt, t);
    const T dvb = rz * (vby - bbt) + (bn * dl - bbt);  // v*.B* - v.B
    dE = o.mul(S, o.mul((e + ps + u * rd) * dl - bn * dvb, iSd));
    const T cA = fabs(bn) * o.rsqrt(rs);
    Ss = left ? SM - cA : SM + cA;
    inner = (left ? lt0<T>(Ss) : ge0<T>(Ss)) && !nonneg_lt<T>(half<T>(bn2), Eps<T>::hlld * pts);
  }
  const T f0 = mu + m1;
  f[0] = f0;
  f[1] = mu * u + (pt - bn2) + sm1;
  f[2] = o.mul(f0, v) - by * C;
  f[3] = o.mul(f0, vw) - bz * C;
  f[4] = o.mul(e + pt, u) - bn * (u * bn + vby) + dE;
  f[5] = o.mul(by, A) - bn * v;
  f[6] = o.mul(bz, A) - bn * vw;
  if (inner) {
    // the increments Ss (U** - U*) of the double-star region: with the star
    // states of both sides, Delta = v** - v* = (sgn(B_n) (B*_R - B*_L) +-
    // sqrt(rho*') (v*_R - v*_L)) / (sqrt(rho*_L) + sqrt(rho*_R)), rho*' the
    // other side's, + on the left, and B** - B* = g Delta, g = +- sqrt(rho*)
    // sgn(B_n), + on the left
    const T* wo = left ? wr : wl;
    const T rdo = left ? rdR : rdL;
    const T Sdo = (left ? SR : SL) - SM;
    const T rso = rdo * o.rcp(Sdo);
    const T Do = rdo * Sdo - bn2;
    const T zo = abs_lt<T>(Do, Eps<T>::hlld * pts) ? T(0) : (left ? dlR : dlL) * o.rcp(Do);
    const T t = bn * z, q = T(1) + rd * z;
    const T to = bn * zo, qo = T(1) + rdo * zo;
    const T vs = v - by * t, ws = vw - bz * t, bys = by * q, bzs = bz * q;
    const T sq = rs * o.rsqrt(rs), sqo = rso * o.rsqrt(rso);
    const T inv = o.rcp(sq + sqo);
    const T sg = (gt0<T>(bn) == left) ? T(1) : T(-1);
    // (differences other minus own: both terms change sign with the side)
    const T Dy = (times_sign<T>(wo[5] * qo - bys, sg) + sqo * ((wo[2] - wo[5] * to) - vs)) * inv;
    const T Dz = (times_sign<T>(wo[6] * qo - bzs, sg) + sqo * ((wo[3] - wo[6] * to) - ws)) * inv;
    const T g = times_sign<T>(sq, sg);
    const T ay = Ss * Dy, az = Ss * Dz;
    f[2] = f[2] + rs * ay;
    f[3] = f[3] + rs * az;
    f[4] = f[4] + g * (ay * (bys + g * (vs + Dy)) + az * (bzs + g * (ws + Dz)));
    f[5] = f[5] + g * ay;
    f[6] = f[6] + g * az;
  }
}

template <class T>
__device__ __noinline__ void hlld_again(T gamma, T gm1i, const T* wl, const T* wr, T bn, T* f) {
  Ops<T> o;
  hlld_diff<T>(o, gamma, gm1i, wl, wr, bn, f);
}
template <class T>
__device__ __forceinline__ void hlld(T gamma, T gm1i, const T* wl, const T* wr, T bn, T* f) {
  if constexpr (sizeof(T) == 4) {
    hlld_jump<T>(gamma, gm1i, wl, wr, bn, f);
  } else {
    TryOps<T> o;
    hlld_diff<T>(o, gamma, gm1i, wl, wr, bn, f);
    if constexpr (std::is_same<T, double>::value) {
      if (__any_sync(__activemask(), o.bad)) {
        if (o.bad) {
          T a[7], b[7], c[7];
#pragma unroll
          for (int q = 0; q < 7; ++q) {
            a[q] = wl[q];
            b[q] = wr[q];
          }
          hlld_again<T>(gamma, gm1i, a, b, bn, c);
#pragma unroll
          for (int q = 0; q < 7; ++q) f[q] = c[q];
        }
      }
    }
  }
}

// ------------------------------------------------ characteristic projection --
// Primitive eigen-system (rho, u, v, w, P, B_t1, B_t2) of one cell with its
// cell-centred longitudinal field bn.  Waves ordered u-cf, u-ca, u-cs, u,
// u+cs, u+ca, u+cf.  beta = (1,1)/sqrt2 for B_t = 0; alpha_f = 1, alpha_s = 0
// when cf2 = cs2; S = sgn(bn) with sgn(0) = +1.  The left eigenvectors are the
// closed-form inverse of the right ones (rows scaled by 1/(2 a^2) for the
// magnetosonic waves, 1/2 for the Alfven waves).
template <class T> struct Eig {
  T rho, ir, sr, isr, a, a2, ia2, af, as, cf, cs, Qf, Qs, Af, As, b1, b2, sg;
  T rcf;  // 1/c_f (for the reverse sweep)
};

// Square roots and divisions are folded into five reciprocal square roots
// and one square root: 1/sqrt(rho), 1/a, 1/c_f, 1/|B_t|, and
// q = 1/sqrt(2 s (s + |D|)) with s = c_f^2 - c_s^2, D = a^2 - b^2, giving
// c_s = a c_a / c_f and the alpha pair (s + |D|) q, 2 a |b_t| q.
template <class T, class O> __device__ __forceinline__ void eig_build(O& o, T gamma, const T* w, T bn, Eig<T>& E) {
  E.rho = w[0];
  E.isr = o.rsqrt(w[0]);
  E.sr = o.mul(w[0], E.isr);
  E.ir = o.mul(E.isr, E.isr);
  E.a2 = o.mul(o.mul(gamma, w[4]), E.ir);
  const T ra = o.rsqrt(E.a2);
  E.a = o.mul(E.a2, ra);
  E.ia2 = o.mul(ra, ra);
  const T ca2 = o.mul(o.mul(bn, bn), E.ir);
  const T bt2r = w[5] * w[5] + w[6] * w[6];
  const T bt2 = o.mul(bt2r, E.ir);
  const T b2 = ca2 + bt2;
  const T D = E.a2 - b2;
  const T sd = o.sqrt(D * D + o.mul(o.quad(E.a2), bt2));
  const T cf2 = half<T>(E.a2 + b2 + sd);
  const T rcf = o.rsqrt(cf2);
  E.rcf = rcf;
  E.cf = o.mul(cf2, rcf);
  E.cs = o.mul(o.mul(o.mul(E.a, fabs(bn)), E.isr), rcf);
  const T ibt = gt0<T>(bt2r) ? o.rsqrt(bt2r) : T(0);
  const T btn = o.mul(o.mul(bt2r, ibt), E.isr);  // |B_t| / sqrt(rho)
  // one formula for both signs of D (only the assignment of the two members
  // to alpha_f and alpha_s depends on it), so neighbouring cells with
  // different signs share one path through the FP64 pipe
  if (is0<T>(sd)) {
    E.af = T(1);
    E.as = T(0);
  } else {
    const bool dpos = ge0<T>(D);
    const T sa = sd + absv<T>(D);
    const T q = o.rsqrt(o.mul(o.twice(sd), sa));
    const T big = o.mul(sa, q), small = o.mul(o.mul(o.twice(E.a), btn), q);
    E.af = dpos ? big : small;
    E.as = dpos ? small : big;
  }
  if (is0<T>(bt2r)) {
    E.b1 = T(0.70710678118654752440);
    E.b2 = T(0.70710678118654752440);
  } else {
    E.b1 = o.mul(w[5], ibt);
    E.b2 = o.mul(w[6], ibt);
  }
  E.sg = ge0<T>(bn) ? T(1) : T(-1);
  const T a = E.a;
  E.Qf = times_sign<T>(o.mul(E.cf, E.af), E.sg);
  E.Qs = times_sign<T>(o.mul(E.cs, E.as), E.sg);
  E.Af = o.mul(o.mul(a, E.af), E.sr);
  E.As = o.mul(o.mul(a, E.as), E.sr);
}

template <class T> __device__ __forceinline__ void eig_build(T gamma, const T* w, T bn, Eig<T>& E) {
  Ops<T> o;
  eig_build<T>(o, gamma, w, bn, E);
}

// characteristic amplitudes q = L dw
//
// Double and float pairs take products of the eigensystem's fields, formed
// once for all projections of a cell (EigCoef), as coefficients: 23 operations per projection against 35 in the form
// below, which float keeps (its rounding fixes the FP32-bulk mode's results).
// With the shorter limiter below: FP64 PLMC 256^3 61.8 -> 56.1 ms per step,
// double-float PPMC 512^3 193 -> 182 ms.
// EigCoef: the fast and slow amplitudes of dP (fp, sp), of dB along beta (fb,
// sb) and of du (fu, su; of dv along beta su, fu), the Alfven ones of dv (h)
// and dB (z).
template <class T> struct EigCoef {
  T fp, sp, fb, sb, fu, su, h1, h2, z1, z2;
};
template <class T, class O> __device__ __forceinline__ EigCoef<T> eig_coef(O& o, const Eig<T>& E) {
  EigCoef<T> C;
  if constexpr (sizeof(T) != 4) {
    const T n = half<T>(E.ia2);
    const T naf = o.mul(n, E.af), nas = o.mul(n, E.as), ai = o.mul(E.a, E.isr);
    const T z = times_sign<T>(E.isr, E.sg);
    C.fp = o.mul(naf, E.ir);
    C.sp = o.mul(nas, E.ir);
    C.fb = o.mul(nas, ai);
    C.sb = o.mul(naf, ai);
    C.fu = o.mul(naf, E.cf);
    C.su = o.mul(nas, E.cs);
    C.h1 = half<T>(E.b1);
    C.h2 = half<T>(E.b2);
    C.z1 = o.mul(C.h1, z);
    C.z2 = o.mul(C.h2, z);
  }
  return C;
}
// (float)
template <class T> __device__ __forceinline__ void eig_left_narrow(const Eig<T>& E, const T* dw, T* q) {
  const T n = T(0.5) * E.ia2;
  const T ir = E.ir;
  const T bv = E.b1 * dw[2] + E.b2 * dw[3];
  const T bb = (E.b1 * dw[5] + E.b2 * dw[6]) * E.isr;
  const T sa = E.a;
  const T Xf = E.af * dw[4] * ir + E.as * sa * bb;
  const T Yf = -E.af * E.cf * dw[1] + E.Qs * bv;
  const T Xs = E.as * dw[4] * ir - E.af * sa * bb;
  const T Ys = -E.as * E.cs * dw[1] - E.Qf * bv;
  const T Z = T(0.5) * (-E.b2 * dw[2] + E.b1 * dw[3]);
  const T Zb = T(0.5) * E.sg * (-E.b2 * dw[5] + E.b1 * dw[6]) * E.isr;
  q[0] = n * (Xf + Yf);
  q[1] = Z + Zb;
  q[2] = n * (Xs + Ys);
  q[3] = dw[0] - dw[4] * E.ia2;
  q[4] = n * (Xs - Ys);
  q[5] = Z - Zb;
  q[6] = n * (Xf - Yf);
}
template <class T, class O>
__device__ __forceinline__ void eig_left(O& o, const Eig<T>& E, const EigCoef<T>& C, const T* dw, T* q) {
  if constexpr (sizeof(T) != 4) {
    const T bv = times_sign<T>(o.mul(E.b1, dw[2]) + E.b2 * dw[3], E.sg);
    const T bb = o.mul(E.b1, dw[5]) + E.b2 * dw[6];
    const T Xf = o.mul(C.fp, dw[4]) + C.fb * bb, Yf = o.mul(C.su, bv) - C.fu * dw[1];
    const T Xs = o.mul(C.sp, dw[4]) - C.sb * bb, Ys = o.mul(C.su, dw[1]) + C.fu * bv;
    const T Z = o.mul(C.h1, dw[3]) - C.h2 * dw[2];
    const T Zb = o.mul(C.z1, dw[6]) - C.z2 * dw[5];
    q[0] = Xf + Yf;
    q[1] = Z + Zb;
    q[2] = Xs - Ys;
    q[3] = dw[0] - dw[4] * E.ia2;
    q[4] = Xs + Ys;
    q[5] = Z - Zb;
    q[6] = Xf - Yf;
  } else {
    eig_left_narrow<T>(E, dw, q);
  }
}

template <class T> __device__ __forceinline__ void eig_left(const Eig<T>& E, const EigCoef<T>& C, const T* dw, T* q) {
  Ops<T> o;
  eig_left<T>(o, E, C, dw, q);
}

// The eigensystem and its coefficients.  A cell whose operands leave the range
// of the integer-pipe functions here (a field below 1e-154) has these evaluated
// again out of line, and not its whole reconstruction.  Measured at 128^3 (FP64,
// fields of 1e-160 everywhere), ms per step with the whole cell evaluated again,
// and as here: PLMC 10.69 and 9.55 (library functions throughout: 10.59), PPMC
// 13.15 and 11.21 (12.52); with fields of order one 5.93 and 5.85, 7.28 and 7.24.
template <class T> struct EigSystem {
  Eig<T> E;
  EigCoef<T> C;
};
template <class T> __device__ __noinline__ void eig_again(T gamma, const T* w, T bn, EigSystem<T>& S) {
  Ops<T> o;
  eig_build<T>(o, gamma, w, bn, S.E);
  S.C = eig_coef<T>(o, S.E);
}
// (with a range test of its own: o's may be set already)
template <class T, class O>
__device__ __forceinline__ EigCoef<T> eig_system(const O&, T gamma, const T* w, T bn, Eig<T>& E) {
  O o;
  eig_build<T>(o, gamma, w, bn, E);
  EigCoef<T> C = eig_coef<T>(o, E);
  if constexpr (std::is_same<O, TryOps<double>>::value) {
    if (__any_sync(__activemask(), o.bad)) {
      if (o.bad) {
        T a[7];
#pragma unroll
        for (int q = 0; q < 7; ++q) a[q] = w[q];
        EigSystem<T> S;
        eig_again<T>(gamma, a, bn, S);
        E = S.E;
        C = S.C;
      }
    }
  }
  return C;
}

// primitive increments dw = R q
template <class T> __device__ __forceinline__ void eig_right(const Eig<T>& E, const T* q, T* dw) {
  const T fp = q[0] + q[6], fm = q[0] - q[6];
  const T sp = q[2] + q[4], sm = q[2] - q[4];
  const T ap = q[1] + q[5], am = q[1] - q[5];
  const T cfa = E.cf * E.af, csa = E.cs * E.as;
  const T K = E.af * fp + E.as * sp;
  dw[0] = E.rho * K + q[3];
  dw[1] = -cfa * fm - csa * sm;
  dw[2] = E.b1 * (E.Qs * fm - E.Qf * sm) - E.b2 * ap;
  dw[3] = E.b2 * (E.Qs * fm - E.Qf * sm) + E.b1 * ap;
  dw[4] = E.rho * E.a2 * K;
  const T ms = E.As * fp - E.Af * sp;
  const T ssr = times_sign<T>(E.sr, E.sg) * am;
  dw[5] = E.b1 * ms - E.b2 * ssr;
  dw[6] = E.b2 * ms + E.b1 * ssr;
}

template <class T> __device__ __forceinline__ T sgn0(T x) { return x > T(0) ? T(1) : (x < T(0) ? T(-1) : T(0)); }

// Sign tests and magnitude minima of the limiters.  The generic forms use
// floating-point instructions; for double they run on the bit patterns
// (integer pipes), because the FP64 pipe bounds the FP64 step on this GPU.
// Both give the same result for finite values whose products do not
// underflow.
template <class T> __device__ __forceinline__ bool pos_prod(T a, T b) { return a * b > T(0); }
template <class T> __device__ __forceinline__ bool neg_prod(T a, T b) { return a * b < T(0); }
template <class T> __device__ __forceinline__ T min_abs(T a, T b) { return fmin(fabs(a), fabs(b)); }
// sgn0(s) m for m >= 0
template <class T> __device__ __forceinline__ T with_sign(T s, T m) { return sgn0<T>(s) * m; }
template <class T> __device__ __forceinline__ bool abs_ge_twice(T a, T b) { return fabs(a) >= T(2) * fabs(b); }

// float pairs: on the signs of the leading floats (a product of pairs and its
// comparison take 8 instructions), and a sign flip for with_sign: PPMC
// reconstruction 12.1 -> 10.0 ms at 256^3
template <> __device__ __forceinline__ bool pos_prod<df>(df a, df b) {
  return ((__float_as_int(a.hi) ^ __float_as_int(b.hi)) >= 0) & (a.hi != 0.0f) & (b.hi != 0.0f);
}
template <> __device__ __forceinline__ bool neg_prod<df>(df a, df b) {
  return ((__float_as_int(a.hi) ^ __float_as_int(b.hi)) < 0) & (a.hi != 0.0f) & (b.hi != 0.0f);
}
template <> __device__ __forceinline__ df with_sign<df>(df s, df m) {
  const df r = s.hi < 0.0f ? df(-m.hi, -m.lo) : m;
  return s.hi == 0.0f ? df(0.0f, 0.0f) : r;
}
template <> __device__ __forceinline__ bool abs_ge_twice<df>(df a, df b) {
  return !(fabs(a) < df(2.0f * fabsf(b.hi), b.hi < 0.0f ? -2.0f * b.lo : 2.0f * b.lo));
}
template <> __device__ __forceinline__ bool pos_prod<double>(double a, double b) {
  const long long x = dbits(a), y = dbits(b);
  return ((x ^ y) >= 0) & ((x & kAbsBits) != 0) & ((y & kAbsBits) != 0);
}
template <> __device__ __forceinline__ bool neg_prod<double>(double a, double b) {
  const long long x = dbits(a), y = dbits(b);
  return ((x ^ y) < 0) & ((x & kAbsBits) != 0) & ((y & kAbsBits) != 0);
}
template <> __device__ __forceinline__ double min_abs<double>(double a, double b) {
  const int ha = __double2hiint(a) & 0x7fffffff, hb = __double2hiint(b) & 0x7fffffff;
  const int la = __double2loint(a), lb = __double2loint(b);
  const bool first = ha < hb || (ha == hb && (unsigned)la < (unsigned)lb);
  return __hiloint2double(first ? ha : hb, first ? la : lb);
}
template <> __device__ __forceinline__ double with_sign<double>(double s, double m) {
  const int hi = __double2hiint(s);
  const bool zero = ((hi & 0x7fffffff) | __double2loint(s)) == 0;
  return __hiloint2double(zero ? 0 : __double2hiint(m) | (hi & (int)0x80000000), zero ? 0 : __double2loint(m));
}
// |a| >= 2 |b|: the exponent of |b| raised by one (normal b; b = 0 stays 0)
template <> __device__ __forceinline__ bool abs_ge_twice<double>(double a, double b) {
  const long long x = dbits(a) & kAbsBits, y = dbits(b) & kAbsBits;
  return x >= (y ? y + (1LL << 52) : 0LL);
}

// ------------------------------------------------------- PLMC (Sec. 2.2.6) --
// wm, w0, wp: primitive 7-vectors of cells i-1, i, i+1; bn: cell-centred
// longitudinal field of cell i.  Outputs W_{L,i+1/2} and W_{R,i-1/2}.
// van Leer differences dG = 2 dL dR / (dL + dR) where dL dR > 0, else 0
// (reading D-5), for the 7 fields of one cell
template <class T, class O> __device__ __forceinline__ void van_leer7(O& o, const T* dL, const T* dR, T* dG) {
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    if constexpr (std::is_same<T, double>::value) {
      // a product that underflows gives 0, also where 1/s would overflow
      const bool act = pos_prod<T>(dL[q], dR[q]);
      const T pr = dL[q] * dR[q];
      const T g = twice_n<T>(pr) * o.rcp(act ? dL[q] + dR[q] : 1.0);
      dG[q] = (act && !is0<T>(pr)) ? g : T(0);
    } else if constexpr (std::is_same<T, df>::value) {
      // the sign from the product's leading float: pos_prod<df> holds for a
      // product that underflows, too, where 1/s may leave the float range
      const dfx pr = dL[q] * dR[q];
      dG[q] = pr.hi > 0.0f ? T(T(2) * pr * o.rcp(dL[q] + dR[q])) : T(0);
    } else {
      dG[q] = pos_prod<T>(dL[q], dR[q]) ? T(2) * (dL[q] * dR[q]) * o.rcp(dL[q] + dR[q]) : T(0);
    }
  }
}
template <class T> __device__ __forceinline__ void van_leer7(const T* dL, const T* dR, T* dG) {
  Ops<T> o;
  van_leer7<T>(o, dL, dR, dG);
}

template <class T, class O>
__device__ __forceinline__ void plmc(O& o, T gamma, const T* wm, const T* w0, const T* wp, T bn, T* wl, T* wr) {
  T dL[7], dR[7], dG[7];
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    dL[q] = w0[q] - wm[q];
    dR[q] = wp[q] - w0[q];
  }
  van_leer7<T>(o, dL, dR, dG);
  Eig<T> E;
  const EigCoef<T> C = eig_system<T>(o, gamma, w0, bn, E);
  T aL[7], aR[7], aC[7], aG[7], am[7], dW[7];
  eig_left<T>(o, E, C, dL, aL);
  eig_left<T>(o, E, C, dR, aR);
  eig_left<T>(o, E, C, dG, aG);
  // the centred difference (W_{i+1} - W_{i-1})/2 projected: L is linear, so
  // its amplitudes are the mean of the left and right ones
#pragma unroll
  for (int q = 0; q < 7; ++q) aC[q] = half<T>(aL[q] + aR[q]);
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    if (pos_prod<T>(aL[q], aR[q])) {
      const T m = min_abs<T>(min_abs<T>(twice_n<T>(aL[q]), twice_n<T>(aR[q])), min_abs<T>(aC[q], aG[q]));
      am[q] = with_sign<T>(aC[q], m);
    } else {
      am[q] = T(0);
    }
  }
  eig_right<T>(E, am, dW);
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    wl[q] = w0[q] + half_f<T>(dW[q]);
    wr[q] = w0[q] - half_f<T>(dW[q]);
  }
}

// PLM with the limiter applied to the primitive differences themselves (the
// variant named at the end of Sec. 2.2.6): the same slopes and limiter as
// plmc, without the characteristic projection.
template <class T>
__device__ __forceinline__ void plm_prim(const T* wm, const T* w0, const T* wp, T* wl, T* wr) {
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    const T dL = w0[q] - wm[q], dR = wp[q] - w0[q], dC = T(0.5) * (wp[q] - wm[q]);
    const T pr = dL * dR;
    T dm = T(0);
    if (pr > T(0)) {
      const T dG = T(2) * pr * trcp<T>(dL + dR);
      dm = sgn0<T>(dC) * fmin(fmin(T(2) * fabs(dL), T(2) * fabs(dR)), fmin(fabs(dC), fabs(dG)));
    }
    wl[q] = w0[q] + T(0.5) * dm;
    wr[q] = w0[q] - T(0.5) * dm;
  }
}

// ------------------------------------------------------- PPMC (Sec. 2.2.6) --
// Fourth-order interface values, Colella & Sekora (2008) interface limiter,
// McCorquodale & Colella (2011) cell limiter (C = 1.25), in characteristic
// deviations q_m - q_0 = L (W_m - W_0) of cell i.
// sgn(x) min(|x|, C|y|, C|z|) when x, y, z share a strict sign, else 0 (C = 1.25)
// (C min(|y|, |z|) is min(C|y|, C|z|) exactly: a rounded product is monotone)
template <class T> __device__ __forceinline__ T d2lim3(T x, T y, T z) {
  if (pos_prod<T>(x, y) && pos_prod<T>(x, z))
    return with_sign<T>(x, min_abs<T>(x, T(1.25) * min_abs<T>(y, z)));
  return T(0);
}
template <class T> __device__ __forceinline__ T d2lim4(T x, T y, T z, T t) {
  if (pos_prod<T>(x, y) && pos_prod<T>(x, z) && pos_prod<T>(x, t))
    return with_sign<T>(x, min_abs<T>(x, T(1.25) * min_abs<T>(y, min_abs<T>(z, t))));
  return T(0);
}

// v (v - x) > 0: v lies beyond x as seen from zero.  (No difference is formed:
// a comparison, for double on the bit patterns.)
template <class T> __device__ __forceinline__ bool beyond(T v, T x) { return gt0<T>(v) ? v > x : (lt0<T>(v) && v < x); }
template <> __device__ __forceinline__ bool beyond<double>(double v, double x) {
  const long long s = dbits(v) & kNegZero, m = dbits(v) & kAbsBits;
  return ((dbits(x) ^ s) < m) & (m != 0);
}

// The limiter for double and float pairs: the interface limiter's
// sgn(u) min(3|u|, C|y|, C|z|)/6 as sgn(u) min(|u|/2, (C/6) min(|y|, |z|)),
// the cell limiter's ratio min(6|s|, C m)/(6|s|) as 1 where |s| <= (C/6) m,
// else (C/6) m / |s|, and the range tests as comparisons.  (An interface
// limit (C/6) min(|y|, |z|) not below |u|/2 leaves x/2 - u/2 = v: the value stays.)
template <class T> __device__ __forceinline__ T lim_face(T x, T v, T y, T z) {
  const T u = sub_twice<T>(x, v);
  const T c = from_d<T>(1.25 / 6.0) * min_abs<T>(y, z);
  if (!(pos_prod<T>(u, y) && pos_prod<T>(u, z))) return half<T>(x);
  return nonneg_lt<T>(c, absv<T>(half<T>(u))) ? T(half<T>(x) - with_sign<T>(u, c)) : v;
}
template <class T> __device__ __forceinline__ void ppm_one_wide(const T* q, T& qm, T& qp) {
  const T c7 = from_d<T>(7.0 / 12.0), c1 = from_d<T>(1.0 / 12.0);
  const T a = q[0], b = q[1], d = q[3], e = q[4];  // cells i-2, i-1, i+1, i+2
  qm = c7 * b - c1 * (a + d);
  qp = c7 * d - c1 * (b + e);
  const T d2m1 = sub_twice<T>(a, b);
  const T d20 = b + d;
  const T d2p1 = sub_twice<T>(e, d);
  // both interfaces share one body (see ppm_one)
  const bool lm = beyond<T>(qm, b), lp = beyond<T>(qp, d);
  if (lm || lp) {
    const T lim = lim_face<T>(pick<T>(lm, b, d), pick<T>(lm, qm, qp), pick<T>(lm, d2m1, d20), pick<T>(lm, d20, d2p1));
    if (lm) qm = lim;
    else qp = lim;
    if (lm && lp) qp = lim_face<T>(d, qp, d20, d2p1);
  }
  if (!neg_prod<T>(qm, qp) || !neg_prod<T>(b, d)) {
    const T s = qm + qp;  // a sixth of the interface values' curvature
    const bool same = pos_prod<T>(s, d2m1) && pos_prod<T>(s, d20) && pos_prod<T>(s, d2p1);
    const T t = from_d<T>(1.25 / 6.0) * min_abs<T>(d2m1, min_abs<T>(d20, d2p1));
    const T sa = absv<T>(s);
    if (!same) {
      qm = T(0);
      qp = T(0);
    } else if (nonneg_lt<T>(t, sa)) {
      const T r = ratio_le1<T>(t, sa);
      qm = r * qm;
      qp = r * qp;
    }
  } else {
    const T m0 = qm;
    if (abs_ge_twice<T>(qm, qp)) qm = neg<T>(twice_n<T>(qp));
    if (abs_ge_twice<T>(qp, m0)) qp = neg<T>(twice_n<T>(m0));
  }
}

// a / b, b != 0
template <class T> __device__ __forceinline__ T ratio_any(T a, T b) { return a / b; }
template <> __device__ __forceinline__ double ratio_any<double>(double a, double b) {
  return ratio_le1<double>(a, b);
}

// q[0..4] = characteristic deviations of cells i-2..i+2 from cell i (q[2] = 0);
// returns the limited deviations of the two interface values.  Written for
// the deviation form: the centre's zero is not added, subtracted or
// multiplied, and sign flips and doublings are exact bit operations, so
// only the arithmetic the limiter needs reaches the FP64 pipe.  Same values
// as the formulas with q[2] kept, up to the sign of zero results.
template <class T> __device__ __forceinline__ void ppm_one_narrow(const T* q, T& qm, T& qp) {
  const T c7 = from_d<T>(7.0 / 12.0), c1 = from_d<T>(1.0 / 12.0), c6 = from_d<T>(1.0 / 6.0);
  const T a = q[0], b = q[1], d = q[3], e = q[4];  // cells i-2, i-1, i+1, i+2
  qm = c7 * b - c1 * (a + d);
  qp = c7 * d - c1 * (b + e);
  const T d2m1 = a - T(2) * b;
  const T d20 = b + d;
  const T d2p1 = e - T(2) * d;
  // interface limiter where the value leaves the range of its two cells.
  // Both interfaces share one body, fed the operands of the lower interface
  // where it needs limiting, else of the upper: a warp whose lanes limit
  // different interfaces runs it once; a second pass runs only where a lane
  // limits both.
  const bool lm = pos_prod<T>(qm - b, qm), lp = neg_prod<T>(qp, d - qp);
  if (lm || lp) {
    const T x = lm ? b : d, v = lm ? qm : qp, y = lm ? d2m1 : d20, z = lm ? d20 : d2p1;
    const T lim = T(0.5) * x - d2lim3<T>(T(3) * (x - T(2) * v), y, z) * c6;
    if (lm) qm = lim;
    else qp = lim;
    if (lm && lp) qp = T(0.5) * d - d2lim3<T>(T(3) * (d - T(2) * qp), d20, d2p1) * c6;
  }
  // cell limiter: at an extremum both deviations scale by the curvature
  // ratio, elsewhere an overshoot is clipped to twice the other deviation
  if (!neg_prod<T>(qm, qp) || !neg_prod<T>(b, d)) {
    const T d2f = T(6) * (qm + qp);
    T r = T(0);
    // (|d2lim4 / d2f| <= 1: a reciprocal where d2f is far from the
    // underflow range, else the division)
    if (!is0<T>(d2f)) r = ratio_le1<T>(d2lim4<T>(d2f, d2m1, d20, d2p1), d2f);
    qm = r * qm;
    qp = r * qp;
  } else {
    const T m0 = qm;
    if (abs_ge_twice<T>(qm, qp)) qm = neg<T>(twice_n<T>(qp));
    if (abs_ge_twice<T>(qp, m0)) qp = neg<T>(twice_n<T>(m0));
  }
}

template <class T> __device__ __forceinline__ void ppm_one(const T* q, T& qm, T& qp) {
  if constexpr (sizeof(T) != 4) ppm_one_wide<T>(q, qm, qp);
  else ppm_one_narrow<T>(q, qm, qp);
}

// The limiter as a call (double and float pairs): seven inlined copies outgrow
// the instruction cache (1.2 warps stalled on instruction fetch per issue in
// the FP64 kernel).  Measured at 256^3: float pairs 10.0 -> 9.4 ms, FP64 45.1 ->
// 40.6 ms with the inlined products of the eigensystem.
template <class T> struct LimitedPair {
  T m, p;
};
template <class T> __device__ __noinline__ LimitedPair<T> ppm_one_call(T a, T b, T d, T e) {
  const T q[5] = {a, b, T(0), d, e};
  LimitedPair<T> r;
  ppm_one<T>(q, r.m, r.p);
  return r;
}

template <class T, class O>
__device__ __forceinline__ void ppmc(O& o, T gamma, const T (*w)[7], T bn, T* wl, T* wr) {
  Eig<T> E;
  const EigCoef<T> C = eig_system<T>(o, gamma, w[2], bn, E);
  T qs[5][7];
#pragma unroll
  for (int m = 0; m < 5; ++m) {
    if (m == 2) {
#pragma unroll
      for (int c = 0; c < 7; ++c) qs[2][c] = T(0);
      continue;
    }
    T d[7];
#pragma unroll
    for (int c = 0; c < 7; ++c) d[c] = w[m][c] - w[2][c];
    eig_left<T>(o, E, C, d, qs[m]);
  }
  T dm[7], dp[7];
#pragma unroll
  for (int c = 0; c < 7; ++c) {
    const T col[5] = {qs[0][c], qs[1][c], T(0), qs[3][c], qs[4][c]};
    T qm, qp;
    if constexpr (sizeof(T) != 4) {
      const LimitedPair<T> r = ppm_one_call<T>(col[0], col[1], col[3], col[4]);
      qm = r.m;
      qp = r.p;
    } else {
      ppm_one<T>(col, qm, qp);
    }
    dm[c] = qm;
    dp[c] = qp;
  }
  T Wm[7], Wp[7];
  eig_right<T>(E, dm, Wm);
  eig_right<T>(E, dp, Wp);
#pragma unroll
  for (int c = 0; c < 7; ++c) {
    wl[c] = w[2][c] + Wp[c];
    wr[c] = w[2][c] + Wm[c];
  }
}

}  // namespace mhd
