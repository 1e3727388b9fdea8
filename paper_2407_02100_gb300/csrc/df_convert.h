// Conversions between double and double-float (a value hi + lo of two
// floats) by integer operations on the IEEE-754 bit patterns.  GB300 runs
// FP64 instructions and the F2F conversions to and from FP64 at about 1/74
// of its FP32 rate, so the double-float sweep of FP64 problems converts its
// inputs and outputs with these integer forms instead.  Host and device
// compile the same code (it is checked on the host against exact
// arithmetic).
//
// to_df: hi is x rounded to 24 significant bits (halves away from zero), lo
//   the remaining signed 29 bits rounded to 24 (|lo| <= ulp(hi) / 2), so
//   hi + lo = x to 2^-49 relative.  Exact
//   integer path for 2^-74 <= |x| < 2^115; other magnitudes (zero aside) take
//   the rounded FP64 path; zero and FP64 subnormals give (0, 0).  The range
//   of double-float is that of float: below |x| = 2^-100 lo is a float
//   subnormal and the error becomes absolute (at most 2^-149); from 2^128 on
//   hi is infinite.
// from_df: hi + lo rounded to double (to 2^-52 relative) for hi normal and at
//   least 2^-75 and |lo| <= ulp(hi); other cases use the FP64 sum.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

namespace gmg {
namespace dfconv {

#if defined(__CUDA_ARCH__)
#define GMG_DFC __device__ __forceinline__
// the FP64 fallbacks live in functions of their own, so that the compiler
// does not predicate their FP64 instructions into the common path
__device__ __noinline__ void to_df_rounded(double x, float& hi, float& lo) {
  if (((uint64_t)__double_as_longlong(x) >> 52 & 0x7FF) == 0) {
    hi = lo = 0.f;
    return;
  }
  hi = __double2float_rn(x);
  lo = __double2float_rn(x - (double)hi);
}
__device__ __noinline__ double from_df_fp64(float hi, float lo) { return (double)hi + (double)lo; }
__device__ __forceinline__ float i2f_rn(int32_t v) { return __int2float_rn(v); }
__device__ __forceinline__ int32_t f2i_rn(float v) { return __float2int_rn(v); }
__device__ __forceinline__ float fmul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ uint64_t dbits(double x) { return (uint64_t)__double_as_longlong(x); }
__device__ __forceinline__ double bitsd(uint64_t b) { return __longlong_as_double((long long)b); }
__device__ __forceinline__ uint32_t fbits(float x) { return __float_as_uint(x); }
__device__ __forceinline__ float bitsf(uint32_t b) { return __uint_as_float(b); }
#else
#define GMG_DFC inline
inline float i2f_rn(int32_t v) { return (float)v; }
inline int32_t f2i_rn(float v) { return (int32_t)std::lrint(v); }
inline float fmul_rn(float a, float b) { return a * b; }
inline uint64_t dbits(double x) { uint64_t b; std::memcpy(&b, &x, 8); return b; }
inline double bitsd(uint64_t b) { double x; std::memcpy(&x, &b, 8); return x; }
inline uint32_t fbits(float x) { uint32_t b; std::memcpy(&b, &x, 4); return b; }
inline float bitsf(uint32_t b) { float x; std::memcpy(&x, &b, 4); return x; }
inline void to_df_rounded(double x, float& hi, float& lo) {
  if ((dbits(x) >> 52 & 0x7FF) == 0) {  // zero or FP64 subnormal (below the float range)
    hi = lo = 0.f;
    return;
  }
  hi = (float)x;
  lo = (float)(x - (double)hi);
}
inline double from_df_fp64(float hi, float lo) { return (double)hi + (double)lo; }
#endif

GMG_DFC void to_df(double x, float& hi, float& lo) {
  const uint64_t b = dbits(x);
  const uint32_t top = (uint32_t)(b >> 32);
  const uint32_t e = (top >> 20) & 0x7FFu;  // biased exponent
  if (e - 949u > 188u) {  // outside the exact integer path: zero, or rounded conversions
    to_df_rounded(x, hi, lo);
    return;
  }
  const uint32_t sign = top & 0x80000000u;
  // exponent and significand of |x|, rounded at bit 29 (a carry moves into the
  // exponent), with the exponent rebased to float's
  const uint64_t m = (b & 0x7FFFFFFFFFFFFFFFull) + (1ull << 28);
  hi = bitsf(sign | ((uint32_t)(m >> 29) - (896u << 23)));
  // x - hi = (low 29 bits, signed) * 2^(e - 1075) with the sign of x; e >= 949
  // keeps the scale 2^(e - 1075) a normal float
  lo = fmul_rn(i2f_rn((int32_t)((uint32_t)b << 3) >> 3), bitsf(sign | ((e - 948u) << 23)));
}

GMG_DFC double from_df(float hi, float lo) {
  const uint32_t hb = fbits(hi);
  // lo in units of the double's last place at hi's exponent, 2^(eh - 127 - 52),
  // negated where hi is negative: an integer of at most 2^29.  306 - eh as an
  // exponent, with hi's sign: the subtraction borrows the sign bit through.
  const float t = fmul_rn(lo, bitsf(0x99000000u - (hb & 0xFF800000u)));
  if ((hb & 0x7FFFFFFFu) - (52u << 23) >= 203u << 23 || !(fabsf(t) <= 536870912.f))
    return from_df_fp64(hi, lo);  // zero, tiny, inf or nan, or a large lo
  int32_t L = f2i_rn(t);
  // below a power of two the last place is half as large
  if ((hb & 0x7FFFFFu) == 0 && L < 0) L *= 2;
  // |hi| as a double's bits (sign apart), plus lo: a carry moves into the exponent
  const uint64_t S = (uint64_t)(hb & 0x7FFFFFFFu) * 0x20000000u + (uint64_t)(int64_t)L;
  return bitsd(S + ((uint64_t)(896u << 20 | (hb & 0x80000000u)) << 32));
}

#undef GMG_DFC

}  // namespace dfconv
}  // namespace gmg
