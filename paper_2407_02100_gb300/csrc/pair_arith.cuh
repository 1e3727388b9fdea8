// Two-wide FP32 arithmetic (add/sub/mul/fma.rn.f32x2) and double-float
// arithmetic on pairs of values built from it.
//
// The FP32 pipe of an SM takes 128 lane operations a cycle whether they come
// as scalar or as two-wide instructions (measured: 1.09 against 2.11 cycles of
// a scheduler per warp instruction), but a two-wide one spends a single issue
// slot on both.  The double-float kernels were bound by issue at 46 % of the
// FP32 pipe: beside every FP32 operation they issue loads, conversions and
// coefficient moves.  A thread that carries the same line of two patches (or
// faces) issues half of the arithmetic and half of the coefficient loads per
// patch, and everything else fits into the slots that frees.
#pragma once
#include "df_arith.cuh"

namespace gmg {
namespace {

// two floats in a 64-bit register pair, x the low half
struct f2 {
  unsigned long long v;
};

__device__ __forceinline__ f2 f2_make(float x, float y) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ f2 f2_dup(float x) { return f2_make(x, x); }
__device__ __forceinline__ float f2_x(f2 a) { return __uint_as_float((unsigned)a.v); }
__device__ __forceinline__ float f2_y(f2 a) { return __uint_as_float((unsigned)(a.v >> 32)); }
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// The rounded product.  The assembler contracts a two-wide multiplication and
// the addition that uses it into one fused operation, .rn or not (seen as a
// lost TwoSum), so a product that has to be rounded by itself is a fused
// operation with a zero that the compiler cannot see.
__constant__ unsigned long long c_zero2 = 0;
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) { return f2_fma(a, b, f2{c_zero2}); }

// Double-float values of two patches; a coefficient shared by both; a Dot2
// accumulator.  The operations are those of df_arith.cuh, lane by lane.
struct df2 {
  f2 hi, lo;
};
struct df2_coef {
  f2 h, l;
};
struct df2_acc {
  f2 s, e;
};

__device__ __forceinline__ df2 df2_make(dfv a, dfv b) { return {f2_make(a.hi, b.hi), f2_make(a.lo, b.lo)}; }
__device__ __forceinline__ dfv df2_x(df2 a) { return {f2_x(a.hi), f2_x(a.lo)}; }
__device__ __forceinline__ dfv df2_y(df2 a) { return {f2_y(a.hi), f2_y(a.lo)}; }

__device__ __forceinline__ df2 df2_norm(f2 a, f2 b) {  // df_fast_two_sum
  const f2 s = f2_add(a, b);
  return {s, f2_sub(b, f2_sub(s, a))};
}
__device__ __forceinline__ df2 df2_add(df2 a, df2 b) {
  const f2 s = f2_add(a.hi, b.hi), bb = f2_sub(s, a.hi);
  const f2 t = f2_add(f2_sub(a.hi, f2_sub(s, bb)), f2_sub(b.hi, bb));
  return df2_norm(s, f2_add(t, f2_add(a.lo, b.lo)));
}
__device__ __forceinline__ df2 df2_sub(df2 a, df2 b) {
  const f2 s = f2_sub(a.hi, b.hi), bb = f2_sub(s, a.hi);
  const f2 t = f2_sub(f2_sub(a.hi, f2_sub(s, bb)), f2_add(b.hi, bb));
  return df2_norm(s, f2_add(t, f2_sub(a.lo, b.lo)));
}
// c x; the negated product's error comes from the product itself (0 - p)
__device__ __forceinline__ df2_acc df2_acc_first(df2_coef c, df2 x) {
  const f2 p = f2_mul(c.h, x.hi);
  f2 e = f2_fma(c.h, x.hi, f2_sub(f2{0}, p));
  e = f2_fma(c.h, x.lo, e);
  return {p, f2_fma(c.l, x.hi, e)};
}
// c x for a coefficient of one float
__device__ __forceinline__ df2_acc df2_acc_scaled(f2 c, df2 x) {
  const f2 p = f2_mul(c, x.hi);
  return {p, f2_fma(c, x.lo, f2_fma(c, x.hi, f2_sub(f2{0}, p)))};
}
// acc += c x (df_acc_add; nb = -b there)
__device__ __forceinline__ void df2_acc_add(df2_acc& a, df2_coef c, df2 x) {
  const f2 p = f2_mul(c.h, x.hi);
  const f2 S = f2_add(a.s, p);
  const f2 nb = f2_sub(a.s, S);
  f2 t = f2_fma(c.h, x.lo, f2_sub(a.s, f2_add(S, nb)));
  t = f2_fma(c.l, x.hi, t);
  a.e = f2_add(a.e, f2_add(t, f2_fma(c.h, x.hi, nb)));
  a.s = S;
}
__device__ __forceinline__ df2 df2_acc_value(df2_acc a) { return df2_norm(a.s, a.e); }

// The arithmetics of the pair kernels, under the same names: a value, an
// accumulator, a coefficient and their forms in shared and constant memory, and
// the patches W that a thread carries.  SoloDF does the operations of a lane of
// PairDF in the same order, bit for bit.
struct PairDF {  // double-float (FP64 problems)
  static constexpr int W = 2;
  using T = double;
  using val = df2;
  using acc = df2_acc;
  using coef = df2_coef;
  using mem = float4;  // (hi, hi, lo, lo)
  using tab = float4;  // (h, h, l, l)
  static __device__ __forceinline__ val load(const mem& a) {
    const ulonglong2 v = reinterpret_cast<const ulonglong2&>(a);
    return {{v.x}, {v.y}};
  }
  static __device__ __forceinline__ void store(mem& a, val v) {
    reinterpret_cast<ulonglong2&>(a) = make_ulonglong2(v.hi.v, v.lo.v);
  }
  static __device__ __forceinline__ coef coefficient(const tab& c) {
    const ulonglong2 v = reinterpret_cast<const ulonglong2&>(c);
    return {{v.x}, {v.y}};
  }
  static void make_tab(tab& c, double, float h, float l) { c = make_float4(h, h, l, l); }
  static __device__ __forceinline__ acc zero() { return {{0}, {0}}; }
  static __device__ __forceinline__ acc first(coef c, val x) { return df2_acc_first(c, x); }
  static __device__ __forceinline__ void add(acc& a, coef c, val x) { df2_acc_add(a, c, x); }
  static __device__ __forceinline__ val value(acc a) { return df2_acc_value(a); }
  static __device__ __forceinline__ val sum(val a, val b) { return df2_add(a, b); }
  static __device__ __forceinline__ val diff(val a, val b) { return df2_sub(a, b); }
  static __device__ __forceinline__ acc scaled(float c, val x) { return df2_acc_scaled(f2_dup(c), x); }
  static __device__ __forceinline__ val pack(T a, T b) { return df2_make(df_from_double(a), df_from_double(b)); }
  static __device__ __forceinline__ val pack_neg(T a, T b) {  // (a negated double would be an FP64 instruction)
    return df2_make(df_neg(df_from_double(a)), df_neg(df_from_double(b)));
  }
  // times entry i of the FD diagonal (n entries, followed by their float pairs)
  static __device__ __forceinline__ val diagonal(const T* dinv, int n, int i, val v) {
    const float2 d = __ldg(reinterpret_cast<const float2*>(dinv + n) + i);
    return value(first({f2_dup(d.x), f2_dup(d.y)}, v));
  }
  static __device__ __forceinline__ T x(val v) { return df_to_double(df2_x(v)); }
  static __device__ __forceinline__ T y(val v) { return df_to_double(df2_y(v)); }
};
struct SoloDF {  // double-float, one patch
  static constexpr int W = 1;
  using T = double;
  using val = dfv;
  using acc = df_acc;
  struct coef {
    float h, l;
  };
  using mem = float2;  // (hi, lo)
  using tab = float2;  // (h, l)
  static __device__ __forceinline__ val load(const mem& a) { return {a.x, a.y}; }
  static __device__ __forceinline__ void store(mem& a, val v) { a = make_float2(v.hi, v.lo); }
  static __device__ __forceinline__ coef coefficient(const tab& c) { return {c.x, c.y}; }
  // a value as a coefficient (of its patch)
  static __device__ __forceinline__ coef weight(const mem& a) { return {a.x, a.y}; }
  static void make_tab(tab& c, double, float h, float l) { c = make_float2(h, l); }
  static __device__ __forceinline__ acc zero() { return {0.f, 0.f}; }
  static __device__ __forceinline__ acc first(coef c, val x) { return df_acc_first(c.h, c.l, x); }
  static __device__ __forceinline__ void add(acc& a, coef c, val x) { df_acc_add(a, c.h, c.l, x); }
  static __device__ __forceinline__ val value(acc a) { return df_acc_value(a); }
  static __device__ __forceinline__ val sum(val a, val b) { return df_add(a, b); }
  static __device__ __forceinline__ val diff(val a, val b) { return df_add(a, df_neg(b)); }
  static __device__ __forceinline__ acc scaled(float c, val x) { return df_acc_scaled(c, x); }
  static __device__ __forceinline__ val pack(T a, T) { return df_from_double(a); }
  static __device__ __forceinline__ val pack_neg(T a, T) { return df_neg(df_from_double(a)); }
  static __device__ __forceinline__ val diagonal(const T* dinv, int n, int i, val v) {
    const float2 d = __ldg(reinterpret_cast<const float2*>(dinv + n) + i);
    return value(first({d.x, d.y}, v));
  }
  static __device__ __forceinline__ T x(val v) { return df_to_double(v); }
  static __device__ __forceinline__ T y(val v) { return df_to_double(v); }
};
struct PairF32 {  // single precision
  static constexpr int W = 2;
  using T = float;
  using val = f2;
  using acc = f2;
  using coef = f2;
  using mem = float2;
  using tab = float2;  // (c, c)
  static __device__ __forceinline__ val load(const mem& a) { return {reinterpret_cast<const unsigned long long&>(a)}; }
  static __device__ __forceinline__ void store(mem& a, val v) { reinterpret_cast<unsigned long long&>(a) = v.v; }
  static __device__ __forceinline__ coef coefficient(const tab& c) { return load(c); }
  static __device__ __forceinline__ coef weight(const mem& a) { return load(a); }
  static void make_tab(tab& c, double v, float, float) { c.x = c.y = (float)v; }
  static __device__ __forceinline__ acc zero() { return {0}; }
  static __device__ __forceinline__ acc first(coef c, val x) { return f2_fma(c, x, f2{0}); }
  static __device__ __forceinline__ void add(acc& a, coef c, val x) { a = f2_fma(c, x, a); }
  static __device__ __forceinline__ val value(acc a) { return a; }
  static __device__ __forceinline__ val sum(val a, val b) { return f2_add(a, b); }
  static __device__ __forceinline__ val diff(val a, val b) { return f2_sub(a, b); }
  static __device__ __forceinline__ acc scaled(float c, val x) { return f2_fma(f2_dup(c), x, f2{0}); }
  static __device__ __forceinline__ val pack(T a, T b) { return f2_make(a, b); }
  static __device__ __forceinline__ val pack_neg(T a, T b) { return f2_make(-a, -b); }
  static __device__ __forceinline__ val diagonal(const T* dinv, int, int i, val v) {
    return f2_fma(f2_dup(__ldg(dinv + i)), v, f2{0});
  }
  static __device__ __forceinline__ T x(val v) { return f2_x(v); }
  static __device__ __forceinline__ T y(val v) { return f2_y(v); }
};

}  // namespace
}  // namespace gmg
