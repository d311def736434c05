// Double-float ("df64") arithmetic on the FP32 pipe: a value is hi + lo with two floats, |lo| <=
// ulp(hi)/2, about 48 significant bits.  Built from the published error-free transformations:
// Knuth's two-sum (TAOCP vol. 2, 4.2.2) and the FMA form of Dekker's two-product (Dekker 1971).
// Products are accumulated lazily: the exact rounding error of each hi*hi product and the hi*lo
// cross terms go into the low word, which is renormalised once at the end of a sum.
#pragma once
#include <cuda_runtime.h>

namespace fthms {

struct df {
  float hi, lo;
};

// Complex double-float, laid out as float4 (re.hi, re.lo, im.hi, im.lo).
__device__ __forceinline__ float4 df_split2(double2 v) {
  const float rh = __double2float_rn(v.x);
  const float ih = __double2float_rn(v.y);
  return make_float4(rh, __double2float_rn(v.x - (double)rh), ih, __double2float_rn(v.y - (double)ih));
}

__device__ __forceinline__ double2 df_join2(float4 v) {
  return make_double2((double)v.x + (double)v.y, (double)v.z + (double)v.w);
}

// The _rn intrinsics keep every operation of the error-free transformations separately rounded (the
// compiler never contracts them into FMAs).
// s + e exactly (Knuth two-sum).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float v = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
}

// s + e exactly for |a| >= |b|.
__device__ __forceinline__ void quick_two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
}

// Running compensated sum: hi carries the rounded sum, lo the accumulated errors and low parts.
struct dfacc {
  float hi = 0.f, lo = 0.f;
  // += (ah + al) * (bh + bl), dropping al * bl
  __device__ __forceinline__ void mac(float ah, float al, float bh, float bl) {
    const float p = __fmul_rn(ah, bh);
    float e = fmaf(ah, bh, -p);
    e = fmaf(ah, bl, e);
    e = fmaf(al, bh, e);
    float s, t;
    two_sum(hi, p, s, t);
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(t, e));
  }
  __device__ __forceinline__ void add(float h, float l) {
    float s, t;
    two_sum(hi, h, s, t);
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(t, l));
  }
  __device__ __forceinline__ df value() const {
    df r;
    quick_two_sum(hi, lo, r.hi, r.lo);
    return r;
  }
};

// Double-float scalar arithmetic (a value is hi + lo): products from the FMA two-product with the
// cross terms, sums from two Knuth two-sums (the accurate form, safe under cancellation).
__device__ __forceinline__ df df_from(double v) {
  const float h = __double2float_rn(v);
  return df{h, __double2float_rn(v - (double)h)};
}
__device__ __forceinline__ df df_mul(df a, df b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  df r;
  quick_two_sum(p, e, r.hi, r.lo);
  return r;
}
__device__ __forceinline__ df df_add(df a, df b) {
  float s, e, t, f;
  two_sum(a.hi, b.hi, s, e);
  two_sum(a.lo, b.lo, t, f);
  e = __fadd_rn(e, t);
  quick_two_sum(s, e, s, e);
  e = __fadd_rn(e, f);
  df r;
  quick_two_sum(s, e, r.hi, r.lo);
  return r;
}
__device__ __forceinline__ df df_neg(df a) { return df{-a.hi, -a.lo}; }
__device__ __forceinline__ df df_sub(df a, df b) { return df_add(a, df_neg(b)); }

// a * b + c * d with one two-sum on the rounded products (their exact errors and the hi * lo cross
// terms added to the low word): error about 2^-46 (|ab| + |cd|).  Enough where accuracy is judged
// against the norm of a whole vector, as in the butterflies of an FFT.
__device__ __forceinline__ df df_dot2(df a, df b, df c, df d) {
  const float p = __fmul_rn(a.hi, b.hi), q = __fmul_rn(c.hi, d.hi);
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  float f = fmaf(c.hi, d.hi, -q);
  f = fmaf(c.hi, d.lo, f);
  f = fmaf(c.lo, d.hi, f);
  float s, t;
  two_sum(p, q, s, t);
  t = __fadd_rn(t, __fadd_rn(e, f));
  df r;
  quick_two_sum(s, t, r.hi, r.lo);
  return r;
}
// a + b with one two-sum on the high words; error about 2^-46 (|a| + |b|), as df_dot2.
__device__ __forceinline__ df df_add_fast(df a, df b) {
  float s, t;
  two_sum(a.hi, b.hi, s, t);
  t = __fadd_rn(t, __fadd_rn(a.lo, b.lo));
  df r;
  quick_two_sum(s, t, r.hi, r.lo);
  return r;
}

// a / b: the FP32 quotient corrected once with the double-float remainder (error about 2^-46).
__device__ __forceinline__ df df_div(df a, df b) {
  const float q1 = __fdiv_rn(a.hi, b.hi);
  const df r = df_sub(a, df_mul(b, df{q1, 0.f}));
  df q;
  quick_two_sum(q1, __fdiv_rn(r.hi, b.hi), q.hi, q.lo);
  return q;
}

// Complex double-float (float4 layout) for the mixed-form FFT butterflies.
__device__ __forceinline__ float4 dfc_mul(float4 a, float4 b) {
  const df re = df_dot2(df{a.x, a.y}, df{b.x, b.y}, df{-a.z, -a.w}, df{b.z, b.w});
  const df im = df_dot2(df{a.x, a.y}, df{b.z, b.w}, df{a.z, a.w}, df{b.x, b.y});
  return make_float4(re.hi, re.lo, im.hi, im.lo);
}
__device__ __forceinline__ float4 dfc_add(float4 a, float4 b) {
  const df re = df_add_fast(df{a.x, a.y}, df{b.x, b.y}), im = df_add_fast(df{a.z, a.w}, df{b.z, b.w});
  return make_float4(re.hi, re.lo, im.hi, im.lo);
}
__device__ __forceinline__ float4 dfc_sub(float4 a, float4 b) {
  const df re = df_add_fast(df{a.x, a.y}, df{-b.x, -b.y}), im = df_add_fast(df{a.z, a.w}, df{-b.z, -b.w});
  return make_float4(re.hi, re.lo, im.hi, im.lo);
}

// A double constant as a double-float pair, folded at compile time when used in a constant expression.
__host__ __device__ constexpr df df_const(double v) { return df{(float)v, (float)(v - (double)(float)v)}; }

// sin x and cos x for |x| <= 1 in double-float: the Taylor series (truncation below 2e-20, as for the
// FP64 version) by Horner's rule in u = x^2 with the coefficients (-1)^k/(2k+1)! and (-1)^k/(2k)!.
__device__ __forceinline__ void df_sincos_taylor(df x, df& s, df& c) {
  constexpr double f3 = 6.0, f5 = f3 * 20.0, f7 = f5 * 42.0, f9 = f7 * 72.0, f11 = f9 * 110.0,
                   f13 = f11 * 156.0, f15 = f13 * 210.0, f17 = f15 * 272.0, f19 = f17 * 342.0;
  constexpr double f2 = 2.0, f4 = f2 * 12.0, f6 = f4 * 30.0, f8 = f6 * 56.0, f10 = f8 * 90.0,
                   f12 = f10 * 132.0, f14 = f12 * 182.0, f16 = f14 * 240.0, f18 = f16 * 306.0,
                   f20 = f18 * 380.0;
  constexpr df ks[9] = {df_const(-1.0 / f19), df_const(1.0 / f17), df_const(-1.0 / f15), df_const(1.0 / f13),
                        df_const(-1.0 / f11), df_const(1.0 / f9),  df_const(-1.0 / f7),  df_const(1.0 / f5),
                        df_const(-1.0 / f3)};
  constexpr df kc[10] = {df_const(1.0 / f20),  df_const(-1.0 / f18), df_const(1.0 / f16), df_const(-1.0 / f14),
                         df_const(1.0 / f12),  df_const(-1.0 / f10), df_const(1.0 / f8),  df_const(-1.0 / f6),
                         df_const(1.0 / f4),   df_const(-1.0 / f2)};
  const df u = df_mul(x, x);
  df ps = ks[0];
#pragma unroll
  for (int k = 1; k < 9; ++k) ps = df_add(df_mul(ps, u), ks[k]);
  s = df_add(x, df_mul(df_mul(x, u), ps));
  df pc = kc[0];
#pragma unroll
  for (int k = 1; k < 10; ++k) pc = df_add(df_mul(pc, u), kc[k]);
  c = df_add(df{1.f, 0.f}, df_mul(u, pc));
}

// sin(pi D / den) for |D| < den < 2^24, den divisible by 4, in double-float: the fraction reduced in
// integers to a = Da / den in [0, 1/4] (sin(pi (1 - t)) = sin(pi t), sin(pi t) = cos(pi (1/2 - t))),
// the quotient formed exactly to double-float (FMA remainder), then the Taylor series at pi a.
__device__ __forceinline__ df df_sinpi_frac(int D, int den) {
  int a = D < 0 ? -D : D;
  if (2 * a > den) a = den - a;
  const bool use_cos = 4 * a > den;
  if (use_cos) a = den / 2 - a;
  const float fa = (float)a, fd = (float)den;
  const float q0 = __fdiv_rn(fa, fd);
  const float r = fmaf(-q0, fd, fa);
  df q;
  quick_two_sum(q0, __fdiv_rn(r, fd), q.hi, q.lo);
  constexpr df kPi = df_const(3.14159265358979323846);
  df s, c;
  df_sincos_taylor(df_mul(kPi, q), s, c);
  const df v = use_cos ? c : s;
  return D < 0 ? df_neg(v) : v;
}

// Complex compensated multiply-accumulate: acc += a * b with a, b complex df64 (float4 layout).
__device__ __forceinline__ void cdf_mac(dfacc& re, dfacc& im, float4 a, float4 b) {
  re.mac(a.x, a.y, b.x, b.y);
  re.mac(-a.z, -a.w, b.z, b.w);
  im.mac(a.x, a.y, b.z, b.w);
  im.mac(a.z, a.w, b.x, b.y);
}

// Two floats in one register pair: one instruction per operation on both (the FP32 pipe's rate is the same, the issue
// slots are half).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// dfacc for two sums at once; (na, nal) is the negated factor, so that the product's error comes out negated.
struct dfacc2 {
  f32x2 hi = 0ull, lo = 0ull;
  __device__ __forceinline__ void mac(f32x2 ah, f32x2 nah, f32x2 nal, f32x2 bh, f32x2 bl) {
    const f32x2 p = mul2(ah, bh);
    f32x2 ne = fma2(nah, bh, p);
    ne = fma2(nah, bl, ne);
    ne = fma2(nal, bh, ne);
    const f32x2 s = add2(hi, p), v = sub2(s, hi);
    const f32x2 t = add2(sub2(hi, sub2(s, v)), sub2(p, v));
    hi = s;
    lo = add2(lo, sub2(t, ne));
  }
};

}  // namespace fthms
