// Fixed point for sums of products: values as integers of up to 60 bits in two halves, multiplied and summed exactly by
// 32 x 32 + 64 -> 64-bit multiply-adds.  GB300 issues 64 of those a clock and SM against 2 FP64 lanes and, with its
// compensation, the equivalent of 2.7 double-float ones: 12 per complex product instead of 4 FP64 FMAs (256 issue
// slots' worth) or 48 FP32 instructions, so a matvec runs at the speed of its 16 bytes an entry.  A row shares one power
// of two (a bound of its entries), a vector another.  What is rounded: each value once, to the last place below its bound,
// and the sum once at the end (the products of two low halves are dropped, below that place); FP64 sums round at every
// step.
#pragma once
#include <cuda_runtime.h>

namespace fthms {

// v = (x 2^kLow + y) 2^(s - fix_bits) for |v| < 2^s, |x| and |y| <= 2^(kLow - 1), rounded to the last place.
__host__ __device__ constexpr int fix_bits(int low) { return 2 * low - 1; }   // |X| < 2^fix_bits
// Products between carries: one adds at most 2^(2 low - 1) to the cross sum, 2^63 in all (at the positive end less
// than that by more than the carry leaves).
__host__ __device__ constexpr int fix_run(int low) { return 1 << (64 - 2 * low); }
// Stored cross rows and their densities: 58 bits, 64 products a carry.  Against FP64 FMAs over the same entries (nodes 33 to
// 800, near and far rows): the sums' error is 1/2 to 1/20 of theirs.
constexpr int kRowLow = 29;
// Matrices kept for the refinement and the corrections they meet: 60 bits, 16 products a carry.  A row's entries lie up
// to 2^6 below its diagonal entry, so 60 bits add 0.1 to 0.25 of the rounding that FP64 entries carry anyway (N = 96 to
// 1024; 56 bits: 1.6 to 4 times it).
constexpr int kMatLow = 30;
constexpr int kLuLow = 30;              // LU updates (sums of eight products): 60 bits

template <int kLow>
__device__ __forceinline__ int2 fix_split(long long X) {
  const int x = (int)((X + (1ll << (kLow - 1))) >> kLow);
  return make_int2(x, (int)(X - ((long long)x << kLow)));
}
template <int kLow>
__device__ __forceinline__ int2 fix_f64(double v, int s) {
  const unsigned h = (unsigned)__double2hiint(v);
  const int e = (int)((h >> 20) & 0x7FFu);
  unsigned long long m = ((unsigned long long)((h & 0xFFFFFu) | 0x100000u) << 32) | (unsigned)__double2loint(v);
  const int sh = e - 1075 + fix_bits(kLow) - s;         // <= fix_bits - 53
  if (e == 0 || sh < -60) m = 0ull;
  else if (sh >= 0) m <<= min(sh, 8);
  else m = (m + (1ull << (-sh - 1))) >> -sh;
  return fix_split<kLow>((h >> 31) ? -(long long)m : (long long)m);
}
// The same for a double-float value (c = 2^(kLow - 1 - s)).
template <int kLow>
__device__ __forceinline__ int2 fix_df(float hi, float lo, float c) {
  const float y = __fmul_rn(hi, c);                     // exact
  const int a = __float2int_rn(y);
  const float t = fmaf(lo, c, __fsub_rn(y, (float)a));  // |t| < 20
  const float q = rintf(t);
  return make_int2(a + (int)q, __float2int_rn(__fmul_rn(__fsub_rn(t, q), (float)(1 << kLow))));
}

// A float |v| < 2^s (c = 2^(kLow - 1 - s)).
template <int kLow>
__device__ __forceinline__ int2 fix_f32(float v, float c) {
  const float y = __fmul_rn(v, c);                      // exact
  const int a = __float2int_rn(y);
  return make_int2(a, __float2int_rn(__fmul_rn(__fsub_rn(y, (float)a), (float)(1 << kLow))));
}

// (double)t by two FP64 additions (the bits of both halves placed under 2^84 and 2^52).
__device__ __forceinline__ double ll_to_double(long long t) {
  const double h = __hiloint2double(0x45300000, (int)(t >> 32) ^ (int)0x80000000u);
  const double l = __hiloint2double(0x43300000, (int)(unsigned)t);
  return (h - 19342822341709703277445120.0) + l;        // 2^84 + 2^63 + 2^52
}

// One warp: N values of a density vector in fixed point, and their unit.  A vector with a value that is not finite gets
// the unit NaN, so that every sum it enters is NaN.
__device__ __forceinline__ void fix_vector(const double2* v, int N, double scale, int4* out, double* unit, int lane) {
  unsigned m = 0u;
  for (int i = lane; i < N; i += 32)
    m = max(m, max((unsigned)__double2hiint(v[i].x) & 0x7FFFFFFFu, (unsigned)__double2hiint(v[i].y) & 0x7FFFFFFFu));
  m = __reduce_max_sync(0xffffffffu, m);
  const int e = max((int)(m >> 20), 100);               // (zero or tiny: any unit does)
  const int s = e - 1022;
  for (int i = lane; i < N; i += 32) {
    const int2 a = fix_f64<kRowLow>(v[i].x, s), b = fix_f64<kRowLow>(v[i].y, s);
    out[i] = make_int4(a.x, a.y, b.x, b.y);
  }
  if (lane == 0)
    *unit = e >= 0x7FF ? __longlong_as_double(0x7FF8000000000000ll)
                       : scale * __hiloint2double((e - 1022 - fix_bits(kRowLow) + 1023) << 20, 0);
}

// Sum of products, exact but for the products of two low halves; at most fix_run(kLow) products between carries.
template <int kLow>
struct fixacc {
  long long a = 0, b = 0, c = 0;          // high products, cross products (2^kLow below), carries (2^32 above)
  __device__ __forceinline__ void mac(int x0, int x1, int y0, int y1) {
    a += (long long)x0 * y0;
    b += (long long)x0 * y1;
    b += (long long)x1 * y0;
  }
  __device__ __forceinline__ void carry() {
    a += b >> kLow;
    b &= (1ll << kLow) - 1;
    c += a >> 32;
    a &= 0xFFFFFFFFll;
  }
  __device__ __forceinline__ double value() {           // in units of 2^(2 kLow)
    carry();
    return fma((double)c, 4294967296.0, (double)a + (1.0 / (1ll << kLow)) * (double)b);
  }
  // A short sum without carries, to the nearest of the same units.  (Cut instead of rounded, every panel of a
  // factorisation moves an entry the same way: 2e-14 of the matrix at N = 400 where FP64 gives 3.5e-15.)
  __device__ __forceinline__ long long nearest() const { return a + ((b + (1ll << (kLow - 1))) >> kLow); }
};

// LU updates: multipliers below 2 and a column of U12 below 2^e, eight complex products a sum.  |l| <= sqrt(2) (partial
// pivoting on |re| + |im|), so with 2^29 for either half's bound a sum stays below 8 x 3 x 2^58 < 2^63 and needs no
// carry.  The unit of a sum: 2^(2 kLuLow) 2^(1 - bits) 2^(e - bits); NaN for a column that is not finite.
__device__ __forceinline__ double lu_unit(int e) {
  return e > 1000 ? __longlong_as_double(0x7FF8000000000000ll) : __hiloint2double((e + 3 - 2 * kLuLow + 1023) << 20, 0);
}

}  // namespace fthms
