// The Hankel kernel of one (target, source) pair along a run of frequencies l, in double-float on the FP32 pipe
// (mixed forms).  With T = h R/(2 pi) the pair's turns per frequency index, z = 2 pi l T and w = 1/z:
//   z < 20 : J0 and Yhat0 from Taylor expansions about the centres of 160 intervals of width 1/8 (the expansions of
//            bessel_taylor.cuh shifted on the host), the terms n <= 4 in double-float, n = 5..8 in FP32 (|d| <= 1/16,
//            so they lie below 2^-26 of the sum);
//   z >= 20: modulus and phase, H0^(1)(z) = sqrt(2/(pi z)) m(w) e^{i(z - pi/4 + phi(w))}.  The phase z/(2 pi) = l T mod 1
//            is an exact 64-bit integer multiple of T's fraction, so no recurrence, no re-seeding and no FP64
//            reduction: -w/8 and its cubic correction join it as integers, the top 10 bits pick (cos, sin) from
//            a table of 1024 angles and the rest (|x| <= pi/1024) needs three Taylor terms.
//            phi = -(w/8)(1 - s (25/48 - s rho(s))), m = 1 - s/16 + s^2 kappa(s), s = w^2 (the leading terms of
//            DLMF 10.18.17-18), rho and kappa polynomials fitted to the exact modulus and phase on s <= 1/400 at 60
//            digits (their fit errors enter below 2^-52 of the result).
// About 135 FP32-pipe instructions an entry above z = 20 against ~225 of the rotated P + iQ recurrence this
// replaces, and the set-up per pair needs no sine or cosine, so short bands cost no more per entry than long ones.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "bessel.cuh"
#include "bits64.cuh"
#include "df64.cuh"
#include "kernels.h"

namespace fthms {

constexpr int kAngles = 1024;           // (cos, sin)(2 pi k/1024)
constexpr int kTayFine = 160;           // Taylor intervals of width 1/8 on [0, 20)
__device__ float4 c_angle_df[kAngles];          // cos hi, lo, sin hi, lo
__device__ float4 c_tayfine_df[kTayFine][7];    // J0: c8..c5 | c4 c3 | c2 c1 (pairs) | c0, Yhat0: see tayfine_pack
__device__ float4 c_log_df[128];                // reciprocal rc (9 bits) of the 128th's centre, -ln rc (hi, lo)

// Per-frequency constants: 2 pi l, 1/(2 pi l); 1/sqrt(l), ln l + ln pi + gamma (so that ln(z/2) + gamma = ln T + it).
struct FreqDf {
  float4 a, b;
  double lnz, rs;             // ln l + ln pi + gamma and 1/sqrt(l) in FP64
};
static_assert(sizeof(FreqDf) == kFreqDfBytes, "size of the per-frequency constants");

__device__ __forceinline__ FreqDf make_freq(int l) {
  const double x = l > 0 ? (double)l : 1.0;
  FreqDf f;
  f.lnz = log(x) + 1.7219455507509330;      // ln pi + gamma
  f.rs = rsqrt(x);
  const df a = df_from(6.28318530717958647692 * x), b = df_from(0.5 * kInvPi / x), c = df_from(f.rs), d = df_from(f.lnz);
  f.a = make_float4(a.hi, a.lo, b.hi, b.lo);
  f.b = make_float4(c.hi, c.lo, d.hi, d.lo);
  return f;
}

// One pair: everything that its frequencies share.  T = h R/(2 pi) carries no unit and lies in FP32's range (a pair below
// 2^-126 turns is taken as z = 0 with the logarithm's FP64 value in the FP64 forms, above 2^127 it gives NaN).
struct PairTurns {
  unsigned long long v;   // fraction of T in units of 2^-64 turns
  df T, iu, aw;           // T, 1/T, (w/(4 pi)) / sqrt(T)
};

// hi + lo ~ a to 2^-47 by integer operations and selects alone (an FP64 branch for the rare ranges would occupy the
// FP64 pipe even when no lane takes it: 10 of its slots a pair): below FP32's normal range zero, above it NaN.
__device__ __forceinline__ df df_split_bits(double a) {
  const unsigned uh = (unsigned)__double2hiint(a), ul = (unsigned)__double2loint(a);
  const int e = (int)((uh >> 20) & 0x7FFu);
  const unsigned sign = uh & 0x80000000u, rem = ul & 0x1FFFFFFFu;
  const float h = __uint_as_float(sign | ((unsigned)(e - 896) << 23) | (__funnelshift_l(ul, uh, 3) & 0x007FFFFFu));
  const float r = __uint_as_float(__float_as_uint(__uint2float_rn(rem)) + ((unsigned)(e - 1075) << 23));
  const bool lo_ok = rem != 0u && e > 1023 - 70;
  df v;
  v.hi = e < 1023 - 126 ? 0.f : e > 1023 + 127 ? __uint_as_float(0x7FFFFFFFu) : h;
  v.lo = lo_ok ? __uint_as_float(__float_as_uint(r) | sign) : 0.f;
  return v;
}

__device__ __forceinline__ unsigned long long turn_fraction(double T) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(T);
  const int s = (int)((u >> 52) & 0x7FF) - 1011;            // T = m 2^(e - 1075), m the 53-bit significand
  const unsigned long long m = (u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  return s >= 0 ? (s < 64 ? m << s : 0ull) : (s > -64 ? m >> -s : 0ull);
}

// a b without the final renormalisation (|low word| a few ulp of the high one)
__device__ __forceinline__ df df_mulq(df a, df b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  return df{p, fmaf(a.lo, b.hi, e)};
}

__device__ __forceinline__ PairTurns pair_turns(double T, df camp4) {   // camp4 = w/(4 pi)
  PairTurns p;
  p.v = turn_fraction(T);
  p.T = df_split_bits(T);
  // 1/sqrt(T): y = rsqrt(T) (2^-22), then y (1 + e/2 + 3 e^2/8) with e = 1 - T y^2 in double-float
  const float y = rsqrtf(p.T.hi);
  const float q = __fmul_rn(y, y), qe = fmaf(y, y, -q);
  const float t = __fmul_rn(p.T.hi, q);
  const float te = fmaf(p.T.lo, q, fmaf(p.T.hi, qe, fmaf(p.T.hi, q, -t)));
  const float e = __fsub_rn(__fsub_rn(1.f, t), te);
  df r;
  quick_two_sum(y, __fmul_rn(y, __fmul_rn(e, fmaf(0.375f, e, 0.5f))), r.hi, r.lo);
  p.iu = df_mul(r, r);
  p.aw = df_mul(r, camp4);
  return p;
}

// ln T for T > 0 (a normal float range): T = 2^e m, r = m rc - 1 (|r| < 0.006), the series of ln(1 + r) with its first
// two terms in double-float.  Error about 2^-47.
__device__ __forceinline__ df df_log(df T) {
  const unsigned u = __float_as_uint(T.hi);
  const int ex = (int)(u >> 23) - 127;
  const float mh = __uint_as_float((u & 0x7FFFFFu) | 0x3F800000u);
  const float ml = __fmul_rn(T.lo, __uint_as_float((unsigned)(127 - ex) << 23));
  const float4 tb = __ldg(&c_log_df[(u >> 16) & 127u]);
  const float p = __fmul_rn(mh, tb.x);
  float rl = fmaf(ml, tb.x, fmaf(mh, tb.x, -p));
  float rh = __fsub_rn(p, 1.f);                               // exact
  quick_two_sum(rh, rl, rh, rl);
  const float h = __fmul_rn(rh, rh), hl = fmaf(2.f * rh, rl, fmaf(rh, rh, -h));
  const float c = __fmul_rn(__fmul_rn(h, rh), fmaf(rh, fmaf(rh, fmaf(rh, -1.f / 6.f, 0.2f), -0.25f), 1.f / 3.f));
  df v;
  quick_two_sum(rh, -0.5f * h, v.hi, v.lo);
  v.lo = __fadd_rn(v.lo, __fadd_rn(fmaf(-0.5f, hl, rl), c));
  constexpr float kLn2Hi = 0x1.62e4p-1f;                      // 15 bits: ex kLn2Hi is exact
  constexpr double kLn2Rest = 0.69314718055994530941723212145817657 - 0.693145751953125;
  constexpr df kLn2Lo = df_const(kLn2Rest);
  const float fe = (float)ex;
  df s, t;
  two_sum(__fmul_rn(fe, kLn2Hi), tb.y, s.hi, s.lo);
  s.lo = __fadd_rn(s.lo, tb.z);
  two_sum(s.hi, v.hi, t.hi, t.lo);
  t.lo = __fadd_rn(t.lo, __fadd_rn(s.lo, v.lo));
  const float k = __fmul_rn(fe, kLn2Lo.hi);
  two_sum(t.hi, k, s.hi, s.lo);
  s.lo = __fadd_rn(__fadd_rn(s.lo, t.lo), fmaf(fe, kLn2Lo.lo, fmaf(fe, kLn2Lo.hi, -k)));
  df r;
  quick_two_sum(s.hi, s.lo, r.hi, r.lo);
  if (!(T.hi > 0.f)) r = df{__uint_as_float(0xFF800000u), 0.f};
  return r;
}

// J0 and Yhat0 at 0 <= z < 20.
__device__ __forceinline__ df tayfine_eval(const float4 f, df c4, df c3, df c2, df c1, df c0, df d) {
  const float t = fmaf(fmaf(fmaf(f.x, d.hi, f.y), d.hi, f.z), d.hi, f.w);   // c8..c5
  df s = df_add_fast(df{__fmul_rn(t, d.hi), 0.f}, c4);
  s = df_add_fast(df_mulq(s, d), c3);
  s = df_add_fast(df_mulq(s, d), c2);
  s = df_add_fast(df_mulq(s, d), c1);
  return df_add_fast(df_mulq(s, d), c0);
}
__device__ __forceinline__ void bessel0_tayfine_df(df z, df& J0, df& Yh) {
  const int k = min((int)(8.f * z.hi), kTayFine - 1);
  const df d = df_add_fast(z, df{-(0.0625f + 0.125f * (float)k), 0.f});
  const float4* t = c_tayfine_df[k];
  const float4 a = __ldg(&t[0]), b = __ldg(&t[1]), c = __ldg(&t[2]), e = __ldg(&t[3]), f = __ldg(&t[4]),
               g = __ldg(&t[5]), h = __ldg(&t[6]);
  J0 = tayfine_eval(a, df{b.x, b.y}, df{b.z, b.w}, df{c.x, c.y}, df{c.z, c.w}, df{e.x, e.y}, d);
  Yh = tayfine_eval(f, df{g.x, g.y}, df{g.z, g.w}, df{h.x, h.y}, df{h.z, h.w}, df{e.z, e.w}, d);
}

// Angle and modulus at z >= 20: the table index, the residual angle x = xh + ... as sin x = xh + sx and
// cos x - 1 = ch + cl, and 1 - m = mh + ml; p = l v - 1/8 turn.  The second-order terms stay in
// double-float (rho(0), kappa(0) as pairs): phase and modulus to 2^-52 near z = 20; in FP32 they reach 2^-45 there, which
// ill-conditioned precision-1 jobs show (densities 1.2e-11 off instead of 7.4e-12) for 5% of the assembly's time.
struct FarAngle {
  unsigned idx;
  float xh, sx, ch, cl, mh, ml;
};
__device__ __forceinline__ FarAngle far_angle(df iu, unsigned long long p, df iv) {
  FarAngle r;
  const df w = df_mul(iu, iv);
  const float sh = __fmul_rn(w.hi, w.hi), sl = fmaf(2.f * w.hi, w.lo, fmaf(w.hi, w.hi, -sh));
  // g = s (25/48 - s rho)
  constexpr df kG = df_const(25.0 / 48.0), kR = df_const(1.67656249910766316), kK = df_const(0.103515624983438744);
  float rho = fmaf(sh, 109818.0144f, -4218.12863f);
  rho = fmaf(sh, rho, 187.743036f);
  rho = fmaf(sh, rho, -13.1045092f);
  const float th = __fmul_rn(sh, kR.hi);                        // s rho(0)
  const float tl = fmaf(sh, fmaf(sh, rho, kR.lo), fmaf(sl, kR.hi, fmaf(sh, kR.hi, -th)));
  df c;
  quick_two_sum(kG.hi, -th, c.hi, c.lo);
  c.lo = __fadd_rn(c.lo, __fsub_rn(kG.lo, tl));
  const df g = df_mul(df{sh, sl}, c);
  const float gh = g.hi, gl = g.lo;
  // phi = -w/8 + (w/8) g = -q + (ah + al)
  const float qh = 0.125f * w.hi, ql = 0.125f * w.lo;
  const float ah = __fmul_rn(qh, gh), al = fmaf(ql, gh, fmaf(qh, gl, fmaf(qh, gh, -ah)));
  // both high parts join the phase as integers of 2^-31 turns (|.| < 2^22: rounded by the FP32 add of 1.5 2^23)
  constexpr double kTurn = 6.28318530717958647692 / 4294967296.0;    // 2^-32 turns in radians
  constexpr df kT = df_const(kTurn), kT2 = df_const(2.0 * kTurn);
  constexpr float kPerRad = (float)(0.5 / kTurn), kMagic = 12582912.f;
  const float m1 = fmaf(qh, -kPerRad, kMagic), m2 = fmaf(ah, kPerRad, kMagic);
  const float f1 = __fsub_rn(m1, kMagic), f2 = __fsub_rn(m2, kMagic);
  const int n = (int)(__float_as_uint(m1) + __float_as_uint(m2) - 2u * 0x4B400000u) * 2;
  float res = __fadd_rn(fmaf(f1, -kT2.hi, -qh), fmaf(f2, -kT2.hi, ah));
  res = __fadd_rn(res, fmaf(-__fadd_rn(f1, f2), kT2.lo, __fsub_rn(al, ql)));
  const unsigned hi = (unsigned)(p >> 32) + (unsigned)n;
  r.idx = ((hi + 0x200000u) >> 22);
  // integers below 2^21 and 2^23 to float by an exponent and a subtraction (the conversion unit is slower)
  const float fr = __fsub_rn(__uint_as_float(0x4B400000u + (hi - (r.idx << 22))), kMagic);
  const float fl = __fsub_rn(__uint_as_float(0x4B000000u | ((unsigned)p >> 9)), 8388608.f);
  constexpr float kLow = (float)(kTurn / 8388608.0);
  r.idx &= kAngles - 1;
  const float xh = __fmul_rn(fr, kT.hi);
  float xl = fmaf(fr, kT.lo, fmaf(fr, kT.hi, -xh));
  xl = __fadd_rn(fmaf(fl, kLow, xl), res);
  const float uh = __fmul_rn(xh, xh), ul = fmaf(2.f * xh, xl, fmaf(xh, xh, -uh));
  r.xh = xh;
  r.ch = -0.5f * uh;
  r.sx = fmaf(xh, __fmul_rn(uh, fmaf(uh, 1.f / 120.f, -1.f / 6.f)), fmaf(xl, r.ch, xl));
  r.cl = fmaf(__fmul_rn(uh, uh), 1.f / 24.f, -0.5f * ul);
  float kap = fmaf(sh, 2366.77002f, -105.650777f);
  kap = fmaf(sh, kap, 5.84762562f);
  kap = fmaf(sh, kap, -0.542846348f);
  r.mh = 0.0625f * sh;
  const float t = __fmul_rn(sh, sh), te = fmaf(2.f * sh, sl, fmaf(sh, sh, -t));
  const float kh = __fmul_rn(t, kK.hi);
  const float kl = fmaf(t, fmaf(sh, kap, kK.lo), fmaf(te, kK.hi, fmaf(t, kK.hi, -kh)));
  quick_two_sum(r.mh, -kh, r.mh, r.ml);
  r.ml = __fadd_rn(r.ml, fmaf(0.0625f, sl, -kl));
  return r;
}

// cos or sin of (table angle + x) minus the table value, as an unrenormalised pair: a ch -+ b x, with (a, b) the
// table's value and its partner.
__device__ __forceinline__ df angle_step(float ah, float al, float bh, float bl, const FarAngle& f) {
  const float A = __fmul_rn(bh, f.xh), B = __fmul_rn(ah, f.ch);
  const float Ae = fmaf(bl, f.xh, fmaf(bh, f.sx, fmaf(bh, f.xh, -A)));
  const float Be = fmaf(al, f.ch, fmaf(ah, f.cl, fmaf(ah, f.ch, -B)));
  df d;
  quick_two_sum(A, B, d.hi, d.lo);
  d.lo = __fadd_rn(d.lo, __fadd_rn(Ae, Be));
  return d;
}

// Entry E = (amp (beta cos - sin), amp cos) at z >= 20; ang: the angle table (shared memory).
__device__ __forceinline__ float4 hankel_far_df(const PairTurns& pr, unsigned long long p, const float4* ang, df iv,
                                                df rs, df beta, bool near) {
  const FarAngle f = far_angle(pr.iu, p, iv);
  const float4 t = ang[f.idx];
  const df dc = angle_step(t.x, t.y, -t.z, -t.w, f), ds = angle_step(t.z, t.w, t.x, t.y, f);
  df co, si;
  quick_two_sum(t.x, dc.hi, co.hi, co.lo);
  co.lo = __fadd_rn(__fadd_rn(co.lo, t.y), dc.lo);
  quick_two_sum(t.z, ds.hi, si.hi, si.lo);
  si.lo = __fadd_rn(__fadd_rn(si.lo, t.w), ds.lo);
  const df a0 = df_mulq(pr.aw, rs);                             // amp (1 - mu)
  const float b = __fmul_rn(a0.hi, f.mh), be = fmaf(a0.lo, f.mh, fmaf(a0.hi, f.ml, fmaf(a0.hi, f.mh, -b)));
  df amp;
  quick_two_sum(a0.hi, -b, amp.hi, amp.lo);
  amp.lo = __fadd_rn(amp.lo, __fsub_rn(a0.lo, be));
  const df im = df_mulq(amp, co);
  const df mr = near ? df_dot2(df_neg(beta), co, df{1.f, 0.f}, si) : si;     // -(beta cos - sin)
  const df re = df_mulq(amp, mr);
  return make_float4(-re.hi, -re.lo, im.hi, im.lo);
}

// Entry at z < 20: re = -(w/4) [((2/pi) Lz - beta) J0 + Yhat0], im = (w/4) J0 with Lz = ln(z/2) + gamma.
__device__ __forceinline__ float4 hankel_near_df(df z, df Lz, df beta, bool near, df qw) {
  constexpr df k2Pi = df_const(0.63661977236758134307553505349005745);
  df J0, Yh;
  bessel0_tayfine_df(z, J0, Yh);
  df a = df_mul(Lz, k2Pi);
  if (near) a = df_sub(a, beta);
  const df re = df_mul(qw, df_dot2(a, J0, df{1.f, 0.f}, Yh));
  const df im = df_mul(qw, J0);
  return make_float4(-re.hi, -re.lo, im.hi, im.lo);
}

// ---- FP64 entries with the FP64 pipe (two lanes a clock and SM) kept for the last additions --------------------
// Only what reaches the result's leading bits needs FP64: the table values and the final sums and products.  The
// corrections to a table value are small -- the angle step below 2^-8, the Taylor terms beyond the constant below
// 2^-6 -- so double-float corrections (2^-46 relative and better) leave the result at FP64's own rounding.  9 FP64
// instructions an entry against 25 to 45 of the plain FP64 series and rotated recurrence.
constexpr int kTay64 = 408;             // Taylor intervals of 1/128 turn on [0, 20/(2 pi))
struct Tay64 {                          // n = 7..5 in FP32, 4..1 double-float (in turns), 0 in FP64
  float4 hi, c43, c21;
  double c0, pad;
};
__device__ double2 c_angle_f64[kAngles];
__device__ Tay64 c_tay64[kTay64 + 1][2];        // J0, Yhat0
__device__ double2 c_log_f64[1024];             // reciprocal (12 bits) of the 1024th's centre, -ln of it

template <bool kF64>
struct AngleTab {                       // shared-memory copy (the FP64 values for FP64 entries only)
  float4 d[kAngles];
  double2 f[kF64 ? kAngles : 1];
};
template <bool kF64>
__device__ __forceinline__ void load_angles(AngleTab<kF64>& t) {
  for (int k = threadIdx.x; k < kAngles; k += blockDim.x) {
    t.d[k] = c_angle_df[k];
    if (kF64) t.f[k] = c_angle_f64[k];
  }
}

// ln x for a normal x > 0 (-inf at 0): x = 2^e m, r = m rc - 1 exact in one FMA (|r| < 2^-10), ln(1 + r) - r in double-
// float.  Five FP64 operations.
__device__ __forceinline__ double log_f64(double x) {
  const int h = __double2hiint(x);
  const int ex = ((h >> 20) & 0x7FF) - 1023;
  const double m = __hiloint2double((h & 0xFFFFF) | 0x3FF00000, __double2loint(x));
  const double2 tb = __ldg(&c_log_f64[(h >> 10) & 1023]);
  const double r = fma(m, tb.x, -1.0);
  const df rd = df_split_bits(r);
  const float u = __fmul_rn(rd.hi, rd.hi), ul = fmaf(2.f * rd.hi, rd.lo, fmaf(rd.hi, rd.hi, -u));
  const float c = __fmul_rn(__fmul_rn(u, rd.hi), fmaf(rd.hi, fmaf(rd.hi, 0.2f, -0.25f), 1.f / 3.f));
  const double q = f2d_bits(-0.5f * u) + f2d_bits(fmaf(-0.5f, ul, c));
  const double v = (fma((double)ex, 0.69314718055994530941723212145817657, tb.y) + r) + q;
  return x > 0.0 ? v : __longlong_as_double(0xFFF0000000000000ll);
}

struct PairF64 {
  unsigned long long v;   // fraction of T in 2^-64 turns
  unsigned long long v62; // T in 2^-62 turns (below 4 turns; for z < 20)
  double T, aw;           // turns, (w/(4 pi)) / sqrt(T)
  df iu;                  // 1/T
  float th;
};
__device__ __forceinline__ PairF64 pair_f64(double T, double camp4) {
  PairF64 p;
  p.T = T;
  p.v = turn_fraction(T);
  p.v62 = turn_fraction(0.25 * T);                     // (exact scaling)
  const df t = df_split_bits(T);
  p.th = t.hi;
  const float y = rsqrtf(t.hi);
  const float q = __fmul_rn(y, y), qe = fmaf(y, y, -q);
  const float a = __fmul_rn(t.hi, q);
  const float ae = fmaf(t.lo, q, fmaf(t.hi, qe, fmaf(t.hi, q, -a)));
  const float e = __fsub_rn(__fsub_rn(1.f, a), ae);
  df r;
  quick_two_sum(y, __fmul_rn(y, __fmul_rn(e, fmaf(0.375f, e, 0.5f))), r.hi, r.lo);
  p.iu = df_mul(r, r);
  const double s = f2d_bits(r.hi) + f2d_bits(r.lo);    // one Newton step on the pair: 2^-46 -> FP64
  p.aw = camp4 * fma(fma(-T * s, s, 1.0), 0.5 * s, s);
  return p;
}

// z >= 20; p = l v - 1/8 turn, rs = 1/sqrt(l).
__device__ __forceinline__ double2 hankel_far_f64(const PairF64& pr, unsigned long long p, const float4* ang,
                                                  const double2* ang64, df iv, double rs, double beta, bool near) {
  const FarAngle f = far_angle(pr.iu, p, iv);
  const float4 t = ang[f.idx];
  const double2 t64 = ang64[f.idx];
  const df dc = angle_step(t.x, t.y, -t.z, -t.w, f), ds = angle_step(t.z, t.w, t.x, t.y, f);
  const double co = t64.x + (f2d_bits(dc.hi) + f2d_bits(dc.lo)), si = t64.y + (f2d_bits(ds.hi) + f2d_bits(ds.lo));
  const double a0 = pr.aw * rs;
  const double amp = fma(-a0, f2d_bits(f.mh) + f2d_bits(f.ml), a0);
  return make_double2(amp * (near ? fma(beta, co, -si) : -si), amp * co);
}

// J0 and Yhat0 at z = 2 pi u / 2^62 < 20 (u = l v62): interval and offset are bits of u.
__device__ __forceinline__ double tay64_eval(const Tay64* __restrict__ tab, df d) {
  const float4 h = __ldg(&tab->hi), a = __ldg(&tab->c43), b = __ldg(&tab->c21);
  const double c0 = __ldg(&tab->c0);
  const float q = fmaf(fmaf(h.x, d.hi, h.y), d.hi, h.z);
  df s = df_add_fast(df{__fmul_rn(q, d.hi), 0.f}, df{a.x, a.y});
  s = df_add_fast(df_mul(s, d), df{a.z, a.w});
  s = df_add_fast(df_mul(s, d), df{b.x, b.y});
  s = df_add_fast(df_mul(s, d), df{b.z, b.w});
  s = df_mulq(s, d);
  return c0 + (f2d_bits(s.hi) + f2d_bits(s.lo));
}
__device__ __forceinline__ void bessel0_f64(unsigned long long u, double& J0, double& Yh) {
  const int k = min((int)(u >> 55), kTay64);
  const long long rem = (long long)(u - ((unsigned long long)k << 55)) - (1ll << 54);
  df d;                                                 // in turns: |d| <= 2^-8
  quick_two_sum((float)(int)(rem >> 32) * 0x1p-30f, (float)((unsigned)rem >> 8) * 0x1p-54f, d.hi, d.lo);
  J0 = tay64_eval(&c_tay64[k][0], d);
  Yh = tay64_eval(&c_tay64[k][1], d);
}

// Entry at z < 20, the sum of hankel_near_df in FP64; L = ln(z/2) + gamma.
__device__ __forceinline__ double2 hankel_near_f64(unsigned long long u, double L, double beta, bool near, double qw) {
  double J0, Yh;
  bessel0_f64(u, J0, Yh);
  const double a = near ? fma(kTwoOverPi, L, -beta) : kTwoOverPi * L;
  return make_double2(-qw * fma(a, J0, Yh), qw * J0);
}
__device__ __forceinline__ float4 split2_bits(double2 v) {
  const df a = df_split_bits(v.x), b = df_split_bits(v.y);
  return make_float4(a.hi, a.lo, b.hi, b.lo);
}

// Fills the tables above and bessel.cuh's on device dev (current), once: the first caller of any thread computes and
// uploads them while the others wait, and returns when they are on the device (a stream of the caller's own does not wait
// for the copies by itself).
inline cudaError_t init_tables(int dev) {
  static std::mutex mu;
  static bool done[64];
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(mu);
  if (done[dev]) return cudaSuccess;
  double ha[20];
  ha[0] = 1.0;
  for (int k = 1; k < 20; ++k) ha[k] = ha[k - 1] * (double)((2 * k - 1) * (2 * k - 1)) / (8.0 * k);
  static float4 ang[kAngles], lg[128], tf[kTayFine][7];
  auto hi = [](double v) { return (float)v; };
  auto lo = [](double v) { return (float)(v - (double)(float)v); };
  for (int k = 0; k < kAngles; ++k) {
    // the first octant's values, moved by symmetry, so that multiples of a quarter turn are exact
    const int q = 4 * k / kAngles, r = k % (kAngles / 4), h = kAngles / 8;
    const double a = 2.0 * 3.14159265358979323846 * (r <= h ? r : 2 * h - r) / kAngles;
    const double c0 = r <= h ? std::cos(a) : std::sin(a), s0 = r <= h ? std::sin(a) : std::cos(a);
    const double c = q == 0 ? c0 : q == 1 ? -s0 : q == 2 ? -c0 : s0, s = q == 0 ? s0 : q == 1 ? c0 : q == 2 ? -s0 : -c0;
    ang[k] = make_float4(hi(c), lo(c), hi(s), lo(s));
  }
  for (int k = 0; k < 128; ++k) {
    const double c = 1.0 + (k + 0.5) / 128.0, rc = std::nearbyint(512.0 / c) / 512.0, l = -std::log(rc);
    lg[k] = make_float4((float)rc, hi(l), lo(l), 0.f);
  }
  double src[2][kTaylorIntervals][kTaylorDegree + 1];
  cudaError_t e = cudaMemcpyFromSymbol(src[0], kTaylorJ0, sizeof src[0]);
  if (e == cudaSuccess) e = cudaMemcpyFromSymbol(src[1], kTaylorYh, sizeof src[1]);
  if (e != cudaSuccess) return e;
  for (int k = 0; k < kTayFine; ++k) {
    const double shift = (0.0625 + 0.125 * k) - (0.25 + 0.5 * (k / 4));
    double c[2][9];
    for (int f = 0; f < 2; ++f)
      for (int n = 0; n <= 8; ++n) {      // c_n = sum_m binom(m, n) a_m shift^(m - n)
        double v = 0.0, binom = 1.0, pw = 1.0;
        for (int m = n; m <= kTaylorDegree; ++m) {
          v += binom * src[f][k / 4][m] * pw;
          binom = binom * (m + 1) / (m + 1 - n);
          pw *= shift;
        }
        c[f][n] = v;
      }
    const double *j = c[0], *y = c[1];
    tf[k][0] = make_float4(hi(j[8]), hi(j[7]), hi(j[6]), hi(j[5]));
    tf[k][1] = make_float4(hi(j[4]), lo(j[4]), hi(j[3]), lo(j[3]));
    tf[k][2] = make_float4(hi(j[2]), lo(j[2]), hi(j[1]), lo(j[1]));
    tf[k][3] = make_float4(hi(j[0]), lo(j[0]), hi(y[0]), lo(y[0]));
    tf[k][4] = make_float4(hi(y[8]), hi(y[7]), hi(y[6]), hi(y[5]));
    tf[k][5] = make_float4(hi(y[4]), lo(y[4]), hi(y[3]), lo(y[3]));
    tf[k][6] = make_float4(hi(y[2]), lo(y[2]), hi(y[1]), lo(y[1]));
  }
  static double2 ang64[kAngles], lg64[1024];
  static Tay64 t64[kTay64 + 1][2];
  for (int k = 0; k < kAngles; ++k) {
    const int q = 4 * k / kAngles, r = k % (kAngles / 4), h = kAngles / 8;
    const double a = 2.0 * 3.14159265358979323846 * (r <= h ? r : 2 * h - r) / kAngles;
    const double c0 = r <= h ? std::cos(a) : std::sin(a), s0 = r <= h ? std::sin(a) : std::cos(a);
    ang64[k] = make_double2(q == 0 ? c0 : q == 1 ? -s0 : q == 2 ? -c0 : s0, q == 0 ? s0 : q == 1 ? c0 : q == 2 ? -s0 : -c0);
  }
  for (int k = 0; k < 1024; ++k) {
    const double rc = std::nearbyint(4096.0 / (1.0 + (k + 0.5) / 1024.0)) / 4096.0;
    lg64[k] = make_double2(rc, -std::log(rc));
  }
  const double tau = 6.28318530717958647692;
  for (int k = 0; k <= kTay64; ++k) {
    const double z = tau * (k + 0.5) / 128.0;
    const int K = std::min((int)(2.0 * z), kTaylorIntervals - 1);
    const long double shift = (long double)tau * (k + 0.5L) / 128.0L + 2.4492935982947064e-16L * (k + 0.5L) / 128.0L -
                              (0.25L + 0.5L * K);          // (2 pi as the sum of two doubles)
    for (int f = 0; f < 2; ++f) {
      double c[8];
      long double sc = 1.0L;
      for (int n = 0; n <= 7; ++n, sc *= tau) {
        long double v = 0.0L, binom = 1.0L, pw = 1.0L;
        for (int m = n; m <= kTaylorDegree; ++m) {
          v += binom * src[f][K][m] * pw;
          binom = binom * (m + 1) / (m + 1 - n);
          pw *= shift;
        }
        c[n] = (double)(v * sc);
      }
      t64[k][f].hi = make_float4((float)c[7], (float)c[6], (float)c[5], 0.f);
      t64[k][f].c43 = make_float4(hi(c[4]), lo(c[4]), hi(c[3]), lo(c[3]));
      t64[k][f].c21 = make_float4(hi(c[2]), lo(c[2]), hi(c[1]), lo(c[1]));
      t64[k][f].c0 = c[0];
      t64[k][f].pad = 0.0;
    }
  }
  if ((e = cudaMemcpyToSymbol(c_angle_f64, ang64, sizeof ang64)) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_log_f64, lg64, sizeof lg64)) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_tay64, t64, sizeof t64)) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_angle_df, ang, sizeof ang)) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_log_df, lg, sizeof lg)) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_tayfine_df, tf, sizeof tf)) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_hank_a, ha, sizeof ha)) != cudaSuccess) return e;
  if ((e = cudaStreamSynchronize(nullptr)) != cudaSuccess) return e;
  done[dev] = true;
  return cudaSuccess;
}

}  // namespace fthms
