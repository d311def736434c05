// CUDA kernels (sm_103a) of the FTH-MS open-arc hot path.
//
// Stages (one job):
//   tables         FFT twiddles, recentring phases, self log-weight tables, restriction tables
//   assemble_self  log-split Chebyshev Nystrom matrices A_j(omega_l)        (Section 4.2-4.3)
//   lu             A = P L U per (arc, omega), reused for every step and window (Algorithm 1)
//   cross_assemble stored S_Gamma_j rows at the other arcs' transfer nodes   (eq. FDsolk-interior)
//   incident       g_{k,1} = sign chi_k u^i on the transfer meshes, slow transform (eqs.
//                  criterion_int1, Fourierk)
//   restrict       transfer-mesh spectra -> data on the N_k(omega_l) solve nodes
//   per step m:
//     solve        phi = A^{-1} G                                             (eq. FDBIEk-interior)
//     cross_apply  W_k = sum_{j != k, masked} S_j[phi_j] (eq. vtilde) and the observation sum
//     synth_fwd    recentred inverse transform (eq. TDsol), g = -chi_k w (eq. criterion_int2),
//                  windowed slow transform (eq. Fourierk) -- one CTA per transfer node, in shared
//                  memory, with a half-length FFT per window
//   traces         u_M(z, t) at the output times (eq. mult-scatt-int)
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <type_traits>

#include "bessel.cuh"
#include "cplx.cuh"
#include "df64.cuh"
#include "fixed.cuh"
#include "hankel_df.cuh"
#include "kernels.h"
#include "lu_common.cuh"

namespace fthms {

cudaError_t init_constants(int dev) { return init_tables(dev); }

namespace {


// ---------------------------------------------------------------------------------------------
// Special functions on an array

// z/(2 pi) for 1e-30 <= z < 2^20 as (t 2^64 + s) 2^-k: the 53-bit significand times 128 bits of 1/(2 pi), exact to 2^-63
// of a turn whatever z.
__device__ __forceinline__ void turns_of(double z, unsigned long long& t, unsigned long long& s, int& k) {
  constexpr unsigned long long c0 = 0x28BE60DB9391054Aull, c1 = 0x7F09D5F47D4D3770ull;   // 1/(2 pi) 2^128
  const unsigned long long u = (unsigned long long)__double_as_longlong(z);
  const unsigned long long m = (u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  k = 1075 - (int)(u >> 52);
  const unsigned long long lo = m * c0, h1 = __umul64hi(m, c1);
  s = lo + h1;
  t = __umul64hi(m, c0) + (s < lo ? 1ull : 0ull);
}
__device__ __forceinline__ unsigned long long shift_down(unsigned long long t, unsigned long long s, int k) {
  if (k >= 128) return 0ull;
  if (k >= 64) return t >> (k - 64);
  return k > 0 ? (s >> k) | (t << (64 - k)) : s;
}

// J0, Y0 and Yhat0 = Y0 - (2/pi)(ln(z/2) + gamma) J0.  The series and expansions of hankel_df.cuh keep the FP64 pipe to
// ~20 instructions a value (bessel0's take ~150 where a warp's values fall on both sides of z = 20); arguments outside
// [1e-30, 2^20) go through bessel0.  One value a thread, the angles through L1 (a shared copy and runs of four values a
// thread: 14.5 us at 1000 values and 72 at 10^6), narrow CTAs for the small calls (256 threads: 9.4 us).  1000 values
// 12.4 -> 7.3 us, 10^6 between 1e-3 and 2000: 248 -> 64 us.
constexpr int kBesselThreads = 64;
__global__ void __launch_bounds__(kBesselThreads) k_bessel0(const double* __restrict__ z, double* j0, double* y0, double* yh,
                                                            int n) {
  const df iv = df_const(0.5 * kInvPi);
  const long long i = (long long)blockIdx.x * kBesselThreads + threadIdx.x;
  if (i >= n) return;
  const double zz = z[i];
  double J0, Y0, Yh;
  if (zz >= 1e-30 && zz < 1048576.0) {
    unsigned long long t, s;
    int k;
    turns_of(zz, t, s, k);
    const double lg = kTwoOverPi * (log_f64(zz) - 0.11593151565841244881);      // ln 2 - gamma
    if (zz < kBesselLarge) {
      bessel0_f64(shift_down(t, s, k + 2), J0, Yh);
      Y0 = fma(lg, J0, Yh);
    } else {
      PairF64 p = pair_f64(0.5 * kInvPi * zz, kInvPi);
      const double2 E = hankel_far_f64(p, shift_down(t, s, k) - (1ull << 61), c_angle_df, c_angle_f64, iv, 1.0, 0.0, false);
      J0 = E.y;
      Y0 = -E.x;
      Yh = fma(-lg, J0, Y0);
    }
  } else {
    const Bessel0 b = bessel0(zz);
    const double lg = kTwoOverPi * (log(0.5 * zz) + kEulerGamma);
    J0 = b.j0;
    Y0 = b.has_yhat ? fma(lg, b.j0, b.y) : b.y;
    Yh = b.has_yhat ? b.y : fma(-lg, b.j0, b.y);
  }
  if (j0) j0[i] = J0;
  if (y0) y0[i] = Y0;
  if (yh) yh[i] = Yh;
}

// ---------------------------------------------------------------------------------------------
// Tables

__global__ void k_fft_tw(double2* tw, float4* tw_df, int K) {
  int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= K / 2) return;
  double s, c;
  sincospi(2.0 * r / K, &s, &c);
  tw[r] = make_double2(c, -s);   // e^{-2 pi i r/K}
  if (tw_df) tw_df[r] = df_split2(make_double2(c, -s));
}

// syn_tw[q][l] = (w_l/pi) e^{-i l c_q} e^{-2 pi i (l nlo_q mod K)/K},  fwd_tw[q][l] = dt e^{i l c_q}
__global__ void k_freq_tw(DevJob J) {
  int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= J.Q * J.L) return;
  int q = idx / J.L, l = idx % J.L;
  double s, c;
  sincos((double)l * J.c_q[q], &s, &c);
  long long m = ((long long)l * J.nlo[q]) % J.K;
  double s2, c2;
  sincospi(2.0 * (double)m / J.K, &s2, &c2);
  double wl = J.wl[l] * kInvPi;
  double2 e1 = make_double2(c, -s), e2 = make_double2(c2, -s2);
  double2 sy = cmul(e1, e2);
  J.syn_tw[idx] = make_double2(wl * sy.x, wl * sy.y);
  J.fwd_tw[idx] = make_double2(J.dt * c, J.dt * s);
}

// Per-frequency constants of the Hankel entries.
__global__ void k_freq_df(DevJob J) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l < J.L) J.freq_df[l] = make_freq(l);
}

// Cosine sums F(m) = sum_{n=1}^{N-1} cos(n m pi/N)/n, m = 0..N, of the self log weights
//   Rlog_il = -(pi/N) [ln 2 + F(|i-l|) + F(i+l+1)],  F(2N - m) = F(m)
// (the product-to-sum form of -(pi/N)[ln 2 + 2 sum_n T_n(t_i) T_n(t_l)/n]); the assembly adds the two F values
// itself (rlog_at), so no N x N table is written or read.  Grid: (distinct N, blocks of kRlogRows values m), eight
// lanes per m.  Bound by the FP64 pipe (N DFMA a value plus the cosine table of each block); one block per N
// that also wrote the N x N table took 1.1 ms at N = 777, this split 0.02 ms.
constexpr int kRlogRows = 32;
__global__ void __launch_bounds__(8 * kRlogRows) k_rlog(DevJob J) {
  extern __shared__ double sh[];
  const int N = J.rlogN[blockIdx.x], m0 = blockIdx.y * kRlogRows;
  if (m0 > N) return;
  double* cosr = sh;           // 2N: cos(r pi/N), the first quadrant evaluated, the rest by symmetry
  double* invn = sh + 2 * N;   // N
  for (int r = threadIdx.x; 2 * r <= N; r += blockDim.x) {
    const double c = cospi((double)r / N);
    cosr[r] = c;
    cosr[N - r] = -c;
    if (r) {
      cosr[2 * N - r] = c;
      cosr[N + r] = -c;
    }
  }
  for (int n = threadIdx.x; n < N; n += blockDim.x) invn[n] = n ? 1.0 / n : 0.0;
  __syncthreads();
  const int m = m0 + (threadIdx.x >> 3), sub = threadIdx.x & 7;
  double acc = 0.0;
  if (m <= N) {
    const int mod = 2 * N, step = (8 * m) % mod;
    int idx = ((1 + sub) * m) % mod;
    for (int n = 1 + sub; n < N; n += 8) {
      acc = fma(cosr[idx], invn[n], acc);
      idx += step;
      if (idx >= mod) idx -= mod;
    }
  }
  for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (sub == 0 && m <= N) J.rlog[J.rlog_off_N[blockIdx.x] + m] = acc;
}

// Rlog_il from the cosine sums F of its N.
__device__ __forceinline__ double rlog_at(const double* __restrict__ F, int N, int i, int l) {
  const double ln2 = 0.69314718055994530941723212145817657;
  const int d = i > l ? i - l : l - i, s = i + l + 1 <= N ? i + l + 1 : 2 * N - (i + l + 1);
  return (-kPiD / N) * (ln2 + __ldg(&F[d]) + __ldg(&F[s]));
}

// Transposed restriction tables RT[x][i] = l_x(t_i): the Lagrange basis of the first-kind grid of
// size M evaluated at the first-kind nodes of size N, in the closed form
//   l_x(t_i) = T_M(t_i) sin(beta_x) (-1)^x / (M (t_i - tau_x))
// with the phases reduced exactly through D = (2i+1)M - (2x+1)N and S = (2i+1)M + (2x+1)N:
//   l_x(t_i) = sin(beta_x) sinpi(D/(2N)) / (2M sinpi(S/(4NM)) sinpi(D/(4NM))),  = 1 when D = 0,
// where sinpi(D/(2N)) = (-1)^(x+1) cospi((2i+1)M/(2N)) (the argument reduced mod 4N in integers) and
// sinpi(S/(4NM)) = sin(a_i + g_x), a_i = pi(2i+1)/(4N), g_x = pi(2x+1)/(4M), both in (0, pi/2), so
// only sinpi(D/(4NM)) is evaluated per entry.  One CTA per (N, M) pair; node tables in shared memory.
__global__ void k_restr(DevJob J) {
  extern __shared__ double shq[];
  const int t = blockIdx.x;
  const int N = J.restr_N[2 * t], M = J.restr_N[2 * t + 1];
  double* RT = J.restr + J.restr_off[t];
  double* cA = shq;          // N: cospi((2i+1)M / (2N))
  double* sa = cA + N;       // N: sin(a_i)
  double* ca = sa + N;       // N: cos(a_i)
  double* sb = ca + N;       // M: (-1)^(x+1) sin(beta_x)
  double* sg = sb + M;       // M: sin(g_x)
  double* cg = sg + M;       // M: cos(g_x)
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    const long long A = ((long long)(2 * i + 1) * M) % (4LL * N);
    cA[i] = cospi((double)A / (2.0 * N));
    sincospi((double)(2 * i + 1) / (4.0 * N), &sa[i], &ca[i]);
  }
  for (int x = threadIdx.x; x < M; x += blockDim.x) {
    const double sbeta = sinpi((double)(2 * x + 1) / (2.0 * M));
    sb[x] = (x & 1) ? sbeta : -sbeta;
    sincospi((double)(2 * x + 1) / (4.0 * M), &sg[x], &cg[x]);
  }
  __syncthreads();
  const long long total = (long long)N * M;
  if (J.mixed) {
    // Mixed form: only the double-float table, computed on the FP32 pipe from the node tables
    // (converted in place, 8 bytes either way) with the exact fraction D / (4NM) for the sine.
    df* td = reinterpret_cast<df*>(shq);
    for (int k = threadIdx.x; k < 3 * (N + M); k += blockDim.x) td[k] = df_from(shq[k]);
    __syncthreads();
    const df *cAd = td, *sad = cAd + N, *cad = sad + N, *sbd = cad + N, *sgd = sbd + M, *cgd = sgd + M;
    const df m2d{(float)(2 * M), 0.f};
    const int den = 4 * N * M;
    float2* out = J.restr_df + J.restr_off[t];
    for (long long e = threadIdx.x; e < total; e += blockDim.x) {
      const int x = (int)(e / N), i = (int)(e % N);
      const int D = (2 * i + 1) * M - (2 * x + 1) * N;
      df v{1.f, 0.f};
      if (D != 0) {
        const df ssum = df_dot2(sad[i], cgd[x], cad[i], sgd[x]);
        v = df_div(df_mul(sbd[x], cAd[i]), df_mul(df_mul(m2d, ssum), df_sinpi_frac(D, den)));
      }
      out[e] = make_float2(v.hi, v.lo);
    }
    return;
  }
  const double nm4 = 4.0 * (double)N * (double)M, m2 = 2.0 * M;
  for (long long e = threadIdx.x; e < total; e += blockDim.x) {
    const int x = (int)(e / N), i = (int)(e % N);
    const long long D = (long long)(2 * i + 1) * M - (long long)(2 * x + 1) * N;
    double v = 1.0;
    if (D != 0) {
      const double ssum = fma(sa[i], cg[x], ca[i] * sg[x]);
      v = sb[x] * cA[i] / (m2 * ssum * sinpi((double)D / nm4));
    }
    RT[e] = v;
  }
}

// ---------------------------------------------------------------------------------------------
// A self-matrix entry: FP64, or (mixed form) the double-float pair the refinement reads plus its FP32
// rounding for the FP32 factorisation -- what a separate split of the FP64 matrix would give -- or (the
// FP64-kept form) the FP64 value, which k_afix turns into fixed point for the residual, plus its FP32 rounding.
// Mixed forms: systems that keep FP64 matrices and residuals (all in the FP64-kept form; N >= f64_min_n in
// the mixed form, whose large systems' conditioning would amplify a double-float matrix's rounding).
__device__ __forceinline__ bool sys_f64(const DevJob& J, int N) { return J.fp64keep || N >= J.f64_min_n; }

__device__ __forceinline__ void store_self(const DevJob& J, long long off, double2 v, bool f64) {
  if (f64) {
    J.A[off] = v;
    J.LU32[off] = make_float2(__double2float_rn(v.x), __double2float_rn(v.y));
  } else if (J.mixed) {
    const float4 d = df_split2(v);
    reinterpret_cast<float4*>(J.A)[off] = d;
    J.LU32[off] = make_float2(d.x, d.z);
  } else {
    J.A[off] = v;
  }
}

// Self assembly: A_ic = K1(t_i,t_c) Rlog_ic + K2(t_i,t_c) pi/N, symmetric in (i, c), for a band of consecutive
// frequencies sharing N (nodes, log weights, |t - s| and its logarithm are shared).  With K1 = -J0/(2 pi) an
// off-diagonal entry is the near rule's E = amp (beta cos - sin, cos) with beta = (2/pi)(ln|t_i - t_c| - Rlog_ic/w),
// below and above z = 20 alike (hankel_df.cuh).  kDf: double-float entries for the mixed form's systems that keep
// double-float matrices; else FP64 entries, bound by the FP64 pipe (84% busy) at 9 of its instructions an entry and ~30 a pair
// (the series and rotated recurrence before took 25 to 45 an entry): 6 arcs x 384 frequencies, N = 512: 24.6 -> 11.8 ms
// with the row bounds.
template <bool kDf>
__global__ void __launch_bounds__(256) k_assemble_self(DevJob J) {
  const SelfTile tile = J.tiles[blockIdx.x];
  const SysDesc s0 = J.sys[tile.sys];
  const int N = s0.N, nb = tile.nsys;
  if (kDf == (!J.mixed || sys_f64(J, N))) return;       // the other launch's systems
  __shared__ AngleTab<!kDf> ang;
  __shared__ FreqDf fr[kSelfBand];
  load_angles(ang);
  if (threadIdx.x < nb) fr[threadIdx.x] = J.freq_df ? J.freq_df[s0.l + threadIdx.x] : make_freq(s0.l + threadIdx.x);
  __syncthreads();
  const int i = tile.ti * kSelfTile + (threadIdx.x % kSelfTile);
  const int c = tile.tl * kSelfTile + (threadIdx.x / kSelfTile);
  if (i >= N || c >= N) return;
  if (tile.ti == tile.tl && i > c) return;
  const Panel pn = J.panels[s0.panel];
  const double rl = rlog_at(J.rlog + s0.rlog_off, N, i, c);
  const double w = kPiD / N, qw = 0.25 * w;
  const long long e1 = (long long)c * N + i, e2 = (long long)i * N + c;
  long long mo = s0.mat_off;                            // the band's matrices follow one another
  const long long nn = (long long)N * N;
  if (i == c) {
    // limit t -> s: K2 = i/4 - (1/(2 pi)) [gamma + ln(kappa |x'|/2)]
    const double lsp = log(0.5 * J.h * J.node_sp[pn.off + i]) - 1.1447298858494002;   // - ln pi (part of lnz)
    for (int b = 0; b < nb; ++b, mo += nn)
      store_self(J, mo + e1, make_double2(-0.5 * kInvPi * fma(w, fr[b].lnz + lsp, rl), qw), !kDf && J.mixed);
    return;
  }
  const double dx = J.node_x[pn.off + i] - J.node_x[pn.off + c];
  const double dy = J.node_y[pn.off + i] - J.node_y[pn.off + c];
  const double T = (J.h * (0.5 * kInvPi)) * dist_f64(fma(dx, dx, dy * dy));
  const double beta = kTwoOverPi * (log_f64(fabs(J.node_t[pn.off + i] - J.node_t[pn.off + c])) - rl * (N * kInvPi));
  if constexpr (kDf) {
    const PairTurns pt = pair_turns(T, df_from(qw * kInvPi));
    const df bd = df_split_bits(beta), qd = df_from(qw);
    df lnT{0.f, 0.f};
    if (pt.T.hi * fr[0].a.x < (float)kBesselLarge) lnT = df_log(pt.T);
    unsigned long long ph = pt.v * (unsigned long long)s0.l - (1ull << 61);
    for (int b = 0; b < nb; ++b, mo += nn, ph += pt.v) {
      const FreqDf& f = fr[b];
      const float4 d = pt.T.hi * f.a.x < (float)kBesselLarge
                           ? hankel_near_df(df_mul(pt.T, df{f.a.x, f.a.y}), df_add_fast(lnT, df{f.b.z, f.b.w}), bd, true, qd)
                           : hankel_far_df(pt, ph, ang.d, df{f.a.z, f.a.w}, df{f.b.x, f.b.y}, bd, true);
      const float2 h = make_float2(d.x, d.z);
      reinterpret_cast<float4*>(J.A)[mo + e1] = d;
      reinterpret_cast<float4*>(J.A)[mo + e2] = d;
      J.LU32[mo + e1] = h;
      J.LU32[mo + e2] = h;
    }
  } else {
    const PairF64 pt = pair_f64(T, qw * kInvPi);
    double lnT = 0.0;
    if (pt.th * fr[0].a.x < (float)kBesselLarge) lnT = log_f64(T);
    unsigned long long ph = pt.v * (unsigned long long)s0.l - (1ull << 61), u = pt.v62 * (unsigned long long)s0.l;
    for (int b = 0; b < nb; ++b, mo += nn, ph += pt.v, u += pt.v62) {
      const FreqDf& f = fr[b];
      const double2 v = pt.th * f.a.x < (float)kBesselLarge
                            ? hankel_near_f64(u, lnT + f.lnz, beta, true, qw)
                            : hankel_far_f64(pt, ph, ang.d, ang.f, df{f.a.z, f.a.w}, f.rs, beta, true);
      store_self(J, mo + e1, v, J.mixed);
      store_self(J, mo + e2, v, J.mixed);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Blocked right-looking LU with partial pivoting (pivot: max |re| + |im|, first index on ties),
// one CTA of 256 threads (small FP64 systems: 128) per system, panel width 8 in shared memory, column-major factor in HBM.
constexpr int kNB = 8;
constexpr int kPS = kNB + 1;   // padded panel row stride (bank-conflict-free column access)
constexpr int kLuThreads = 256;
constexpr int kLuNarrow = 135;   // FP64 jobs of systems up to this size: 128 threads (launch_lu says why)

// C = double2 (plain form: factors J.A in place) or float2 (mixed form: factors J.LU32 in place).  One system
// by the whole CTA (NT threads); shl_raw: lu_smem bytes of shared memory.
//
// FP64 trailing update in fixed point (fixed.cuh): A22 -= L21 U12 took 32 FP64 FMAs an entry and panel, the whole FP64
// pipe (75% of the kernel's time at its rate).  The multipliers are below 2 (partial pivoting on |re| + |im|) and a column
// of U12 shares one unit, so both become 60-bit integers in the same shared memory and the eight products sum in
// integers (low x low halves dropped), rounded once to 2^-57 of the column's largest entry; only the final conversion
// and subtraction are FP64: 6 instructions an entry and panel.  One FP64 rounding a panel in place of sixteen: |LU - PA|
// over |A| at N = 400 2.7e-16 against 9.3e-16 of the FMAs (oracle's self matrices), entry by entry 3.9e-16 against 1.3e-15
// of |L||U|.  A thread takes two columns of a row, so that each multiplier is read once for both.  8192 systems of N
// 48..259: 31.0 -> 16.6 ms; the FP64 pipe is still 73% busy (panels, U12, the conversions), and warps wait at the
// panels' barriers.
template <class C>
__host__ __device__ constexpr size_t lu_smem(int N) {
  const size_t panel = (size_t)N * (kNB + kPS) * sizeof(C) + (sizeof(C) == sizeof(double2) ? (size_t)N * sizeof(double) : 0);
  const size_t finish = (size_t)2 * kSB * kSB * sizeof(C);
  return panel > finish ? panel : finish;
}
template <class C, int NT>
__device__ void lu_one(const DevJob& J, int sidx, unsigned char* shl_raw) {
  C* shl = reinterpret_cast<C*>(shl_raw);
  const SysDesc s = J.sys[sidx];
  const int N = s.N;
  C* A = (sizeof(C) == sizeof(double2) ? reinterpret_cast<C*>(J.A) : reinterpret_cast<C*>(J.LU32)) + s.mat_off;
  int* piv = J.piv + s.piv_off;
  C* Pn = shl;                       // [N][kPS] panel rows
  C* U = shl + (size_t)N * kPS;      // [kNB][N] U12 rows
  [[maybe_unused]] double* unit = reinterpret_cast<double*>(U + (size_t)kNB * N);   // FP64: per column of U12
  __shared__ int spiv[kNB];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int k0 = 0; k0 < N; k0 += kNB) {
    const int w = min(kNB, N - k0);
    const int nr = N - k0;
    for (int idx = tid; idx < nr * w; idx += NT) {
      int c = idx / nr, r = idx % nr;
      Pn[r * kPS + c] = A[(long long)(k0 + c) * N + k0 + r];
    }
    __syncthreads();
    // The panel's columns by one warp (warp barriers only).
    if (wid == 0) {
      panel_factor_warp<C>(Pn, kPS, nr, w, spiv, lane);
      __syncwarp();
      if (lane < w) piv[k0 + lane] = k0 + spiv[lane];
    }
    __syncthreads();
    for (int idx = tid; idx < nr * w; idx += NT) {
      int c = idx / nr, r = idx % nr;
      A[(long long)(k0 + c) * N + k0 + r] = Pn[r * kPS + c];
    }
    // Row interchanges on the columns outside the panel.
    for (int col = tid; col < N; col += NT) {
      if (col >= k0 && col < k0 + w) continue;
      C* Ac = A + (long long)col * N + k0;
      for (int c = 0; c < w; ++c) {
        int p = spiv[c];
        if (p != c) { C t = Ac[c]; Ac[c] = Ac[p]; Ac[p] = t; }
      }
    }
    __syncthreads();
    const int nc = N - k0 - w;
    if (nc > 0) {
      // U12 = L11^{-1} A12 (unit lower triangular solve), one column per thread.
      for (int j = tid; j < nc; j += NT) {
        C* Ac = A + (long long)(k0 + w + j) * N + k0;
        C xv[kNB];
#pragma unroll
        for (int r = 0; r < kNB; ++r) {
          if (r < w) {
            C v = Ac[r];
            for (int c = 0; c < r; ++c) v = cfms(Pn[r * kPS + c], xv[c], v);
            xv[r] = v;
            Ac[r] = v;
            if constexpr (sizeof(C) == sizeof(float2)) U[r * N + j] = v;
          }
        }
        if constexpr (sizeof(C) == sizeof(double2)) {   // (w = kNB here: columns remain)
          unsigned top = 0u;
#pragma unroll
          for (int r = 0; r < kNB; ++r)
            top = max(top, max((unsigned)__double2hiint(xv[r].x) & 0x7FFFFFFFu, (unsigned)__double2hiint(xv[r].y) & 0x7FFFFFFFu));
          const int e = max((int)(top >> 20), 100) - 1022;
#pragma unroll
          for (int r = 0; r < kNB; ++r) {
            const int2 x = fix_f64<kLuLow>(xv[r].x, e), y = fix_f64<kLuLow>(xv[r].y, e);
            reinterpret_cast<int4*>(U)[r * N + j] = make_int4(x.x, x.y, y.x, y.y);
          }
          unit[j] = lu_unit(e);
        }
      }
      __syncthreads();
      // A22 -= L21 U12.
      const int mr = nr - w;
      if constexpr (sizeof(C) == sizeof(double2)) {
        int4* L = reinterpret_cast<int4*>(Pn) + w * kPS;          // multipliers, converted in place
        const int4* Ui = reinterpret_cast<const int4*>(U);
        for (int idx = tid; idx < mr * kNB; idx += NT) {
          const int o = (idx / kNB) * kPS + idx % kNB;
          const C v = Pn[w * kPS + o];
          const int2 x = fix_f64<kLuLow>(v.x, 1), y = fix_f64<kLuLow>(v.y, 1);
          L[o] = make_int4(x.x, x.y, y.x, y.y);
        }
        __syncthreads();
        const int np = (nc + 1) / 2;
        for (int idx = tid; idx < mr * np; idx += NT) {
          const int r = idx % mr, j0 = 2 * (idx / mr), j1 = min(j0 + 1, nc - 1);
          C* a0 = A + (long long)(k0 + w + j0) * N + k0 + w + r;
          C* a1 = A + (long long)(k0 + w + j1) * N + k0 + w + r;
          C v0 = *a0, v1 = *a1;
          fixacc<kLuLow> re0, im0, re1, im1;
#pragma unroll
          for (int c = 0; c < kNB; ++c) {
            const int4 l = L[r * kPS + c], p = Ui[c * N + j0], q = Ui[c * N + j1];
            const int n0 = -l.z, n1 = -l.w;
            re0.mac(l.x, l.y, p.x, p.y);
            im0.mac(l.x, l.y, p.z, p.w);
            re1.mac(l.x, l.y, q.x, q.y);
            im1.mac(l.x, l.y, q.z, q.w);
            re0.mac(n0, n1, p.z, p.w);
            im0.mac(l.z, l.w, p.x, p.y);
            re1.mac(n0, n1, q.z, q.w);
            im1.mac(l.z, l.w, q.x, q.y);
          }
          auto less = [](double v, double u, const fixacc<kLuLow>& s) { return fma(-u, ll_to_double(s.nearest()), v); };
          const double u0 = unit[j0], u1 = unit[j1];
          v0 = make_double2(less(v0.x, u0, re0), less(v0.y, u0, im0));
          v1 = make_double2(less(v1.x, u1, re1), less(v1.y, u1, im1));
          *a0 = v0;
          if (j1 > j0) *a1 = v1;
        }
      } else
      for (long long idx = tid; idx < (long long)mr * nc; idx += NT) {
        int j = (int)(idx / mr), r = (int)(idx % mr);
        C* a = A + (long long)(k0 + w + j) * N + k0 + w + r;
        C v = *a;
#pragma unroll
        for (int c = 0; c < kNB; ++c)
          if (c < w) v = cfms(Pn[(w + r) * kPS + c], U[c * N + j], v);
        *a = v;
      }
    }
    __syncthreads();
  }
  lu_finish<C, NT>(A, N,
                           (sizeof(C) == sizeof(double2) ? reinterpret_cast<C*>(J.dinv) : reinterpret_cast<C*>(J.dinv32)) +
                               s.piv_off,
                           shl);
}

// Threads per system: the panel's columns are one warp's work, so an FP64 system below about a hundred nodes, whose
// shared memory lets six share an SM, runs faster on fewer (768 systems of N = 96: 1.73 -> 1.47 ms at 128 threads).  The
// FP32 form fits 48 registers, five CTAs an SM (8192 systems of N 48..259: three 5.53 ms, four 4.63, five 4.22).
template <class C, int NT>
__global__ void __launch_bounds__(NT, sizeof(C) == sizeof(double2) ? 768 / NT : 5) k_lu(DevJob J, const int* __restrict__ list) {
  extern __shared__ __align__(16) unsigned char shl_raw[];
  lu_one<C, NT>(J, list[blockIdx.x], shl_raw);
}

// ---------------------------------------------------------------------------------------------
// Triangular solves, one warp per system, all Q right-hand sides together, in blocks of kSB = 32
// rows: x_b = T_b^{-1} b_b with the inverted diagonal block (a 32 x 32 GEMV, lane = row), then the
// rows beyond the block are updated with the block's columns (independent loads, lane = row).
// ceil(N/32) dependent steps per sweep instead of N.  Both factors have a unit diagonal (U was scaled
// and D^{-1} is applied between the sweeps).  C = double2 (FP64 factors) or float2 (FP32 factors).
constexpr int kSolveWarps = 4;

// Rows i0 and i0 + 32 of every window's b_q -= T[:, r0..r0+w) x_q with x_q = b_q[r0..r0+w), column-major T
// of leading dimension N: each factor entry is loaded once for all QT windows.  Each batch of columns
// issues the loads of both rows before their FMAs, so a lane has 2 x kCols independent loads in flight
// instead of walking its rows one after another.  A second row past `end` is computed on the first and
// not stored.
template <class C, int QT, bool kLean>
__device__ __forceinline__ void tri_update2(C* b, int N, const C* __restrict__ A, int r0, int w, int i0, int end) {
  const int i1 = i0 + 32 < end ? i0 + 32 : i0;
  // columns per load batch: 16 FP32 or 8 FP64 entries per row, halved for 3-4 windows and in lean builds
  // (registers)
  constexpr int kCols = (sizeof(C) == 8 ? 16 : 8) / (QT > 2 ? 2 : 1) / (kLean ? 2 : 1);
  C a0[QT], a1[QT];
#pragma unroll
  for (int q = 0; q < QT; ++q) {
    a0[q] = b[q * N + i0];
    a1[q] = b[q * N + i1];
  }
#pragma unroll 1
  for (int c0 = 0; c0 < kSB; c0 += kCols) {
    C v0[kCols], v1[kCols];
#pragma unroll
    for (int k = 0; k < kCols; ++k) {
      if (c0 + k < w) {
        const C* col = A + (long long)(r0 + c0 + k) * N;
        v0[k] = __ldg(&col[i0]);
        v1[k] = __ldg(&col[i1]);
      }
    }
#pragma unroll
    for (int k = 0; k < kCols; ++k) {
      if (c0 + k < w) {
#pragma unroll
        for (int q = 0; q < QT; ++q) {
          const C x = b[q * N + r0 + c0 + k];
          a0[q] = cfms(v0[k], x, a0[q]);
          a1[q] = cfms(v1[k], x, a1[q]);
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < QT; ++q) {
    b[q * N + i0] = a0[q];
    if (i0 + 32 < end) b[q * N + i0 + 32] = a1[q];
  }
}

// x_q = T_kk^{-1} b_q on the block rows r0 .. r0+w (the diagonal block stored inverted, so a GEMV): lane =
// row, the block's entries loaded once for all QT windows.  lower: the unit-lower block (entries left of
// the diagonal); else the unit-upper one (right of it).
template <class C, int QT, bool kLean>
__device__ __forceinline__ void tri_diag(C* b, int N, const C* __restrict__ A, int r0, int w, int lane, bool lower) {
  constexpr int kH = kLean ? 8 : 16;
  C x[QT];
  if (lane < w) {
#pragma unroll
    for (int q = 0; q < QT; ++q) x[q] = b[q * N + r0 + lane];
#pragma unroll 1
    for (int h = 0; h < kSB; h += kH) {        // kH loads in flight, then their FMAs
      C v[kH];
#pragma unroll
      for (int k = 0; k < kH; ++k) {
        const bool use = lower ? h + k < lane : (h + k > lane && h + k < w);
        if (use) v[k] = __ldg(&A[(long long)(r0 + h + k) * N + r0 + lane]);
      }
#pragma unroll
      for (int k = 0; k < kH; ++k) {
        const bool use = lower ? h + k < lane : (h + k > lane && h + k < w);
        if (use) {
#pragma unroll
          for (int q = 0; q < QT; ++q) x[q] = cfms(make_neg(v[k]), b[q * N + r0 + h + k], x[q]);
        }
      }
    }
  }
  __syncwarp();
  if (lane < w) {
#pragma unroll
    for (int q = 0; q < QT; ++q) b[q * N + r0 + lane] = x[q];
  }
  __syncwarp();
}

// Both triangular sweeps of one system for its QT windows b[q * N + i] (shared memory), one warp (kLean:
// smaller load batches, for kernels with a tighter register budget).
template <class C, int QT, bool kLean = false>
__device__ void tri_solve(C* b, int N, const C* __restrict__ A, const int* __restrict__ piv,
                          const C* __restrict__ dinv, int lane) {
  if (lane < QT) {
    C* bq = b + lane * N;
    for (int k = 0; k < N; ++k) {
      const int p = __ldg(&piv[k]);
      if (p != k) { C t = bq[k]; bq[k] = bq[p]; bq[p] = t; }
    }
  }
  __syncwarp();
  for (int r0 = 0; r0 < N; r0 += kSB) {           // forward, unit lower
    const int w = min(kSB, N - r0), r1 = r0 + w;
    tri_diag<C, QT, kLean>(b, N, A, r0, w, lane, true);
#pragma unroll 1
    for (int i0 = r1 + lane; i0 < N; i0 += 64) tri_update2<C, QT, kLean>(b, N, A, r0, w, i0, N);
    __syncwarp();
  }
  for (int e = lane; e < QT * N; e += 32) b[e] = cmul(b[e], __ldg(&dinv[e % N]));
  __syncwarp();
  for (int r0 = ((N - 1) / kSB) * kSB; r0 >= 0; r0 -= kSB) {   // backward, unit upper
    const int w = min(kSB, N - r0);
    tri_diag<C, QT, kLean>(b, N, A, r0, w, lane, false);
#pragma unroll 1
    for (int i0 = lane; i0 < r0; i0 += 64) tri_update2<C, QT, kLean>(b, N, A, r0, w, i0, r0);
    __syncwarp();
  }
}

// Both sweeps of one system's FP64 factors for all QT windows of step m, by one warp (b: QT x N double2 of
// shared memory), then its densities, their running sum and (kept densities) step m's copy.
template <int QT, bool kLean = false>
__device__ void solve_one(const DevJob& J, int sidx, int m, double2* b, int lane) {
  const SysDesc s = J.sys[sidx];
  const int N = s.N;
  const double2* G = J.G + s.vec_off;
  for (int e = lane; e < QT * N; e += 32) b[e] = G[e];
  __syncwarp();
  tri_solve<double2, QT, kLean>(b, N, J.A + s.mat_off, J.piv + s.piv_off, J.dinv + s.piv_off, lane);
  double2* out = J.phi + s.vec_off;
  double2* sum = J.phi_sum + s.vec_off;
  double2* all = J.phi_all ? J.phi_all + (long long)(m - 1) * J.vec_total + s.vec_off : nullptr;
  for (int e = lane; e < QT * N; e += 32) {
    double2 v = b[e];
    out[e] = v;
    sum[e] = m == 1 ? v : cadd(sum[e], v);
    if (all) all[e] = v;
  }
  if (!J.otf) {
    __syncwarp();
#pragma unroll 1
    for (int q = 0; q < QT; ++q)
      fix_vector(b + q * N, N, 1.0, reinterpret_cast<int4*>(J.phi_df) + s.vec_off + (long long)q * N,
                 J.phi_unit + 4ll * sidx + q, lane);
  }
}

template <int QT>
__global__ void __launch_bounds__(32 * kSolveWarps) k_solve(DevJob J, int m) {
  extern __shared__ double2 shs[];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int slot = blockIdx.x * (blockDim.x >> 5) + wid;
  if (slot >= J.nsys) return;
  solve_one<QT>(J, J.sys_order[slot], m, shs + (size_t)wid * QT * J.max_n, lane);
}

// The FP64 self matrix of one system (plain form) by one CTA: every entry of the upper triangle (diagonal
// included) evaluated for the system's own frequency and stored at both mirror positions -- the log-split rule of
// k_assemble_self with other arithmetic: all in FP64, Taylor series below z = 20 and Hankel's asymptotic series above
// (bessel.cuh) instead of hankel_df.cuh's, and nothing shared across a band of frequencies.  The two matrices agree to
// FP64's rounding, not bit for bit.
__device__ void assemble_one(const DevJob& J, int sidx) {
  const SysDesc s = J.sys[sidx];
  const int N = s.N;
  const Panel pn = J.panels[s.panel];
  const double l = (double)s.l, lnl = log(l);
  const double w = kPiD / N, qw = 0.25 * w;
  const long long ntri = (long long)N * (N + 1) / 2;
  for (long long t = threadIdx.x; t < ntri; t += blockDim.x) {
    // t -> (i, c) with i <= c, column by column: c (c + 1) / 2 <= t < (c + 1) (c + 2) / 2
    int c = (int)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
    while ((long long)(c + 1) * (c + 2) / 2 <= t) ++c;
    while ((long long)c * (c + 1) / 2 > t) --c;
    const int i = (int)(t - (long long)c * (c + 1) / 2);
    const double rl = rlog_at(J.rlog + s.rlog_off, N, i, c);
    const long long e1 = (long long)c * N + i, e2 = (long long)i * N + c;
    double2 v;
    if (i == c) {
      const double lsp = log(0.5 * J.h * J.node_sp[pn.off + i]);
      v = make_double2(fma(-0.5 * kInvPi, rl, -0.5 * kInvPi * (kEulerGamma + lnl + lsp) * w), qw);
    } else {
      const double dx = J.node_x[pn.off + i] - J.node_x[pn.off + c];
      const double dy = J.node_y[pn.off + i] - J.node_y[pn.off + c];
      const double R = sqrt(fma(dx, dx, dy * dy));
      const double dts = fabs(J.node_t[pn.off + i] - J.node_t[pn.off + c]);
      const double hR = J.h * R, z = l * hR;
      if (z < kBesselLarge) {
        double J0, Yh;
        bessel0_taylor(z, J0, Yh);
        const double alpha = -0.5 * kInvPi * fma(w, lnl + log(hR / (2.0 * dts)) + kEulerGamma, rl);
        v = make_double2(fma(alpha, J0, -qw * Yh), qw * J0);
      } else {
        double J0, Y0;
        bessel0_asym(z, J0, Y0);
        const double alpha = -0.5 * kInvPi * (rl - w * log(dts));
        v = make_double2(fma(alpha, J0, -qw * Y0), qw * J0);
      }
    }
    J.A[s.mat_off + e1] = v;
    J.A[s.mat_off + e2] = v;
  }
}

// The fused kernel's step-1 solve, one window per warp (a single-window sweep needs few registers), as a
// separate call so that it keeps its own register allocation.
__device__ __noinline__ void fused_solve(const DevJob& J, int sidx, int q, double2* b, int lane) {
  const SysDesc s = J.sys[sidx];
  const int N = s.N;
  const long long o = s.vec_off + (long long)q * N;
  for (int e = lane; e < N; e += 32) b[e] = J.G[o + e];
  __syncwarp();
  tri_solve<double2, 1, true>(b, N, J.A + s.mat_off, J.piv + s.piv_off, J.dinv + s.piv_off, lane);
  double2* all = J.phi_all ? J.phi_all + o : nullptr;   // step 1's copy when densities are kept
  for (int e = lane; e < N; e += 32) {
    const double2 v = b[e];
    J.phi[o + e] = v;
    J.phi_sum[o + e] = v;
    if (all) all[e] = v;
  }
  if (!J.otf) {
    __syncwarp();
    fix_vector(b, N, 1.0, reinterpret_cast<int4*>(J.phi_df) + o, J.phi_unit + 4ll * sidx + q, lane);
  }
}

// Batching form, plain FP64: one persistent launch assembles, factors and solves (step 1) every (arc, omega)
// system.  Each CTA takes the next system from a work counter (systems by decreasing N, so the largest start
// first and the small ones fill the tail), assembles its matrix, factors it (lu_one) and solves its step-1
// windows, one warp per window; the counter is reset by the host before the launch.
constexpr int kFusedThreads = 256;
template <int QT>
__global__ void __launch_bounds__(kFusedThreads, 2) k_fused_asf(DevJob J, int* counter) {
  extern __shared__ __align__(16) unsigned char shf_raw[];
  __shared__ int s_item;
  for (;;) {
    if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
    __syncthreads();
    const int item = s_item;
    if (item >= J.nsys) return;
    const int sidx = J.sys_order[item];
    assemble_one(J, sidx);
    __syncthreads();
    lu_one<double2, kFusedThreads>(J, sidx, shf_raw);
    __syncthreads();
    const int wid = threadIdx.x >> 5;
    if (wid < QT) fused_solve(J, sidx, wid, reinterpret_cast<double2*>(shf_raw) + (size_t)wid * J.max_n, threadIdx.x & 31);
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------
// Cross assembly: stored rows of S_Gamma_j for one (pair, frequency band, 8-row chunk).
constexpr int kAsmThreads = 128;   // small blocks: an 8-row task leaves a short last pass
constexpr int kAsmMaxThreads = 256;   // largest cross-assembly block a tuned launch may use
constexpr int kAsmRows = 8;

constexpr int kAsmBand = 64;   // frequencies per assembly task (matches the planner's band cap)

// Near-rule corrections of the rows of one task at N source nodes (block-wide, all threads call), in FP64:
// beta[r * N + i] = -(2/pi)(W_i/w - ln|t* - t_i|) for the near rows r, with the product-integration weights
// W_i = (lambda_0 + 2 sum_{n<N} lambda_n T_n(t_i)) / N, lambda_n(t*) = int log|t* - s| T_n(s)/sqrt(1-s^2) ds for
// |t*| > 1, = -pi zeta^n / n (n >= 1).  The whole series sums to ln|t* - t_i| (beta is its tail from n = N on), so a row
// with |zeta|^N < 1e-18 has beta = 0 and is marked by +0.0 at every node without any sum (an exact zero of the formula
// would come out as -0.0): of the near rows only those next to the arc's ends keep the N-term sums and the
// logarithms.  12-arc cavity, table of all rows: 13.9 -> 1.9 ms.  tn: the nodes t_i; ctab: 2N + 1 doubles, lam:
// kAsmRows x N doubles of shared memory; beta may be shared or global memory.
__device__ void near_beta_block(const CrossTgt* tg, int nrows, int N, const double* __restrict__ tn, double* ctab,
                                double* lam, double* beta) {
  __shared__ int s_full[kAsmRows], s_any;
  if (threadIdx.x == 0) s_any = 0;
  __syncthreads();
  if (threadIdx.x < nrows) {
    int full = 0;
    if (tg[threadIdx.x].near) {
      const double ts = tg[threadIdx.x].tstar;
      const double rt = sqrt(fma(ts, ts, -1.0));
      const double zeta = ts > 0 ? ts - rt : ts + rt;
      if (!(N * log(fabs(zeta)) < -41.4465)) {            // |zeta|^N >= 1e-18 (or not a number)
        full = 1;
        s_any = 1;
        double* lr = lam + threadIdx.x * N;
        lr[0] = kPiD * log(0.5 * (fabs(ts) + rt));
        double pw = 1.0;
        for (int n = 1; n < N; ++n) {
          pw *= zeta;
          lr[n] = -kPiD * pw / n;
        }
      }
    }
    s_full[threadIdx.x] = full;
  }
  __syncthreads();
  if (s_any) {
    for (int r = threadIdx.x; r <= 2 * N; r += blockDim.x) ctab[r] = cospi((double)r / (2.0 * N));
    __syncthreads();
  }
  for (int e = threadIdx.x; e < nrows * N; e += blockDim.x) {
    const int r = e / N, i = e % N;
    if (!tg[r].near) continue;
    double v = 0.0;
    if (s_full[r]) {
      const double* lr = lam + r * N;
      const int step = 2 * i + 1, mod = 4 * N;
      double acc = 0.0;
      int ph = 0;
      for (int n = 1; n < N; ++n) {
        ph += step;
        if (ph >= mod) ph -= mod;
        acc = fma(lr[n], ctab[ph <= 2 * N ? ph : mod - ph], acc);
      }
      v = -kTwoOverPi * fma(lr[0] + 2.0 * acc, kInvPi, -log(fabs(tg[r].tstar - tn[i])));
    }
    beta[r * N + i] = v;
  }
  __syncthreads();
}

// kNear: the launch over the tasks with near rows (shared memory for their corrections); otherwise over the far-only
// tasks, which need only the tables (more CTAs per SM).  Each launch skips the other kind of task.  kF64: the FP64 form;
// else the mixed forms (FP64 below z = 20, double-float above).  A thread owns (row, source) pairs and walks the
// band's frequencies.  Bound by the FP64 pipe in the FP64 form (84% busy: 9 instructions an entry, ~25 a pair, which a
// band of about five frequencies shares on the obstacles; 8 arcs, 4.8e8 entries: 34 -> 12.4 ms); in the mixed forms by
// issue (68%, ~135 FP32 instructions an entry) and the FP64 of the pairs and of the entries below z = 20 (60%) together
// (12 -> 5.3 ms; N = 512 with 2.6e9 entries: 29.3 -> 17.1 ms).
template <bool kNear, bool kF64>
__global__ void __launch_bounds__(kAsmMaxThreads) k_cross_assemble(DevJob J) {
  extern __shared__ __align__(16) double sha[];
  const CrossAsm task = J.asms[blockIdx.x];
  const PairDesc pr = J.pairs[task.pair];
  const int N = task.N;
  const Panel pn = J.panels[task.panel];
  const CrossTgt* tg = J.tgts + pr.tgt_off + task.row0;
  const int nl = task.l1 - task.l0 + 1;
  FreqDf* fr = reinterpret_cast<FreqDf*>(sha);       // kAsmBand
  double* bt = sha + kAsmBand * (sizeof(FreqDf) / sizeof(double));   // near launch: kAsmRows x N corrections,
  double* lam = bt + kAsmRows * N;                   // kAsmRows x N and
  double* ctab = lam + kAsmRows * N;                 // 2N + 1 doubles of near_beta_block
  __shared__ AngleTab<kF64> ang;
  __shared__ int any_near;
  __shared__ unsigned s_r2[kAsmRows], s_beta[kAsmRows];   // smallest R^2 (FP64 high word), largest |beta| of a row (FP32 bits)
  __shared__ short s_exp[kAsmRows][kAsmBand];             // entries of (row, frequency) stay below 2^s_exp
  if (threadIdx.x == 0) {
    int a = 0;
    for (int r = 0; r < task.nrows; ++r) a |= tg[r].near;
    any_near = a;
  }
  __syncthreads();
  if ((any_near != 0) != kNear) return;
  load_angles(ang);
  for (int b = threadIdx.x; b < nl; b += blockDim.x) fr[b] = J.freq_df[task.l0 + b];
  if (threadIdx.x < kAsmRows) {
    s_r2[threadIdx.x] = 0x7FF00000u;
    s_beta[threadIdx.x] = 0u;
  }
  if (kNear) near_beta_block(tg, task.nrows, N, J.node_t + pn.off, ctab, lam, bt);
  __syncthreads();
  const double qw = 0.25 * kPiD / N, camp4 = qw * kInvPi, turns = J.h * (0.5 * kInvPi);
  // Fixed-point unit per row and frequency: |E| <= (w/4) |H0(z_min)| (1 + max |beta|), |H0(z)| <= sqrt(2/(pi z)) for
  // every z > 0 (z |H0|^2 increases to 2/pi), and <= 1.5 - 0.64 ln z below 1.  A row through a node, or with a
  // distance that is not finite, gets the unit NaN, as its entries would be.
  for (int e = threadIdx.x; e < task.nrows * N; e += blockDim.x) {
    const int r = e % task.nrows, i = e / task.nrows;
    const double dx = tg[r].x - J.node_x[pn.off + i], dy = tg[r].y - J.node_y[pn.off + i];
    const unsigned h = (unsigned)__double2hiint(fma(dx, dx, dy * dy));
    atomicMin(&s_r2[r], h - 0x100000u < 0x7FE00000u ? h : 0u);      // normal and finite
    if (kNear && tg[r].near) atomicMax(&s_beta[r], __float_as_uint(fabsf((float)bt[r * N + i])));
  }
  __syncthreads();
  for (int e = threadIdx.x; e < task.nrows * nl; e += blockDim.x) {
    const int r = e / nl, b = e % nl;
    const double T = turns * dist_f64(__hiloint2double((int)s_r2[r], 0));
    const float z = (float)T * fr[b].a.x * 0.99999f;
    float hb = sqrtf(0.63661978f / z);
    if (z < 1.f) hb = fminf(hb, 1.5f - 0.64f * ((float)(log_f64(T) + fr[b].lnz) + 0.1159f));   // (ln z, ln 2 - gamma)
    const float bound = (float)qw * hb * (1.f + __uint_as_float(s_beta[r])) * 1.0001f;
    const int s = max((int)(__float_as_uint(bound) >> 23) - 126, -64);
    s_exp[r][b] = (short)s;
    J.e_unit[J.row_off[(long long)task.pair * J.L + task.l0 + b] + task.row0 + r] =
        s_r2[r] != 0u && z < 3e38f && s < 120 ? __uint_as_float((unsigned)(s - fix_bits(kRowLow) + 127) << 23)
                                              : __uint_as_float(0x7FFFFFFFu);
  }
  __syncthreads();
  const df cd = df_from(camp4);
  const int ld = pr.nrows;   // blocks are stored source-major: E[i * nrows + row]
  const long long* eo = J.e_off + (long long)task.pair * J.L + task.l0;
  for (int e = threadIdx.x; e < task.nrows * N; e += blockDim.x) {
    const int r = e % task.nrows, i = e / task.nrows;
    const CrossTgt t = tg[r];
    const double dx = t.x - J.node_x[pn.off + i], dy = t.y - J.node_y[pn.off + i];
    const double T = turns * dist_f64(fma(dx, dx, dy * dy));
    const double beta = kNear && t.near ? bt[r * N + i] : 0.0;
    const bool near = kNear && beta != 0.0;
    int4* Ep = reinterpret_cast<int4*>(J.E) + (long long)i * ld + task.row0 + r;
    auto put = [&](int b, double2 v) {
      const int s = s_exp[r][b];
      const int2 x = fix_f64<kRowLow>(v.x, s), y = fix_f64<kRowLow>(v.y, s);
      Ep[eo[b]] = make_int4(x.x, x.y, y.x, y.y);
    };
    if constexpr (kF64) {
      const PairF64 pt = pair_f64(T, camp4);
      const double lnT = pt.th * fr[0].a.x < (float)kBesselLarge ? log_f64(T) : 0.0;
      unsigned long long ph = pt.v * (unsigned long long)task.l0 - (1ull << 61),
                         u = pt.v62 * (unsigned long long)task.l0;
      for (int b = 0; b < nl; ++b, ph += pt.v, u += pt.v62) {
        const FreqDf& f = fr[b];
        put(b, pt.th * f.a.x < (float)kBesselLarge ? hankel_near_f64(u, lnT + f.lnz, beta, near, qw)
                                                   : hankel_far_f64(pt, ph, ang.d, ang.f, df{f.a.z, f.a.w}, f.rs, beta, near));
      }
    } else {
      const PairTurns pt = pair_turns(T, cd);
      const df bd = kNear ? df_split_bits(beta) : df{0.f, 0.f};
      double lnT = 0.0;
      unsigned long long v62 = 0ull;
      if (pt.T.hi * fr[0].a.x < (float)kBesselLarge) {
        lnT = log_f64(T);
        v62 = turn_fraction(0.25 * T);
      }
      unsigned long long ph = pt.v * (unsigned long long)task.l0 - (1ull << 61);
      for (int b = 0; b < nl; ++b, ph += pt.v) {
        const FreqDf& f = fr[b];
        if (pt.T.hi * f.a.x < (float)kBesselLarge) {
          put(b, hankel_near_f64(v62 * (unsigned long long)(task.l0 + b), lnT + f.lnz, beta, near, qw));
          continue;
        }
        const float4 d = hankel_far_df(pt, ph, ang.d, df{f.a.z, f.a.w}, df{f.b.x, f.b.y}, bd, near);
        const float c = __uint_as_float((unsigned)(kRowLow - 1 - s_exp[r][b] + 127) << 23);
        const int2 x = fix_df<kRowLow>(d.x, d.y, c), y = fix_df<kRowLow>(d.z, d.w, c);
        Ep[eo[b]] = make_int4(x.x, x.y, y.x, y.y);
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Cross rows evaluated every step (cross_mode 1), nothing stored.  Near corrections beta first, once per job,
// into a table (one slab of nrows x N per assembly task with near rows).
__global__ void __launch_bounds__(kAsmThreads) k_near_weights(DevJob J) {
  const long long off = J.wn_off[blockIdx.x];
  if (off < 0) return;
  extern __shared__ double shn[];
  const CrossAsm task = J.asms[blockIdx.x];
  const CrossTgt* tg = J.tgts + J.pairs[task.pair].tgt_off + task.row0;
  near_beta_block(tg, task.nrows, task.N, J.node_t + J.panels[task.panel].off, shn,
                  shn + 2 * task.N + 1, J.wn + off);
}

constexpr int kOtfThreads = 32 * kAsmRows;

// V sums of a warp's lanes added over the lanes (V a power of two <= 32): each halving step keeps one half of the values
// and hands the other to the partner lane, so lane e << log2(32/V) ends with sum e.
template <int V>
__device__ __forceinline__ void warp_sums(double (&a)[V], int lane) {
  int w = 16;
#pragma unroll
  for (int n = V / 2; n >= 1; n >>= 1, w >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int e = 0; e < n; ++e) {
      const double keep = up ? a[e + n] : a[e], give = up ? a[e] : a[e + n];
      a[e] = keep + __shfl_xor_sync(0xffffffffu, give, w);
    }
  }
  for (; w >= 1; w >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], w);
}

// FP64 form: one CTA of kAsmRows warps per (assembly task, band of at most kOtfBand frequencies), warp = target row,
// lane = source node, frequencies in register blocks; each entry (hankel_df.cuh: 9 FP64 instructions) goes straight
// into the lane's FP64 sums, which are added over the lanes once per block.  Bound by the FP64 pipe; the rotated
// recurrences summed through shared memory before took 25 to 45 FP64 instructions an entry besides the 4 a window:
// 8 obstacle arcs, 256 frequencies, 2 steps: 23.3 -> 12.3 ms; 3 arcs of a disk at N = 96, 2 steps: 2.26 -> 0.88 ms.
__host__ __device__ constexpr int otf64_regs(int Q) { return Q == 1 ? 4 : Q == 2 ? 2 : 1; }
template <int Q>
__global__ void __launch_bounds__(kOtfThreads, 2) k_cross_otf(DevJob J) {
  constexpr int NB = otf64_regs(Q), V = NB * (Q == 3 ? 4 : Q) * 2;
  __shared__ AngleTab<true> ang;
  __shared__ FreqDf fr[kOtfBand];
  __shared__ long long vo[kOtfBand];
  const CrossOtf ot = J.otf_tasks[(int)((long long)blockIdx.x * J.otf_stride % J.n_otf)];
  const CrossAsm task = J.asms[ot.task];
  const PairDesc pr = J.pairs[task.pair];
  const int N = task.N, nl = ot.l1 - ot.l0 + 1;
  const Panel pn = J.panels[task.panel];
  const long long woff = J.wn_off[ot.task];
  const int tid = threadIdx.x, lane = tid & 31, r = tid >> 5;
  load_angles(ang);
  if (tid < nl) {
    fr[tid] = J.freq_df[ot.l0 + tid];
    vo[tid] = J.sys[(long long)pr.j * (J.L - 1) + (ot.l0 + tid - 1)].vec_off;
  }
  __syncthreads();
  if (r >= task.nrows) return;
  const CrossTgt t = J.tgts[pr.tgt_off + task.row0 + r];
  const double* __restrict__ bt = t.near ? J.wn + woff + (long long)r * N : nullptr;
  const bool near = bt && __double_as_longlong(__ldg(bt)) != 0;     // (+0.0: beta vanishes on the whole row)
  const double qw = 0.25 * kPiD / N, camp4 = qw * kInvPi, turns = J.h * (0.5 * kInvPi);
  const double* __restrict__ nx = J.node_x + pn.off;
  const double* __restrict__ ny = J.node_y + pn.off;
#pragma unroll 1
  for (int b0 = 0; b0 < nl; b0 += NB) {
    const int nb = min(NB, nl - b0);
    double acc[V];                                    // [frequency][window][re, im]
#pragma unroll
    for (int e = 0; e < V; ++e) acc[e] = 0.0;
#pragma unroll 1
    for (int i = lane; i < N; i += 32) {
      const double dx = t.x - __ldg(&nx[i]), dy = t.y - __ldg(&ny[i]);
      const double T = turns * dist_f64(fma(dx, dx, dy * dy));
      const PairF64 pt = pair_f64(T, camp4);
      const double beta = near ? __ldg(&bt[i]) : 0.0;
      const double lnT = pt.th * fr[b0].a.x < (float)kBesselLarge ? log_f64(T) : 0.0;
      unsigned long long ph = pt.v * (unsigned long long)(ot.l0 + b0) - (1ull << 61),
                         u = pt.v62 * (unsigned long long)(ot.l0 + b0);
#pragma unroll
      for (int k = 0; k < NB; ++k, ph += pt.v, u += pt.v62) {
        if (k < nb) {
          const FreqDf& f = fr[b0 + k];
          const double2 e = pt.th * f.a.x < (float)kBesselLarge
                                ? hankel_near_f64(u, lnT + f.lnz, beta, near, qw)
                                : hankel_far_f64(pt, ph, ang.d, ang.f, df{f.a.z, f.a.w}, f.rs, beta, near);
          const double2* __restrict__ pd = J.phi + vo[b0 + k] + i;
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            const double2 s = cfma(e, pd[(long long)q * N], make_double2(acc[(k * Q + q) * 2], acc[(k * Q + q) * 2 + 1]));
            acc[(k * Q + q) * 2] = s.x;
            acc[(k * Q + q) * 2 + 1] = s.y;
          }
        }
      }
    }
    warp_sums<V>(acc, lane);
    constexpr int kShift = V == 32 ? 0 : V == 16 ? 1 : V == 8 ? 2 : V == 4 ? 3 : 4;
    const int e = lane >> kShift, k = e / (2 * Q), q = (e / 2) % Q;
    if ((lane & ((1 << kShift) - 1)) == 0 && k < nb) {
      const long long row = J.row_off[(long long)task.pair * J.L + ot.l0 + b0 + k] + task.row0 + r;
      reinterpret_cast<double*>(J.apply_res)[(row * Q + q) * 2 + (e & 1)] = acc[0];
    }
  }
}

// Mixed forms, cross rows evaluated every step in double-float (on the FP32 pipe).  One CTA of kAsmRows warps per
// (assembly task of kAsmRows target rows, band of at most kOtfBand frequencies): warp = target row, lane = source
// node (s0 + lane, so node coordinates and densities load coalesced and the near rule is warp-uniform), frequencies
// in register blocks of otf_regs(Q).  A lane sets its pair up in turns (PairTurns), evaluates each entry and multiplies
// it straight into its own compensated double-float sums, one per (frequency, window); the 32 lanes' sums are added
// once per block of frequencies.  Entries never leave registers.  An earlier form wrote them to shared memory and
// summed with one thread per (row, frequency): at bands of one or two frequencies (N grows with every step of omega)
// 8 to 16 of its 128 threads worked, and each pair paid two sine/cosine series; 12-arc cavity, 5.7e8 pairs x 5 steps,
// four windows: 501 -> 89 ms; 6 arcs at N = 1024, two windows: 499 -> 329 ms.  At four windows bound by the FP64
// pipe (85% busy, issue 59%): a pair's set-up takes ~11 FP64 instructions (differences, distance, scaling), and blocks of
// one frequency share it with no other entry.  At two windows blocks of four share it: FMA pipe 62%, FP64 45%, issue 68%
// at two CTAs an SM, no pipe full.  (~135 FP32 instructions an entry and 24 to 48 a window.)
// kKeep64 (the FP64-kept form): entries below z = 20 in FP64.
__host__ __device__ constexpr int otf_regs(int Q) { return Q == 1 ? 8 : Q == 2 ? 4 : 1; }
// blocks per SM: 16 warps of 128 registers, or 24 of 80 where the few sums leave room (measured per Q)
constexpr int otf_blocks(int Q) { return Q <= 2 ? 2 : 3; }

// V double-float sums of a warp's lanes added over the lanes (V a power of two <= 32): each halving step keeps one
// half of the values and hands the other to the partner lane, so lane e << s (s = log2(32/V)) ends with sum e.
template <int V>
__device__ __forceinline__ void df_warp_sums(dfacc (&a)[V], int lane) {
  int w = 16;
#pragma unroll
  for (int n = V / 2; n >= 1; n >>= 1, w >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int e = 0; e < n; ++e) {
      const dfacc lo = a[e], hi = a[e + n];
      const float gh = up ? lo.hi : hi.hi, gl = up ? lo.lo : hi.lo;
      a[e] = up ? hi : lo;
      a[e].add(__shfl_xor_sync(0xffffffffu, gh, w), __shfl_xor_sync(0xffffffffu, gl, w));
    }
  }
  for (; w >= 1; w >>= 1) {
    const float gh = a[0].hi, gl = a[0].lo;
    a[0].add(__shfl_xor_sync(0xffffffffu, gh, w), __shfl_xor_sync(0xffffffffu, gl, w));
  }
}

template <int Q, bool kKeep64>
__global__ void __launch_bounds__(kOtfThreads, otf_blocks(Q)) k_cross_otf_df(DevJob J) {
  constexpr int B = kOtfBand, NB = otf_regs(Q);
  constexpr int V = NB * (Q == 3 ? 4 : Q) * 2;                      // sums per warp, a power of two
  __shared__ float4 ang[kAngles];
  __shared__ FreqDf fr[B];
  __shared__ long long vo[B];                                       // density offsets of the band's systems
  __shared__ df s_qw, s_camp4;                                      // w/4, w/(4 pi), one thread's FP64
  // blocks in a strided order: the low-frequency tasks (FP64 Taylor range of the FP64-kept form) are neighbours in
  // the list and spread over the launch, so the FP64 pipe works beside the other blocks' FP32
  const long long nt = J.n_otf, stride = J.otf_stride;
  const CrossOtf ot = J.otf_tasks[(int)((long long)blockIdx.x * stride % nt)];
  const CrossAsm task = J.asms[ot.task];
  const PairDesc pr = J.pairs[task.pair];
  const int N = task.N, nl = ot.l1 - ot.l0 + 1;
  const Panel pn = J.panels[task.panel];
  const long long woff = J.wn_off[ot.task];
  const int tid = threadIdx.x, lane = tid & 31, r = tid >> 5;
  for (int k = tid; k < kAngles; k += kOtfThreads) ang[k] = c_angle_df[k];
  if (tid < nl) {
    fr[tid] = J.freq_df[ot.l0 + tid];
    vo[tid] = J.sys[(long long)pr.j * (J.L - 1) + (ot.l0 + tid - 1)].vec_off;
  }
  if (tid == kOtfThreads - 1) {
    const double w4 = 0.25 * kPiD / N;
    s_qw = df_from(w4);
    s_camp4 = df_from(w4 * kInvPi);
  }
  __syncthreads();
  if (r >= task.nrows) return;
  const CrossTgt t = J.tgts[pr.tgt_off + task.row0 + r];
  const double* __restrict__ bt = t.near ? J.wn + woff + (long long)r * N : nullptr;
  const bool near = bt && __double_as_longlong(__ldg(bt)) != 0;     // (+0.0: beta vanishes on the whole row)
  const double qw64 = kKeep64 ? 0.25 * kPiD / N : 0.0, turns = J.h * (0.5 * kInvPi);
  const df qw = s_qw, camp4 = s_camp4;
  const double* __restrict__ nx = J.node_x + pn.off;
  const double* __restrict__ ny = J.node_y + pn.off;
#pragma unroll 1
  for (int b0 = 0; b0 < nl; b0 += NB) {
    const int nb = min(NB, nl - b0);
    dfacc acc[V];
    dfacc2 acc2[NB][Q / 2 > 0 ? Q / 2 : 1][2];      // windows in pairs: (re, im)
    // T one step ahead: its chain of dependent FP64 operations runs beside the current pair's entries
    auto turns_at = [&](int i) {
      const double dx = t.x - __ldg(&nx[i]), dy = t.y - __ldg(&ny[i]);
      return turns * dist_f64(fma(dx, dx, dy * dy));
    };
    double Tn = turns_at(min(lane, N - 1));
#pragma unroll 1
    for (int i = lane; i < N; i += 32) {
      const double T = Tn;
      if (i - lane + 32 < N) Tn = turns_at(min(i + 32, N - 1));
      const PairTurns pt = pair_turns(T, camp4);
      double beta64 = 0.0;
      df beta{0.f, 0.f};
      if (near) {
        beta64 = __ldg(&bt[i]);
        beta = df_split_bits(beta64);
      }
      df lnT{0.f, 0.f};
      double lnT64 = 0.0;
      unsigned long long v62 = 0ull;
      if (pt.T.hi * fr[b0].a.x < (float)kBesselLarge) {             // the block's first entry is below z = 20
        if (kKeep64) {
          lnT64 = log_f64(T);
          v62 = turn_fraction(0.25 * T);
        } else {
          lnT = df_log(pt.T);
        }
      }
      unsigned long long ph = pt.v * (unsigned long long)(ot.l0 + b0) - (1ull << 61);
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        if (k < nb) {
          const FreqDf& f = fr[b0 + k];
          // densities: windows in pairs (re hi hi lo lo, im hi hi lo lo), an odd last one alone
          float4 pv[Q], e;
          const float4* __restrict__ pd = J.phi_df + vo[b0 + k];
#pragma unroll
          for (int q = 0; q < Q; ++q)
            pv[q] = __ldg(&pd[q < (Q & ~1) ? (long long)(q & ~1) * N + 2 * i + (q & 1) : (long long)q * N + i]);
          if (pt.T.hi * f.a.x < (float)kBesselLarge) {
            if (kKeep64) {
              e = split2_bits(hankel_near_f64(v62 * (unsigned long long)(ot.l0 + b0 + k), lnT64 + f.lnz, beta64, near, qw64));
            } else {
              e = hankel_near_df(df_mul(pt.T, df{f.a.x, f.a.y}), df_add_fast(lnT, df{f.b.z, f.b.w}), beta, near, qw);
            }
          } else {
            e = hankel_far_df(pt, ph, ang, df{f.a.z, f.a.w}, df{f.b.x, f.b.y}, beta, near);
          }
          if constexpr (Q >= 2) {
            const f32x2 xr = pack2(e.x, e.x), nxr = pack2(-e.x, -e.x), nlr = pack2(-e.y, -e.y), lr = pack2(e.y, e.y);
            const f32x2 xi = pack2(e.z, e.z), nxi = pack2(-e.z, -e.z), nli = pack2(-e.w, -e.w), li = pack2(e.w, e.w);
#pragma unroll
            for (int g = 0; g < Q / 2; ++g) {
              const float4 a = pv[2 * g], b = pv[2 * g + 1];
              const f32x2 rh = pack2(a.x, a.y), rl = pack2(a.z, a.w), ih = pack2(b.x, b.y), il = pack2(b.z, b.w);
              acc2[k][g][0].mac(xr, nxr, nlr, rh, rl);
              acc2[k][g][0].mac(nxi, xi, li, ih, il);
              acc2[k][g][1].mac(xr, nxr, nlr, ih, il);
              acc2[k][g][1].mac(xi, nxi, nli, rh, rl);
            }
          }
          if constexpr (Q & 1) cdf_mac(acc[(k * Q + Q - 1) * 2], acc[(k * Q + Q - 1) * 2 + 1], e, pv[Q - 1]);
        }
        ph += pt.v;
      }
    }
#pragma unroll
    for (int k = 0; k < NB; ++k)
#pragma unroll
      for (int g = 0; g < Q / 2; ++g)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          dfacc &a = acc[(k * Q + 2 * g) * 2 + c], &b = acc[(k * Q + 2 * g + 1) * 2 + c];
          unpack2(acc2[k][g][c].hi, a.hi, b.hi);
          unpack2(acc2[k][g][c].lo, a.lo, b.lo);
        }
    df_warp_sums<V>(acc, lane);
    constexpr int kShift = V == 32 ? 0 : V == 16 ? 1 : V == 8 ? 2 : V == 4 ? 3 : 4;
    const int e = lane >> kShift, k = e / (2 * Q), q = (e / 2) % Q;
    if ((lane & ((1 << kShift) - 1)) == 0 && k < nb) {
      const df v = acc[0].value();
      const long long row = J.row_off[(long long)task.pair * J.L + ot.l0 + b0 + k] + task.row0 + r;
      reinterpret_cast<double*>(J.apply_res)[(row * Q + q) * 2 + (e & 1)] = (double)v.hi + (double)v.lo;
    }
  }
}

constexpr int kApplyThreads = 256;

// ---------------------------------------------------------------------------------------------
// Mixed-precision solve: an FP32 blocked solve with the FP32 factors, then refinement steps, each a
// residual r = G - A phi (A kept as double-float, about 48 bits, and the residual too; systems that keep
// FP64: A in 60-bit fixed point, the residual an exact sum rounded to FP64) and an FP32 correction, until the error estimated to remain is below
// J.refine_tol, or J.refine_max steps.  Each step shrinks the error by a factor rho (the FP32 solve's
// relative accuracy), so what remains after a correction of relative size rel is about rho * rel; rho is
// estimated by the ratio of the last two corrections, or after the first step by kFirstRhoSafety * rel
// (that correction is the FP32 solution's own error, about rho times the solution for a generic
// right-hand side; the factor covers large systems, where one right-hand side underestimates rho by up
// to ~10x).  A system still above the tolerance after J.refine_max steps is counted as unconverged.
// A step is two launches over the
// systems still refining: k_mresid (fixed point) or k_mresid_df (double-float) streams the kept matrix with
// one thread per row (many warps in flight per SM), k_msolve runs the triangular solves with one warp per system and little
// register state.  Until a system finishes, its densities sit in its phi slots as double-float pairs
// (16 bytes, the size of the FP64 value written there at the end).
constexpr int kRefineCap = 16;          // largest refine_max accepted
constexpr double kFirstRhoSafety = 10.0;
constexpr int kResidThreads = 128;

// Asynchronous 16-byte copies global -> shared (bypassing L1), for streams whose loads would otherwise
// occupy registers until they land.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(kPending) : "memory");
}

// One thread's row of a fixed-point product: sums over N sources of entry (at src + i stride) times the densities
// den[q N + i] of every window.  The entries stream through the thread's own ring of kStages batches in shared memory
// (ring + k blockDim.x, cp.async): the next batches are in flight while one is summed and hold no registers; a thread
// reads only the slots it filled itself (no barrier).  The densities are the same for the whole warp: one cached load
// per column.
constexpr int kFixStages = 2;
__host__ __device__ constexpr int fix_batch(int Q) { return Q <= 2 ? 8 : 4; }   // entries a batch
constexpr size_t fix_ring_bytes(int Q, int threads) { return (size_t)kFixStages * fix_batch(Q) * threads * sizeof(int4); }
template <int Q, int kLow>
__device__ __forceinline__ void fix_row(const int4* __restrict__ src, long long stride, int N, const int4* __restrict__ den,
                                        int4* ring, fixacc<kLow> (&re)[Q], fixacc<kLow> (&im)[Q]) {
  constexpr int kB = fix_batch(Q);
  const int T = blockDim.x, nbat = N / kB;
  auto mac = [&](const int4 e, int i) {
    const int n0 = -e.z, n1 = -e.w;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int4 p = __ldg(&den[q * N + i]);
      re[q].mac(e.x, e.y, p.x, p.y);
      im[q].mac(e.x, e.y, p.z, p.w);
      re[q].mac(n0, n1, p.z, p.w);
      im[q].mac(e.z, e.w, p.x, p.y);
    }
  };
  auto issue = [&](int bi) {
    int4* dst = ring + (bi % kFixStages) * kB * T;
    const int4* s = src + (long long)bi * kB * stride;
#pragma unroll
    for (int k = 0; k < kB; ++k) cp_async16(dst + k * T, s + k * stride);
  };
#pragma unroll
  for (int bi = 0; bi < kFixStages - 1; ++bi) {
    if (bi < nbat) issue(bi);
    cp_async_commit();
  }
#pragma unroll 1
  for (int bi = 0; bi < nbat; ++bi) {
    if (bi + kFixStages - 1 < nbat) issue(bi + kFixStages - 1);
    cp_async_commit();                          // (empty near the end: keeps the group count uniform)
    cp_async_wait<kFixStages - 1>();            // batch bi has landed
    const int4* s = ring + (bi % kFixStages) * kB * T;
#pragma unroll
    for (int k = 0; k < kB; ++k) mac(s[k * T], bi * kB + k);
    // a source adds two products to a sum
    if ((bi + 1) % (fix_run(kLow) / 2 / kB) == 0) {
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        re[q].carry();
        im[q].carry();
      }
    }
  }
  for (int i = nbat * kB; i < N; ++i) mac(__ldg(&src[(long long)i * stride]), i);
}

// The FP64-kept matrices in fixed point (fixed.cuh) for the refinement, converted in place once per job after the assembly:
// every entry of row i as a 60-bit integer in units of a power of two just above the row's largest component (rounding
// below 2^-60 of it; a row with an entry that is not finite gets the unit NaN).  A block stages kRows rows of one
// system in shared memory, so the matrix is read and written once: bound by HBM.
constexpr int kFixThreads = 256;
template <int kRows>
__global__ void __launch_bounds__(kFixThreads) k_afix(DevJob J) {
  extern __shared__ __align__(16) double2 shx[];        // [N][kRows]
  __shared__ unsigned s_max[kRows];
  const ResidChunk c = J.rchunks[blockIdx.x];
  const SysDesc s = J.sys[c.sys];
  const int N = s.N, r = threadIdx.x % kRows, j0 = threadIdx.x / kRows;
  if (!sys_f64(J, N)) return;
  double2* A = J.A + s.mat_off;
  for (int row0 = c.row0; row0 < min(c.row0 + 32, N); row0 += kRows) {
    if (threadIdx.x < kRows) s_max[threadIdx.x] = 0u;
    __syncthreads();
    const bool on = row0 + r < N;
    if (on) {
      unsigned m = 0u;
      for (int j = j0; j < N; j += kFixThreads / kRows) {
        const double2 v = __ldcs(&A[(long long)j * N + row0 + r]);
        shx[j * kRows + r] = v;
        m = max(m, max((unsigned)__double2hiint(v.x) & 0x7FFFFFFFu, (unsigned)__double2hiint(v.y) & 0x7FFFFFFFu));
      }
      atomicMax(&s_max[r], m);
    }
    __syncthreads();
    if (on) {
      const int e = max((int)(s_max[r] >> 20) - 1022, -60);         // every |component| < 2^e
      for (int j = j0; j < N; j += kFixThreads / kRows) {
        const double2 v = shx[j * kRows + r];
        const int2 x = fix_f64<kMatLow>(v.x, e), y = fix_f64<kMatLow>(v.y, e);
        __stcs(reinterpret_cast<int4*>(A) + (long long)j * N + row0 + r, make_int4(x.x, x.y, y.x, y.y));
      }
      if (j0 == 0)
        J.a_unit[s.piv_off + row0 + r] =
            e > 60 ? __uint_as_float(0x7FFFFFFFu) : __uint_as_float((unsigned)(e - fix_bits(kMatLow) + 127) << 23);
    }
    __syncthreads();
  }
}

// Refinement residuals of the systems that keep FP64, one thread per row (rows past N recompute the last row and store
// nothing), all Q windows of the row: pass 1 r = G - A phi_0, later passes r <- r - A d with the last correction (the same value: phi grew by d).
// Matrix and vector are fixed-point and the sum is exact (low x low halves dropped), rounded once to FP64 and once more in
// the subtraction -- below an FP64 accumulation's error; all residuals run in units of a power of two of the right-hand side (exact).  Bound by HBM (16
// bytes an entry, 0.68 of a copy's rate; issue 37%); the FP64 and anchored FP32 sums (first pass) and double-float sums (later ones) before, 96 to 225
// instructions an entry at two windows, were issue-bound: N = 512, 2304 systems, 8 steps: 30.5 + 20.6 -> 15.8 + 16.5 ms.
template <int Q>
__global__ void __launch_bounds__(kResidThreads, 4) k_mresid(DevJob J, int pass) {
  const int chunk = blockIdx.x * (kResidThreads / 32) + (threadIdx.x >> 5);
  if (chunk >= J.n_rchunks) return;
  const ResidChunk c = J.rchunks[chunk];
  if (J.mdone[c.sys]) return;
  const SysDesc s = J.sys[c.sys];
  const int N = s.N;
  if (!sys_f64(J, N)) return;                 // double-float systems: k_mresid_df
  const int i = c.row0 + (threadIdx.x & 31);
  const int row = i < N ? i : N - 1;
  extern __shared__ __align__(16) int4 she[];
  fixacc<kMatLow> re[Q], im[Q];
  fix_row<Q, kMatLow>(reinterpret_cast<const int4*>(J.A) + s.mat_off + row, N, N, reinterpret_cast<const int4*>(J.phi_df) + s.vec_off,
             she + threadIdx.x, re, im);
  if (i >= N) return;
  const double ua = (double)J.a_unit[s.piv_off + i] * (double)(1ll << 2 * kMatLow);
  const double isc = pass == 1 ? 1.0 / J.mscale[c.sys] : 0.0;   // a power of two: exact
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const long long o = s.vec_off + (long long)q * N + i;
    double2 r;
    if (pass == 1) {
      const double2 g = J.G[o];
      r = make_double2(g.x * isc, g.y * isc);
    } else {
      r = J.rres64[o];
    }
    const double u = ua * J.phi_unit[4ll * c.sys + q];
    r.x = fma(-u, re[q].value(), r.x);
    r.y = fma(-u, im[q].value(), r.y);
    J.rres64[o] = r;
    J.rres[o] = make_float2(__double2float_rn(r.x), __double2float_rn(r.y));
  }
}

// The same for the mixed form's systems that keep double-float matrices: r = G - A phi in compensated double-float sums
// (one window: HBM-bound already, and no conversion of the matrix).
template <int Q>
__global__ void __launch_bounds__(kResidThreads) k_mresid_df(DevJob J) {
  const int chunk = blockIdx.x * (kResidThreads / 32) + (threadIdx.x >> 5);
  if (chunk >= J.n_rchunks) return;
  const ResidChunk c = J.rchunks[chunk];
  if (J.mdone[c.sys]) return;
  const SysDesc s = J.sys[c.sys];
  const int N = s.N;
  if (sys_f64(J, N)) return;                  // these: k_mresid
  const int i = c.row0 + (threadIdx.x & 31);
  const int row = i < N ? i : N - 1;
  const float4* __restrict__ Adf = reinterpret_cast<const float4*>(J.A) + s.mat_off;
  const float4* __restrict__ ph = reinterpret_cast<const float4*>(J.phi + s.vec_off);
  const double2* __restrict__ G = J.G + s.vec_off;
  const double isc = 1.0 / J.mscale[c.sys];   // a power of two: exact
  dfacc re[Q], im[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const double2 g = G[q * N + row];
    const float4 gd = df_split2(make_double2(g.x * isc, g.y * isc));
    re[q].add(gd.x, gd.y);
    im[q].add(gd.z, gd.w);
  }
  int j0 = 0;
  if (Q == 1) {
    // 16 matrix entries of the row loaded before their sums; the 16 densities (the same for the whole
    // warp) loaded once by 16 lanes and handed round by shuffles.  Same order of sums as below.
    constexpr int kB = 16;
    const int lane = threadIdx.x & 31;
    for (; j0 + kB <= N; j0 += kB) {
      float4 a[kB];
#pragma unroll
      for (int k = 0; k < kB; ++k) a[k] = __ldg(&Adf[(long long)(j0 + k) * N + row]);
      const float4 pv = ph[j0 + (lane & (kB - 1))];
#pragma unroll
      for (int k = 0; k < kB; ++k) {
        const float4 x = make_float4(__shfl_sync(0xffffffffu, pv.x, k), __shfl_sync(0xffffffffu, pv.y, k),
                                     __shfl_sync(0xffffffffu, pv.z, k), __shfl_sync(0xffffffffu, pv.w, k));
        cdf_mac(re[0], im[0], make_float4(-a[k].x, -a[k].y, -a[k].z, -a[k].w), x);
      }
    }
  }
  constexpr int kUnroll = Q == 1 ? 8 : Q == 2 ? 4 : 2;   // loads in flight without spilling
#pragma unroll kUnroll
  for (int j = j0; j < N; ++j) {
    const float4 a = __ldg(&Adf[(long long)j * N + row]);
    const float4 na = make_float4(-a.x, -a.y, -a.z, -a.w);
#pragma unroll
    for (int q = 0; q < Q; ++q) cdf_mac(re[q], im[q], na, ph[q * N + j]);
  }
  if (i < N) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const df rr = re[q].value(), ri = im[q].value();
      J.rres[s.vec_off + q * N + i] = make_float2(rr.hi + rr.lo, ri.hi + ri.lo);
    }
  }
}

// One warp: the FP32 solution (or correction) b[0..N) of one window in fixed point for the next residual.
__device__ __forceinline__ void fix_correction(const float2* b, int N, int4* out, double* unit, int lane) {
  unsigned m = 0u;
  for (int i = lane; i < N; i += 32)
    m = max(m, max(__float_as_uint(b[i].x) & 0x7FFFFFFFu, __float_as_uint(b[i].y) & 0x7FFFFFFFu));
  m = __reduce_max_sync(0xffffffffu, m);
  const int e = max((int)(m >> 23), 30) - 126;          // every |component| < 2^e (subnormal and tiny: any unit does)
  const bool bad = m >= 0x7F800000u || e > 120;
  const float c0 = __uint_as_float((unsigned)(127 - e / 2) << 23), c1 = __uint_as_float((unsigned)(kMatLow - 1 - (e - e / 2) + 127) << 23);
  for (int i = lane; i < N; i += 32) {                  // (scaled in two steps: 2^(29 - e) may leave FP32's range)
    const int2 x = fix_f32<kMatLow>(__fmul_rn(b[i].x, c0), c1), y = fix_f32<kMatLow>(__fmul_rn(b[i].y, c0), c1);
    out[i] = make_int4(x.x, x.y, y.x, y.y);
  }
  if (lane == 0)
    *unit = bad ? __longlong_as_double(0x7FF8000000000000ll) : __hiloint2double((e - fix_bits(kMatLow) + 1023) << 20, 0);
}

// pass 0: solve with FP32 G, store phi as double-float (systems that keep FP64: as FP64, and in fixed point for the
// residual), mark the system as refining.  pass p >= 1: solve for the correction from the residual, add it in
// double-float (FP64), and finish the system (FP64 densities, their copy for the cross rows, their running sum, the
// statistics) once the correction is small enough or p = J.refine_max.
template <int QT>
__global__ void __launch_bounds__(32 * kSolveWarps, 3) k_msolve(DevJob J, int m, int pass) {
  extern __shared__ __align__(16) unsigned char shm_raw[];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nw = blockDim.x >> 5;
  const int slot = blockIdx.x * nw + wid;
  if (slot >= J.nsys) return;
  const int sidx = J.sys_order[slot];
  if (pass > 0 && J.mdone[sidx]) return;
  const SysDesc s = J.sys[sidx];
  const int N = s.N, Q = QT;
  const bool f64 = sys_f64(J, N);            // densities refined in FP64 (FP64 residual)
  float2* b = reinterpret_cast<float2*>(shm_raw) + (size_t)wid * Q * J.max_n;
  const float2* __restrict__ L32 = J.LU32 + s.mat_off;
  const int* __restrict__ piv = J.piv + s.piv_off;
  const float2* __restrict__ dinv = J.dinv32 + s.piv_off;
  float4* ph = reinterpret_cast<float4*>(J.phi + s.vec_off);
  double scale;
  if (pass == 0) {
    // the refinement runs in units of scale = 2^k >= max |G| (exact), so that no data underflow FP32
    const double2* __restrict__ G = J.G + s.vec_off;
    double gmax = 0.0;
    for (int e = lane; e < Q * N; e += 32) gmax = fmax(gmax, fmax(fabs(G[e].x), fabs(G[e].y)));
    for (int o = 16; o > 0; o >>= 1) gmax = fmax(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
    int ex = 0;
    frexp(gmax, &ex);
    scale = gmax > 0.0 ? ldexp(1.0, ex) : 1.0;
    if (lane == 0) J.mscale[sidx] = scale;
    const double isc = 1.0 / scale;
    for (int e = lane; e < Q * N; e += 32) {
      const double2 g = G[e];
      b[e] = make_float2(__double2float_rn(g.x * isc), __double2float_rn(g.y * isc));
    }
  } else {
    scale = J.mscale[sidx];
    const float2* __restrict__ r = J.rres + s.vec_off;
    for (int e = lane; e < Q * N; e += 32) b[e] = r[e];
  }
  __syncwarp();
  tri_solve<float2, QT>(b, N, L32, piv, dinv, lane);
  double2* ph64 = J.phi + s.vec_off;
  auto keep = [&] {                           // b for the next residual
#pragma unroll 1
    for (int q = 0; q < QT; ++q)
      fix_correction(b + q * N, N, reinterpret_cast<int4*>(J.phi_df) + s.vec_off + (long long)q * N,
                     J.phi_unit + 4ll * sidx + q, lane);
  };
  if (pass == 0) {
    for (int e = lane; e < Q * N; e += 32) {
      if (f64) ph64[e] = make_double2(b[e].x, b[e].y);
      else ph[e] = make_float4(b[e].x, 0.f, b[e].y, 0.f);
    }
    if (f64) keep();
    if (lane == 0) J.mdone[sidx] = 0;
    return;
  }
  float dmax = 0.f, pmax = 0.f;
  for (int e = lane; e < Q * N; e += 32) {
    const float2 d = b[e];
    if (f64) {
      double2 p = ph64[e];
      p.x += (double)d.x;
      p.y += (double)d.y;
      ph64[e] = p;
      pmax = fmaxf(pmax, fmaxf(fabsf((float)p.x), fabsf((float)p.y)));
    } else {
      float4 p = ph[e];
      float sh, sl;
      two_sum(p.x, d.x, sh, sl);
      quick_two_sum(sh, sl + p.y, p.x, p.y);
      two_sum(p.z, d.y, sh, sl);
      quick_two_sum(sh, sl + p.w, p.z, p.w);
      ph[e] = p;
      pmax = fmaxf(pmax, fmaxf(fabsf(p.x), fabsf(p.z)));
    }
    dmax = fmaxf(dmax, fmaxf(fabsf(d.x), fabsf(d.y)));
  }
  for (int o = 16; o > 0; o >>= 1) {
    dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    pmax = fmaxf(pmax, __shfl_xor_sync(0xffffffffu, pmax, o));
  }
  const double rel = pmax > 0.f ? (double)dmax / (double)pmax : 0.0;
  // contraction factor: after the first correction, twice the largest one measured for this system in an
  // earlier step, else kFirstRhoSafety x rel; later, the ratio of the last two corrections (remembered)
  double rho;
  if (pass == 1) {
    const float known = J.mrho[sidx];
    rho = known > 0.f ? 2.0 * (double)known : kFirstRhoSafety * rel;
  } else {
    rho = rel / fmax((double)J.mrel[sidx], 1e-300);
    if (lane == 0) J.mrho[sidx] = fmaxf(J.mrho[sidx], fminf((float)rho, 1.0f));
  }
  const double left = rel * rho;
  if (left >= J.refine_tol && pass < J.refine_max) {
    if (f64) keep();
    if (lane == 0) J.mrel[sidx] = (float)rel;
    return;
  }
  if (lane == 0) {
    J.mdone[sidx] = 1;
    // non-negative doubles and floats order like their bit patterns
    atomicMax(reinterpret_cast<unsigned long long*>(J.refine_resid), (unsigned long long)__double_as_longlong(left));
    atomicAdd(reinterpret_cast<unsigned long long*>(J.refine_resid) + 1, (unsigned long long)pass);
    if (!(left < J.refine_tol)) atomicAdd(reinterpret_cast<unsigned long long*>(J.refine_resid) + 2, 1ULL);
    atomicMax(reinterpret_cast<int*>(J.sys_err) + sidx, __float_as_int(fminf((float)left, 3.0e38f)));
  }
  // Each lane reads back the values it wrote itself (in units of scale) and replaces them by FP64.
  double2* out = J.phi + s.vec_off;
  double2* sum = J.phi_sum + s.vec_off;
  double2* all = J.phi_all ? J.phi_all + (long long)(m - 1) * J.vec_total + s.vec_off : nullptr;
  float4* pdf = J.phi_df + s.vec_off;
  for (int e = lane; e < Q * N; e += 32) {
    double2 v = f64 ? out[e] : df_join2(ph[e]);
    v = make_double2(v.x * scale, v.y * scale);
    if (J.otf) {                              // windows in pairs, as k_cross_otf_df reads them
      const float4 d = df_split2(v);
      const int q = e / N, i = e % N;
      if (q < (QT & ~1)) {
        float* p = reinterpret_cast<float*>(pdf + (long long)(q & ~1) * N + 2 * i) + (q & 1);
        p[0] = d.x;
        p[2] = d.y;
        p[4] = d.z;
        p[6] = d.w;
      } else {
        pdf[e] = d;
      }
    }
    out[e] = v;
    sum[e] = m == 1 ? v : cadd(sum[e], v);
    if (all) all[e] = v;
  }
  if (!J.otf) {
    __syncwarp();
#pragma unroll 1
    for (int q = 0; q < QT; ++q)
      fix_vector(out + q * N, N, 1.0, reinterpret_cast<int4*>(pdf) + (long long)q * N, J.phi_unit + 4ll * sidx + q, lane);
  }
}

// Cross apply: W_k(x, q, l) = sum_j sum_i E_{l,k,j}[i, r] phi_j[q, i]; observation sums accumulate.  First half: one CTA
// per slice of kApplySlice rows of a group (the rows of all its source blocks, concatenated), one thread per row, the
// source-major blocks read coalesced.  Entries and densities are fixed-point (fixed.cuh), the sums exact integers,
// so one kernel serves every form (fix_row).  Bound by HBM (16 bytes an entry): 8 obstacle arcs, 4.8e8 entries, 12 steps: 42.7 (FP64 FMAs) ->
// 17.2 ms, 0.84 of a copy's rate; the mixed forms' double-float sums took 16.8 (N = 512, two windows: 70 either way).
template <int Q>
__global__ void __launch_bounds__(kApplySlice, Q == 1 ? 3 : 2) k_cross_rows(DevJob J) {
  extern __shared__ __align__(16) int4 she[];
  const ApplySlice sl = J.slices[blockIdx.x];
  if ((int)threadIdx.x >= sl.nrows) return;
  const int row = sl.row0 + threadIdx.x;
  // the thread's source block: the slice's blocks hold consecutive rows of the group
  int b = sl.b0, r = row - sl.rowb0;
  while (r >= J.blks[b].nrows) {
    r -= J.blks[b].nrows;
    ++b;
  }
  const CrossBlk B = J.blks[b];
  fixacc<kRowLow> re[Q], im[Q];
  fix_row<Q, kRowLow>(reinterpret_cast<const int4*>(J.E + B.e_off) + r, B.nrows, B.N,
             reinterpret_cast<const int4*>(J.phi_df) + J.sys[B.sys].vec_off, she + threadIdx.x, re, im);
  const long long rr = J.grp_res_off[sl.grp] + row;
  const double unit = (double)J.e_unit[rr] * (double)(1ll << 2 * kRowLow);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const double u = unit * J.phi_unit[4ll * B.sys + q];
    J.apply_res[rr * Q + q] = make_double2(re[q].value() * u, im[q].value() * u);
  }
}

// Second half: per group, the row sums of every source block added to their targets in
// the fixed block order (deterministic), then W (transfer nodes) or the observation spectra.
template <int Q>
__global__ void __launch_bounds__(kApplyThreads) k_cross_reduce(DevJob J) {
  extern __shared__ __align__(16) unsigned char shd_raw[];
  const CrossGrp g = J.grps[blockIdx.x];
  const int l = g.l;
  const bool obs = g.k == J.P;
  const int nout = obs ? J.n_obs : J.panels[J.tpanel[g.k]].N;
  double2* acc = reinterpret_cast<double2*>(shd_raw);      // [Q][nout]
  for (int e = threadIdx.x; e < Q * nout; e += kApplyThreads) acc[e] = make_double2(0.0, 0.0);
  __syncthreads();
  const double2* res = J.apply_res + J.grp_res_off[blockIdx.x] * Q;
  int row0 = 0;
  for (int bb = g.blk_begin; bb < g.blk_end; ++bb) {
    const CrossBlk B = J.blks[bb];
    for (int r = threadIdx.x; r < B.nrows; r += kApplyThreads) {
      const int o = J.tgts[B.tgt_off + r].out;
#pragma unroll
      for (int q = 0; q < Q; ++q) acc[q * nout + o] = cadd(acc[q * nout + o], res[(row0 + r) * Q + q]);
    }
    row0 += B.nrows;
    __syncthreads();
  }
  if (obs) {
    for (int e = threadIdx.x; e < Q * nout; e += kApplyThreads) {
      int q = e / nout, z = e % nout;
      double2* v = J.Vobs + ((long long)z * Q + q) * J.L + l;
      *v = cadd(*v, acc[e]);
    }
  } else {
    const long long base = J.tr_off[g.k];
    for (int e = threadIdx.x; e < Q * nout; e += kApplyThreads) {
      int q = e / nout, x = e % nout;
      J.W[((base + x) * Q + q) * J.L + l] = acc[e];
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Time-domain kernels: one CTA per active transfer node.
constexpr int kTimeThreads = 256;
constexpr int kTimeMaxThreads = 512;   // largest time-transform block a tuned launch may use

// The transforms' complex arithmetic: FP64, or double-float on the FP32 pipe (mixed form; complex values as float4:
// re.hi, re.lo, im.hi, im.lo).
struct FftF64 {
  using T = double2;
  static __device__ __forceinline__ const T* tw(const DevJob& J) { return J.fft_tw; }
  static __device__ __forceinline__ T mul(T a, T b) { return cmul(a, b); }
  static __device__ __forceinline__ T add(T a, T b) { return cadd(a, b); }
  static __device__ __forceinline__ T sub(T a, T b) { return csub(a, b); }
  static __device__ __forceinline__ T neg(T a) { return make_double2(-a.x, -a.y); }
  static __device__ __forceinline__ T conj(T a) { return make_double2(a.x, -a.y); }
  static __device__ __forceinline__ T times_i(T a) { return make_double2(-a.y, a.x); }
  static __device__ __forceinline__ T from(double2 a) { return a; }
  static __device__ __forceinline__ double2 to(T a) { return a; }
};
struct FftDf {
  using T = float4;
  static __device__ __forceinline__ const T* tw(const DevJob& J) { return J.fft_tw_df; }
  static __device__ __forceinline__ T mul(T a, T b) { return dfc_mul(a, b); }
  static __device__ __forceinline__ T add(T a, T b) { return dfc_add(a, b); }
  static __device__ __forceinline__ T sub(T a, T b) { return dfc_sub(a, b); }
  static __device__ __forceinline__ T neg(T a) { return make_float4(-a.x, -a.y, -a.z, -a.w); }
  static __device__ __forceinline__ T conj(T a) { return make_float4(a.x, a.y, -a.z, -a.w); }
  static __device__ __forceinline__ T times_i(T a) { return make_float4(-a.z, -a.w, a.x, a.y); }
  static __device__ __forceinline__ T from(double2 a) { return df_split2(a); }
  static __device__ __forceinline__ double2 to(T a) { return df_join2(a); }
};

// In-place decimation-in-time FFT of n = 2^logn points, y_r = sum_b X_b e^{-2 pi i b r/n}, input in bit-reversed order,
// two radix-2 stages at a time (three complex products per four points; a single stage first when logn is odd).
// tw: e^{-2 pi i r/K}, r < K/2, K a multiple of n.
template <class O>
__device__ void block_fft(typename O::T* buf, int logn, const typename O::T* __restrict__ tw, int K) {
  using T = typename O::T;
  const int n = 1 << logn;
  int half = 1;
  if (logn & 1) {
    for (int j = threadIdx.x; j < n / 2; j += blockDim.x) {
      const T a = buf[2 * j], c = buf[2 * j + 1];
      buf[2 * j] = O::add(a, c);
      buf[2 * j + 1] = O::sub(a, c);
    }
    __syncthreads();
    half = 2;
  }
  for (; half < n; half *= 4) {
    const int ts = K / (4 * half);          // twiddle stride of the second stage
    for (int j = threadIdx.x; j < n / 4; j += blockDim.x) {
      const int pos = j & (half - 1), i0 = ((j & ~(half - 1)) << 2) + pos;
      T* p = buf + i0;
      const T x0 = p[0];
      T t1 = p[half], t2 = p[2 * half], t3 = p[3 * half];
      if (half > 1) {
        const int k = pos * ts, k3 = 3 * k;
        t1 = O::mul(t1, tw[2 * k]);
        t2 = O::mul(t2, tw[k]);
        t3 = O::mul(t3, k3 < K / 2 ? tw[k3] : O::neg(tw[k3 - K / 2]));
      }
      const T y0 = O::add(x0, t1), y1 = O::sub(x0, t1), u = O::add(t2, t3), v = O::times_i(O::sub(t2, t3));
      p[0] = O::add(y0, u);
      p[half] = O::sub(y1, v);
      p[2 * half] = O::sub(y0, u);
      p[3 * half] = O::add(y1, v);
    }
    __syncthreads();
  }
}

__device__ __forceinline__ int bitrev(int b, int logK) { return (int)(__brev((unsigned)b) >> (32 - logK)); }

// Both transforms work on real samples of one period K, so each window takes one complex FFT of K/2 points: even
// samples in the real part and odd ones in the imaginary part.  FP64 form: bound by the FP64 pipe, about half of the
// full-length radix-2 transforms' work (4096 samples, two windows, 2 700 nodes: 31.3 -> 14.3 ms a job of 7 steps).

// Windowed slow transforms of g[0..NT) into out[q*L + l] (eq. Fourierk with the exact phase split): with C the FFT of
// x[2n] + i x[2n+1], bin k of the real sequence is (C_k + C*_{-k})/2 - (i/2) e^{-2 pi i k/K} (C_k - C*_{-k}).
template <class O>
__device__ void forward_all(const DevJob& J, const double* g, double2* sbuf, double2* out) {
  using T = typename O::T;
  T* buf = reinterpret_cast<T*>(sbuf);
  const int K = J.K, K2 = K / 2, NT = J.NT, L = J.L;
  const T* __restrict__ tw = O::tw(J);
  for (int q = 0; q < J.Q; ++q) {
    const double* wq = J.win + (long long)q * NT;
    for (int b = threadIdx.x; b < K2; b += blockDim.x) {
      double2 acc = make_double2(0.0, 0.0);
      for (int n = 2 * b; n < NT; n += K) {
        acc.x = fma(g[n], wq[n], acc.x);
        if (n + 1 < NT) acc.y = fma(g[n + 1], wq[n + 1], acc.y);
      }
      buf[bitrev(b, J.logK - 1)] = O::from(acc);
    }
    __syncthreads();
    block_fft<O>(buf, J.logK - 1, tw, K);
    for (int l = threadIdx.x; l < L; l += blockDim.x) {
      double2 v = make_double2(0.0, 0.0);
      if (l > 0) {
        const int k = l & (K - 1), kk = k & (K2 - 1);
        const T c = buf[kk], d = O::conj(buf[(K2 - kk) & (K2 - 1)]);
        const T t = k < K2 ? tw[kk] : O::neg(tw[kk]);
        const T y = O::sub(O::add(c, d), O::times_i(O::mul(t, O::sub(c, d))));   // twice the bin
        const double2 yy = O::to(y);
        v = cmul(J.fwd_tw[q * L + l], make_double2(0.5 * yy.x, -0.5 * yy.y));
      }
      out[q * L + l] = v;
    }
    __syncthreads();
  }
}

// g[nlo_q + r] += Re sum_l syn_tw[l] W_l e^{-2 pi i l r/K} for one window: with S the spectrum folded to one period,
// the real part's spectrum is H_b = (S_b + S*_{-b})/2, and the K/2-point FFT of (H_b + H_{b+K/2}) + i e^{-2 pi i b/K}
// (H_b - H_{b+K/2}) gives the samples in pairs.
template <class O>
__device__ void synth_window(const DevJob& J, int q, const double2* __restrict__ Wq, double2* sbuf, double* g) {
  using T = typename O::T;
  T* buf = reinterpret_cast<T*>(sbuf);
  const int K = J.K, K2 = K / 2, L = J.L, NT = J.NT;
  const T* __restrict__ tw = O::tw(J);
  const double2* __restrict__ st = J.syn_tw + (long long)q * L;
  auto fold = [&](int b, double2& s) {        // S_b; l = 0 (the constant) is not solved
    bool any = false;
    for (int l = (b == 0 ? K : b); l < L; l += K) {
      s = any ? cfma(st[l], Wq[l], s) : cmul(st[l], Wq[l]);
      any = true;
    }
    return any;
  };
  for (int b = threadIdx.x; b < K2; b += blockDim.x) {
    // twice H_b and H_{b+K/2}: S_b + S*_{K-b} and S_{b+K/2} + S*_{K/2-b}
    double2 s0{}, s1{}, s2{}, s3{};
    bool lo = fold(b, s0), hi = fold(b + K2, s1);
    if (fold((K - b) & (K - 1), s2)) {
      s0 = lo ? cadd(s0, make_double2(s2.x, -s2.y)) : make_double2(s2.x, -s2.y);
      lo = true;
    }
    if (fold(K2 - b, s3)) {
      s1 = hi ? cadd(s1, make_double2(s3.x, -s3.y)) : make_double2(s3.x, -s3.y);
      hi = true;
    }
    T v = O::from(make_double2(0.0, 0.0));
    if (lo || hi) {
      const T a = O::from(s0), c = O::from(s1);
      const T e = !hi ? a : !lo ? c : O::add(a, c), o = !hi ? a : !lo ? O::neg(c) : O::sub(a, c);
      v = O::add(e, O::times_i(O::mul(tw[b], o)));
    }
    buf[bitrev(b, J.logK - 1)] = v;
  }
  __syncthreads();
  block_fft<O>(buf, J.logK - 1, tw, K);
  const int n0 = J.nlo[q];
  for (int r = threadIdx.x; r < K2; r += blockDim.x) {
    const double2 v = O::to(buf[r]);
    const int n = n0 + 2 * r;
    if (n < NT) g[n] = fma(0.5, v.x, g[n]);
    if (n + 1 < NT) g[n + 1] = fma(0.5, v.y, g[n + 1]);
  }
  __syncthreads();
}

// Sampled signal: the degree-7 Lagrange interpolant through the samples i0 .. i0 + 7, i0 = floor(s) - 3,
// s = (t - t0)/dt (missing samples count as zero), and 0 outside [t0, t0 + (n_t - 1) dt].  With x = s - i0
// in [3, 4), the weight of sample i0 + k is prod_{m != k} (x - m) / prod_{m != k} (k - m), the numerator
// from prefix and suffix products.
__device__ double sampled_f(const DevJob& J, double t) {
  const double tend = J.sig_t0 + (double)(J.sig_nt - 1) * J.sig_dt;
  if (!(t >= J.sig_t0 && t <= tend)) return 0.0;
  const double s = (t - J.sig_t0) / J.sig_dt;
  const double fl = floor(s);
  const int i0 = (int)fl - 3;
  const double x = s - fl + 3.0;
  constexpr double kDen[8] = {-5040.0, 720.0, -240.0, 144.0, -144.0, 240.0, -720.0, 5040.0};
  double pre[8], suf[8];
  pre[0] = 1.0;
#pragma unroll
  for (int k = 1; k < 8; ++k) pre[k] = pre[k - 1] * (x - (double)(k - 1));
  suf[7] = 1.0;
#pragma unroll
  for (int k = 6; k >= 0; --k) suf[k] = suf[k + 1] * (x - (double)(k + 1));
  double acc = 0.0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int i = i0 + k;
    const double fi = (i >= 0 && i < J.sig_nt) ? __ldg(&J.sig_f[i]) : 0.0;
    acc = fma(pre[k] * suf[k] / kDen[k], fi, acc);
  }
  return acc;
}

__device__ __forceinline__ double signal_f(const DevJob& J, double t) {
  if (J.sig_nt > 0) return sampled_f(J, t);
  const double a = (t - J.centre) / J.width;
  return J.amp * sin(J.carrier * t) * exp(-a * a);
}

// u^i at (X, Y) and time t (plane wave, or point source by the trapezoid rule in v).
__device__ double incident_u(const DevJob& J, double X, double Y, double t) {
  if (J.sig_kind == 1) return signal_f(J, t - fma(Y, J.diry, X * J.dirx));
  const double dx = X - J.z0x, dy = Y - J.z0y;
  const double r = sqrt(fma(dx, dx, dy * dy));
  // f(t - tau) can be nonzero for tau in [t - (end of f), t - (start of f)]
  const bool smp = J.sig_nt > 0;
  const double tau_hi = smp ? t - J.sig_t0 : t - J.centre + 8.0 * J.width;
  if (tau_hi <= r) return 0.0;
  const double tau_lo = fmax(r, smp ? t - (J.sig_t0 + (double)(J.sig_nt - 1) * J.sig_dt)
                                    : t - J.centre - 8.0 * J.width);
  if (tau_lo >= tau_hi) return 0.0;
  const double v_lo = acosh(tau_lo / r), v_hi = acosh(tau_hi / r);
  const double band = smp ? J.sig_band : fabs(J.carrier) + 8.0 / J.width;
  const double rate = band * r * sinh(v_hi) + 1.0;
  const int n = (int)ceil((v_hi - v_lo) * (1.25 * rate + 24.0) / (2.0 * kPiD) * 2.0) + 16;
  const double dv = (v_hi - v_lo) / n;
  double acc = 0.5 * (signal_f(J, t - r * cosh(v_lo)) + signal_f(J, t - r * cosh(v_hi)));
  for (int k = 1; k < n; ++k) acc += signal_f(J, t - r * cosh(v_lo + k * dv));
  return acc * dv * (0.5 * kInvPi);
}

// Incident time samples g[a][n] = sign chi_k u^i(x, t_n) at the active transfer nodes, t_n = -H + n dt.
//
// Point source with the analytic signal (k_incident_ps): the trapezoid rule in v for a run of kIncRun consecutive
// samples on the run's common range [v_lo(t_first), v_hi(t_last)] (it contains every sample's own range, outside
// of which f < e^{-64}) with the step of the run's largest rate.  With rho = r cosh v, t_c the run's middle
// sample, d = t_c - centre - rho and delta = dt, the signal at t_c + j delta is
//   f = amp Im(e^{i carrier (t_c - rho)} e^{-(d/width)^2} b^j Gamma_j),   b = e^{-2 delta d/width^2},
//   Gamma_j = e^{i carrier j delta} e^{-(j delta/width)^2},
// so a term costs one seed (cosh, sincos, two exp) per run and three FP64 operations per sample (b^j by repeated
// multiplication from the middle outwards, at most kIncRun / 2 of them), Gamma_j entering after the sum.  One warp
// per (row, run), the terms split over its lanes: a row's runs are few in a small job, and one thread per run left
// the GPU empty (45 nodes, 256 samples: 1.45 ms; 0.1 ms so).  Runs whose Gaussian factor could change by more
// than e^{-64} within the run (dt kIncRun > 2 width) and sampled signals evaluate every sample directly.
//
// Rows are the active nodes, or (J.inc_m > 0) inc_m first-kind Chebyshev points of the interval of distances
// r = |x - z0| that the active nodes span: u^i depends on the node through r alone and is analytic in it, so its
// interpolant in r gives every node's samples (k_inc_interp, one small FP64 product) to below rounding; the number of
// points follows from the signal's growth on a Bernstein ellipse (incident_points).  12-arc cavity with 2 500
// active nodes: 76 rows instead of 2 500.
constexpr int kIncRun = 16;
constexpr int kIncThreads = 128;

__device__ __forceinline__ double inc_point(const DevJob& J, int i) {
  return fma(J.inc_half, cospi((2.0 * i + 1.0) / (2.0 * J.inc_m)), J.inc_mid);
}

// Direct form: one thread per sample.
__global__ void __launch_bounds__(kIncThreads) k_incident_u(DevJob J) {
  const int a = blockIdx.x;
  const int n = blockIdx.y * kIncThreads + threadIdx.x;
  if (n >= J.NT) return;
  const int k = J.act_arc[a], x = J.act_idx[a];
  const Panel pn = J.panels[J.tpanel[k]];
  const double pref = J.sign * J.chi[J.tr_off[k] + x];
  J.ginc[(long long)a * J.NT + n] =
      pref * incident_u(J, J.node_x[pn.off + x], J.node_y[pn.off + x], -J.H + n * J.dt);
}

__global__ void __launch_bounds__(kIncThreads) k_incident_ps(DevJob J) {
  const int row = blockIdx.x, lane = threadIdx.x & 31;
  const int n0 = (blockIdx.y * (kIncThreads / 32) + (threadIdx.x >> 5)) * kIncRun;
  if (n0 >= J.NT) return;
  const int nr = min(kIncRun, J.NT - n0);
  double r, pref, *out;
  if (J.inc_m > 0) {
    r = inc_point(J, row);
    pref = 1.0;
    out = J.inc_u;
  } else {
    const int k = J.act_arc[row], x = J.act_idx[row];
    const Panel pn = J.panels[J.tpanel[k]];
    const double dx = J.node_x[pn.off + x] - J.z0x, dy = J.node_y[pn.off + x] - J.z0y;
    r = sqrt(fma(dx, dx, dy * dy));
    pref = J.sign * J.chi[J.tr_off[k] + x];
    out = J.ginc;
  }
  out += (long long)row * J.NT + n0;
  constexpr int kMid = kIncRun / 2;
  const double t_first = -J.H + n0 * J.dt, t_last = -J.H + (n0 + nr - 1) * J.dt;
  double v[2 * kIncRun];   // [2 j] real, [2 j + 1] imaginary part of sum_k T_k b_k^(j - kMid)
#pragma unroll
  for (int j = 0; j < 2 * kIncRun; ++j) v[j] = 0.0;
  double sc = 0.0;
  const double tau_hi = t_last - J.centre + 8.0 * J.width;
  const double tau_lo = fmax(r, t_first - J.centre - 8.0 * J.width);
  if (tau_hi > r && tau_lo < tau_hi) {
    const double v_lo = acosh(tau_lo / r), v_hi = acosh(tau_hi / r);
    const double rate = (fabs(J.carrier) + 8.0 / J.width) * r * sinh(v_hi) + 1.0;
    const int n = (int)ceil((v_hi - v_lo) * (1.25 * rate + 24.0) / (2.0 * kPiD) * 2.0) + 16;
    const double dv = (v_hi - v_lo) / n;
    const double iw2 = 1.0 / (J.width * J.width);
    const double t_c = -J.H + (n0 + kMid) * J.dt;
    for (int kk = lane; kk <= n; kk += 32) {
      const double rho = r * cosh(fma((double)kk, dv, v_lo));
      const double wgt = (kk == 0 || kk == n) ? 0.5 : 1.0;
      const double d = t_c - J.centre - rho;
      double sp, cp;
      sincos(J.carrier * (t_c - rho), &sp, &cp);
      const double e0 = wgt * exp(-d * d * iw2), x = 2.0 * J.dt * d * iw2;
      const double b = exp(-x), ib = exp(x);
      cp *= e0;
      sp *= e0;
      v[2 * kMid] += cp;
      v[2 * kMid + 1] += sp;
      double p = b, m = ib;
#pragma unroll
      for (int j = 1; j <= kMid; ++j) {
        if (kMid + j < kIncRun) {
          v[2 * (kMid + j)] = fma(p, cp, v[2 * (kMid + j)]);
          v[2 * (kMid + j) + 1] = fma(p, sp, v[2 * (kMid + j) + 1]);
          p *= b;
        }
        v[2 * (kMid - j)] = fma(m, cp, v[2 * (kMid - j)]);
        v[2 * (kMid - j) + 1] = fma(m, sp, v[2 * (kMid - j) + 1]);
        m *= ib;
      }
    }
    sc = pref * J.amp * dv * (0.5 * kInvPi);
  }
  // sum over the lanes: each step keeps half of the values, so lane e ends with value e (j = e / 2)
#pragma unroll
  for (int w = kIncRun; w >= 1; w >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int e = 0; e < w; ++e) {
      const double keep = up ? v[e + w] : v[e], give = up ? v[e] : v[e + w];
      v[e] = keep + __shfl_xor_sync(0xffffffffu, give, w);
    }
  }
  const double im = __shfl_down_sync(0xffffffffu, v[0], 1);
  const int j = lane >> 1;
  if ((lane & 1) == 0 && j < nr) {
    const double y = (j - kMid) * J.dt, g = exp(-(y / J.width) * (y / J.width));
    double s, c;
    sincos(J.carrier * y, &s, &c);
    out[j] = sc * g * fma(s, v[0], c * im);
  }
}

// Lagrange basis of the inc_m Chebyshev points at every active node's distance, times sign chi_k (barycentric
// form, weights (-1)^i sin((2i+1) pi/(2m))); one warp per node.
__global__ void __launch_bounds__(kIncThreads) k_inc_basis(DevJob J) {
  const int a = blockIdx.x * (kIncThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (a >= J.n_act) return;
  const int k = J.act_arc[a], x = J.act_idx[a], m = J.inc_m;
  const Panel pn = J.panels[J.tpanel[k]];
  const double dx = J.node_x[pn.off + x] - J.z0x, dy = J.node_y[pn.off + x] - J.z0y;
  const double r = sqrt(fma(dx, dx, dy * dy));
  const double pref = J.sign * J.chi[J.tr_off[k] + x];
  double* L = J.inc_basis + (long long)a * m;
  double den = 0.0;
  int hit = -1;
  for (int i = lane; i < m; i += 32) {
    double s, c;
    sincospi((2.0 * i + 1.0) / (2.0 * m), &s, &c);
    const double d = r - fma(J.inc_half, c, J.inc_mid);
    if (d == 0.0) hit = i;
    const double q = ((i & 1) ? -s : s) / (d == 0.0 ? 1.0 : d);
    L[i] = q;
    den += q;
  }
  for (int o = 16; o > 0; o >>= 1) {
    den += __shfl_xor_sync(0xffffffffu, den, o);
    hit = max(hit, __shfl_xor_sync(0xffffffffu, hit, o));
  }
  const double sc = pref / den;
  for (int i = lane; i < m; i += 32) L[i] = hit >= 0 ? (i == hit ? pref : 0.0) : L[i] * sc;
}

// ginc[a][n] = sum_i basis[a][i] u[i][n]: 64 x 64 tiles, 4 x 4 values a thread, 16 points staged at a time.  FP64-pipe
// bound (2 n_act m NT flops: 2.3 GFLOP, 2 ms, for the 12-arc cavity with four windows).
constexpr int kItpTile = 64, kItpK = 16;
__global__ void __launch_bounds__(256) k_inc_interp(DevJob J) {
  __shared__ double As[kItpK][kItpTile + 1], Bs[kItpK][kItpTile];
  const int a0 = blockIdx.y * kItpTile, n0 = blockIdx.x * kItpTile, m = J.inc_m;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[4][4] = {};
  for (int k0 = 0; k0 < m; k0 += kItpK) {
    for (int e = threadIdx.x; e < kItpK * kItpTile; e += 256) {
      const int ka = e % kItpK, a = e / kItpK, kb = e / kItpTile, n = e % kItpTile;
      As[ka][a] = a0 + a < J.n_act && k0 + ka < m ? J.inc_basis[(long long)(a0 + a) * m + k0 + ka] : 0.0;
      Bs[kb][n] = n0 + n < J.NT && k0 + kb < m ? J.inc_u[(long long)(k0 + kb) * J.NT + n0 + n] : 0.0;
    }
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < kItpK; ++k) {
      double av[4], bv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        av[i] = As[k][ty + 16 * i];
        bv[i] = Bs[k][tx + 16 * i];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int a = a0 + ty + 16 * i;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx + 16 * j;
      if (a < J.n_act && n < J.NT) J.ginc[(long long)a * J.NT + n] = acc[i][j];
    }
  }
}

// Slow transforms of the incident samples of one active transfer node (eq. Fourierk per window).
template <bool DF>
__global__ void __launch_bounds__(kTimeMaxThreads) k_incident(DevJob J) {
  extern __shared__ double2 sht[];
  const int a = blockIdx.x;
  const int k = J.act_arc[a], x = J.act_idx[a];
  double2* buf = sht;                                   // K/2
  double* g = reinterpret_cast<double*>(sht + J.K / 2); // NT
  const double* src = J.ginc + (long long)a * J.NT;
  for (int n = threadIdx.x; n < J.NT; n += blockDim.x) g[n] = src[n];
  __syncthreads();
  forward_all<std::conditional_t<DF, FftDf, FftF64>>(J, g, buf, J.Gt + (J.tr_off[k] + x) * J.Q * J.L);
}

// PART = 0: the whole step at one transfer node (synthesis, -chi_k, windowed forward transforms).  In a
// frequency-partitioned job the synthesis sums only this rank's frequencies: PART = 1 writes those partial
// samples to J.ginc, the ranks add them, and PART = 2 reads the sums back and finishes the step.
template <bool DF, int PART>
__global__ void __launch_bounds__(kTimeMaxThreads) k_synth_fwd(DevJob J) {
  extern __shared__ double2 sht[];
  const int a = blockIdx.x;
  const int k = J.act_arc[a], x = J.act_idx[a];
  using O = std::conditional_t<DF, FftDf, FftF64>;
  const int L = J.L, NT = J.NT;
  double2* buf = sht;                                   // K/2
  double* g = reinterpret_cast<double*>(sht + J.K / 2); // NT
  const long long base = (J.tr_off[k] + x) * J.Q * L;
  double* gpart = J.ginc + (long long)a * NT;
  if (PART == 2) {
    for (int n = threadIdx.x; n < NT; n += blockDim.x) g[n] = gpart[n];
  } else {
    for (int n = threadIdx.x; n < NT; n += blockDim.x) g[n] = 0.0;
    __syncthreads();
    for (int q = 0; q < J.Q; ++q) synth_window<O>(J, q, J.W + base + (long long)q * L, buf, g);
    if (PART == 1) {
      for (int n = threadIdx.x; n < NT; n += blockDim.x) gpart[n] = g[n];
      return;
    }
  }
  const double mchi = -J.chi[J.tr_off[k] + x];
  for (int n = threadIdx.x; n < NT; n += blockDim.x) g[n] *= mchi;
  __syncthreads();
  forward_all<O>(J, g, buf, J.Gt + base);
}

// ---------------------------------------------------------------------------------------------
// Restriction of transfer-mesh spectra to the solve nodes of every system.
constexpr int kRestrThreads = 128;
constexpr int kRestrMaxThreads = 256;   // largest restriction block a tuned launch may use

template <bool DF>
__global__ void __launch_bounds__(kRestrMaxThreads) k_restrict(DevJob J) {
  extern __shared__ double2 shr[];
  const int sidx = J.sys_order[blockIdx.x];
  const SysDesc s = J.sys[sidx];
  const int k = s.arc, l = s.l, N = s.N, Q = J.Q, L = J.L;
  const long long base = J.tr_off[k];
  double2* G = J.G + s.vec_off;
  const long long off = J.restr_of_sys[sidx];
  if (off < 0) {
    for (int e = threadIdx.x; e < Q * N; e += blockDim.x) {
      int q = e / N, i = e % N;
      G[e] = J.Gt[((base + i) * Q + q) * L + l];
    }
    return;
  }
  const int a0 = J.act_off[k], na = J.act_off[k + 1] - a0;
  if constexpr (DF) {
    // Mixed form: the same sums in double-float (spectra split once, compensated sums).
    float4* sh4 = reinterpret_cast<float4*>(shr);
    for (int e = threadIdx.x; e < Q * na; e += blockDim.x) {
      int q = e / na, a = e % na;
      sh4[e] = df_split2(J.Gt[((base + J.act_idx[a0 + a]) * Q + q) * L + l]);
    }
    __syncthreads();
    const float2* RTd = J.restr_df + off;
    for (int e = threadIdx.x; e < Q * N; e += blockDim.x) {
      int q = e / N, i = e % N;
      dfacc re, im;
      for (int a = 0; a < na; ++a) {
        const float2 rv = RTd[(long long)J.act_idx[a0 + a] * N + i];
        const float4 gv = sh4[q * na + a];
        re.mac(rv.x, rv.y, gv.x, gv.y);
        im.mac(rv.x, rv.y, gv.z, gv.w);
      }
      const df vr = re.value(), vi = im.value();
      G[e] = make_double2((double)vr.hi + (double)vr.lo, (double)vi.hi + (double)vi.lo);
    }
  } else {
    for (int e = threadIdx.x; e < Q * na; e += blockDim.x) {
      int q = e / na, a = e % na;
      shr[e] = J.Gt[((base + J.act_idx[a0 + a]) * Q + q) * L + l];
    }
    __syncthreads();
    const double* RT = J.restr + off;
    for (int e = threadIdx.x; e < Q * N; e += blockDim.x) {
      int q = e / N, i = e % N;
      double2 acc = make_double2(0.0, 0.0);
      for (int a = 0; a < na; ++a) {
        const double rv = RT[(long long)J.act_idx[a0 + a] * N + i];
        const double2 gv = shr[q * na + a];
        acc.x = fma(rv, gv.x, acc.x);
        acc.y = fma(rv, gv.y, acc.y);
      }
      G[e] = acc;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Output traces u_M(z, t) = sum_q [valid] (1/pi) Re sum_l w_l Vobs(z, q, l) e^{-i l h (t - s_q)}.
constexpr int kTraceThreads = 128;

// One block per (observation point, output time): the threads split the frequencies, then a
// fixed-order tree sums their partial sums (deterministic).
__global__ void __launch_bounds__(kTraceThreads) k_traces(DevJob J) {
  __shared__ double part[kTraceThreads];
  const int idx = blockIdx.x;
  const int z = idx / J.n_tout, it = idx % J.n_tout;
  const double t = J.tout[it];
  double acc = 0.0;
  for (int q = 0; q < J.Q; ++q) {
    const double rel = t - J.s_q[q];
    if (!(rel >= -J.H && rel < J.period - J.H)) continue;
    const double c = J.h * (t - J.s_q[q]);
    const double2* V = J.Vobs + ((long long)z * J.Q + q) * J.L;
    for (int l = 1 + threadIdx.x; l < J.L; l += kTraceThreads) {
      double sn, cs;
      sincos((double)l * c, &sn, &cs);
      acc = fma(J.wl[l], fma(V[l].x, cs, V[l].y * sn), acc);
    }
  }
  part[threadIdx.x] = acc;
  __syncthreads();
  for (int w = kTraceThreads / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) J.traces[idx] = part[0] * kInvPi;
}

// Window q of every system's density block [q][i], one block per system, as one array in system order.  A system's
// block starts at vec_off, Q N complex values after its predecessor's, so its place in the array is
// (vec_off - first vec_off) / Q.  One copy call per frequency took 3.7 us each, 30 ms for 8 arcs x 1024
// frequencies; this launch is a few microseconds an arc.
__global__ void __launch_bounds__(128) k_gather_density(const SysDesc* __restrict__ sys, const double2* __restrict__ vec,
                                                        int Q, int q, double* __restrict__ out) {
  const SysDesc s = sys[blockIdx.x];
  const double* src = reinterpret_cast<const double*>(vec + s.vec_off + (long long)q * s.N);
  double* dst = out + 2 * ((s.vec_off - sys[0].vec_off) / Q);
  for (int e = threadIdx.x; e < 2 * s.N; e += blockDim.x) dst[e] = src[e];
}

inline int cdiv(long long a, int b) { return (int)((a + b - 1) / b); }

}  // namespace

// ---------------------------------------------------------------------------------------------
// Launch wrappers

cudaError_t launch_bessel0(const double* z, double* j0, double* y0, double* yh, int n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_bessel0<<<cdiv(n, kBesselThreads), kBesselThreads, 0, st>>>(z, j0, y0, yh, n);
  return cudaGetLastError();
}

cudaError_t launch_tables(const DevJob& J, cudaStream_t st, int* launches) {
  k_fft_tw<<<cdiv(J.K / 2, 256), 256, 0, st>>>(J.fft_tw, J.fft_tw_df, J.K);
  k_freq_tw<<<cdiv((long long)J.Q * J.L, 256), 256, 0, st>>>(J);
  k_freq_df<<<cdiv(J.L, 128), 128, 0, st>>>(J);
  *launches += 3;
  if (J.n_rlogN > 0) {
    cudaError_t e = launch_tables_rlog_only(J, st, launches);
    if (e != cudaSuccess) return e;
  }
  if (J.n_restr > 0) {
    const size_t sh = (size_t)3 * (J.max_n + J.max_nmax) * sizeof(double);   // <= 38 KB
    k_restr<<<J.n_restr, 256, sh, st>>>(J);
    *launches += 1;
  }
  return cudaGetLastError();
}

cudaError_t launch_tables_rlog_only(const DevJob& J, cudaStream_t st, int* launches) {
  const size_t sh = (size_t)3 * J.max_n * sizeof(double);
  cudaError_t e = cudaFuncSetAttribute(k_rlog, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
  if (e != cudaSuccess) return e;
  k_rlog<<<dim3(J.n_rlogN, cdiv(J.max_n + 1, kRlogRows)), 8 * kRlogRows, sh, st>>>(J);
  *launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_assemble_self(const DevJob& J, cudaStream_t st, int* launches) {
  if (J.n_tiles > 0) {
    if (!J.mixed || J.fp64keep || J.max_n >= J.f64_min_n) {
      k_assemble_self<false><<<J.n_tiles, 256, 0, st>>>(J);
      *launches += 1;
    }
    if (J.mixed && !J.fp64keep) {
      k_assemble_self<true><<<J.n_tiles, 256, 0, st>>>(J);
      *launches += 1;
    }
  }
  // the FP64-kept systems' fixed-point matrices (rows staged: 8 while two blocks fit an SM, else 4)
  if (J.mixed && J.n_rchunks > 0 && (J.fp64keep || J.max_n >= J.f64_min_n)) {
    const bool wide = J.max_n <= 800;
    const size_t sh = (size_t)(wide ? 8 : 4) * J.max_n * sizeof(int4);
    cudaError_t e = cudaFuncSetAttribute(wide ? k_afix<8> : k_afix<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
    if (e != cudaSuccess) return e;
    if (wide) k_afix<8><<<J.n_rchunks, kFixThreads, sh, st>>>(J);
    else k_afix<4><<<J.n_rchunks, kFixThreads, sh, st>>>(J);
    *launches += 1;
  }
  return cudaGetLastError();
}

cudaError_t launch_lu(const DevJob& J, cudaStream_t st, int* launches) {
  cudaError_t e = launch_lu_small(J, st, launches);
  if (e != cudaSuccess || !J.mixed) return e;
  return launch_lu_large(J, st, launches);
}

cudaError_t launch_lu_small(const DevJob& J, cudaStream_t st, int* launches) {
  if (J.mixed) {
    // k_assemble_self already wrote the FP32 matrix and the double-float pairs (or FP64 values)
    if (J.n_lu_small > 0) {
      int small_max = 0;   // systems above kLuBigMin go to the tensor-core path; J.max_n bounds the rest
      small_max = std::min(J.max_n, kLuBigMin - 1);
      size_t sh = lu_smem<float2>(small_max);
      cudaError_t e = cudaFuncSetAttribute(k_lu<float2, kLuThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
      if (e != cudaSuccess) return e;
      k_lu<float2, kLuThreads><<<J.n_lu_small, kLuThreads, sh, st>>>(J, J.lu_small);
      *launches += 1;
      return cudaGetLastError();
    }
    return cudaSuccess;
  }
  // FP64: every system, whatever the split of the mixed form (a job that falls back keeps its split)
  if (J.nsys == 0) return cudaSuccess;
  const size_t sh = lu_smem<double2>(J.max_n);
  auto go = [&](auto nt) {
    constexpr int NT = decltype(nt)::value;
    cudaError_t e = cudaFuncSetAttribute(k_lu<double2, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
    if (e != cudaSuccess) return e;
    k_lu<double2, NT><<<J.nsys, NT, sh, st>>>(J, J.sys_order);
    return cudaGetLastError();
  };
  *launches += 1;
  // A small system's panel keeps one warp busy while the others wait, so more and narrower CTAs an SM win; a large
  // system's trailing update wants the wide one.  768 systems, 128 against 256 threads: N = 64 0.77 / 0.93 ms, N = 96
  // 1.47 / 1.73, N = 128 2.56 / 2.90, N = 144 4.05 / 3.61, N = 256 15.7 / 13.6 (the factors are the same bit for bit).
  return J.max_n <= kLuNarrow ? go(std::integral_constant<int, 128>{}) : go(std::integral_constant<int, kLuThreads>{});
}

template <int QT>
static cudaError_t launch_fused_q(const DevJob& J, int* counter, size_t sh, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_fused_asf<QT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fused_asf<QT>, kFusedThreads, sh);
  if (e != cudaSuccess) return e;
  const int grid = std::max(1, std::min(J.nsys, sms * std::max(per_sm, 1)));
  e = cudaMemsetAsync(counter, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  k_fused_asf<QT><<<grid, kFusedThreads, sh, st>>>(J, counter);
  return cudaGetLastError();
}

cudaError_t launch_fused_asf(const DevJob& J, int* counter, cudaStream_t st, int* launches) {
  if (J.nsys == 0) return cudaSuccess;
  const size_t sh = lu_smem<double2>(J.max_n);
  *launches += 1;
  switch (J.Q) {
    case 1: return launch_fused_q<1>(J, counter, sh, st);
    case 2: return launch_fused_q<2>(J, counter, sh, st);
    case 3: return launch_fused_q<3>(J, counter, sh, st);
    default: return launch_fused_q<4>(J, counter, sh, st);
  }
}

cudaError_t launch_cross_assemble(const DevJob& J, cudaStream_t st, int* launches) {
  if (J.n_asm == 0) return cudaSuccess;
  const size_t sh_far = (size_t)kAsmBand * sizeof(FreqDf);   // (the far-only launch: the band's constants alone)
  const size_t sh = sh_far + (size_t)((2 * kAsmRows + 2) * J.max_n + 1) * sizeof(double);
  const int nt = J.shape_asm > 0 ? J.shape_asm : kAsmThreads;
  auto go = [&](auto form) {
    constexpr bool F = decltype(form)::value;
    cudaError_t e = cudaFuncSetAttribute(k_cross_assemble<true, F>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
    if (e != cudaSuccess) return e;
    k_cross_assemble<true, F><<<J.n_asm, nt, sh, st>>>(J);
    k_cross_assemble<false, F><<<J.n_asm, nt, sh_far, st>>>(J);
    return cudaGetLastError();
  };
  *launches += 2;
  return J.mixed ? go(std::false_type{}) : go(std::true_type{});
}

// one window's K/2 complex points and the samples
static size_t time_smem(const DevJob& J) { return (size_t)J.K * sizeof(double) + (size_t)J.NT * sizeof(double); }

bool incident_recurrent(const DevJob& J) {
  return J.sig_kind == 0 && J.sig_nt == 0 && J.dt * kIncRun <= 2.0 * J.width;
}

cudaError_t launch_incident(const DevJob& J, cudaStream_t st, int* launches) {
  if (J.n_act == 0) return cudaSuccess;
  if (incident_recurrent(J)) {
    const int runs = cdiv(J.NT, kIncRun), rows = J.inc_m > 0 ? J.inc_m : J.n_act;
    k_incident_ps<<<dim3(rows, cdiv(runs, kIncThreads / 32)), kIncThreads, 0, st>>>(J);
    *launches += 1;
    if (J.inc_m > 0) {
      k_inc_basis<<<cdiv(J.n_act, kIncThreads / 32), kIncThreads, 0, st>>>(J);
      k_inc_interp<<<dim3(cdiv(J.NT, kItpTile), cdiv(J.n_act, kItpTile)), 256, 0, st>>>(J);
      *launches += 2;
    }
  } else {
    k_incident_u<<<dim3(J.n_act, cdiv(J.NT, kIncThreads)), kIncThreads, 0, st>>>(J);
    *launches += 1;
  }
  size_t sh = time_smem(J);
  const int nt = J.shape_time > 0 ? J.shape_time : kTimeThreads;
  const bool df = J.mixed && !J.fp64keep;   // double-float FFT butterflies
  cudaError_t e = cudaFuncSetAttribute(df ? k_incident<true> : k_incident<false>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
  if (e != cudaSuccess) return e;
  if (df) k_incident<true><<<J.n_act, nt, sh, st>>>(J);
  else k_incident<false><<<J.n_act, nt, sh, st>>>(J);
  *launches += 1;
  return cudaGetLastError();
}

template <int PART>
static cudaError_t launch_synth_part(const DevJob& J, cudaStream_t st, int* launches) {
  if (J.n_act == 0) return cudaSuccess;
  size_t sh = time_smem(J);
  const int nt = J.shape_time > 0 ? J.shape_time : kTimeThreads;
  const bool df = J.mixed && !J.fp64keep;   // double-float FFT butterflies
  cudaError_t e = cudaFuncSetAttribute(df ? k_synth_fwd<true, PART> : k_synth_fwd<false, PART>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
  if (e != cudaSuccess) return e;
  if (df) k_synth_fwd<true, PART><<<J.n_act, nt, sh, st>>>(J);
  else k_synth_fwd<false, PART><<<J.n_act, nt, sh, st>>>(J);
  *launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_synth_fwd(const DevJob& J, cudaStream_t st, int* launches) {
  return launch_synth_part<0>(J, st, launches);
}
cudaError_t launch_synth_partial(const DevJob& J, cudaStream_t st, int* launches) {
  return launch_synth_part<1>(J, st, launches);
}
cudaError_t launch_fwd_after_sum(const DevJob& J, cudaStream_t st, int* launches) {
  return launch_synth_part<2>(J, st, launches);
}

cudaError_t launch_restrict(const DevJob& J, cudaStream_t st, int* launches) {
  size_t sh = (size_t)J.Q * J.max_nmax * sizeof(double2);
  const int nt = J.shape_restr > 0 ? J.shape_restr : kRestrThreads;
  cudaError_t e = cudaFuncSetAttribute(J.mixed ? k_restrict<true> : k_restrict<false>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
  if (e != cudaSuccess) return e;
  if (J.nsys == 0) return cudaSuccess;
  if (J.mixed) k_restrict<true><<<J.nsys, nt, sh, st>>>(J);
  else k_restrict<false><<<J.nsys, nt, sh, st>>>(J);
  *launches += 1;
  return cudaGetLastError();
}

// Warps (systems) per solve block: kSolveWarps, fewer when their right-hand sides would not fit in the
// 227 KB of shared memory a block may use (large Q x N).
static int solve_warps(size_t bytes_per_warp, int wanted) {
  const size_t cap = 227 * 1024;
  int nw = wanted > 0 && wanted < kSolveWarps ? wanted : kSolveWarps;
  while (nw > 1 && (size_t)nw * bytes_per_warp > cap) --nw;
  return nw;
}

int refine_passes(const DevJob& J) {
  return J.mixed && J.n_rchunks > 0 ? std::min(std::max(J.refine_max, 1), kRefineCap) : 0;
}

// Mixed forms: the triangular solves of refinement pass `pass` (0: the FP32 solution) for every system
// still refining.
template <int QT>
static cudaError_t launch_msolve_q(const DevJob& J, int m, int pass, cudaStream_t st, int* launches) {
  const size_t per = (size_t)QT * J.max_n * sizeof(float2);
  const int nw = solve_warps(per, J.shape_solve);
  const size_t sh = (size_t)nw * per;
  cudaError_t e = cudaFuncSetAttribute(k_msolve<QT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
  if (e != cudaSuccess) return e;
  k_msolve<QT><<<cdiv(J.nsys, nw), 32 * nw, sh, st>>>(J, m, pass);
  *launches += 1;
  return cudaGetLastError();
}

// Mixed forms: the residuals before refinement pass `pass` >= 1.
template <int QT>
static cudaError_t launch_resid_q(const DevJob& J, int pass, cudaStream_t st, int* launches) {
  const int rgrid = cdiv(J.n_rchunks, kResidThreads / 32);
  if (rgrid == 0) return cudaSuccess;
  if (J.fp64keep || J.max_n >= J.f64_min_n) {
    const size_t sh = fix_ring_bytes(QT, kResidThreads);
    cudaError_t e = cudaFuncSetAttribute(k_mresid<QT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
    if (e != cudaSuccess) return e;
    k_mresid<QT><<<rgrid, kResidThreads, sh, st>>>(J, pass);
    *launches += 1;
  }
  if (!J.fp64keep) {
    k_mresid_df<QT><<<rgrid, kResidThreads, 0, st>>>(J);
    *launches += 1;
  }
  return cudaGetLastError();
}

template <int QT>
static cudaError_t launch_solve_q(const DevJob& J, int m, cudaStream_t st, int* launches) {
  if (J.mixed) {
    cudaError_t e = launch_msolve_q<QT>(J, m, 0, st, launches);
    for (int pass = 1; pass <= refine_passes(J) && e == cudaSuccess; ++pass) {
      e = launch_resid_q<QT>(J, pass, st, launches);
      if (e == cudaSuccess) e = launch_msolve_q<QT>(J, m, pass, st, launches);
    }
    return e;
  }
  const size_t per = (size_t)QT * J.max_n * sizeof(double2);
  const int nw = solve_warps(per, J.shape_solve);
  size_t sh = (size_t)nw * per;
  cudaError_t e = cudaFuncSetAttribute(k_solve<QT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
  if (e != cudaSuccess) return e;
  k_solve<QT><<<cdiv(J.nsys, nw), 32 * nw, sh, st>>>(J, m);
  *launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_solve(const DevJob& J, int m, cudaStream_t st, int* launches) {
  switch (J.Q) {
    case 1: return launch_solve_q<1>(J, m, st, launches);
    case 2: return launch_solve_q<2>(J, m, st, launches);
    case 3: return launch_solve_q<3>(J, m, st, launches);
    default: return launch_solve_q<4>(J, m, st, launches);
  }
}

cudaError_t launch_msolve(const DevJob& J, int m, int pass, cudaStream_t st, int* launches) {
  switch (J.Q) {
    case 1: return launch_msolve_q<1>(J, m, pass, st, launches);
    case 2: return launch_msolve_q<2>(J, m, pass, st, launches);
    case 3: return launch_msolve_q<3>(J, m, pass, st, launches);
    default: return launch_msolve_q<4>(J, m, pass, st, launches);
  }
}

cudaError_t launch_resid(const DevJob& J, int pass, cudaStream_t st, int* launches) {
  switch (J.Q) {
    case 1: return launch_resid_q<1>(J, pass, st, launches);
    case 2: return launch_resid_q<2>(J, pass, st, launches);
    case 3: return launch_resid_q<3>(J, pass, st, launches);
    default: return launch_resid_q<4>(J, pass, st, launches);
  }
}

template <int Q>
static cudaError_t launch_cross_apply_q(const DevJob& J, cudaStream_t st) {
  // the row kernel's ring of entry batches (the densities come through the L1 cache)
  const size_t sh_rows = fix_ring_bytes(Q, kApplySlice);
  const size_t sh_red = (size_t)Q * J.acc_cap * sizeof(double2);
  cudaError_t e = cudaFuncSetAttribute(k_cross_rows<Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh_rows);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_cross_reduce<Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh_red);
  if (e != cudaSuccess) return e;
  if (J.n_slices > 0) k_cross_rows<Q><<<J.n_slices, kApplySlice, sh_rows, st>>>(J);
  k_cross_reduce<Q><<<J.n_grp, kApplyThreads, sh_red, st>>>(J);
  return cudaGetLastError();
}

cudaError_t launch_cross_apply(const DevJob& J, cudaStream_t st, int* launches) {
  if (J.n_grp == 0) return cudaSuccess;
  *launches += 2;
  switch (J.Q) {
    case 1: return launch_cross_apply_q<1>(J, st);
    case 2: return launch_cross_apply_q<2>(J, st);
    case 3: return launch_cross_apply_q<3>(J, st);
    default: return launch_cross_apply_q<4>(J, st);
  }
}

cudaError_t launch_near_weights(const DevJob& J, cudaStream_t st, int* launches) {
  if (J.n_asm == 0) return cudaSuccess;
  const size_t sh = (size_t)((2 + kAsmRows) * J.max_n + 1) * sizeof(double);   // ctab 2N + 1, lam kAsmRows N
  cudaError_t e = cudaFuncSetAttribute(k_near_weights, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
  if (e != cudaSuccess) return e;
  k_near_weights<<<J.n_asm, kAsmThreads, sh, st>>>(J);
  *launches += 1;
  return cudaGetLastError();
}

template <int Q>
static cudaError_t launch_cross_otf_q(const DevJob& J, cudaStream_t st) {
  const size_t sh_red = (size_t)Q * J.acc_cap * sizeof(double2);
  cudaError_t e = cudaFuncSetAttribute(k_cross_reduce<Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh_red);
  if (e != cudaSuccess) return e;
  if (J.n_otf > 0) {
    if (J.mixed) {
      if (J.fp64keep) k_cross_otf_df<Q, true><<<J.n_otf, kOtfThreads, 0, st>>>(J);
      else k_cross_otf_df<Q, false><<<J.n_otf, kOtfThreads, 0, st>>>(J);
    } else {
      k_cross_otf<Q><<<J.n_otf, kOtfThreads, 0, st>>>(J);
    }
  }
  k_cross_reduce<Q><<<J.n_grp, kApplyThreads, sh_red, st>>>(J);
  return cudaGetLastError();
}

cudaError_t launch_cross_otf(const DevJob& J, cudaStream_t st, int* launches) {
  if (J.n_grp == 0) return cudaSuccess;
  *launches += 2;
  switch (J.Q) {
    case 1: return launch_cross_otf_q<1>(J, st);
    case 2: return launch_cross_otf_q<2>(J, st);
    case 3: return launch_cross_otf_q<3>(J, st);
    default: return launch_cross_otf_q<4>(J, st);
  }
}

cudaError_t launch_gather_density(const SysDesc* sys, int n, const double2* vec, int Q, int q, double* out,
                                  cudaStream_t st) {
  k_gather_density<<<n, 128, 0, st>>>(sys, vec, Q, q, out);
  return cudaGetLastError();
}

cudaError_t launch_traces(const DevJob& J, cudaStream_t st, int* launches) {
  int n = J.n_obs * J.n_tout;
  if (n == 0) return cudaSuccess;
  k_traces<<<n, kTraceThreads, 0, st>>>(J);
  *launches += 1;
  return cudaGetLastError();
}

}  // namespace fthms
