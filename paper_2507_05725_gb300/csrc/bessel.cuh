// FP64 Bessel functions of order 0 for the Helmholtz kernel (i/4) H0^(1)(z) = (i/4)(J0 + i Y0)
// of Section 2.1, in two regimes:
//   0 <= z < 20  : J0 and the regular part Yhat0 = Y0 - (2/pi)(ln(z/2) + gamma) J0, both entire
//                  (J0 = sum_k (-z^2/4)^k/(k!)^2, Yhat0 = (2/pi) sum_{k>=1} (-1)^{k+1} H_k (z^2/4)^k/(k!)^2,
//                  Abramowitz-Stegun 9.1.12-9.1.13), by 13-term Taylor expansions about the centres
//                  0.25 + 0.5 k of 40 intervals of width 1/2 (coefficients: bessel_taylor.cuh).
//   z >= 20      : Hankel's asymptotic expansion with 10 + 10 terms,
//                  H0^(1)(z) ~ sqrt(2/(pi z)) e^{i(z - pi/4)} sum_k (-i)^k a_k/z^k,
//                  a_k = 1^2 3^2 ... (2k-1)^2/(k! 8^k)  (A-S 9.2.7-9.2.10, DLMF 10.17.5).
// Accuracy (checked against arbitrary-precision values): <= 1.2e-16 absolute for J0, Yhat0 below 20,
// <= 4e-16 relative to the amplitude sqrt(2/(pi z)) above.
#pragma once
#include <cuda_runtime.h>

#include "bessel_taylor.cuh"

namespace fthms {

constexpr double kEulerGamma = 0.57721566490153286060651209008240243;
constexpr double kPiD = 3.14159265358979323846;
constexpr double kInvPi = 0.31830988618379067153776752674502872;
constexpr double kTwoOverPi = 0.63661977236758134307553505349005745;
constexpr double kSqrtHalf = 0.70710678118654752440084436210484904;
constexpr double kBesselLarge = 20.0;

// Hankel coefficients a_k (filled by init_tables(); this header is included by one translation
// unit only).
__constant__ double c_hank_a[20];

// 0 <= z < 20: piecewise Taylor expansions of J0 and Yhat0 about c_k = 0.25 + 0.5 k (both functions
// are entire), 13 terms each, coefficients from gen_bessel_taylor.py (mpmath).  Every lane runs the
// same instruction stream (two 12-step Horner chains), whatever its interval.
__device__ __forceinline__ void bessel0_taylor(double z, double& J0, double& Yh) {
  const int k = min(max((int)(2.0 * z), 0), kTaylorIntervals - 1);   // (a negative z stays inside the table)
  const double d = z - fma(0.5, (double)k, 0.25);
  const double* cj = kTaylorJ0[k];
  const double* cy = kTaylorYh[k];
  double j = __ldg(&cj[kTaylorDegree]), y = __ldg(&cy[kTaylorDegree]);
#pragma unroll
  for (int n = kTaylorDegree - 1; n >= 0; --n) {
    j = fma(j, d, __ldg(&cj[n]));
    y = fma(y, d, __ldg(&cy[n]));
  }
  J0 = j;
  Yh = y;
}

// Hankel asymptotics given w = 1/z, amp = sqrt(2/(pi z)) and (s, c) = (sin z, cos z).
__device__ __forceinline__ void hankel_asym_phase(double w, double amp, double s, double c, double& J0,
                                                  double& Y0) {
  const double w2 = -w * w;
  double P = c_hank_a[18], Qa = c_hank_a[19];
#pragma unroll
  for (int k = 8; k >= 0; --k) {
    P = fma(P, w2, c_hank_a[2 * k]);
    Qa = fma(Qa, w2, c_hank_a[2 * k + 1]);
  }
  Qa *= w;
  const double cx = (c + s) * kSqrtHalf;   // cos(z - pi/4)
  const double sx = (s - c) * kSqrtHalf;   // sin(z - pi/4)
  J0 = amp * fma(P, cx, Qa * sx);
  Y0 = amp * fma(P, sx, -Qa * cx);
}

// Hankel asymptotics on z >= 20: J0 and Y0.
__device__ __forceinline__ void bessel0_asym(double z, double& J0, double& Y0) {
  const double w = 1.0 / z;
  double s, c;
  sincos(z, &s, &c);
  hankel_asym_phase(w, sqrt(kTwoOverPi * w), s, c, J0, Y0);
}

// Kernel pieces used by the Nystrom rules:
//  J0(z) and either Yhat0(z) (z < 20, has_yhat = true) or Y0(z) (z >= 20, has_yhat = false).
struct Bessel0 {
  double j0;
  double y;      // Yhat0 if has_yhat else Y0
  bool has_yhat;
};

__device__ __forceinline__ Bessel0 bessel0(double z) {
  Bessel0 b;
  if (z < kBesselLarge) {
    bessel0_taylor(z, b.j0, b.y);
    b.has_yhat = true;
  } else {
    bessel0_asym(z, b.j0, b.y);
    b.has_yhat = false;
  }
  return b;
}

}  // namespace fthms
