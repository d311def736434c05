"""The kernels' fixed-point and bit arithmetic (csrc/fixed.cuh, csrc/bits64.cuh) compiled for the host and compared with the
FP64 arithmetic whose place it takes, both against a higher precision."""
import ctypes as ct
import os
import subprocess

import numpy as np
import pytest
from scipy import special

import workloads as wl
from oracle import geometry as geo
from oracle import kernels as oker

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_05725_gb300", "csrc")

SHIM = r"""
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <utility>
#include <vector>

// the device intrinsics that the headers use
static long long bits(double v) { long long u; std::memcpy(&u, &v, 8); return u; }
static double dbl(long long u) { double v; std::memcpy(&v, &u, 8); return v; }
static int __double2hiint(double v) { return (int)(bits(v) >> 32); }
static int __double2loint(double v) { return (int)bits(v); }
static double __hiloint2double(int h, int l) { return dbl(((long long)h << 32) | (unsigned)l); }
static double __longlong_as_double(long long u) { return dbl(u); }
static float __fmul_rn(float a, float b) { return a * b; }
static float __fadd_rn(float a, float b) { return a + b; }
static float __fdiv_rn(float a, float b) { return a / b; }
static double rsqrt(double v) { return 1.0 / std::sqrt(v); }
static long long __double_as_longlong(double v) { return bits(v); }
static float __fsub_rn(float a, float b) { return a - b; }
static unsigned __float_as_uint(float v) { unsigned u; std::memcpy(&u, &v, 4); return u; }
static float __uint_as_float(unsigned u) { float v; std::memcpy(&v, &u, 4); return v; }
static float rsqrtf(float v) { return 1.f / std::sqrt(v); }
static float __double2float_rn(double v) { return (float)v; }
static float __uint2float_rn(unsigned v) { return (float)v; }
static unsigned __funnelshift_l(unsigned l, unsigned h, int k) { return (unsigned)(((((unsigned long long)h) << 32 | l) << k) >> 32); }
template <class T> static T __ldg(const T* p) { return *p; }
static uint3 threadIdx, blockDim;
static int __float2int_rn(float a) { return (int)std::nearbyintf(a); }
static unsigned __reduce_max_sync(unsigned, unsigned m) { return m; }
using std::max;
using std::min;
"""

SOURCE = SHIM + r"""
// (bessel.cuh reads its tables through this: the addresses are recorded, not read)
static const double *g_low, *g_high;
static double watched(const double* p) {
  g_low = g_low ? min(g_low, p) : p;
  g_high = max(g_high, p);
  return 1.0;
}
#define __ldg watched
#include "bessel.cuh"
#undef __ldg
#include "bits64.cuh"
#include "cplx.cuh"
#include "fixed.cuh"
using namespace fthms;
#ifdef __SIZEOF_FLOAT128__
using quad = __float128;
#else
using quad = long double;   // (128 bits where there is no __float128)
#endif

extern "C" void dist(const double* R2, double* r, int n) {
  for (int i = 0; i < n; ++i) r[i] = dist_f64(R2[i]);
}

// Whether bessel0(z) reads inside its two tables (or nothing).
extern "C" int taylor_reads_inside(double z) {
  const double *a = &kTaylorJ0[0][0], *b = &kTaylorYh[0][0];
  g_low = g_high = nullptr;
  bessel0(z);
  return !g_low || (g_low >= min(a, b) && g_high < max(a, b) + sizeof kTaylorJ0 / sizeof(double));
}

// One factorisation as the one-CTA kernel makes it: panels of 8 columns in FP64 with partial pivoting, and the trailing
// updates by FP64 FMAs (fixed = 0) or in fixed point.
extern "C" void lu(double2* A, int* perm, int N, int fixed) {
  auto at = [&](int r, int c) -> double2& { return A[(size_t)c * N + r]; };
  for (int i = 0; i < N; ++i) perm[i] = i;
  for (int k0 = 0; k0 < N; k0 += 8) {
    const int w = min(8, N - k0), k1 = k0 + w;
    for (int k = k0; k < k1; ++k) {
      int p = k;
      auto size = [&](int r) { return std::fabs(at(r, k).x) + std::fabs(at(r, k).y); };
      for (int r = k + 1; r < N; ++r) if (size(r) > size(p)) p = r;
      if (p != k) {
        for (int j = 0; j < N; ++j) std::swap(at(k, j), at(p, j));
        std::swap(perm[k], perm[p]);
      }
      const double2 inv = crecip(at(k, k));
      for (int r = k + 1; r < N; ++r) {
        const double2 l = at(r, k) = cmul(at(r, k), inv);
        for (int c = k + 1; c < k1; ++c) at(r, c) = cfms(l, at(k, c), at(r, c));
      }
    }
    std::vector<int4> L((size_t)8 * (N - k1));
    for (int r = k1; r < N; ++r)
      for (int c = 0; c < 8; ++c) {
        const int2 x = fix_f64<kLuLow>(at(r, k0 + c).x, 1), y = fix_f64<kLuLow>(at(r, k0 + c).y, 1);
        L[(size_t)8 * (r - k1) + c] = make_int4(x.x, x.y, y.x, y.y);
      }
    for (int j = k1; j < N; ++j) {
      unsigned top = 0u;
      for (int r = k0; r < k1; ++r) {
        for (int c = k0; c < r; ++c) at(r, j) = cfms(at(r, c), at(c, j), at(r, j));
        top = max(top, max(__double2hiint(at(r, j).x) & 0x7FFFFFFFu, __double2hiint(at(r, j).y) & 0x7FFFFFFFu));
      }
      const int e = max((int)(top >> 20), 100) - 1022;
      int4 U[8];
      for (int c = 0; c < 8; ++c) {
        const int2 x = fix_f64<kLuLow>(at(k0 + c, j).x, e), y = fix_f64<kLuLow>(at(k0 + c, j).y, e);
        U[c] = make_int4(x.x, x.y, y.x, y.y);
      }
      for (int r = k1; r < N; ++r) {
        double2& v = at(r, j);
        if (!fixed) {
          for (int c = k0; c < k1; ++c) v = cfms(at(r, c), at(c, j), v);
          continue;
        }
        fixacc<kLuLow> re, im;
        for (int c = 0; c < 8; ++c) {
          const int4 l = L[(size_t)8 * (r - k1) + c], p = U[c];
          re.mac(l.x, l.y, p.x, p.y);
          im.mac(l.x, l.y, p.z, p.w);
          re.mac(-l.z, -l.w, p.z, p.w);
          im.mac(l.z, l.w, p.x, p.y);
        }
        v.x = fma(-lu_unit(e), ll_to_double(re.nearest()), v.x);
        v.y = fma(-lu_unit(e), ll_to_double(im.nearest()), v.y);
      }
    }
  }
}

// Sums over N sources with the row kernels' carries; X, Y: [N][2] values as integers of fix_bits(low) bits.  Returns how many
// of the two sums differ from the exact sums of the products kept.
template <int kLow>
static int exact_sums(const long long* X, const long long* Y, int N) {
  fixacc<kLow> re, im;
  __int128 er = 0, ei = 0;
  auto kept = [](int2 a, int2 b) { return ((__int128)a.x * b.x << kLow) + (__int128)a.x * b.y + (__int128)a.y * b.x; };
  for (int i = 0; i < N; ++i) {
    const int2 a = fix_split<kLow>(X[2 * i]), b = fix_split<kLow>(X[2 * i + 1]);
    const int2 c = fix_split<kLow>(Y[2 * i]), d = fix_split<kLow>(Y[2 * i + 1]), n = make_int2(-b.x, -b.y);
    re.mac(a.x, a.y, c.x, c.y);
    im.mac(a.x, a.y, d.x, d.y);
    re.mac(n.x, n.y, d.x, d.y);
    im.mac(b.x, b.y, c.x, c.y);
    er += kept(a, c) + kept(n, d);
    ei += kept(a, d) + kept(b, c);
    if ((i + 1) % (fix_run(kLow) / 2) == 0) {
      re.carry();
      im.carry();
    }
  }
  auto same = [](fixacc<kLow>& s, __int128 want) {
    s.carry();
    return (((((__int128)s.c) << 32) + s.a) << kLow) + s.b == want;
  };
  return !same(re, er) + !same(im, ei);
}
extern "C" int sums_differ(const long long* X, const long long* Y, int N, int low) {
  return low == kRowLow ? exact_sums<kRowLow>(X, Y, N) : exact_sums<kMatLow>(X, Y, N);
}
extern "C" int lows(int* out) { out[0] = kRowLow; out[1] = kMatLow; return 0; }

// R rows of N entries (bounds 2^s[r]) times p (bound 2^sp): errors of FP64 FMAs and of the fixed-point sums over sum |E||p|.
extern "C" void row_errors(const double2* E, const int* s, const double2* p, int sp, int R, int N, double* out) {
  for (int r = 0; r < R; ++r, E += N) {
    quad x = 0, y = 0;
    double2 f = make_double2(0, 0);
    fixacc<kRowLow> re, im;
    double size = 0;
    for (int i = 0; i < N; ++i) {
      const double2 e = E[i], v = p[i];
      x += (quad)e.x * v.x - (quad)e.y * v.y;
      y += (quad)e.x * v.y + (quad)e.y * v.x;
      f = cfma(e, v, f);
      size += std::hypot(e.x, e.y) * std::hypot(v.x, v.y);
      const int2 a = fix_f64<kRowLow>(e.x, s[r]), b = fix_f64<kRowLow>(e.y, s[r]);
      const int2 c = fix_f64<kRowLow>(v.x, sp), d = fix_f64<kRowLow>(v.y, sp);
      re.mac(a.x, a.y, c.x, c.y);
      im.mac(a.x, a.y, d.x, d.y);
      re.mac(-b.x, -b.y, d.x, d.y);
      im.mac(b.x, b.y, c.x, c.y);
      if ((i + 1) % (fix_run(kRowLow) / 2) == 0) {
        re.carry();
        im.carry();
      }
    }
    const double u = std::ldexp(1.0, 2 * kRowLow + s[r] + sp - 2 * fix_bits(kRowLow));
    out[2 * r] = std::hypot((double)(x - f.x), (double)(y - f.y)) / size;
    out[2 * r + 1] = std::hypot((double)(x - (quad)(re.value() * u)), (double)(y - (quad)(im.value() * u))) / size;
  }
}

// Root mean square over a row (bound 2^e) of the matrices' fixed-point rounding.
extern "C" double kept_error(const double* v, int n, int e) {
  double sum = 0;
  for (int i = 0; i < n; ++i) {
    const int2 x = fix_f64<kMatLow>(v[i], e);
    const quad w = ((quad)((long long)x.x << kMatLow) + x.y) * std::ldexp(1.0, e - fix_bits(kMatLow));
    const double d = (double)(w - v[i]);
    sum += d * d;
  }
  return std::sqrt(sum / n);
}

// P A - L U: Frobenius norm over |A|'s, largest entry over |L||U|'s, and the mean (re, im) over the mean |a|.
extern "C" void lu_error(const double2* A, const double2* F, const int* perm, int N, double* out) {
  double num = 0, den = 0, big = 0, re = 0, im = 0, sum = 0;
  for (int j = 0; j < N; ++j)
    for (int i = 0; i < N; ++i) {
      quad x = 0, y = 0;
      double size = 0;
      for (int k = 0; k <= min(i, j); ++k) {
        const double2 l = k == i ? make_double2(1, 0) : F[(size_t)k * N + i], u = F[(size_t)j * N + k];
        x += (quad)l.x * u.x - (quad)l.y * u.y;
        y += (quad)l.x * u.y + (quad)l.y * u.x;
        size += std::hypot(l.x, l.y) * std::hypot(u.x, u.y);
      }
      const double2 a = A[(size_t)j * N + perm[i]];
      const double dx = (double)(x - a.x), dy = (double)(y - a.y);
      num += dx * dx + dy * dy;
      den += a.x * a.x + a.y * a.y;
      big = max(big, std::hypot(dx, dy) / size);
      re += dx;
      im += dy;
      sum += std::hypot(a.x, a.y);
    }
  out[0] = std::sqrt(num / den);
  out[1] = big;
  out[2] = re / sum;
  out[3] = im / sum;
}
"""


TABLES = SHIM + r"""
#include <atomic>
#include <thread>
#include <unistd.h>

#include "hankel_df.cuh"

// A runtime that takes its time and counts the copies under way.
static std::atomic<int> inside, most, to_device, waits;
static void slow() {
  const int n = ++inside;
  for (int m = most; n > m && !most.compare_exchange_weak(m, n);) {}
  usleep(2000);
  --inside;
}
extern "C" cudaError_t cudaMemcpyToSymbol(const void* d, const void* s, size_t n, size_t, cudaMemcpyKind) {
  slow();
  ++to_device;
  std::memcpy(const_cast<void*>(d), s, n);
  return cudaSuccess;
}
extern "C" cudaError_t cudaMemcpyFromSymbol(void* d, const void* s, size_t n, size_t, cudaMemcpyKind) {
  slow();
  std::memcpy(d, s, n);
  return cudaSuccess;
}
extern "C" cudaError_t cudaStreamSynchronize(cudaStream_t) { ++waits; return cudaSuccess; }

// Four threads' first calls on a device, then a call on another one: copies at once, copies and waits after each part,
// tables missing when a thread's call returned.
extern "C" void first_calls(int* out) {
  std::atomic<int> missing{0};
  std::vector<std::thread> t;
  for (int k = 0; k < 4; ++k)
    t.emplace_back([&] {
      if (fthms::init_tables(3) != cudaSuccess || fthms::c_hank_a[0] != 1.0 || fthms::c_angle_f64[0].x != 1.0 || waits == 0) ++missing;
    });
  for (auto& x : t) x.join();
  out[0] = most;
  out[1] = to_device;
  out[2] = missing;
  const int bad = fthms::init_tables(4) != cudaSuccess || fthms::init_tables(4) != cudaSuccess ||
                  fthms::init_tables(-1) == cudaSuccess || fthms::init_tables(64) == cudaSuccess;
  out[3] = to_device;
  out[4] = bad;
  out[5] = waits;
}
"""


def _compile(tmp_path_factory, name, source):
    d = tmp_path_factory.mktemp(name)
    src, so = d / f"{name}.cpp", d / f"{name}.so"
    src.write_text(source)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-pthread", "-shared", "-fPIC", "-Wl,-Bsymbolic",
                    "-I", CSRC, "-I", os.path.join(cuda, "include"), str(src), "-o", str(so)], check=True)
    return ct.CDLL(str(so))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return _compile(tmp_path_factory, "fixed", SOURCE)


def _ptr(a):
    return ct.c_void_p(a.ctypes.data)


@pytest.mark.parametrize("N,kappa", [(17, 5.0), (48, 12.0), (136, 3.0), (136, 34.0), (259, 65.0)])
def test_lu_updates_are_no_less_accurate_than_fp64(lib, N, kappa):
    """Trailing updates of the FP64 LU on the oracle's self matrices.  One rounding to the column's unit and one FP64
    rounding a panel take the place of sixteen FP64 roundings and the panels are the same, so the error may not exceed that
    of the FMAs: in norm, entry by entry (a quarter more: a maximum over N^2 values), and without a direction (the
    rounding is to the nearest: the mean error stays below a tenth of the error's own size)."""
    A = np.asfortranarray(oker.self_matrix(geo.Arc(0, 0, wl.kite(0.1, 0.2), -1.3, 1.1), N, kappa).astype(complex))
    err = []
    for fixed in (0, 1):
        F, perm, out = A.copy(order="F"), np.zeros(N, np.int32), np.zeros(4)
        lib.lu(_ptr(F), _ptr(perm), N, fixed)
        lib.lu_error(_ptr(A), _ptr(F), _ptr(perm), N, _ptr(out))
        err.append(out)
    fma, fix = err
    assert fix[0] <= fma[0]
    assert fix[1] <= 1.25 * fma[1]
    assert max(abs(fix[2]), abs(fix[3])) <= 0.1 * fix[0]


def test_distances_in_any_unit_of_length(lib):
    """dist_f64 over the whole range of R^2: two Newton steps leave less than half a unit in the last place, the last
    rounding adds half of one (2^-52 together); zero stays zero, and what is not a finite number gives none."""
    rng = np.random.default_rng(3)
    R2 = np.concatenate([np.exp2(rng.uniform(-1021.0, 1023.0, 20000)), np.exp2(rng.uniform(-60.0, 60.0, 5000)),
                         np.exp2(np.arange(-1022.0, 1024.0)), np.nextafter(np.exp2(np.arange(-1021.0, 1024.0)), 0.0), [0.0]])
    r = np.full_like(R2, np.nan)
    lib.dist(_ptr(R2), _ptr(r), R2.size)
    want = np.sqrt(R2.astype(np.longdouble))
    assert np.all(np.abs(r - want) <= want * 2.0 ** -52)
    bad, out = np.array([np.inf, np.nan, -1.0]), np.zeros(3)
    lib.dist(_ptr(bad), _ptr(out), 3)
    assert not np.any(np.isfinite(out[:2]))


def test_tables_are_filled_once_whoever_calls_first(tmp_path_factory):
    """The tables of a device are computed and uploaded by one thread while the others' first calls wait for them, once
    per device, and the upload is waited for."""
    out = (ct.c_int * 6)()
    _compile(tmp_path_factory, "tables", TABLES).first_calls(out)
    at_once, copies, missing, copies2, bad, waits = out
    assert at_once == 1 and missing == 0 and bad == 0
    assert copies > 0 and copies2 == 2 * copies and waits == 2


@pytest.mark.parametrize("z", [0.0, 19.999, -0.3, -0.6, -7.0, -1e9, -np.inf, np.inf, np.nan])
def test_bessel_tables_are_read_inside_whatever_the_argument(lib, z):
    """fthms_bessel0 asks for z > 0, but an argument on the device cannot be refused: it must not lead outside the
    tables."""
    lib.taylor_reads_inside.argtypes = [ct.c_double]
    assert lib.taylor_reads_inside(z)


@pytest.mark.parametrize("which", [0, 1])
def test_sums_are_exact_up_to_the_largest_values(lib, which):
    """Sums of 2 048 sources with a carry after each run, at the largest values either half can hold (every sign), random
    ones, and mixtures: no overflow, nothing lost."""
    low = (ct.c_int * 2)()
    lib.lows(low)
    low = low[which]
    top, half = 1 << (2 * low - 1), 1 << (low - 1)
    edge = [top, -top, top - half, half - top, top - half - 1, half - 1, -half, 0, 1, -1]
    rng = np.random.default_rng(low)
    N = 2048
    sets = [np.full(2 * N, v, np.int64) for v in edge]
    for a in edge:
        for b in edge:
            sets.append(np.array([a, b] * N, np.int64))
    sets += [rng.integers(-top, top, 2 * N, endpoint=True) for _ in range(4)] + [rng.choice(np.array(edge), 2 * N) for _ in range(8)]
    for X in sets:
        for Y in sets[::3]:
            assert lib.sums_differ(_ptr(np.ascontiguousarray(X)), _ptr(np.ascontiguousarray(Y)), N, low) == 0


def _near_beta(ts, N):
    """-(2/pi)(W_i/w - ln|t* - t_i|) of the near rule for a target continued to t*."""
    t, n = geo.cheb_nodes(N), np.arange(1, N)
    rt = np.sqrt(ts * ts - 1.0)
    zeta = ts - rt if ts > 0 else ts + rt
    W = (np.pi * np.log(0.5 * (abs(ts) + rt)) + 2.0 * np.cos(np.outer(np.arccos(t), n)) @ (-np.pi * zeta ** n / n)) / N
    return -(2.0 / np.pi) * (W * N / np.pi - np.log(np.abs(ts - t)))


@pytest.mark.parametrize("N", [33, 96, 259, 800])
@pytest.mark.parametrize("rate", [0.02, 0.15, 0.3])
def test_stored_row_sums_are_no_less_accurate_than_fp64(lib, N, rate):
    """Rows of cross entries (next to the arc's ends with their near corrections, and far ones) times a density, sums in
    fixed point against FP64 FMAs over the same FP64 entries.  N roundings of the running sum become one rounding a value
    of 2^-58 of the bound, so the error may not be larger: root mean square over the near and over the far rows, and the
    largest."""
    rng = np.random.default_rng(N)
    kappa, curve, w = rate * N, wl.kite(0.1, 0.2), np.pi / N
    X = geo.Arc(0, 0, curve, -1.3, 1.1).point(geo.cheb_nodes(N))[0]
    ts = rng.choice([-1.0, 1.0], 40) * (1.0 + np.exp(rng.uniform(np.log(1e-4), np.log(2.0), 40)))
    th, k = -0.1 + 1.2 * ts, np.arange(3)[:, None]
    near = np.stack([np.dot(curve[a], np.cos(k * th)) + np.dot(curve[b], np.sin(k * th)) for a, b in (("ax", "bx"), ("ay", "by"))], 1)
    tg = np.concatenate([near, rng.uniform(-8.0, 8.0, (40, 2))])
    beta = np.concatenate([np.array([_near_beta(t, N) for t in ts]), np.zeros((40, N))])
    z = kappa * np.linalg.norm(tg[:, None] - X[None], axis=-1)
    J = special.j0(z)
    E = np.ascontiguousarray(0.25 * w * (beta * J - special.y0(z) + 1j * J))
    zm = z.min(1)
    h0 = np.where(zm < 1.0, np.minimum(np.sqrt(0.6367 / zm), 1.5 - 0.64 * np.log(zm)), np.sqrt(0.6367 / zm))
    s = (np.floor(np.log2(0.25 * w * h0 * (1.0 + np.abs(beta).max(1)))) + 1).astype(np.int32)      # the kernel's row bound
    assert np.all(np.abs(E).max(1) < np.exp2(s))
    p = np.exp(1j * kappa * X[:, 0]) * (1.0 + 0.3 * np.polynomial.chebyshev.chebval(geo.cheb_nodes(N), rng.normal(size=12) + 1j * rng.normal(size=12)))
    sp = int(np.floor(np.log2(max(np.abs(p.real).max(), np.abs(p.imag).max())))) + 1
    out = np.zeros((80, 2))
    lib.row_errors(_ptr(E), _ptr(s), _ptr(p), sp, 80, N, _ptr(out))
    for rows in (out[:40], out[40:]):
        fma, fix = np.sqrt(np.mean(rows ** 2, 0))
        assert fix <= fma and rows[:, 1].max() <= rows[:, 0].max()


@pytest.mark.parametrize("N,kappa", [(96, 20.0), (259, 65.0), (512, 150.0), (1024, 150.0)])
def test_kept_matrices_hold_what_fp64_holds(lib, N, kappa):
    """The refinement's matrices: their fixed-point rounding against the half unit in the last place that every FP64 entry
    carries from its own computation.  A row's entries lie up to 2^6 below its largest, which 60 bits (2^-60 of it) cover:
    below a half of it in the root mean square."""
    lib.kept_error.restype = ct.c_double
    A = oker.self_matrix(geo.Arc(0, 0, wl.kite(0.1, 0.2), -1.3, 1.1), N, kappa)
    kept = own = 0.0
    for row in A:
        v = np.ascontiguousarray(np.stack([row.real, row.imag], 1)).ravel()
        e = int(np.floor(np.log2(np.abs(v).max()))) + 1
        kept += lib.kept_error(_ptr(v), v.size, e) ** 2
        own += float(np.mean(np.spacing(np.abs(v)) ** 2)) / 12.0
    assert np.sqrt(kept) <= 0.5 * np.sqrt(own)
