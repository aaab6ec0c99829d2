"""The error bounds that certify the cutoff decisions of fixed-point items, on the host (the device
headers compiled as C++ with the handful of CUDA intrinsics that they use): differences of
to_fixed values are within one unit of the exact ones, and cutoff_filter, given that bound,
returns only decisions (and exponents of the adaptive C_T) that hold for every sequence within it."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2010_13289_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
#define asm(...) (void)0
using std::fabs;
template <class A, class B> static A bits_of(B b) { A a; std::memcpy(&a, &b, sizeof a); return a; }
static long long __double_as_longlong(double x) { return bits_of<long long>(x); }
static double __longlong_as_double(long long x) { return bits_of<double>(x); }
static int __double2hiint(double x) { return (int)(__double_as_longlong(x) >> 32); }
static int __double2loint(double x) { return (int)__double_as_longlong(x); }
static double __hiloint2double(int h, int l) { return __longlong_as_double((long long)h << 32 | (unsigned)l); }
static float __uint_as_float(unsigned x) { return bits_of<float>(x); }
static float __int_as_float(int x) { return bits_of<float>(x); }
static unsigned __float_as_uint(float x) { return bits_of<unsigned>(x); }
static float __fdividef(float a, float b) { return a / b; }
static float rsqrtf(float x) { return 1.0f / std::sqrt(x); }
static long long __mul64hi(long long a, long long b) { return (long long)(((__int128)a * b) >> 64); }
static float __ll2float_rz(long long x) {
  const unsigned long long m = x < 0 ? 0ull - (unsigned long long)x : (unsigned long long)x;
  const int s = m ? 64 - __builtin_clzll(m) - 24 : 0;
  const float f = s > 0 ? std::ldexp((float)(m >> s), s) : (float)m;
  return x < 0 ? -f : f;
}
#include "tenom_fixed.cuh"
using namespace tenom;
typedef long double real;

static std::mt19937_64 rng(20);
static double uni(double a, double b) { return a + (b - a) * std::generate_canonical<double, 53>(rng); }

/* chi_k >= C_T and [beta] in long double from the differences D */
template <int K>
static void decide(const real* D, const SchemeDev& S, unsigned& bits, int& ex, real& margin) {
  constexpr int c = K / 2 - 1, nk = K - 2;
  real b[6] = {beta0<c - 1, false, real>(D), beta1<c, false, real>(D), beta2<c - 2, false, real>(D),
               beta3<c, false, real>(D)}, bK;
  if constexpr (K == 8) {
    b[4] = beta4<c - 3, false, real>(D);
    b[5] = beta5<c, false, real>(D);
    bK = betaK8<0, false, real>(D);
  } else {
    bK = betaK6<0, false, real>(D);
  }
  const real tau = std::fabs(bK - (b[1] + b[2] + 4 * b[0]) / 6);
  real g[6], sum = 0;
  for (int k = 0; k < nk; ++k) sum += g[k] = std::pow(1 + tau / (b[k] + 1e-40L), 6);
  real CT = S.ct_const;
  margin = 1e30L;
  ex = 7;
  if (S.ct_mode == CT_ADAPTIVE) {
    const real xi = 1e-3L, Cr = 0.23L, eps = 0.9L * Cr / (1 - 0.9L * Cr) * xi * xi;
    real eh = 1e30L;
    for (int q = 0; q < 4; ++q) {
      const real p = D[c + q - 1], m = D[c + q - 2];
      eh = std::fmin(eh, (std::fabs(2 * p * m) + eps) / (p * p + m * m + eps));
    }
    const real m = 1 - std::fmin((real)1, eh / Cr), om = 1 - m, gg = om * om * om * om * (1 + 4 * m);
    const real beta = 10.5L - 3.5L * (1 - gg);
    ex = (int)std::floor(beta);
    ex = ex < 7 ? 7 : (ex > 10 ? 10 : ex);
    CT = std::pow((real)10, -ex);
    for (int e = 8; e <= 10; ++e) margin = std::fmin(margin, std::fabs(beta - e) / 1e-2L);
  }
  bits = 0;
  for (int k = 0; k < nk; ++k) {
    if (g[k] >= CT * sum) bits |= 1u << k;
    margin = std::fmin(margin, std::fabs(std::log(g[k] / (CT * sum))) / 0.1L);
  }
}

/* one fixed-point item's side: the differences and their bound, as the kernel forms them */
template <int K>
static int item(const double* v, const SchemeDev& S, bool want_decided, int& undecided, int& decided) {
  double big = 0;
  for (int q = 0; q < K; ++q) big = std::fmax(big, std::fabs(v[q]));
  int em;
  std::frexp(big, &em);
  em += 1022;                                        /* biased exponent: |v| < 2^(em - 1022) */
  const float unit = std::ldexp(1.0f, em - 1076);    /* of the values given to to_fixed */
  float d[K - 1];
  real D[K - 1];
  unsigned zero = 0;
  long long x0 = to_fixed(v[0], em);
  for (int t = 0; t < K - 1; ++t) {
    const long long x1 = to_fixed(v[t + 1], em);
    D[t] = (real)v[t + 1] - (real)v[t];
    const real off = std::fabs((real)(x1 - x0) - D[t] / (real)unit);
    if (off > 1.01L) {
      std::printf("difference off by %.4Lf units: %.17g %.17g\n", off, v[t], v[t + 1]);
      return 1;
    }
    d[t] = __ll2float_rz(x1 - x0) * unit;
    zero |= v[t + 1] == v[t] ? 1u << t : 0u;
    x0 = x1;
  }
  unsigned b = 0, rb;
  int e = 0, re;
  real margin;
  decide<K>(D, S, rb, re, margin);
  const bool ok = cutoff_filter<K>(d, 1.01f * unit, zero, S, b, e);
  if (ok) {
    ++decided;
    if (b != rb || (S.ct_mode == CT_ADAPTIVE && e != re)) {
      std::printf("K %d decided %x [%d], exact %x [%d]\n", K, b, e, rb, re);
      return 1;
    }
  } else {
    ++undecided;
    if (want_decided && margin > 1) {
      std::printf("K %d refused at scale %g, margin %.3Lg\n", K, big, margin);
      return 1;
    }
  }
  return 0;
}

template <int K>
static int run() {
  SchemeDev S = {};
  S.default_d = S.screen = S.fixed = 1;
  int bad = 0, und = 0, dec = 0;
  for (int mode = 0; mode < 2; ++mode) {
    S.ct_mode = mode;
    S.ct_const = 1e-5;
    S.ct_const_f = 1e-5f;
    /* values of both signs, a few units each, beside a slope of any size */
    for (int i = 0; i < 200000 && !bad; ++i) {
      double v[K];
      const double u = std::ldexp(1.0, -53 + (int)uni(0, 4)), slope = std::ldexp(uni(0.5, 1.0), -(int)uni(0, 50));
      const int at = (int)uni(0, K);
      const bool left = uni(0, 1) < 0.5;
      for (int q = 0; q < K; ++q) {
        const bool s = left ? q < at : q > at;
        v[q] = (q & 1 ? -1 : 1) * u * uni(0.02, 0.98) + (s ? slope * (q - at) : 0.0);
      }
      v[left ? 0 : K - 1] = left ? -0.999 : 0.999;
      bad += item<K>(v, S, false, und, dec);
    }
    /* waves of any size: what is decided at size 1 is decided at every size */
    for (int i = 0; i < 100000 && !bad; ++i) {
      double v[K];
      const double s = std::ldexp(1.0, (int)uni(-8, 36)), ph = uni(0, 6.3), k = uni(0.05, 1.5), off = uni(-2, 2);
      for (int q = 0; q < K; ++q) v[q] = s * (off + std::sin(ph + k * q) + (q > K / 2 && i % 3 == 0 ? 1.0 : 0.0));
      double least = 1e300;
      for (int t = 0; t + 1 < K; ++t) least = std::fmin(least, std::fabs(v[t + 1] - v[t]));
      bad += item<K>(v, S, least > 1e-3 * s, und, dec);
    }
    /* a bound E near the largest for which eta is certain: [beta] holds for every sequence within it */
    for (int i = 0; i < 200000 && !bad && mode == CT_ADAPTIVE; ++i) {
      float d[K - 1];
      const double s = std::ldexp(1.0, (int)uni(-12, 30));
      const float E = (float)(std::fmax(s * 0.05, 5e-4) * std::exp(uni(std::log(1e-9), std::log(1e-5))));
      for (int t = 0; t < K - 1; ++t) d[t] = (float)(s * uni(0.02, 1.0) * (uni(0, 1) < 0.3 ? -1 : 1));
      unsigned b;
      int e;
      if (!cutoff_filter<K>(d, E, 0u, S, b, e)) continue;
      for (int r = 0; r < 8 && !bad; ++r) {
        real D[K - 1], margin;
        unsigned rb;
        int re;
        for (int t = 0; t < K - 1; ++t) D[t] = (real)d[t] + (real)E * (uni(0, 1) < 0.5 ? -1 : 1);
        decide<K>(D, S, rb, re, margin);
        if (rb != b || re != e) {
          std::printf("K %d E %g s %g: decided %x [%d], within E %x [%d]\n", K, E, s, b, e, rb, re);
          ++bad;
        }
      }
    }
  }
  std::printf("K %d: %d decided, %d undecided\n", K, dec, und);
  return bad;
}

int main() { return run<6>() + run<8>() ? 1 : 0; }
"""


def test_fixed_point_decisions_hold_within_their_bound(tmp_path):
    src, exe = tmp_path / "fixed_filter.cpp", tmp_path / "fixed_filter"
    src.write_text(PROGRAM)
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-w", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    if r.returncode != 0:
        pytest.fail("g++ failed:\n" + r.stderr[-3000:])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
