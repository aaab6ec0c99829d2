/* The limiter's part of a reconstruction in 64-bit fixed point.
 *
 * With the cutoff decisions taken, fhat = sum_k d_k f_k + sum_{k nonsmooth} d_k (limited_k - f_k);
 * the first sum is the central scheme, and the correction depends only on the differences of
 * the sequence: every term is a combination with rational coefficients, a minimum or a
 * maximum.  On integers v_q = floor(value / unit), unit = 2^-54 of a power of two above the
 * largest |v_q|, those are exact (a few floor divisions lose one unit each), so the correction
 * carries the rounding of FP64 values of the sequence's size, and runs on the integer pipe:
 * about 250 instructions a side where the FP64 form has 50-80 operations of 64 issue slots
 * each on GB300's FP64 pipe, paid by the whole warp when one lane needs them.
 *
 * Overflow: |v| <= 2^54, differences <= 2^55, second differences < 2^56, 4 d - d' < 5 2^56,
 * bounds (alpha, beta/3 <= 8, scheme's fixed flag) < 2^60; the candidates' numerators and the TVD5
 * terms in 60ths at most 130 2^55 (candidate 4) + 60 2^55 < 2^62.6. */
#pragma once
#include "tenom_recon.cuh"

namespace tenom {

/* floor(v 2^(1076 - em)) for a finite v with biased exponent at most em: |result| <= 2^54.  Floored and
   not truncated, so that a difference of two results is within one unit of the exact one whatever
   their signs: the filter is given that bound.  (Subnormal v: 0.) */
__device__ __forceinline__ long long to_fixed(double v, int em) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const int e = (int)((hi >> 20) & 0x7ffu), sh = em - e;
  long long m = (long long)((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 1;
  m = (int)hi < 0 ? -m : m;
  return e == 0 ? 0 : m >> (sh < 63 ? sh : 63);
}

/* D q 2^-60 for a coefficient q = coef 2^60 (coef <= 8 exclusive), |D| < 2^58 */
__device__ __forceinline__ long long mul_q60(long long D, long long q) { return __mul64hi(D * 16, q); }

__device__ __forceinline__ long long lmin2(long long a, long long b) { return a < b ? a : b; }
__device__ __forceinline__ long long lmax2(long long a, long long b) { return a > b ? a : b; }

__device__ __forceinline__ long long lminmod(long long a, long long b) {
  const long long lo = lmin2(a, b), hi = lmax2(a, b);
  return lo > 0 ? lo : (hi < 0 ? hi : 0);
}

/* 60 (f_k - f_i) of candidate k (Table 1) from the differences D, c = index of f_i */
template <int c>
__device__ __forceinline__ long long cand60(int k, const long long* D) {
  switch (k) {
    case 0: return 10 * D[c - 1] + 20 * D[c];
    case 1: return 40 * D[c] - 10 * D[c + 1];
    case 2: return 50 * D[c - 1] - 20 * D[c - 2];
    case 3: return 45 * D[c] - 20 * D[c + 1] + 5 * D[c + 2];
    case 4: return 65 * D[c - 1] - 50 * D[c - 2] + 15 * D[c > 2 ? c - 3 : 0];
    default: return 48 * D[c] - 29 * D[c + 1] + 14 * D[c + 2] - 3 * D[c + 3];
  }
}

/* floor((60 (f_k - f_i)) / 60) within one unit, through the candidate's own denominator (so that
   the numerator stays below 2^62) */
template <int c>
__device__ __forceinline__ long long cand_unit(int k, const long long* D) {
  const long long q6 = 0x2aaaaaaaaaaaaaaall;   /* 2^64 / 6 */
  const long long q12 = 0x1555555555555555ll;  /* 2^64 / 12 */
  const long long q60 = 0x0444444444444444ll;  /* 2^64 / 60 */
  switch (k) {
    case 0: return __mul64hi(D[c - 1] + 2 * D[c], q6);
    case 1: return __mul64hi(4 * D[c] - D[c + 1], q6);
    case 2: return __mul64hi(5 * D[c - 1] - 2 * D[c - 2], q6);
    case 3: return __mul64hi(9 * D[c] - 4 * D[c + 1] + D[c + 2], q12);
    case 4: return __mul64hi(13 * D[c - 1] - 10 * D[c - 2] + 3 * D[c > 2 ? c - 3 : 0], q12);
    default: return __mul64hi(48 * D[c] - 29 * D[c + 1] + 14 * D[c + 2] - 3 * D[c + 3], q60);
  }
}

/* a running sum of small-integer multiples of 64-bit values, in two 64-bit words (hi 2^32 + lo) */
struct Acc96 {
  long long hi = 0, lo = 0;
  __device__ __forceinline__ void add(int w, long long x) {
    lo += (long long)w * (long long)(unsigned)x;
    hi += (long long)w * (long long)(int)(x >> 32);
  }
  __device__ __forceinline__ double value() const { return fma((double)hi, 4294967296.0, (double)lo); }
};

/* maximal-order d_k = fixed_weight / fixed_den */
template <int K>
__host__ __device__ constexpr int fixed_weight(int k) {
  if (K == 6) return k == 0 ? 9 : (k == 1 ? 6 : (k == 2 ? 1 : 4));
  return k == 0 ? 30 : (k == 1 ? 18 : (k == 2 ? 4 : (k == 3 ? 12 : (k == 4 ? 1 : 5))));
}
template <int K, int LIM>
__host__ __device__ constexpr double fixed_den() {
  return (K == 6 ? 20.0 : 70.0) * (LIM == LIM_TVD5 ? 60.0 : 1.0);
}

/* Adds fixed_den() sum_{k nonsmooth} d_k (limited_k - f_k) of one side, in units, to acc:
   MP (Eqs. maximal_curvature-value_min_max, mp_flux; everything relative to f_i, where
   f^min <= 0 <= f^max, so the median is a clamp) or TVD5. */
template <int K, int LIM>
__device__ __forceinline__ void fixed_correction(const long long (&D)[K - 1], unsigned bits, const SchemeDev& S,
                                                 Acc96& acc) {
  constexpr int c = K / 2 - 1, nk = K - 2;
  if constexpr (LIM == LIM_TVD5) {
    const long long D0 = D[c - 1], Dp = D[c];
    const long long B = -2 * D[c - 2] + 11 * D0 + 24 * Dp - 3 * D[c + 1];  /* 30 B */
    const long long lo = lmin2(lmin2(60 * D0, 60 * Dp), B), hi = lmax2(lmax2(60 * D0, 60 * Dp), B);
    const long long pd = D0 > 0 ? lmax2(lo, 0) : (D0 < 0 ? lmin2(hi, 0) : 0);  /* 60 (f - f_i) */
#pragma unroll
    for (int k = 0; k < nk; ++k)
      if (!(bits >> k & 1u)) acc.add(fixed_weight<K>(k), pd - cand60<c>(k, D));
  } else {
    const long long dm = D[c - 1] - D[c - 2], d0 = D[c] - D[c - 1], dp = D[c + 1] - D[c];
    long long hp, hm;
    if (S.mp_curv == CURV_M4) {
      hp = lminmod(lminmod(4 * d0 - dp, 4 * dp - d0), lminmod(d0, dp));
      hm = lminmod(lminmod(4 * dm - d0, 4 * d0 - dm), lminmod(dm, d0));
    } else {
      hp = lminmod(d0, dp);
      hm = lminmod(dm, d0);
    }
    const long long md = (D[c] - hp) >> 1, ul = mul_q60(D[c - 1], S.alpha_q60);
    const long long lc = (D[c - 1] >> 1) + mul_q60(hm, S.beta_third_q60);
    const long long fmin = lmax2(lmin2(lmin2(0, D[c]), md), lmin2(lmin2(0, ul), lc));
    const long long fmax = lmin2(lmax2(lmax2(0, D[c]), md), lmax2(lmax2(0, ul), lc));
#pragma unroll
    for (int k = 0; k < nk; ++k)
      if (!(bits >> k & 1u)) {
        const long long x = cand_unit<c>(k, D);
        acc.add(fixed_weight<K>(k), lmin2(lmax2(x, fmin), fmax) - x);
      }
  }
}

}  // namespace tenom
