/* Face sweep, first half: the central flux of every face and an FP32 certificate that the
 * nonlinear reconstruction would return exactly it (Sections 2.2, 3.3 and 4 of arXiv
 * 2010.13289).
 *
 * Where every candidate of both split sides of a characteristic field is smooth (delta_k = 1,
 * Eq. cut-off) and the optimal weights are the maximal-order d_k, the field's reconstruction
 * is the K-point central formula on both sides; the mirrored f- stencil carries the same
 * symmetric coefficients c_q, so f+ + f- = sum_q c_q (g+_q + g-_q) = sum_q c_q G_q = l_s . Fc
 * with Fc = sum_q c_q F(U_q): the LLF terms cancel, and when every field of the face is such
 * a field the back-projection returns Fc itself (R L = I).  screen_kernel writes Fc to every
 * face, certifies per face and field that all candidates are smooth, and appends the faces
 * with an uncertified field to the axis's work list; nonlinear_kernel (tenom_nonlinear.cuh)
 * then works through the lists of all axes in FP64.
 *
 * The FP64 pipe of GB300 runs at 1/64 of the FP32 rate, so a face that is certified costs the
 * K nvar FMAs of Fc and a share of its points' fluxes; everything the certificate needs --
 * Roe average, differences, projections, indicators -- runs in FP32 and on the integer pipe
 * with rigorous error bounds.  What bounds it (ncu, 2D 1024^2 TENO8): FP64 pipe 57 % and issue
 * 65 % busy, 0.124 ms for 1.05 M faces (16 FP64 pipe cycles a face, 93 instructions issued per
 * warp and face).  The single kernel this pair replaced formed Roe state, eigenvectors and the
 * composition in FP64 for every warp that held an uncertified face and waited for its own
 * queue at CTA barriers: 1024^2 TENO8 sweeps 0.72 ms against 0.43 ms for the pair, one step of
 * 2048^2 TENO8-TVD5 17.8 -> 5.8 ms, TENO6-MP 13.2 -> 5.3, 256^3 TENO8-MP 133 -> 52 with the
 * nonlinear kernel's later forms. */
#pragma once
#include "tenom_recon.cuh"
#include "tenom_face.cuh"
#include "tenom_adjoint.cuh"

namespace tenom {

/* Certificate that every candidate of one split side is smooth (delta_k = 1 for every k).
   d: the K - 1 differences of the characteristic sequence up to a common factor, each within
   E of its exact value.  With x_k = 1 + tau/beta_k (gamma_k = x_k^6, chi_k = gamma_k / sum),
   sum <= nk x_max^6 gives
     x_max <= R x_min  =>  chi_k >= 1/(nk R^6) >= C_T,   R = (nk C_T)^(-1/6) (quick_r, rounded down),
   and with beta_min >= L, beta_max <= U, tau <= T (bounds on the exact values) either of
     T <= (R - 1) L,     T (U - R L) <= (R - 1) L U
   implies x_max <= R x_min (1 + tau/L - R (1 + tau/U) is linear in tau and negative at 0).
   Bounds: each form beta = sum_j w_j t_j^2 is evaluated with t_j within Eb sum_i |m_ji| of its
   exact value, Eb = E + 10 u max|d| (dot product of at most 7 terms with rounded
   coefficients), so |sqrt(beta) - sqrt(beta_exact)| <= sqrt(kk) Eb, and 2 sqrt(beta kk) Eb <=
   s beta + kk Eb^2 / s turns that into beta (1 -+ s) -+ kk (1 + 1/s) Eb^2, with s = 1/32 for the
   beta_k and s = 2^-11 for tau (tau's bound is what a candidate near a critical point, with a
   beta_k far below the others', is compared with); the constants below (0.966, 1.0315, 4.95e-4,
   1.04) add the 20 u relative rounding of the sums of squares.  No square root, division or interval arithmetic: about a third of the work of
   bounding every gamma_k, and it fails on few smooth sides (per face of the 256^3 solenoidal
   state 0.17 fields are truly nonsmooth).
   Adaptive C_T (TENO8A): 1e-7, the largest, always holds; where the least of the four eta is
   at least 0.2 (beta >= 10 for eta >= 0.1984, Eqs. shock_indicator, cut-off_adjust; the
   epsilon only raises eta) C_T is 1e-10 and R larger; need_ex (the flag byte holds [beta])
   certifies only those. */
template <int K>
__device__ __forceinline__ bool quick_smooth(const float (&d)[K - 1], float E, const SchemeDev& S, bool need_ex) {
  constexpr int c = K / 2 - 1;
  const float u = 5.9604645e-8f;
  float dm = 0.f;
#pragma unroll
  for (int t = 0; t < K - 1; ++t) dm = fmaxf(dm, fabsf(d[t]));
  const float Eb = fmaf(10.f * u, dm, E);
  const float eb2 = Eb * Eb, e2 = 33.f * eb2;
  const float b0 = beta0<c - 1, false, float>(d), b1 = beta1<c, false, float>(d), b2 = beta2<c - 2, false, float>(d);
  const float b3 = beta3<c, false, float>(d);
  float lo = fminf(fmaf(-1.04f * beta_norm(0), e2, b0), fmaf(-1.04f * beta_norm(1), e2, fminf(b1, b2)));
  float hi = fmaxf(fmaxf(b0, b1), fmaxf(b2, b3));
  float bK;
  if constexpr (K == 8) {
    const float b4 = beta4<c - 3, false, float>(d), b5 = beta5<c, false, float>(d);
    lo = fminf(lo, fminf(fmaf(-1.04f * beta_norm(3), e2, fminf(b3, b4)), fmaf(-1.04f * beta_norm(5), e2, b5)));
    hi = fmaxf(hi, fmaxf(b4, b5));
    bK = betaK8<0, false, float>(d);
  } else {
    lo = fminf(lo, fmaf(-1.04f * beta_norm(3), e2, b3));
    bK = betaK6<0, false, float>(d);
  }
  const float comb = (b1 + b2 + 4.f * b0) * (1.f / 6.f);
  const float T = fabsf(bK - comb) + fmaf(4.95e-4f, bK + comb, (2060.f * (BetaNorm<K>::kK + 6.f)) * eb2);
  float R = S.quick_r[0];
  if (S.ct_mode == CT_ADAPTIVE) {
    /* 2 |a b| - 0.2 (a^2 + b^2) over the four neighbouring pairs, |a|, |b| known to within Eb */
    float m = 1e30f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float a = d[c + q - 1], b = d[c + q - 2];
      m = fminf(m, 2.f * fabsf(a * b) - 0.2f * fmaf(a, a, b * b));
    }
    const bool ten = m >= 5.f * Eb * dm;  /* [beta] = 10 */
    R = ten ? S.quick_r[1] : (need_ex ? 1.f : R);
  }
  const float L = 0.966f * lo, U = fmaf(1.0315f, hi, (1.04f * BetaNorm<K>::kmax) * e2);
  const float r1 = (R - 1.f) * L;
  /* written so that a NaN fails; dm <= 1e15 keeps every form finite, and the product form
     needs its factors away from under- and overflow */
  return dm <= 1e15f && lo >= 1e-30f &&
         (T <= r1 || (lo >= 1e-18f && U <= 1e15f && T <= 1e17f && T * (U - R * L) <= r1 * U));
}

/* FP32 data of a staged point (component c of point p at c * NP + p): rho, velocity, p and c as
   hi + lo (hi the FP64 value truncated to FP32, lo the rest), a check word of the state's low
   bits, and the differences of rho, velocity, p, c to the next point along the axis */
template <int NV>
struct ScreenLayout {
  static constexpr int D = NV - 2, NQ = NV + 1;
  static constexpr int R = 0, V = 1, P = 1 + D, C = 2 + D;   /* quantity order */
  static constexpr int hi = 0, lo = NQ, chk = 2 * NQ, df = 2 * NQ + 1, NF = 3 * NQ + 1;
};

/* x - hi for hi = f32_rz(x), on the integer and FP32 pipes: the 29 mantissa bits below hi's, as a
   signed float of at most 24 bits (within 2^-47 |x|) */
__device__ __forceinline__ float f32_rest(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7ffu) - 1023 - 52;        /* value of the last mantissa bit: 2^e */
  const float m = (float)(lo & 0x1fffffffu);
  if (e < -126 || e > 127) return 0.f;                          /* far outside the FP32 range: hi is 0 or inf, or the rest is below 2^-97 */
  const float r = m * __int_as_float((e + 127) << 23);
  return (int)hi < 0 ? -r : r;
}

/* the screen's data of point p, and (once all points are there) its differences to point p + step */
template <int NV>
__device__ __forceinline__ void stage_screen_point(const double (&u)[NV], const double (&vel)[NV - 2], double pr, double cs,
                                                   float* sf, int NP, int p) {
  using L = ScreenLayout<NV>;
  unsigned chk = 0u;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const unsigned x = (unsigned)__double2loint(u[v]);
    chk ^= __funnelshift_l(x, x, 6 * v);
  }
  sf[L::chk * NP + p] = __uint_as_float(chk);
  auto put = [&](int c, double x) {
    sf[(L::hi + c) * NP + p] = f32_rz(x);
    sf[(L::lo + c) * NP + p] = f32_rest(x);
  };
  put(L::R, u[0]);
#pragma unroll
  for (int d = 0; d < NV - 2; ++d) put(L::V + d, vel[d]);
  put(L::P, pr);
  put(L::C, cs);
}
template <int NV>
__device__ __forceinline__ void stage_screen_differences(float* sf, int NP, int p, int step) {
  using L = ScreenLayout<NV>;
  float any = 0.f;
#pragma unroll
  for (int c = L::NQ - 1; c >= 0; --c) {  /* rho (c = 0) last */
    const float* h = sf + (L::hi + c) * NP + p;
    const float* l = sf + (L::lo + c) * NP + p;
    float x = (h[step] - h[0]) + (l[step] - l[0]);
    any += fabsf(x);  /* a sum, which keeps a NaN */
    if (c == 0) {
      /* equal to 47 bits but not bit for bit: not a constant stencil (nor one that can be certified) */
      if (any == 0.f &&
          __float_as_uint(sf[L::chk * NP + p + step]) != __float_as_uint(sf[L::chk * NP + p])) x = 1e-37f;
      /* a point that is not finite in FP32 (infinite here: f32_rz): its maxima would drop the NaN of
         inf - inf, and a stencil of such points would pass for a constant one */
      if (!(any <= 3e38f)) x = __int_as_float(0x7f800000);
    }
    sf[(L::df + c) * NP + p] = x;
  }
}

/* Shared-memory values read again after this point are loaded again: the compiler otherwise keeps
   the tile values of a face's several passes (30-60 of them) in spilled registers, and the local
   memory of 768 threads does not fit L1 beside the tile (2D TENO8 328 -> 108 bytes a thread at 80
   registers, TENO6 128 -> 8; 2048^2 step 6.45 -> 5.98 ms and 5.44 -> 5.17 ms with the
   differences of both sides formed together).  Not in 1D, where few threads wait on latency. */
__device__ __forceinline__ void keep_loads_here() { asm volatile("" ::: "memory"); }

/* Fields of one face that are NOT certified central (bit s); the face's stencil point q is
   tile point p0 + q * LANES.

   In the frame moving with the Roe velocity u~ (w = u - u~) the left eigenvectors are those
   at rest, so with E' = p/(gamma - 1) + rho w^2/2, b1 = (gamma - 1)/c~^2:
     W_{u-+c} = (b1 E' -+ rho w_n/c~)/2,  W_0 = rho - b1 E',  W_t = rho w_t,
     G_s = l_s.F = (u_n + sigma_s c~) W_s + X_s,  sigma = -1, +1 (acoustic), 0,
     2 X_{u-+c} = +-(gamma - 1)/(2 c~) rho w^2 - w_n (rho - b1 p),  X_0 = -b1 p w_n,  X_t = 0,
   and the split sequences are 2 g+-_q = (u_n + sigma c~ +- alpha) W + X.  Their differences are
     (w_{t+1} + off+-) dW_t + R_t,  off+- = u~_n + sigma c~ +- alpha,
   with (dv, drho, dp the point differences, w accumulated from the face outwards, k = rho
   (c^2 - c~^2)/c~^2 + b1 rho w^2/2, d(rho w^2) = drho w1^2 + rho0 (w0 + w1).dv):
     2 dW_{u-+c} = e -+ m,   e = dp/c~^2 + b1 d(rho w^2)/2,   m = (w1 drho + rho0 dv_n)/c~,
     2 R_{u-+c} = k dv_n - w1 (drho - b1 dp) -+ Q,  Q = (rho0 w0 dv_n - (gamma - 1)/2 d(rho w^2))/c~,
     dW_0 = drho - e,  R_0 = -(k dv_n + b1 w1 dp),  dW_t = w1_t drho + rho0 dv_t,  R_t = rho0 w0_t dv_n.
   Every term is a product of differences with quantities known to a relative accuracy, and
   where all speeds of the window have one sign the offset that cancels (alpha against the
   speed itself) is formed from differences too: the sequences of a wave running the other
   way, smaller by the relative change of the speed, keep their relative accuracy.  (Projecting
   U and F loses exactly that: with the differences of U and F the screen certified 1.46 fields
   of a face less on the 2D TENO8 state, where 0.04 are nonsmooth.)

   Error bounds (u = 2^-24, H = K/2; M_x = largest |dx| of the window + 2^-27 |x|, which covers
   the 2^-46 |x| of the hi/lo differences and the FP64 rounding of u, p, c against U):
   wl within 9u, w within 40u M_v (|w| <= H M_v), c~ within 6u th, c - c~ within 60u (M_c + T/c~),
   th = 1 + |cR^2 - cL^2|/c~^2 + 3 T/c~^2, T = (gamma - 1)/2 wl wr |dv|^2 (gated: th <= 2), so that
   dW is within 60u th of its terms' magnitudes MW, R within 80u th of Y, an offset within
   120u (M_n + M_c + T/c~) of differences or 20u th (|u~_n| + c~) more where it does not cancel. */
template <int NV, int K, int AXIS, int LANES>
__device__ __forceinline__ unsigned screen_face(const float* sf, int NP, int p0, float gm1, const SchemeDev& S,
                                                bool need_ex) {
  using L = ScreenLayout<NV>;
  constexpr int D = NV - 2, H = K / 2;
  constexpr unsigned all = (1u << NV) - 1u;
  const float u = 5.9604645e-8f;
  auto at = [&](int comp, int q) -> float { return sf[comp * NP + p0 + q * LANES]; };
  auto val = [&](int comp, int q) -> float { return at(L::hi + comp, q); };
  auto dif = [&](int comp, int t) -> float { return at(L::df + comp, t); };

  /* Roe state of points H - 1 | H */
  const float rl = val(L::R, H - 1), rr = val(L::R, H);
  const float sl = __fsqrt_rn(rl), wl = __fdividef(sl, sl + __fsqrt_rn(rr)), wr = 1.f - wl;
  float dv2 = 0.f, q2 = 0.f, wn[K] = {}, vt[D];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const float dv = dif(L::V + d, H - 1);
    vt[d] = fmaf(wr, dv, val(L::V + d, H - 1));
    dv2 = fmaf(dv, dv, dv2);
    q2 = fmaf(vt[d], vt[d], q2);
  }
  const float cl = val(L::C, H - 1), cr = val(L::C, H);
  const float Tv = 0.5f * gm1 * wl * wr * dv2;
  const float c2 = fmaf(wl * cl, cl, fmaf(wr * cr, cr, Tv));
  const float ic = rsqrtf(c2), i2 = __fdividef(1.f, c2), ct = c2 * ic, b1 = gm1 * i2, hb1 = 0.5f * b1;
  const float dcm = dif(L::C, H - 1);
  const float gl = -__fdividef(fmaf(wr * dcm, cl + cr, Tv), ct + cl);  /* c_{H-1} - c~ */
  const float th = 1.f + fmaf(fabsf(dcm), cl + cr, 3.f * Tv) * i2;
  const float un = vt[AXIS];

  float Mr = 0.f, Mv[D], Mp = 0.f, Mc = 0.f;
#pragma unroll
  for (int d = 0; d < D; ++d) Mv[d] = 0.f;
#pragma unroll
  for (int t = 0; t < K - 1; ++t) {
    Mr = fmaxf(Mr, fabsf(dif(L::R, t)));
    Mp = fmaxf(Mp, fabsf(dif(L::P, t)));
    Mc = fmaxf(Mc, fabsf(dif(L::C, t)));
#pragma unroll
    for (int d = 0; d < D; ++d) Mv[d] = fmaxf(Mv[d], fabsf(dif(L::V + d, t)));
  }
  float mx = fmaxf(Mr, fmaxf(Mp, Mc));
#pragma unroll
  for (int d = 0; d < D; ++d) mx = fmaxf(mx, Mv[d]);
  /* a constant stencil: every sequence is constant, beta = tau = 0, all smooth (and eta = 1, [beta] = 10) */
  if (mx == 0.f) return 0u;
  /* (c2: the fast division returns 0 for divisors above 2^126; mx: not finite) */
  if (!(th <= 2.f && q2 <= 1e8f * c2 && c2 <= 8e37f && mx <= 3e38f)) return all;
  unsigned still = 0u;  /* shear fields with no tangential velocity at all: the sequence is zero */
#pragma unroll
  for (int d = 0; d < D; ++d)
    if (d != AXIS && Mv[d] == 0.f && vt[d] == 0.f) still |= 1u << (2 + (d < AXIS ? d : d - 1));

  /* bounds over the window */
  const float k27 = 7.4505806e-9f;
  const float rh0 = fmaxf(rl, rr), ph0 = fmaxf(val(L::P, H - 1), val(L::P, H));
  Mr = fmaf(k27, rh0, Mr);
  Mp = fmaf(k27, fmaf(rh0, q2, ph0), Mp);
  Mc = fmaf(k27, ct, Mc);
  const float vs = k27 * (__fsqrt_rn(q2) + ct);
  float w2h = 0.f, sv = 0.f;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    Mv[d] += vs;
    w2h = fmaf(Mv[d], Mv[d], w2h);
  }
  sv = (float)H * w2h;                   /* sum_d |w_d| M_v,d */
  w2h *= (float)(H * H);                 /* max |w|^2 */
  const float Mn = Mv[AXIS], whn = (float)H * Mn, rh = fmaf((float)H, Mr, rh0);
  const float gh = fmaf((float)(H + 1), Mc, Tv * ic);   /* max |c - c~| */
  const float B2 = fmaf(Mr, w2h, 2.f * rh * sv);
  const float Me = fmaf(Mp, i2, hb1 * B2), Mm = ic * fmaf(whn, Mr, rh * Mn);
  const float kh = rh * fmaf(gh * (2.f * ct + gh), i2, hb1 * w2h);
  const float dcan = 120.f * u * fmaf(Tv, ic, Mn + Mc);

  if constexpr (NV > 3) keep_loads_here();
  /* differences shared by the acoustic pair and the entropy field */
  float e[K - 1], m[K - 1], Q[K - 1], kn[K - 1];
  float mxm = -1e30f, mnm = 1e30f, mxp = -1e30f, mnp = 1e30f, mx0 = -1e30f, mn0 = 1e30f;
  auto pass = [&](int q, float g) {      /* extremes of w + sigma (c - c~): speeds relative to the face's */
    const float a = wn[q] - g, b = wn[q] + g;
    mxm = fmaxf(mxm, a);
    mnm = fminf(mnm, a);
    mxp = fmaxf(mxp, b);
    mnp = fminf(mnp, b);
    mx0 = fmaxf(mx0, wn[q]);
    mn0 = fminf(mn0, wn[q]);
  };
  /* difference t between points t and t + 1 with w and c - c~ of both */
  auto step = [&](int t, const float (&w0)[D], const float (&w1)[D], float g0) {
    const float r0 = val(L::R, t), dr = dif(L::R, t), dn = dif(L::V + AXIS, t);
    float s0 = 0.f, s1 = 0.f, sd = 0.f;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      s0 = fmaf(w0[d], w0[d], s0);
      s1 = fmaf(w1[d], w1[d], s1);
      sd = fmaf(w0[d] + w1[d], dif(L::V + d, t), sd);
    }
    const float drw2 = fmaf(dr, s1, r0 * sd);
    e[t] = fmaf(dif(L::P, t), i2, hb1 * drw2);
    m[t] = ic * fmaf(w1[AXIS], dr, r0 * dn);
    kn[t] = r0 * fmaf(g0 * (2.f * ct + g0), i2, hb1 * s0) * dn;
    Q[t] = ic * fmaf(r0 * w0[AXIS], dn, -0.5f * gm1 * drw2);
  };
  {
    float w0[D], w1[D], g = gl;  /* outwards to the left from H - 1 */
#pragma unroll
    for (int d = 0; d < D; ++d) w1[d] = -wr * dif(L::V + d, H - 1);
    wn[H - 1] = w1[AXIS];
    pass(H - 1, g);
#pragma unroll
    for (int t = H - 2; t >= 0; --t) {
#pragma unroll
      for (int d = 0; d < D; ++d) w0[d] = w1[d] - dif(L::V + d, t);
      g -= dif(L::C, t);
      wn[t] = w0[AXIS];
      pass(t, g);
      step(t, w0, w1, g);
#pragma unroll
      for (int d = 0; d < D; ++d) w1[d] = w0[d];
    }
    g = gl;                      /* across the face and to the right */
#pragma unroll
    for (int d = 0; d < D; ++d) w0[d] = -wr * dif(L::V + d, H - 1);
#pragma unroll
    for (int t = H - 1; t < K - 1; ++t) {
#pragma unroll
      for (int d = 0; d < D; ++d) w1[d] = (t == H - 1) ? wl * dif(L::V + d, t) : w0[d] + dif(L::V + d, t);
      wn[t + 1] = w1[AXIS];
      step(t, w0, w1, g);
      g += dif(L::C, t);
      pass(t + 1, g);
#pragma unroll
      for (int d = 0; d < D; ++d) w0[d] = w1[d];
    }
  }

  if constexpr (NV > 3) keep_loads_here();
  unsigned bad = 0u;
  float off[2], del[2];  /* side f+, f-: off+- = lambda~ +- alpha and the bound of its error */
  auto offsets = [&](float lam, float lerr, float hi, float lo) {
    const bool pos = lam + lo > lerr, neg = lam + hi < -lerr;
    const float al = fmaxf(fabsf(lam + hi), fabsf(lam + lo));
    off[0] = pos ? 2.f * lam + hi : (neg ? -lo : lam + al);
    off[1] = pos ? -hi : (neg ? 2.f * lam + lo : lam - al);
    del[0] = dcan + (neg ? 0.f : lerr);
    del[1] = dcan + (pos ? 0.f : lerr);
  };
  /* differences of f+ and of f- on its mirrored stencil (the forms are even in d), formed together
     so that the projections' terms are not kept over the two tests */
  float dp[K - 1], dn[K - 1], lm[2];
  auto diff = [&](int t, float dw, float R) {
    const float l0 = wn[t + 1] + off[0], l1 = wn[t + 1] + off[1];
    lm[0] = fmaxf(lm[0], fabsf(l0));
    lm[1] = fmaxf(lm[1], fabsf(l1));
    dp[t] = fmaf(l0, dw, R);
    dn[K - 2 - t] = fmaf(l1, dw, R);
  };
  auto test = [&](float MW, float Y) -> bool {
    const float u80 = 80.f * u * th, u60 = 60.f * u * th;
    const bool ok = quick_smooth<K>(dp, fmaf(fmaf(u60, lm[0], del[0]), MW, u80 * Y), S, need_ex);
    return quick_smooth<K>(dn, fmaf(fmaf(u60, lm[1], del[1]), MW, u80 * Y), S, need_ex) && ok;
  };
  {
    const float lerr = 20.f * u * th * (fabsf(un) + ct);
    const float MW = Me + Mm;
    const float Y = fmaf(kh, Mn, fmaf(whn, fmaf(b1, Mp, Mr), ic * fmaf(rh * whn, Mn, 0.5f * gm1 * B2)));
#pragma unroll 1
    for (int i = 0; i < 2; ++i) {
      const float sg = i ? 1.f : -1.f;
      offsets(fmaf(sg, ct, un), lerr, i ? mxp : mxm, i ? mnp : mnm);
      if constexpr (NV > 3) keep_loads_here();
      lm[0] = lm[1] = 0.f;
#pragma unroll
      for (int t = 0; t < K - 1; ++t)
        diff(t, fmaf(sg, m[t], e[t]), fmaf(sg, Q[t], fmaf(-wn[t + 1], fmaf(-b1, dif(L::P, t), dif(L::R, t)), kn[t])));
      bad |= test(MW, Y) ? 0u : (i ? 1u << (NV - 1) : 1u);
    }
  }
  /* entropy and shear fields: speed u_n */
  offsets(un, 10.f * u * fmaf(4.f, Mn, fabsf(un)), mx0, mn0);
#pragma unroll 1
  for (int s = 1; s <= NV - 2; ++s) {
    float MW, Y;
    if constexpr (NV > 3) keep_loads_here();
    lm[0] = lm[1] = 0.f;
    if (s == 1) {
#pragma unroll
      for (int t = 0; t < K - 1; ++t) diff(t, dif(L::R, t) - e[t], -fmaf(b1 * wn[t + 1], dif(L::P, t), kn[t]));
      MW = Mr + Me;
      Y = fmaf(kh, Mn, b1 * whn * Mp);
    } else {
      const int dt = (s - 2) < AXIS ? (s - 2) : (s - 1);
      const float* sd = sf + (L::df + L::V + dt) * NP + p0;
      float Mt = 0.f;
#pragma unroll
      for (int x = 0; x < D; ++x) Mt = (x == dt) ? Mv[x] : Mt;
      float w1 = -wr * sd[(H - 1) * LANES];
#pragma unroll
      for (int t = H - 2; t >= 0; --t) {
        const float dvt = sd[t * LANES], w0 = w1 - dvt, r0 = val(L::R, t);
        diff(t, fmaf(w1, dif(L::R, t), r0 * dvt), r0 * w0 * dif(L::V + AXIS, t));
        w1 = w0;
      }
      float w0 = -wr * sd[(H - 1) * LANES];
#pragma unroll
      for (int t = H - 1; t < K - 1; ++t) {
        const float dvt = sd[t * LANES], r0 = val(L::R, t);
        w1 = (t == H - 1) ? wl * dvt : w0 + dvt;
        diff(t, fmaf(w1, dif(L::R, t), r0 * dvt), r0 * w0 * dif(L::V + AXIS, t));
        w0 = w1;
      }
      const float wht = (float)H * Mt;
      MW = fmaf(wht, Mr, rh * Mt);
      Y = rh * wht * Mn;
    }
    bad |= ((still >> s & 1u) || test(MW, Y)) ? 0u : 1u << s;
  }
  return bad;
}

/* fs = l_s . Fc of every field, with the FP64 Roe state of cells cl | cr (record kernels) */
template <int NV, int AXIS>
__device__ __forceinline__ void central_fields(const FaceArgs& A, long long cl, long long cr, const double (&Fc)[NV],
                                               double (&fs)[NV]) {
  constexpr int D = NV - 2;
  const double sL = __ldg(A.P + (D + 3) * A.ncell + cl), sR = __ldg(A.P + (D + 3) * A.ncell + cr);
  const double wsum = rcp_nr(sL + sR);
  double ut[D], q2 = 0.0, uF = 0.0;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    ut[d] = (sL * __ldg(A.P + d * A.ncell + cl) + sR * __ldg(A.P + d * A.ncell + cr)) * wsum;
    q2 += ut[d] * ut[d];
    uF = fma(ut[d], Fc[1 + d], uF);
  }
  const double Ht = (sL * __ldg(A.P + (D + 2) * A.ncell + cl) + sR * __ldg(A.P + (D + 2) * A.ncell + cr)) * wsum;
  const double cinv = rsqrt_nr((A.gamma - 1.0) * (Ht - 0.5 * q2));
  const double b1 = (A.gamma - 1.0) * (cinv * cinv), b2 = 0.5 * q2 * b1;
  const double a = fma(b2, Fc[0], b1 * (Fc[NV - 1] - uF));
  const double b = cinv * fma(ut[AXIS], Fc[0], -Fc[1 + AXIS]);
  fs[0] = 0.5 * (a + b);
  fs[1] = Fc[0] - a;
  fs[NV - 1] = 0.5 * (a - b);
#pragma unroll
  for (int s = 2; s <= NV - 2; ++s) {
    const int dt = (s - 2) < AXIS ? (s - 2) : (s - 1);
    fs[s] = fma(-ut[dt], Fc[0], Fc[1 + dt]);
  }
}

/* shared memory of screen_kernel: F of the tile's points in FP64 and their FP32 data */
template <int NV, int K, int AXIS>
constexpr size_t screen_smem() {
  using T = FaceTile<NV, K, AXIS, true>;
  return (sizeof(double) * (size_t)NV + sizeof(float) * (size_t)ScreenLayout<NV>::NF) * T::NP;
}

/* REC: also the linearisation of the certified fields (the record kernels' tape, see
   nonlinear_kernel): sigma_q = c_q, delta_q = 0, omegaW = -0 (kCentralMark), fs = l_s . Fc. */
template <int NV, int K, int AXIS, bool REC>
__global__ void __launch_bounds__(FaceTile<NV, K, AXIS, true>::THREADS,
                                  screen_threads_per_sm(K, NV) / FaceTile<NV, K, AXIS, true>::THREADS)
screen_kernel(const FaceArgs A) {
  using T = FaceTile<NV, K, AXIS, true>;
  using L = ScreenLayout<NV>;
  constexpr int H = T::H, D = NV - 2, NP = T::NP;
  extern __shared__ double sm[];
  double* const sF = sm;
  float* const sf = reinterpret_cast<float*>(sm + NV * NP);
  __shared__ int s_cnt, s_base;
  const int tid = threadIdx.x;
  if (tid == 0) s_cnt = 0;

  const int na = A.n[AXIS];
  int f0, x0 = 0, o1 = 0, o2 = 0;
  f0 = blockIdx.y * T::FACES;
  if (AXIS == 0) {
    const int row = blockIdx.x;          /* y + ny * z */
    o1 = row % A.n[1];
    o2 = row / A.n[1];
  } else {
    x0 = blockIdx.x * T::LANES;
    o2 = blockIdx.z;                     /* AXIS 1: z ; AXIS 2: y */
  }
  const long long sy = A.n[0], sz = (long long)A.n[0] * A.n[1];
  const long long sa = (AXIS == 0) ? 1 : (AXIS == 1 ? sy : sz);

  /* --- stage the tile's points: F in FP64, the screen's point data in FP32 --- */
  for (int p = tid; p < NP; p += T::THREADS) {
    const int lane = (AXIS == 0) ? 0 : (p % T::LANES);
    const int row = (AXIS == 0) ? p : (p / T::LANES);
    const int j = bc_wrap(f0 - H + row, na, A.bc[AXIS]);
    long long base;
    if (AXIS == 0) base = sy * o1 + sz * o2;
    else {
      int x = x0 + lane;
      x = x < A.n[0] ? x : A.n[0] - 1;
      base = x + (AXIS == 1 ? sz * o2 : sy * o2);
    }
    const long long cell = base + sa * j;
    double u[NV], vel[D], pr, cs;
#pragma unroll
    for (int q = 0; q < NV; ++q) u[q] = __ldg(A.U + q * A.ncell + cell);
    /* primitives computed once per cell per stage */
#pragma unroll
    for (int d = 0; d < D; ++d) vel[d] = __ldg(A.P + d * A.ncell + cell);
    pr = __ldg(A.P + D * A.ncell + cell);
    cs = __ldg(A.P + (D + 1) * A.ncell + cell);
    double F[NV];
    F[0] = u[1 + AXIS];
#pragma unroll
    for (int d = 0; d < D; ++d) F[1 + d] = (d == AXIS) ? fma(u[1 + d], vel[AXIS], pr) : u[1 + d] * vel[AXIS];
    F[NV - 1] = (u[NV - 1] + pr) * vel[AXIS];
#pragma unroll
    for (int v = 0; v < NV; ++v) sF[v * NP + p] = F[v];
    stage_screen_point<NV>(u, vel, pr, cs, sf, NP, p);
  }
  __syncthreads();
  for (int p = tid; p < NP - T::LANES; p += T::THREADS) stage_screen_differences<NV>(sf, NP, p, T::LANES);
  __syncthreads();

  /* --- one face per thread --- */
  const int lane = (AXIS == 0) ? 0 : (tid % T::LANES);
  const int jf = (AXIS == 0) ? tid : (tid / T::LANES);
  const int f = f0 + jf;
  const int xg = x0 + lane;
  /* a periodic axis computes faces 0 .. n-1 only: face n has face 0's stencil points, and
     face 0's thread writes it to both places (no nearly empty last tile per line) */
  const bool wrapped = A.bc[AXIS] == 0;
  const bool active = (wrapped ? f < na : f <= na) && (AXIS == 0 || xg < A.n[0]);
  auto face_index = [&](int ff) -> long long {
    if (AXIS == 0) return ff + (long long)(A.n[0] + 1) * (o1 + (long long)A.n[1] * o2);
    if (AXIS == 1) return xg + (long long)A.n[0] * (ff + (long long)(A.n[1] + 1) * o2);
    return xg + (long long)A.n[0] * (o2 + (long long)A.n[1] * ff);
  };
  const long long flin = face_index(f);
  unsigned bad = 0u;
  if (active) {
    const int p0 = jf * T::LANES + lane;
    constexpr unsigned allf = (1u << NV) - 1u;
    const bool adaptive = A.sch.ct_mode == CT_ADAPTIVE;
    bad = A.sch.screen ? screen_face<NV, K, AXIS, T::LANES>(sf, NP, p0, (float)(A.gamma - 1.0), A.sch, A.flags && adaptive)
                       : allf;
    double cw[K], Fc[NV];
    central_weights<K>(cw);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const double* s = sF + v * NP + p0;
      double x = cw[0] * s[0];
#pragma unroll
      for (int q = 1; q < K; ++q) x = fma(cw[q], s[q * T::LANES], x);
      Fc[v] = x;
      A.Fhat[v * A.nface + flin] = x;
    }
    if (wrapped && f == 0) {
      const long long fn = face_index(na);
#pragma unroll
      for (int v = 0; v < NV; ++v) A.Fhat[v * A.nface + fn] = Fc[v];
    }
    if (A.flags) {  /* the certified fields' bytes: every candidate smooth, [beta] = 10 */
      const unsigned allk = ((1u << (K - 2)) - 1u) | (adaptive ? 3u << 6 : 0u);
      for (int r = 0; r < ((wrapped && f == 0) ? 2 : 1); ++r) {
        uint8_t* o = A.flags + (r ? face_index(na) : flin) * NV * 2;
#pragma unroll
        for (int e = 0; e < 2 * NV; ++e) o[e] = (uint8_t)allk;
      }
    }
    if constexpr (REC) {
      if (bad != allf) {
        const long long cell = (AXIS == 0) ? sy * o1 + sz * o2 : xg + (AXIS == 1 ? sz * o2 : sy * o2);
        const long long cl = cell + sa * bc_wrap(f - 1, na, A.bc[AXIS]), cr = cell + sa * bc_wrap(f, na, A.bc[AXIS]);
        double fs[NV];
        central_fields<NV, AXIS>(A, cl, cr, Fc, fs);
        for (int r = 0; r < ((wrapped && f == 0) ? 2 : 1); ++r) {
          double* o = A.lin + (r ? face_index(na) : flin);
#pragma unroll
          for (int s = 0; s < NV; ++s) {
            if (bad >> s & 1u) continue;
            double* os = o + (long long)s * (2 * K + 2) * A.nface;
            os[0] = fs[s];
            os[A.nface] = __longlong_as_double((long long)kCentralMark);  /* -0.0 */
#pragma unroll
            for (int q = 0; q < K; ++q) {
              os[(2 + q) * A.nface] = 0.5 * (cw[q] + cw[K - 1 - q]);
              os[(2 + K + q) * A.nface] = cw[q] - cw[K - 1 - q];
            }
          }
        }
      }
    }
  }
  /* --- append the uncertified faces to the axis's list (one global atomic per CTA) --- */
  const unsigned bal = __ballot_sync(0xffffffffu, bad != 0u);
  int wofs = 0;
  if ((tid & 31) == 0 && bal) wofs = atomicAdd(&s_cnt, __popc(bal));
  wofs = __shfl_sync(0xffffffffu, wofs, 0);
  __syncthreads();
  if (tid == 0 && s_cnt) s_base = (int)atomicAdd(A.count, (unsigned)s_cnt);
  __syncthreads();
  if (bad) {
    const long long pos = (long long)(unsigned)s_base + wofs + __popc(bal & ((1u << (tid & 31)) - 1u));
    if (pos < A.nface) {
      A.list[pos] = (unsigned)flin;
      A.mask[pos] = (uint8_t)bad;
    }
  }
}

}  // namespace tenom
