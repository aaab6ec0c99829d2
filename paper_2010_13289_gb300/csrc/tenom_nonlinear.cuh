/* Face sweep, second half: the faces screen_kernel could not certify, in FP64 (Section 4 of
 * arXiv 2010.13289: Roe-averaged characteristic decomposition, local Lax-Friedrichs
 * splitting, TENO-M per characteristic field and split side, back-projection).
 *
 * One persistent launch works through the lists of every axis.  A CTA takes a chunk of up to
 * NL_THREADS faces of one axis: (0) a thread per face forms the Roe state and the LLF
 * speeds; (1) the uncertified (face, field) pairs of the chunk, ordered by field so that a
 * warp mostly runs one kind of projection, are spread over the CTA's threads: projection of
 * the K points, decisions and reconstruction of both split sides; (2) a thread per face
 * composes the flux.  The list is dense, so every step runs in full warps whatever share of the faces needs it; when there
 * are few faces a chunk is smaller, so that they spread over all SMs.
 *
 * The kernel is written in the axis's own frame: component 1 is the momentum along the axis,
 * 2 .. NV-2 the tangential ones in increasing axis order (fields: 0 u-c, 1 entropy,
 * 2 .. NV-2 shear, NV-1 u+c).
 *
 * FIX: a nonsmooth side only adds its limiter's correction sum_k d_k (limited_k - f_k), in fixed
 * point (tenom_fixed.cuh), and the face flux is Fc + sum_s r_s correction_s (the smooth part of
 * every field sums to Fc, R L = I): what is left of FP64 per field is the projection, in full
 * warps, whatever the decisions.  Items whose stencil reaches across a jump (reaches_jump: the large
 * values beyond it would leave their rounding on a smaller flux) and values outside the
 * fixed-point range take the general FP64 reconstruction, as do all other schemes (!FIX).
 *
 * What bounds it (ncu, 64^3 turbulence TENO8, 4 of 5 fields of 98 % of the faces listed): FP64
 * pipe 69 % busy, then waiting at the CTA's barriers.  Per 3-sweep launch 2.9 ms in FP64 (the
 * limiter's divergent lanes and, for any lane the FP32 filter left undecided, the whole warp in
 * FP64 decisions), 1.9 ms with fixed-point corrections and the second pass, 1.45 ms with the
 * rolled loops and called rare paths (instruction fetch had been the largest stall), 1.19 ms since
 * the filter decides all but 0.01 % of the sides, 1.04 ms with jumps found per face instead of
 * exponents kept per side. */
#pragma once
#include "tenom_recon.cuh"
#include "tenom_face.cuh"
#include "tenom_fixed.cuh"
#include "tenom_adjoint.cuh"

namespace tenom {

struct NonlinArgs {
  const double* U;           /* [NV][ncell] */
  const double* P;           /* cell primitives (velocity, p, c, ..) */
  double* Fhat[3];           /* face fluxes per axis, holding Fc of every face */
  uint8_t* flags[3];         /* [nface][NV][2] or null */
  double* lin[3];            /* linearisation (record kernels) */
  const unsigned* list[3];   /* faces of the axis with an uncertified field, and which (bit s) */
  const uint8_t* mask[3];
  const unsigned* count;     /* list lengths */
  int* status;
  int n[3];
  int bc[3];
  long long ncell;
  long long nface[3];
  double gamma;
  double rgm1;               /* 1 / (gamma - 1) */
  int dim;
  SchemeDev sch;
};

constexpr int NL_THREADS = 128;
constexpr int NL_CTAS_PER_SM = 4;  /* 128 registers a thread */

/* smem rows (doubles per face): Roe state and LLF speeds */
template <int NV>
struct NlRow {
  static constexpr int D = NV - 2;
  static constexpr int u = 0, H = D, ci = D + 1, ct = D + 2, b1 = D + 3, b2 = D + 4, am = D + 5, a0 = D + 6, ap = D + 7,
                       N = D + 8;
};

/* bc_wrap for a point at most half a stencil outside the line (a periodic line has at least
   K/2 cells) */
__device__ __forceinline__ int bc_near(int j, int n, int bc) {
  if (bc == 0) return j < 0 ? j + n : (j >= n ? j - n : j);
  return j < 0 ? 0 : (j >= n ? n - 1 : j);
}

/* face_rows' view of a face of the grid: its line starts at cell `base` with stride sa */
template <int NV, int K>
struct GridFace {
  const double *rho, *vel[NV - 2], *un, *c;
  long long base, sa;
  int f, na, bc;
  __device__ __forceinline__ long long cell(int q) const { return base + sa * bc_near(f - K / 2 + q, na, bc); }
  __device__ __forceinline__ void centre(int e, double& r, double& cs, double (&v)[NV - 2]) const {
    const long long x = cell(K / 2 - 1 + e);
    r = __ldg(rho + x);
    cs = __ldg(c + x);
#pragma unroll
    for (int d = 0; d < NV - 2; ++d) v[d] = __ldg(vel[d] + x);
  }
  __device__ __forceinline__ void speed(int q, double& u, double& cs) const {
    const long long x = cell(q);
    u = __ldg(un + x);
    cs = __ldg(c + x);
  }
  __device__ __forceinline__ void speed32(int, double u, double cs, float& uf, float& cf) const {
    uf = f32_rz(u);
    cf = f32_rz(cs);
  }
};

/* Roe state and LLF speeds of one face into its row (entry r at row[r * TH]).  src.centre(e, rho,
   c, v): density, sound speed and velocity (normal first) of the face's left (0) and right (1)
   cell; src.speed(q, u_n, c): stencil point q, speed32: truncated to FP32.  H~ = h + |u~|^2/2 with h =
   c~^2/(gamma - 1) in its cancellation-free form (weighted c^2 plus (gamma - 1)/2 wl wr |dv|^2), then
   c~^2 = (gamma - 1)(H~ - |u~|^2/2) back from the rounded H~: at Mach M the fields are of size M^2,
   and R L = I has to hold to the rounding of c~^2 against that H~ (a c~^2 that H~ does not give
   leaves M^2 times the rounding of H~ in the pressure: limited near-vacuum steps were up to 5 times
   further off). */
template <int NV, int K, int TH, class Src>
__device__ __forceinline__ void face_rows(const Src& src, double* row, double gm1, double rgm1, int& st) {
  using R = NlRow<NV>;
  constexpr int D = NV - 2;
  double sr[2], cs[2], v[2][D];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    double rho;
    src.centre(e, rho, cs[e], v[e]);
    sr[e] = rho * rsqrt_nr(rho);
  }
  const double ws = rcp_nr(sr[0] + sr[1]), wl = sr[0] * ws, wr = sr[1] * ws;
  double q2 = 0.0, dv2 = 0.0;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const double x = fma(wl, v[0][d], wr * v[1][d]), y = v[1][d] - v[0][d];
    q2 = fma(x, x, q2);
    dv2 = fma(y, y, dv2);
    row[(R::u + d) * TH] = x;
  }
  const double c2f = fma(wl * cs[0], cs[0], fma(wr * cs[1], cs[1], 0.5 * gm1 * (wl * wr) * dv2));
  const double Ht = fma(c2f, rgm1, 0.5 * q2);
  const double c2 = gm1 * (Ht - 0.5 * q2);
  if (!(c2 > 0.0)) st |= ST_ROE;
  const double ci = rsqrt_nr(c2);
  const double b1 = gm1 * (ci * ci);
  row[R::H * TH] = Ht;
  row[R::ci * TH] = ci;
  row[R::ct * TH] = c2 * ci;
  row[R::b1 * TH] = b1;
  row[R::b2 * TH] = 0.5 * q2 * b1;
  /* LLF: alpha_s = max over the K stencil points of |lambda_s|, one per eigenvalue family.  The
     largest |u -+ c| is found in FP32 (each within 5u (|u| + c)) and formed in FP64 where it is
     the only candidate; ties within the error take all K points in FP64 */
  double am = 0.0, a0 = 0.0, ap = 0.0;
  float bm = -1.f, bp = -1.f, sm = -1.f, sp = -1.f, ah = 0.f;
  int qm = 0, qp = 0;
#pragma unroll 1
  for (int q = 0; q < K; ++q) {
    double un, c;
    src.speed(q, un, c);
    a0 = imax_nonneg(a0, iabs(un));
    float uf, cf;
    src.speed32(q, un, c, uf, cf);
    const float xm = fabsf(uf - cf), xp = fabsf(uf + cf);
    ah = fmaxf(ah, fabsf(uf) + cf);
    sm = fmaxf(sm, fminf(xm, bm));
    sp = fmaxf(sp, fminf(xp, bp));
    if (xm > bm) {
      bm = xm;
      qm = q;
    }
    if (xp > bp) {
      bp = xp;
      qp = q;
    }
  }
  const float tie = 10.f * 5.9604645e-8f * ah;
  if (bm - sm > tie && bp - sp > tie && ah < 1e30f && ah > 1e-30f) {
    double un, c;
    src.speed(qm, un, c);
    am = iabs(un - c);
    src.speed(qp, un, c);
    ap = iabs(un + c);
  } else {
#pragma unroll 1
    for (int q = 0; q < K; ++q) {
      double un, c;
      src.speed(q, un, c);
      am = imax_nonneg(am, iabs(un - c));
      ap = imax_nonneg(ap, iabs(un + c));
    }
  }
  row[R::am * TH] = am;
  row[R::a0 * TH] = a0;
  row[R::ap * TH] = ap;
}

/* left eigenvector l_s of a face's row (closed form of R^{-1}; shear: l = e_t - u_t e_0, l[0] only);
   returns alpha_s / 2 */
template <int NV, int TH>
__device__ __forceinline__ double left_vector(const double* face, int s, double (&l)[NV]) {
  using R = NlRow<NV>;
  constexpr int D = NV - 2;
  auto row = [&](int r) -> double { return face[r * TH]; };
  if (s == 0 || s == NV - 1) {
    const double ci = (s == 0) ? 0.5 * row(R::ci) : -0.5 * row(R::ci), b1 = 0.5 * row(R::b1), un = row(R::u);
    l[0] = fma(un, ci, 0.5 * row(R::b2));
    l[1] = -fma(b1, un, ci);
#pragma unroll
    for (int d = 1; d < D; ++d) l[1 + d] = -b1 * row(R::u + d);
    l[NV - 1] = b1;
  } else if (s == 1) {
    const double b1 = row(R::b1);
    l[0] = 1.0 - row(R::b2);
#pragma unroll
    for (int d = 0; d < D; ++d) l[1 + d] = b1 * row(R::u + d);
    l[NV - 1] = -b1;
  } else {
    l[0] = -row(R::u + (s - 1));
#pragma unroll
    for (int v = 1; v < NV; ++v) l[v] = 0.0;
  }
  return 0.5 * row(s == 0 ? R::am : (s == NV - 1 ? R::ap : R::a0));
}

/* Both split sides of a field from its W and G/2 in FP64, through one copy of the decisions and the
   reconstruction: f+ on g+_q = G_q/2 + (alpha/2) W_q, f- on g-_q = G_q/2 - (alpha/2) W_q mirrored
   about x_{i+1/2}; adds f+ + f- to fsum.  REC: op, om receive the frozen linear weights. */
template <int K, int LIM, bool REC>
__device__ __forceinline__ void general_sides(const double (&w)[K], const double (&hg)[K], double ha, const SchemeDev& S,
                                              unsigned& fl, double& fsum, double* op, double* om, int& st) {
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    double v[K];
#pragma unroll
    for (int q = 0; q < K; ++q) v[q] = side ? fma(-ha, w[K - 1 - q], hg[K - 1 - q]) : fma(ha, w[q], hg[q]);
    unsigned b = 0;
    int e = 7;
    if (!teno_decide_fast<K>(v, S, b, e)) teno_decide_fp64<K>(v, S, b, e, st);
    if constexpr (REC) {
      double wt[K];
      fsum += teno_general<K, LIM, true>(v, S, b, wt);
#pragma unroll
      for (int q = 0; q < K; ++q) {
        if (side) om[q] = wt[q];
        else op[q] = wt[q];
      }
    } else {
      fsum += teno_general<K, LIM>(v, S, b);
    }
    fl |= (b | ((unsigned)((e - 7) & 3) << 6)) << (8 * side);
  }
}

template <int NV>
__host__ __device__ constexpr unsigned allshear() { return ((1u << (NV - 1)) - 1u) & ~3u; }

/* Face flux from the central one, F = Fc on entry (components in the axis's frame): Fc + sum_s r_s
   correction_s; when an acoustic or entropy field is direct (dir), sum_s r_s fs with fs = l_s . Fc (+
   correction) for the others.  Where only shear fields are direct their component alone is, F_t = f_t +
   u_t F_rho: l_s . Fc of the other fields, of size M^2 at Mach M, would not cancel against their
   corrections to the rounding of the internal energy.  cm: central fields.  Both sums go through the vectors the eigenvectors share: a =
   (b2, -b1 u, b1) and b = (u_n, -e_n, 0)/c give l_{u-c} = (a + b)/2, l_{u+c} = (a - b)/2,
   l_entropy = e_0 - a, l_shear = e_t - u_t e_0, and with sigma = f_{u-c} + f_{u+c}, delta =
   (f_{u+c} - f_{u-c}) c:  F_0 = sigma + f_1,  F_d = (sigma + f_1) u_d + (delta if d = n, else
   f_shear(d)),  F_E = sigma H + delta u_n + f_1 |u|^2/2 + sum_t f_t u_t. */
template <int NV, int TH>
__device__ __forceinline__ void compose(const double* face, const double* fsv, unsigned cm, unsigned dir,
                                        double (&F)[NV]) {
  using R = NlRow<NV>;
  constexpr int D = NV - 2;
  auto row = [&](int r) -> double { return face[r * TH]; };
  double ut[D], fs[NV], q2 = 0.0;
#pragma unroll
  for (int s = 0; s < NV; ++s) fs[s] = (cm >> s & 1u) ? 0.0 : fsv[s * TH];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    ut[d] = row(R::u + d);
    q2 = fma(ut[d], ut[d], q2);
  }
  const unsigned sh = allshear<NV>();
  double raw[NV > 3 ? NV - 3 : 1];  /* f+ + f- of the direct shear fields */
  if (!(dir & ~sh)) {
#pragma unroll
    for (int s = 2; s <= NV - 2; ++s) {
      raw[s - 2] = fs[s];
      if (dir >> s & 1u) fs[s] -= fma(-ut[s - 1], F[0], F[s]);
    }
  } else {
    double uF = 0.0;
#pragma unroll
    for (int d = 0; d < D; ++d) uF = fma(ut[d], F[1 + d], uF);
    const double a = fma(row(R::b2), F[0], row(R::b1) * (F[NV - 1] - uF));
    const double b = row(R::ci) * fma(ut[0], F[0], -F[1]);
    if (!(dir & 1u)) fs[0] += 0.5 * (a + b);
    if (!(dir >> (NV - 1) & 1u)) fs[NV - 1] += 0.5 * (a - b);
    if (!(dir >> 1 & 1u)) fs[1] += F[0] - a;
#pragma unroll
    for (int s = 2; s <= NV - 2; ++s)
      if (!(dir >> s & 1u)) fs[s] += fma(-ut[s - 1], F[0], F[s]);
#pragma unroll
    for (int v = 0; v < NV; ++v) F[v] = 0.0;
  }
  const double sigma = fs[0] + fs[NV - 1];
  const double delta = (fs[NV - 1] - fs[0]) * row(R::ct);
  const double m = sigma + fs[1];
  double FE = fma(sigma, row(R::H), fma(delta, ut[0], 0.5 * q2 * fs[1]));
  F[0] += m;
  F[1] += fma(m, ut[0], delta);
#pragma unroll
  for (int s = 2; s <= NV - 2; ++s) {
    F[s] = (!(dir & ~sh) && (dir >> s & 1u)) ? fma(ut[s - 1], F[0], raw[s - 2]) : F[s] + fma(m, ut[s - 1], fs[s]);
    FE = fma(ut[s - 1], fs[s], FE);
  }
  F[NV - 1] += FE;
}

/* The rare FP64 paths of the fixed-point kernel, called rather than inlined: they are larger
   than the path every item takes, and instruction fetch is what that path waits for.  w, g: the
   item's W and G of point q at q * NL_THREADS; side 1: the mirrored stencil of f-.  The item keeps
   twice the split sequences (G +- alpha W), which saves a product per point (256^3 TENO8: FP64
   pipe 74 % busy); halving is exact. */
template <int K>
__device__ __forceinline__ void split_side(const double* w, const double* g, double al, int side, double (&v)[K]) {
#pragma unroll
  for (int q = 0; q < K; ++q) {
    const int p = (side ? K - 1 - q : q) * NL_THREADS;
    v[q] = 0.5 * fma(side ? -al : al, w[p], g[p]);
  }
}
template <int K>
__device__ __noinline__ unsigned decide_cold(const double* w, const double* g, double al, int side, const SchemeDev& S,
                                             int& st) {
  double v[K];
  split_side<K>(w, g, al, side, v);
  unsigned b;
  int e;
  teno_decide_fp64<K>(v, S, b, e, st);
  return b | ((unsigned)((e - 7) & 3) << 6);
}
/* f+ + f- with the decisions fl taken: a shear item that turned out to reach across a jump */
template <int K, int LIM>
__device__ __noinline__ double general_cold(const double* w, const double* g, double al, unsigned fl, const SchemeDev& S) {
  constexpr unsigned allk = (1u << (K - 2)) - 1u;
  double f = 0.0;
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    double v[K];
    split_side<K>(w, g, al, side, v);
    f += teno_general<K, LIM>(v, S, fl >> (8 * side) & allk);
  }
  return f;
}
/* an item that takes the FP64 form from the start (a jump face's, or outside the fixed-point range):
   decisions and reconstruction of both sides from the FP64 sequence; returns f+ + f- */
template <int K, int LIM>
__device__ __noinline__ double direct_cold(const double* w, const double* g, double al, const SchemeDev& S, unsigned& fl,
                                           int& st) {
  double f = 0.0;
  unsigned bits = 0u;
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    double v[K];
    split_side<K>(w, g, al, side, v);
    unsigned b = 0u;
    int e = 7;
    if (!teno_decide_fast<K>(v, S, b, e)) teno_decide_fp64<K>(v, S, b, e, st);
    f += teno_general<K, LIM>(v, S, b);
    bits |= (b | ((unsigned)((e - 7) & 3) << 6)) << (8 * side);
  }
  fl = bits;
  return f;
}

/* A field's rows of the tape at o (and at oc, unless null), stride nface: fs, omegaW = sum_q delta_q W_q,
   sigma_q, delta_q with fs = sum_q sigma_q G_q + (alpha/2) delta_q W_q, sigma_q = (op_q +
   om_{K-1-q})/2, delta_q = op_q - om_{K-1-q} (op, om: the frozen linear weights of f+ and f-) */
template <int K, class Wq>
__device__ __forceinline__ void put_tape(const Wq& w, const double* op, const double* om, double fs, bool central,
                                         double* o, double* oc, long long nface) {
  double wW = 0.0;
#pragma unroll
  for (int q = 0; q < K; ++q) wW = fma(op[q] - om[K - 1 - q], w(q), wW);
  for (double* p = o; p; p = p == o ? oc : nullptr) {
    p[0] = fs;
    p[nface] = central ? __longlong_as_double((long long)kCentralMark) : wW + 0.0;
#pragma unroll
    for (int q = 0; q < K; ++q) {
      p[(2 + q) * nface] = 0.5 * (op[q] + om[K - 1 - q]);
      p[(2 + K + q) * nface] = op[q] - om[K - 1 - q];
    }
  }
}
/* The tape of a fixed-point item (a record launch of the 512^2 rollout: 600 us, 470 with FP64 items
   alone, 245 without a tape).  The face flux comes from the same fixed-point form as the forward
   kernel's, so that a recorded step has its bits (a rollout is recomputed from its checkpoints for the
   reverse, and branches frozen on states that differ in the last bits are another trajectory's);
   only the frozen weights are formed in FP64. */
template <int K, int LIM>
__device__ __noinline__ void record_item(const double* w, const double* g, double al, unsigned fl, const SchemeDev& S,
                                         double* o, double* oc, long long nface, bool central) {
  constexpr unsigned allk = (1u << (K - 2)) - 1u;
  double op[K], om[K], f = 0.0;
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    double v[K], wt[K];
    split_side<K>(w, g, al, side, v);
    f += teno_general<K, LIM, true>(v, S, fl >> (8 * side) & allk, wt);
#pragma unroll
    for (int q = 0; q < K; ++q) {
      if (side) om[q] = wt[q];
      else op[q] = wt[q];
    }
  }
  put_tape<K>([&](int q) { return w[q * NL_THREADS]; }, op, om, f, central, o, oc, nface);
}

/* FP32 value of a double from its high word (20 mantissa bits; below the FP32 range 0, above it inf) */
__device__ __forceinline__ float f32_hi(const double* x) {
  const int h = __ldg(reinterpret_cast<const int*>(x) + 1), m = (h & 0x7fffffff) - 0x38000000;
  const int f = m < 0x100000 ? 0 : (m >= 0x0ff00000 ? 0x7f800000 : m << 3);
  return __int_as_float(f | (h & (int)0x80000000));
}

/* Whether the stencil reaches across a jump: a point's density, or its size in the face's frame p +
   (gamma - 1)/2 rho w^2 (w = v - v~; what the acoustic and entropy fields are made of), is more than
   `most` times the larger of the face's two cells.  Up to there the limiters are applied as
   corrections to Fc.  Fc and the corrections carry the rounding of the stencil's largest values, the
   FP64 reconstruction that of the values it keeps, so the correction form is the more exact one where
   the values are of one size and loses with the ratio where they are not: rms errors of the face
   flux against 80-bit, in units of 2^-53 of the cells' |lambda U|, FP64 form | correction (2D, jumps
   of rho and p every 7 cells, TENO6): MP ratio 1 0.71 | 0.50, 2 0.71 | 0.69, 4 0.75 | 1.08, 10 0.73 | 2.4,
   1000 0.76 | 57; TVD5 ratio 1 0.58 | 0.24, 4 0.71 | 0.65 (jumps of p), 10 0.88 | 1.8.  It holds for the
   face, not for a field: beside a field in FP64 another one's l_s . Fc would bring the far values
   back.  What it costs: 2048^2 TENO6-MP, whose discs jump by 2-10, 5.0 -> 5.3 ms a step, TENO8-TVD5 5.6
   -> 5.8; 256^3 nothing.  (A NaN reaches.) */
template <int NV, int K, int LIM, int TH>
__device__ __forceinline__ bool reaches_jump(const GridFace<NV, K>& src, const double* p, const double* row, double gm1) {
  constexpr int D = NV - 2, H = K / 2;
  const float most = LIM == LIM_TVD5 ? 2.8f : 2.f, hg = 0.5f * f32_rz(gm1);
  float ut[D], far[2] = {0.f, 0.f}, near[2] = {0.f, 0.f};
#pragma unroll
  for (int d = 0; d < D; ++d) ut[d] = f32_rz(row[(NlRow<NV>::u + d) * TH]);
  bool nan = false;
#pragma unroll 1
  for (int q = 0; q < K; ++q) {
    const long long x = src.cell(q);
    const float rho = f32_hi(src.rho + x);
    float w2 = 0.f;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const float w = f32_hi(src.vel[d] + x) - ut[d];
      w2 = fmaf(w, w, w2);
    }
    const float s = fmaf(hg * rho, w2, f32_hi(p + x));
    nan |= !(s <= 3e38f);
    far[0] = fmaxf(far[0], rho);
    far[1] = fmaxf(far[1], s);
    if (q == H - 1 || q == H) {
      near[0] = fmaxf(near[0], rho);
      near[1] = fmaxf(near[1], s);
    }
  }
  return nan || !(far[0] <= most * near[0] && far[1] <= most * near[1]);
}

/* The same for a shear field's own terms |u_t rho|, |m_t|, which vanish where the tangential velocity
   does, as a difference of high words: up to 16 the error of the tangential flux stays at that of the
   acoustic fields' part (0.58 | 0.65 at a ratio of 10; 0.77 | 13 at 100 without the rule). */
constexpr unsigned kShearJump = 4u << 20;
constexpr unsigned kJumpFace = 1u << 31;  /* s_dir: no field of the face takes the correction form */
__device__ __forceinline__ unsigned abs_hi(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

/* Both split sides of an item from its projected W and G (columns w, g in shared memory):
   decisions, and the corrections of the nonsmooth sides in fixed point.  Returns false when the
   FP32 filter leaves a side undecided and `defer` is set.  Dx: K - 1 scratch words of the item's
   thread.  em: biased exponent of a power of two above every |G| + |alpha W|.  fp64: the item's
   face takes the FP64 form (reaches_jump); jump: the shear item's corrections would cancel values far
   above the centre's (kShearJump).  The loops over
   the points are rolled and everything rare is called, to keep the code that an item runs
   small (unrolled 4 or 8 times: 256^3 step 64 ms against 59, 64^3 turbulence 5.6 against 5.1). */
template <int K, int LIM>
__device__ __forceinline__ bool fixed_item(const double* w, const double* g, double al, int em, bool fp64, bool jump,
                                           long long* Dx, const SchemeDev& S, bool defer, unsigned& fl, double& fsum,
                                           bool& direct, int& st) {
  constexpr int TH = NL_THREADS;
  constexpr unsigned allk = (1u << (K - 2)) - 1u;
  direct = fp64 || em < 1024 - 40 || em > 1024 + 40;  /* FP64, and at once (no pass can do better) */
  if (direct) {
    fsum = direct_cold<K, LIM>(w, g, al, S, fl, st);
    return true;
  }
  fl = 0u;
  const float unit = __int_as_float((em - 1077 + 127) << 23);  /* 2^(em - 1077): of the halved values */
  Acc96 acc;
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    unsigned zero = 0u, b = 0u;
    int e = 7;
    auto cold = [&]() {
      const unsigned f = decide_cold<K>(w, g, al, side, S, st);
      b = f & allk;
      e = 7 + (int)(f >> 6);
    };
    if (S.exact_decisions) {  /* decided first: a smooth side needs no differences */
      cold();
      if (b == allk) {
        fl |= (b | ((unsigned)((e - 7) & 3) << 6)) << (8 * side);
        continue;
      }
    }
    {
      const int p0 = side ? (K - 1) * TH : 0, dp = side ? -TH : TH;
      const double hs = side ? -al : al;
      double v0 = fma(hs, w[p0], g[p0]);
      long long x0 = to_fixed(v0, em);
#pragma unroll 1
      for (int t = 0; t < K - 1; ++t) {
        const int p = p0 + (t + 1) * dp;
        const double v1 = fma(hs, w[p], g[p]);
        const long long x1 = to_fixed(v1, em);
        Dx[t * TH] = x1 - x0;
        zero |= dbits(v1) == dbits(v0) ? 1u << t : 0u;
        x0 = x1;
        v0 = v1;
      }
    }
    if (!S.exact_decisions) {
      float d[K - 1];
#pragma unroll
      for (int t = 0; t < K - 1; ++t) d[t] = __ll2float_rz(Dx[t * TH]) * unit;
      if (!cutoff_filter<K>(d, 1.01f * unit, zero, S, b, e)) {
        if (defer) return false;
        cold();
      }
    }
    fl |= (b | ((unsigned)((e - 7) & 3) << 6)) << (8 * side);
    if (b != allk) {
      if (jump) {
        direct = true;
      } else {
        long long D[K - 1];
#pragma unroll
        for (int t = 0; t < K - 1; ++t) D[t] = Dx[t * TH];
        fixed_correction<K, LIM>(D, b, S, acc);
      }
    }
  }
  fsum = direct ? general_cold<K, LIM>(w, g, al, fl, S)
                : acc.value() * (__hiloint2double((em - 1077 + 1023) << 20, 0) * (1.0 / fixed_den<K, LIM>()));
  return true;
}

template <int NV, int K, int LIM, bool REC, bool FIX>
__global__ void __launch_bounds__(NL_THREADS, NL_CTAS_PER_SM) nonlinear_kernel(const NonlinArgs A) {
  using R = NlRow<NV>;
  constexpr int D = NV - 2, H = K / 2, TH = NL_THREADS, W = TH / 32;
  constexpr unsigned allk = (1u << (K - 2)) - 1u, allf = (1u << NV) - 1u;
  __shared__ double s_row[R::N * TH];
  __shared__ double s_fs[NV * TH];
  __shared__ long long s_base[TH];
  __shared__ int s_f[TH];
  __shared__ unsigned s_cm[TH];             /* certified and found-central fields */
  __shared__ unsigned s_dir[TH];            /* fields whose s_fs is f+ + f- (else the correction to l_s . Fc) */
  __shared__ unsigned short s_item[NV * TH];
  __shared__ unsigned short s_later[FIX ? NV * TH : 1];
  __shared__ double s_w[FIX ? K * TH : 1], s_g[FIX ? K * TH : 1];  /* an item's W and G */
  __shared__ long long s_D[FIX ? (K - 1) * TH : 1];
  __shared__ int s_nlater;
  constexpr int NS = FIX ? 2 * NV : NV;  /* the item order's sorts: field, and jump faces last */
  __shared__ int s_wc[NS * W + 1];
  const int tid = threadIdx.x, wid = tid >> 5, ln = tid & 31;
  int st = 0;

  long long cnt[3] = {0, 0, 0}, total = 0;
  for (int a = 0; a < A.dim; ++a) {
    const long long c = A.count[a];
    cnt[a] = c < A.nface[a] ? c : A.nface[a];
    total += cnt[a];
  }
  /* faces per chunk: NL_THREADS, or fewer (8 at least) when that leaves CTAs without one */
  int sh = 7;
  while (sh > 3 && (total >> sh) < gridDim.x) --sh;
  const long long chunk = 1ll << sh;
  const long long nch0 = (cnt[0] + chunk - 1) >> sh, nch1 = (cnt[1] + chunk - 1) >> sh, nch2 = (cnt[2] + chunk - 1) >> sh;

#pragma unroll 1
  for (long long ch = blockIdx.x; ch < nch0 + nch1 + nch2; ch += gridDim.x) {
    const int ax = ch < nch0 ? 0 : (ch < nch0 + nch1 ? 1 : 2);
    const long long i0 = (ch - (ax == 0 ? 0 : (ax == 1 ? nch0 : nch0 + nch1))) << sh;
    const int nf = (int)((cnt[ax] - i0) < chunk ? (cnt[ax] - i0) : chunk);  /* faces of this chunk */
    const int na = A.n[ax], bc = A.bc[ax];
    const long long sa = ax == 0 ? 1 : (ax == 1 ? (long long)A.n[0] : (long long)A.n[0] * A.n[1]);
    const long long nface = A.nface[ax];
    /* global component of component v in the axis's frame */
    auto gc = [&](int v) -> int {
      if (v == 0 || v == NV - 1) return v;
      if (v == 1) return 1 + ax;
      const int t = v - 2;
      return 1 + (t < ax ? t : t + 1);
    };
    const double* up[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) up[v] = A.U + gc(v) * A.ncell;
    const double* const Pn = A.P + ax * A.ncell;  /* normal velocity, pressure, sound speed */
    const double* const Pp = A.P + D * A.ncell;
    const double* const Pc = A.P + (D + 1) * A.ncell;

    /* ---- (0) Roe state and LLF speeds, one thread per face ---- */
    unsigned mask = 0u;
    bool jump_face = false;
    long long flin = 0, fcopy = -1;  /* face n of a periodic line is face 0's copy */
    if (tid < nf) {
      const unsigned idx = A.list[ax][i0 + tid];
      mask = A.mask[ax][i0 + tid];
      flin = idx;
      int f;
      long long base;
      if (ax == 0) {
        const unsigned line = idx / (unsigned)(na + 1);
        f = (int)(idx - line * (unsigned)(na + 1));
        base = (long long)line * A.n[0];
      } else {
        const unsigned r = idx / (unsigned)A.n[0], x = idx - r * (unsigned)A.n[0];
        const unsigned m = ax == 1 ? (unsigned)(na + 1) : (unsigned)A.n[1];
        const unsigned hi = r / m, lo = r - hi * m;
        f = (int)(ax == 1 ? lo : hi);
        base = (long long)x + (ax == 1 ? (long long)A.n[0] * A.n[1] * hi : (long long)A.n[0] * lo);
      }
      if (bc == 0 && f == 0) fcopy = flin + na * (ax == 0 ? 1ll : (ax == 1 ? (long long)A.n[0] : sa));
      GridFace<NV, K> src;
      src.rho = up[0];
#pragma unroll
      for (int d = 0; d < D; ++d) src.vel[d] = A.P + (gc(1 + d) - 1) * A.ncell;
      src.un = Pn;
      src.c = Pc;
      src.base = base;
      src.sa = sa;
      src.f = f;
      src.na = na;
      src.bc = bc;
      face_rows<NV, K, TH>(src, s_row + tid, A.gamma - 1.0, A.rgm1, st);
      s_base[tid] = base;
      s_f[tid] = f;
      s_cm[tid] = A.sch.default_d ? (allf & ~mask) : 0u;
      jump_face = FIX && reaches_jump<NV, K, LIM, TH>(src, Pp, s_row + tid, A.gamma - 1.0);
      s_dir[tid] = jump_face ? kJumpFace : 0u;
    }
    /* the chunk's (face, field) items, field after field; those of jump faces, which take the FP64
       form, after the others, in warps of their own */
    auto has_item = [&](int e) -> bool { return (mask >> (e % NV) & 1u) && (!FIX || jump_face == (e >= NV)); };
#pragma unroll
    for (int e = 0; e < NS; ++e) {
      const unsigned b = __ballot_sync(0xffffffffu, has_item(e));
      if (ln == 0) s_wc[e * W + wid] = __popc(b);
    }
    __syncthreads();
    if (wid == 0) {  /* exclusive scan of the NS * W counts, two a lane */
      static_assert(NS * W <= 64, "one warp scans the counts");
      const int c0 = 2 * ln < NS * W ? s_wc[2 * ln] : 0, c1 = 2 * ln + 1 < NS * W ? s_wc[2 * ln + 1] : 0;
      int x = c0 + c1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (ln >= o) x += y;
      }
      if (2 * ln < NS * W) s_wc[2 * ln] = x - c0 - c1;
      if (2 * ln + 1 < NS * W) s_wc[2 * ln + 1] = x - c1;
      if (ln == 31) s_wc[NS * W] = x;
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < NS; ++e) {
      const unsigned b = __ballot_sync(0xffffffffu, has_item(e));
      if (has_item(e)) s_item[s_wc[e * W + wid] + __popc(b & ((1u << ln) - 1u))] = (unsigned short)(tid | ((e % NV) << 8));
    }
    const int nitem = s_wc[NS * W];
    if (tid == 0) s_nlater = 0;
    __syncthreads();

    /* ---- (1) one (face, field) per thread; FIX: what the FP32 filter leaves undecided comes
       again in a second pass, in warps of its own ---- */
#pragma unroll 1
    for (int pass = 0; pass < (FIX ? 2 : 1); ++pass) {
    const int npass = pass ? s_nlater : nitem;
#pragma unroll 1
    for (int it = tid; it < npass; it += TH) {
      const unsigned item = pass ? s_later[it] : s_item[it];
      const int fc = item & 255, s = item >> 8;
      const bool shear = s >= 2 && s <= NV - 2;
      double l[NV];
      const double ha = left_vector<NV, TH>(s_row + fc, s, l);
      const double* const ut = A.U + gc(shear ? s : 1) * A.ncell;
      const long long base = s_base[fc];
      const int f = s_f[fc];
      /* W and G/2 (FIX: G) of stencil point q, G = l . F = u_n W + p (l_n + u_n l_E); term: the larger
         of a shear field's |l_0 rho|, |m_t|, as the sum of the factors' high words (FIX only) */
      auto project = [&](int q, double& w, double& hg, unsigned& term) {
        const long long cell = base + sa * bc_near(f - H + q, na, bc);
        const double un = __ldg(Pn + cell);
        if (shear) {
          const double rho = __ldg(up[0] + cell), m = __ldg(ut + cell);
          w = fma(l[0], rho, m);
          hg = un * w;
          if constexpr (FIX) term = max(abs_hi(l[0]) + abs_hi(rho), 0x3ff00000u + abs_hi(m));
        } else {
          w = l[0] * __ldg(up[0] + cell);
#pragma unroll
          for (int v = 1; v < NV; ++v) w = fma(l[v], __ldg(up[v] + cell), w);
          hg = fma(__ldg(Pp + cell), fma(un, l[NV - 1], l[1]), un * w);
        }
        if constexpr (!FIX) hg *= 0.5;
      };
      unsigned fl = 0u;
      double fsum = 0.0;
      bool direct = !FIX;
      constexpr int KR = REC && !FIX ? K : 1;
      double wv[KR], op[KR], om[KR];  /* W; frozen linear weights of f+ and f- */
      if constexpr (FIX) {
        int eg = 0, ew = 0;
        unsigned far = 0u, near = 0u;
#pragma unroll 1
        for (int q = 0; q < K; ++q) {
          double w, hg;
          unsigned term = 0u;
          project(q, w, hg, term);
          far = max(far, term);
          if (q == H - 1 || q == H) near = max(near, term);
          s_w[q * TH + tid] = w;
          s_g[q * TH + tid] = hg;
          eg = max(eg, (int)((unsigned)__double2hiint(hg) >> 20 & 0x7ffu));
          ew = max(ew, (int)((unsigned)__double2hiint(w) >> 20 & 0x7ffu));
        }
        /* 2 |v| <= |G| + |alpha W| < 2^(em - 1022) */
        const double al = ha + ha;
        const int em = 1 + max(eg, ew + (int)((unsigned)__double2hiint(al) >> 20 & 0x7ffu) - 1022);
        if (!fixed_item<K, LIM>(s_w + tid, s_g + tid, al, em, (s_dir[fc] & kJumpFace) != 0u, far - near > kShearJump,
                                s_D + tid, A.sch, pass == 0 && nitem > TH, fl, fsum, direct, st)) {
          s_later[atomicAdd(&s_nlater, 1)] = (unsigned short)item;
          continue;
        }
      } else {
        double w[K], hg[K];
        unsigned term = 0u;
#pragma unroll
        for (int q = 0; q < K; ++q) {
          project(q, w[q], hg[q], term);
          if constexpr (REC) wv[q] = w[q];
        }
        general_sides<K, LIM, REC>(w, hg, ha, A.sch, fl, fsum, op, om, st);
      }
      s_fs[s * TH + fc] = fsum;
      /* a field found all smooth on both sides is central after all: the flux does not depend on
         which test decided */
      if ((fl & (allk | allk << 8)) == (allk | allk << 8) && A.sch.default_d) atomicOr(&s_cm[fc], 1u << s);
      else if (direct) atomicOr(&s_dir[fc], 1u << s);
      const bool copy = bc == 0 && f == 0;
      const long long fi = A.list[ax][i0 + fc];
      const long long fcp = fi + na * (ax == 0 ? 1ll : (ax == 1 ? (long long)A.n[0] : sa));
      if (A.flags[ax]) {
        for (int r = 0; r < (copy ? 2 : 1); ++r) {
          uint8_t* o = A.flags[ax] + ((r ? fcp : fi) * NV + s) * 2;
          o[0] = (uint8_t)(fl & 0xffu);
          o[1] = (uint8_t)(fl >> 8);
        }
      }
      if constexpr (REC) {
        double* const o = A.lin[ax] + fi + (long long)s * (2 * K + 2) * nface;
        double* const oc = copy ? A.lin[ax] + fcp + (long long)s * (2 * K + 2) * nface : nullptr;
        const bool central = (fl & (allk | allk << 8)) == (allk | allk << 8) && A.sch.default_d;
        if constexpr (FIX) record_item<K, LIM>(s_w + tid, s_g + tid, ha + ha, fl, A.sch, o, oc, nface, central);
        else put_tape<K>([&](int q) { return wv[q]; }, op, om, fsum, central, o, oc, nface);
      }
    }
    __syncthreads();
    }

    /* ---- (2) the face fluxes ---- */
    if (tid < nf && s_cm[tid] != allf) {
      const unsigned cm = s_cm[tid], dir = s_dir[tid] & allf;
      double* const Fo = A.Fhat[ax];
      double Fh[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) Fh[v] = Fo[gc(v) * nface + flin];
      compose<NV, TH>(s_row + tid, s_fs + tid, cm, dir, Fh);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        Fo[gc(v) * nface + flin] = Fh[v];
        if (fcopy >= 0) Fo[gc(v) * nface + fcopy] = Fh[v];
      }
    }
    __syncthreads();  /* the rows are free for the next chunk */
  }
  if (st) atomicOr(A.status, st);
}

}  // namespace tenom
