/* Face sweep, second half: the faces screen_kernel could not certify, in FP64 (Section 4 of
 * arXiv 2010.13289: Roe-averaged characteristic decomposition, local Lax-Friedrichs
 * splitting, TENO-M per characteristic field and split side, back-projection).
 *
 * One persistent launch works through the lists of every axis.  A CTA takes a chunk of up to
 * NL_THREADS faces of one axis: (0) a thread per face forms the Roe state and the LLF
 * speeds; (1) the uncertified (face, field) pairs of the chunk, ordered by field so that a
 * warp mostly runs one kind of projection, are spread over the CTA's threads: projection of
 * the K points, decisions and reconstruction of both split sides; (2) a thread per face
 * composes the flux from those fields and from l_s . Fc of the certified ones.  The list is
 * dense, so every step runs in full warps whatever share of the faces needs it; when there
 * are few faces a chunk is smaller, so that they spread over all SMs.
 *
 * The kernel is written in the axis's own frame: component 1 is the momentum along the axis,
 * 2 .. NV-2 the tangential ones in increasing axis order (fields: 0 u-c, 1 entropy,
 * 2 .. NV-2 shear, NV-1 u+c). */
#pragma once
#include "tenom_recon.cuh"
#include "tenom_face.cuh"

namespace tenom {

struct NonlinArgs {
  const double* U;           /* [NV][ncell] */
  const double* P;           /* cell primitives (velocity, p, c, ..), or null: formed here */
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

template <int NV, int K, int LIM, bool REC>
__global__ void __launch_bounds__(NL_THREADS, NL_CTAS_PER_SM) nonlinear_kernel(const NonlinArgs A) {
  using R = NlRow<NV>;
  constexpr int D = NV - 2, H = K / 2, TH = NL_THREADS, W = TH / 32;
  constexpr unsigned allk = (1u << (K - 2)) - 1u, allf = (1u << NV) - 1u;
  __shared__ double s_row[R::N * TH];
  __shared__ double s_fs[NV * TH];
  __shared__ long long s_base[TH];
  __shared__ int s_f[TH];
  __shared__ unsigned s_cm[TH];             /* certified and found-central fields */
  __shared__ unsigned short s_item[NV * TH];
  __shared__ int s_wc[NV * W + 1];
  const int tid = threadIdx.x, wid = tid >> 5, ln = tid & 31;
  int st = 0;

  long long cnt[3] = {0, 0, 0}, total = 0;
  for (int a = 0; a < A.dim; ++a) {
    const long long c = A.count[a];
    cnt[a] = c < A.nface[a] ? c : A.nface[a];
    total += cnt[a];
  }
  long long chunk = (total + gridDim.x - 1) / gridDim.x;
  chunk = chunk < 8 ? 8 : (chunk > TH ? TH : chunk);
  const long long nch0 = (cnt[0] + chunk - 1) / chunk, nch1 = (cnt[1] + chunk - 1) / chunk,
                  nch2 = (cnt[2] + chunk - 1) / chunk;

#pragma unroll 1
  for (long long ch = blockIdx.x; ch < nch0 + nch1 + nch2; ch += gridDim.x) {
    const int ax = ch < nch0 ? 0 : (ch < nch0 + nch1 ? 1 : 2);
    const long long i0 = (ch - (ax == 0 ? 0 : (ax == 1 ? nch0 : nch0 + nch1))) * chunk;
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
    const double* const Pn = A.P ? A.P + ax * A.ncell : nullptr;
    const double* const Pp = A.P ? A.P + D * A.ncell : nullptr;
    const double* const Pc = A.P ? A.P + (D + 1) * A.ncell : nullptr;
    /* normal velocity and pressure of a cell */
    auto normal = [&](long long cell, const double (&u)[NV], double& un, double& p) {
      if (A.P) {
        un = __ldg(Pn + cell);
        p = __ldg(Pp + cell);
      } else {
        const double rinv = rcp_nr(u[0]);
        double ke = 0.0;
#pragma unroll
        for (int d = 1; d <= D; ++d) ke += u[d] * (u[d] * rinv);
        un = u[1] * rinv;
        p = (A.gamma - 1.0) * (u[NV - 1] - 0.5 * ke);
      }
    };

    /* ---- (0) Roe state and LLF speeds, one thread per face ---- */
    unsigned mask = 0u;
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
      double sr[2], Hh[2], v[2][D];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const long long cell = base + sa * bc_wrap(f - 1 + e, na, bc);
        double u[NV], un, p;
#pragma unroll
        for (int q = 0; q < NV; ++q) u[q] = __ldg(up[q] + cell);
        normal(cell, u, un, p);
        const double rinv = rcp_nr(u[0]);
        Hh[e] = (u[NV - 1] + p) * rinv;
        sr[e] = u[0] * rsqrt_nr(u[0]);
        v[e][0] = un;
#pragma unroll
        for (int d = 1; d < D; ++d) v[e][d] = u[1 + d] * rinv;
      }
      const double wsum = rcp_nr(sr[0] + sr[1]);
      double q2 = 0.0;
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const double x = (sr[0] * v[0][d] + sr[1] * v[1][d]) * wsum;
        q2 += x * x;
        s_row[(R::u + d) * TH + tid] = x;
      }
      const double Ht = (sr[0] * Hh[0] + sr[1] * Hh[1]) * wsum;
      const double c2 = (A.gamma - 1.0) * (Ht - 0.5 * q2);
      if (!ipos(c2)) st |= ST_ROE;
      const double ci = rsqrt_nr(c2);
      const double b1 = (A.gamma - 1.0) * (ci * ci);
      s_row[R::H * TH + tid] = Ht;
      s_row[R::ci * TH + tid] = ci;
      s_row[R::ct * TH + tid] = c2 * ci;
      s_row[R::b1 * TH + tid] = b1;
      s_row[R::b2 * TH + tid] = 0.5 * q2 * b1;
      /* LLF: alpha_s = max over the K stencil points of |lambda_s|, one per eigenvalue family */
      double am = 0.0, a0 = 0.0, ap = 0.0;
#pragma unroll
      for (int q = 0; q < K; ++q) {
        const long long cell = base + sa * bc_wrap(f - H + q, na, bc);
        double un, cs;
        if (A.P) {
          un = __ldg(Pn + cell);
          cs = __ldg(Pc + cell);
        } else {
          double u[NV], vel[D], p;
          int s2 = 0;
#pragma unroll
          for (int w = 0; w < NV; ++w) u[w] = __ldg(up[w] + cell);
          point_prims<NV>(u, A.gamma, vel, p, cs, s2);
          un = vel[0];
        }
        am = imax_nonneg(am, iabs(un - cs));
        a0 = imax_nonneg(a0, iabs(un));
        ap = imax_nonneg(ap, iabs(un + cs));
      }
      s_row[R::am * TH + tid] = am;
      s_row[R::a0 * TH + tid] = a0;
      s_row[R::ap * TH + tid] = ap;
      s_base[tid] = base;
      s_f[tid] = f;
      s_cm[tid] = A.sch.default_d ? (allf & ~mask) : 0u;
    }
    /* the chunk's (face, field) items, field after field */
#pragma unroll
    for (int s = 0; s < NV; ++s) {
      const unsigned b = __ballot_sync(0xffffffffu, mask >> s & 1u);
      if (ln == 0) s_wc[s * W + wid] = __popc(b);
    }
    __syncthreads();
    if (wid == 0) {  /* exclusive scan of the NV * W counts */
      static_assert(NV * W <= 32, "one warp scans the counts");
      const int c = ln < NV * W ? s_wc[ln] : 0;
      int x = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (ln >= o) x += y;
      }
      if (ln < NV * W) s_wc[ln] = x - c;
      if (ln == 31) s_wc[NV * W] = x;
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < NV; ++s) {
      const unsigned b = __ballot_sync(0xffffffffu, mask >> s & 1u);
      if (mask >> s & 1u) s_item[s_wc[s * W + wid] + __popc(b & ((1u << ln) - 1u))] = (unsigned short)(tid | (s << 8));
    }
    const int nitem = s_wc[NV * W];
    __syncthreads();

    /* ---- (1) one (face, field) per thread ---- */
#pragma unroll 1
    for (int it = tid; it < nitem; it += TH) {
      const int fc = s_item[it] & 255, s = s_item[it] >> 8;
      auto row = [&](int r) -> double { return s_row[r * TH + fc]; };
      const bool acoustic = s == 0 || s == NV - 1, shear = s >= 2 && s <= NV - 2;
      const double ha = 0.5 * row(s == 0 ? R::am : (s == NV - 1 ? R::ap : R::a0));
      /* left eigenvector l_s (closed form of R^{-1}); shear: l = e_t - u_t e_0 */
      double l[NV];
      if (acoustic) {
        const double sg = (s == 0) ? 1.0 : -1.0, ci = row(R::ci), b1 = row(R::b1), un = row(R::u);
        l[0] = 0.5 * (row(R::b2) + sg * un * ci);
        l[1] = 0.5 * (-b1 * un - sg * ci);
#pragma unroll
        for (int d = 1; d < D; ++d) l[1 + d] = -0.5 * b1 * row(R::u + d);
        l[NV - 1] = 0.5 * b1;
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
      const double* const ut = A.U + gc(shear ? s : 1) * A.ncell;
      const long long base = s_base[fc];
      const int f = s_f[fc];
      double wv[K], hgv[K];
#pragma unroll
      for (int q = 0; q < K; ++q) {
        const long long cell = base + sa * bc_wrap(f - H + q, na, bc);
        double un, pq, w, kap;
        if (A.P && shear) {
          un = __ldg(Pn + cell);
          w = fma(l[0], __ldg(up[0] + cell), __ldg(ut + cell));
          pq = 0.0;
          kap = 0.0;
        } else {
          double u[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) u[v] = __ldg(up[v] + cell);
          normal(cell, u, un, pq);
          if (shear) {
            w = fma(l[0], u[0], __ldg(ut + cell));
            kap = 0.0;
          } else {
            w = l[0] * u[0];
#pragma unroll
            for (int v = 1; v < NV; ++v) w = fma(l[v], u[v], w);
            kap = fma(un, l[NV - 1], l[1]);
          }
        }
        wv[q] = w;
        hgv[q] = 0.5 * fma(pq, kap, un * w);  /* G/2, G = l . F = u_n W + p (l_n + u_n l_E) */
      }
      /* the two split sides through one copy of the decisions and the reconstruction:
         f+ on g+_q = G_q/2 + (alpha/2) W_q, f- on g-_q = G_q/2 - (alpha/2) W_q mirrored about
         x_{i+1/2} */
      unsigned fl = 0u, sm2 = 0u;
      double fsum = 0.0;
      double op[REC ? K : 1], om[REC ? K : 1];  /* frozen linear weights of f+ and f- */
#pragma unroll 1
      for (int side = 0; side < 2; ++side) {
        double v[K];
#pragma unroll
        for (int q = 0; q < K; ++q) v[q] = side ? fma(-ha, wv[K - 1 - q], hgv[K - 1 - q]) : fma(ha, wv[q], hgv[q]);
        unsigned b = 0;
        int e = 7;
        if (!teno_decide_fast<K>(v, A.sch, b, e)) teno_decide_fp64<K>(v, A.sch, b, e, st);
        if constexpr (REC) {
          double wt[K];
          fsum += teno_general<K, LIM, true>(v, A.sch, b, wt);
#pragma unroll
          for (int q = 0; q < K; ++q) {
            if (side) om[q] = wt[q];
            else op[q] = wt[q];
          }
        } else {
          fsum += teno_general<K, LIM>(v, A.sch, b);
        }
        fl |= (b | ((unsigned)((e - 7) & 3) << 6)) << (8 * side);
        sm2 += (b == allk) ? 1u : 0u;
      }
      s_fs[s * TH + fc] = fsum;
      /* a field found all smooth on both sides is central after all: the flux does not depend on
         which test decided */
      if (sm2 == 2u && A.sch.default_d) atomicOr(&s_cm[fc], 1u << s);
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
        /* the tape's rows of this field: fs, omegaW = sum_q delta_q W_q, sigma_q, delta_q with
           fs = sum_q sigma_q G_q + (alpha/2) delta_q W_q, sigma_q = (op_q + om_{K-1-q})/2,
           delta_q = op_q - om_{K-1-q} */
        for (int r = 0; r < (copy ? 2 : 1); ++r) {
          double* o = A.lin[ax] + (r ? fcp : fi) + (long long)s * (2 * K + 2) * nface;
          double wW = 0.0;
#pragma unroll
          for (int q = 0; q < K; ++q) {
            const double dq = op[q] - om[K - 1 - q];
            o[(2 + q) * nface] = 0.5 * (op[q] + om[K - 1 - q]);
            o[(2 + K + q) * nface] = dq;
            wW = fma(dq, wv[q], wW);
          }
          o[0] = fsum;
          o[nface] = wW;
        }
      }
    }
    __syncthreads();

    /* ---- (2) Fhat = Fc when every field is central, else sum_s r_s fs with fs = l_s . Fc for
       the central fields.  Both sums go through the vectors the eigenvectors share:
       a = (b2, -b1 u, b1) and b = (u_n, -e_n, 0)/c give l_{u-c} = (a + b)/2, l_{u+c} = (a - b)/2,
       l_entropy = e_0 - a, l_shear = e_t - u_t e_0, and with sigma = f_{u-c} + f_{u+c},
       delta = (f_{u+c} - f_{u-c}) c:  F_0 = sigma + f_1,  F_d = (sigma + f_1) u_d + (delta if
       d = n, else f_shear(d)),  F_E = sigma H + delta u_n + f_1 |u|^2/2 + sum_t f_t u_t. ---- */
    if (tid < nf && s_cm[tid] != allf) {
      const unsigned cm = s_cm[tid];
      auto row = [&](int r) -> double { return s_row[r * TH + tid]; };
      double* const Fo = A.Fhat[ax];
      double Fc[NV], ut[D], fs[NV], Fh[NV], q2 = 0.0, uF = 0.0;
#pragma unroll
      for (int v = 0; v < NV; ++v) Fc[v] = Fo[gc(v) * nface + flin];
#pragma unroll
      for (int d = 0; d < D; ++d) {
        ut[d] = row(R::u + d);
        q2 += ut[d] * ut[d];
        uF = fma(ut[d], Fc[1 + d], uF);
      }
      const double a = fma(row(R::b2), Fc[0], row(R::b1) * (Fc[NV - 1] - uF));
      const double b = row(R::ci) * fma(ut[0], Fc[0], -Fc[1]);
      fs[0] = (cm & 1u) ? 0.5 * (a + b) : s_fs[tid];
      fs[NV - 1] = (cm >> (NV - 1) & 1u) ? 0.5 * (a - b) : s_fs[(NV - 1) * TH + tid];
      fs[1] = (cm >> 1 & 1u) ? Fc[0] - a : s_fs[TH + tid];
#pragma unroll
      for (int s = 2; s <= NV - 2; ++s)
        fs[s] = (cm >> s & 1u) ? fma(-ut[s - 1], Fc[0], Fc[s]) : s_fs[s * TH + tid];
      const double sigma = fs[0] + fs[NV - 1];
      const double delta = (fs[NV - 1] - fs[0]) * row(R::ct);
      const double m = sigma + fs[1];
      double FE = fma(sigma, row(R::H), fma(delta, ut[0], 0.5 * q2 * fs[1]));
      Fh[0] = m;
      Fh[1] = fma(m, ut[0], delta);
#pragma unroll
      for (int s = 2; s <= NV - 2; ++s) {
        Fh[s] = fma(m, ut[s - 1], fs[s]);
        FE = fma(ut[s - 1], fs[s], FE);
      }
      Fh[NV - 1] = FE;
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
