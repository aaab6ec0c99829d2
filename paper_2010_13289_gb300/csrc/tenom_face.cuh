/* Tiles, staging and the per-lane face flux shared by the face sweeps (Section 4 of arXiv
 * 2010.13289: Roe-averaged characteristic decomposition, Rusanov / local Lax-Friedrichs
 * splitting, TENO-M per characteristic field and split side, back-projection).
 *
 * A sweep of one axis is screen_kernel (tenom_screen.cuh: the central flux of every face and
 * the certificate that it is the nonlinear one) followed by nonlinear_kernel
 * (tenom_nonlinear.cuh: the faces left over).  A CTA owns a tile of consecutive faces along the
 * sweep axis, one thread per face:
 *   axis x : a run of faces of one row (x is contiguous);
 *   axis y,z: contiguous x-columns (lanes) x faces along the axis.
 * (Tile sizes: FaceTile; the screen's tiles use fx_faces / FWD_LANES.)  The tile's points
 * (faces + K-1 halo points, boundary condition applied at load: periodic wrap or
 * zero-gradient clamp) are staged in shared memory with every point quantity the faces need.
 * Each face flux is written once to the face buffer [nvar][nface_a]; the cell update (flux
 * difference) reads it later, so both neighbouring cells use the same face value.
 */
#pragma once
#include <cstdint>
#include "tenom_recon.cuh"
#include "tenom_stats.cuh"
#include "tenom_fastmath.cuh"

namespace tenom {

struct FaceArgs {
  const double* U;    /* [NV][ncell] */
  double* Fhat;       /* [NV][nface] */
  uint8_t* flags;     /* [nface][NV][2] or null */
  const double* P;    /* point primitives [NV + 2][ncell] (velocity, p, c, H, sqrt rho); the screen reads
                         velocity, p and c only */
  double* lin;        /* linearisation [NV][2K+2][nface] (record kernels only) */
  unsigned* list;     /* screen: faces with an uncertified field ([nface]), the fields (bit s), the count */
  uint8_t* mask;
  unsigned* count;
  int* status;        /* sticky status word (statistics) */
  unsigned long long* stats;  /* decision statistics [SC_COUNT] (statistics kernels only) */
  int n[3];
  int bc[3];
  long long ncell;
  long long nface;
  double gamma;
  SchemeDev sch;
};

/* shared-memory layout of the staged point quantities: component c of point p at c * NP + p */
template <int NV>
struct PointLayout {
  static constexpr int NC = 3 * NV + 3;
  static constexpr int cU = 0, cF = NV, cV = 2 * NV, cH = 3 * NV - 2, cC = 3 * NV - 1, cS = 3 * NV;
  static constexpr int cLm = 3 * NV + 1, cLp = 3 * NV + 2;
};

constexpr int FX_FACES = 128;  /* faces per CTA, x sweeps of the statistics kernels */
/* threads (faces) per CTA of the screen: 256 in 2D and 3D (x sweeps 256 faces of a row, y/z
   sweeps 16 x columns by 16 faces: 1.3-1.4 staged points per face), 128 for 1D grids (the tile
   index is the grid's y: 64 would halve the longest line) */
__host__ __device__ constexpr int fx_faces(int K, int NV) { return (void)K, NV > 3 ? 256 : 128; }
/* faces per CTA along the axis of the statistics kernels, y/z (x 32 lanes): 4, i.e. 128-thread CTAs */
__host__ __device__ constexpr int ft_faces(int K) { return (void)K, 4; }
/* screen, y/z sweeps: FWD_LANES x columns by fx_faces(K, NV) / FWD_LANES faces (a warp takes
   two face rows) */
constexpr int FWD_LANES = 16;
/* resident threads per SM the screen is compiled for.  1024 (64 registers) spill 100 bytes a thread
   in TENO6, 210 in TENO8; 2048^2 steps 5.08 ms against 5.17 (TENO6) and 5.99 against 5.98 (TENO8),
   777x531 TENO8 1.11 ms against 1.06 */
__host__ __device__ constexpr int screen_threads_per_sm(int K, int NV) { return K == 6 && NV > 3 ? 1024 : 768; }
/* statistics kernels: 3 CTAs of 128 threads, 168 registers */
constexpr int FACE_CTAS_PER_SM_STATS = 3;

template <int NV, int K, int AXIS, bool FWDT = false>
struct FaceTile {
  static constexpr int H = K / 2;
  static constexpr int NC = PointLayout<NV>::NC;
  static constexpr int LANES = (AXIS == 0) ? 1 : (FWDT ? FWD_LANES : 32);
  static constexpr int FACES = (AXIS == 0) ? (FWDT ? fx_faces(K, NV) : FX_FACES) : (FWDT ? fx_faces(K, NV) / FWD_LANES : ft_faces(K));
  static constexpr int ROWS = FACES + K - 1;     /* points along the axis */
  static constexpr int NP = ROWS * LANES;        /* points per tile */
  static constexpr int THREADS = FACES * LANES;
  static constexpr size_t SMEM = sizeof(double) * NC * NP;
};

__device__ __forceinline__ int bc_wrap(int j, int n, int bc) {
  if (j >= 0 && j < n) return j;
  if (bc == 0) {
    j %= n;
    return j < 0 ? j + n : j;
  }
  return j < 0 ? 0 : (j >= n ? n - 1 : j);
}

/* Primitive quantities of one point: velocity, pressure p = (gamma - 1)(E - rho|u|^2/2),
   sound speed c = sqrt(gamma p / rho). */
template <int NV>
__device__ __forceinline__ void point_prims(const double (&u)[NV], double gamma, double (&vel)[NV - 2], double& pr,
                                            double& c, int& st) {
  constexpr int D = NV - 2;
  const double rho = u[0];
  const double rinv = rcp_nr(rho);
  double ke = 0.0;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    vel[d] = u[1 + d] * rinv;
    ke += u[1 + d] * vel[d];
  }
  pr = (gamma - 1.0) * (u[NV - 1] - 0.5 * ke);
  c = sqrt(gamma * pr * rinv);
  if (!ipos(rho)) st |= ST_RHO;
  if (!ipos(pr)) st |= ST_P;
}

/* Point quantities of the Euler equations for sweep axis AXIS, written to the tile from U
   and its primitives: U, the physical flux F_AXIS(U), velocity, H, c, sqrt(rho),
   |u_a - c|, |u_a + c|. */
template <int NV, int AXIS>
__device__ __forceinline__ void stage_point_from(const double (&u)[NV], const double (&vel)[NV - 2], double pr,
                                                 double Hh, double c, double sr, double* sm, int NP, int p) {
  using L = PointLayout<NV>;
  constexpr int D = NV - 2;
  const double un = vel[AXIS];
#pragma unroll
  for (int q = 0; q < NV; ++q) sm[(L::cU + q) * NP + p] = u[q];
  sm[(L::cF + 0) * NP + p] = u[0] * un;
#pragma unroll
  for (int d = 0; d < D; ++d) sm[(L::cF + 1 + d) * NP + p] = u[1 + d] * un + (d == AXIS ? pr : 0.0);
  sm[(L::cF + NV - 1) * NP + p] = (u[NV - 1] + pr) * un;
#pragma unroll
  for (int d = 0; d < D; ++d) sm[(L::cV + d) * NP + p] = vel[d];
  sm[L::cH * NP + p] = Hh;
  sm[L::cC * NP + p] = c;
  sm[L::cS * NP + p] = sr;
  sm[L::cLm * NP + p] = iabs(un - c);
  sm[L::cLp * NP + p] = iabs(un + c);
}

/* Decision statistics of the face whose K stencil points are shared-memory points
   (jf + q) * LANES + lane, q = 0..K-1, of a tile laid out by PointLayout<NV> with NP points per
   component: Roe average of points K/2-1 and K/2, characteristic projection, LLF split, both sides
   of every field counted into cnt. */
template <int NV, int K, int LIM, int AXIS, int LANES>
__device__ __forceinline__ void face_stats(const double* sm, int NP, int jf, int lane, double gamma,
                                           const SchemeDev& sch, unsigned (&cnt)[SC_COUNT], int& st) {
  using L = PointLayout<NV>;
  constexpr int D = NV - 2;
  constexpr int H = K / 2;
  auto P = [&](int comp, int q) -> double {
    return sm[comp * NP + (jf + q) * LANES + lane];
  };
  /* Roe average of cells f-1 (point H-1) and f (point H) */
  const double sL = P(L::cS, H - 1), sR = P(L::cS, H);
  const double wsum = rcp_nr(sL + sR);
  double ut[D], q2 = 0.0;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    ut[d] = (sL * P(L::cV + d, H - 1) + sR * P(L::cV + d, H)) * wsum;
    q2 += ut[d] * ut[d];
  }
  const double Ht = (sL * P(L::cH, H - 1) + sR * P(L::cH, H)) * wsum;
  const double c2 = (gamma - 1.0) * (Ht - 0.5 * q2);
  if (!ipos(c2)) st |= ST_ROE;
  const double cinv = rsqrt_nr(c2);
  const double b1 = (gamma - 1.0) * (cinv * cinv);
  const double b2 = 0.5 * q2 * b1;
  const double una = ut[AXIS];
  /* LLF: alpha_s = max over the K stencil points of |lambda_s|, one per eigenvalue family */
  double a_m = 0.0, a_0 = 0.0, a_p = 0.0;
#pragma unroll
  for (int q = 0; q < K; ++q) {
    a_m = imax_nonneg(a_m, P(L::cLm, q));
    a_0 = imax_nonneg(a_0, iabs(P(L::cV + AXIS, q)));
    a_p = imax_nonneg(a_p, P(L::cLp, q));
  }

  /* The acoustic pair and the entropy field share the vectors a = (b2, -b1 u, b1) and
     b = (u_n / c, -e_n / c, 0): l_{u-+c} = (a +- b)/2, l_0 = e_0 - a.  Per stencil point
     A = a.U/2, B = b.U/2, AF = a.F/4, BF = b.F/4 once, then W_{u-+c} = A +- B,
     G_{u-+c}/2 = AF +- BF, W_0 = rho - 2A, G_0/2 = F_rho/2 - 2AF. */
  double pA[K], pB[K], pAF[K], pBF[K];
  {
    double ah[NV], aq[NV];
    ah[0] = 0.5 * b2;
#pragma unroll
    for (int d = 0; d < D; ++d) ah[1 + d] = -0.5 * b1 * ut[d];
    ah[NV - 1] = 0.5 * b1;
#pragma unroll
    for (int v = 0; v < NV; ++v) aq[v] = 0.5 * ah[v];
    const double bh0 = 0.5 * una * cinv, bh1 = -0.5 * cinv;
#pragma unroll
    for (int q = 0; q < K; ++q) {
      double a = ah[0] * P(L::cU, q), af = aq[0] * P(L::cF, q);
#pragma unroll
      for (int v = 1; v < NV; ++v) {
        a = fma(ah[v], P(L::cU + v, q), a);
        af = fma(aq[v], P(L::cF + v, q), af);
      }
      pA[q] = a;
      pAF[q] = af;
      pB[q] = fma(bh1, P(L::cU + 1 + AXIS, q), bh0 * P(L::cU, q));
      pBF[q] = 0.5 * fma(bh1, P(L::cF + 1 + AXIS, q), bh0 * P(L::cF, q));
    }
  }

#pragma unroll 1
  for (int s = 0; s < NV; ++s) {
    const bool acoustic = (s == 0) || (s == NV - 1);
    const double sg = (s == 0) ? 1.0 : -1.0;            /* l: +1 for u-c, -1 for u+c */
    const int dt = (s - 2) < AXIS ? (s - 2) : (s - 1);  /* shear fields: tangential axes in increasing order */
    double utt = 0.0;
#pragma unroll
    for (int d = 0; d < D; ++d) utt = (d == dt) ? ut[d] : utt;
    /* left eigenvector l_s (closed form of R^{-1}) */
    double l[NV];
    if (acoustic) {
      l[0] = 0.5 * (b2 + sg * una * cinv);
#pragma unroll
      for (int d = 0; d < D; ++d) l[1 + d] = 0.5 * (-b1 * ut[d] - (d == AXIS ? sg * cinv : 0.0));
      l[NV - 1] = 0.5 * b1;
    } else if (s == 1) {
      l[0] = 1.0 - b2;
#pragma unroll
      for (int d = 0; d < D; ++d) l[1 + d] = b1 * ut[d];
      l[NV - 1] = -b1;
    } else {
      l[0] = -utt;
#pragma unroll
      for (int d = 0; d < D; ++d) l[1 + d] = (d == dt) ? 1.0 : 0.0;
      l[NV - 1] = 0.0;
    }
    /* characteristic projection of the K stencil points and LLF split
       g+- = (G +- alpha W)/2, evaluated as fma(+-alpha/2, W, G/2) */
    const double ha = 0.5 * ((s == 0) ? a_m : (s == NV - 1 ? a_p : a_0));
    double gp[K], gm[K];
    if (acoustic) {
#pragma unroll
      for (int q = 0; q < K; ++q) {
        const double w = fma(sg, pB[q], pA[q]), hg = fma(sg, pBF[q], pAF[q]);
        gp[q] = fma(ha, w, hg);
        gm[q] = fma(-ha, w, hg);
      }
    } else if (s == 1) {
#pragma unroll
      for (int q = 0; q < K; ++q) {
        const double w = fma(-2.0, pA[q], P(L::cU, q)), hg = fma(-2.0, pAF[q], 0.5 * P(L::cF, q));
        gp[q] = fma(ha, w, hg);
        gm[q] = fma(-ha, w, hg);
      }
    } else {
      /* shear wave: l = (-u_t, e_t, 0) */
#pragma unroll
      for (int q = 0; q < K; ++q) {
        const double w = fma(-utt, P(L::cU, q), P(L::cU + 1 + dt, q));
        const double hg = 0.5 * fma(-utt, P(L::cF, q), P(L::cF + 1 + dt, q));
        gp[q] = fma(ha, w, hg);
        gm[q] = fma(-ha, w, hg);
      }
    }
    /* f+ on the upwind stencil, f- on the stencil mirrored about x_{i+1/2} */
    double vm[K];
#pragma unroll
    for (int q = 0; q < K; ++q) vm[q] = gm[K - 1 - q];
    side_stats<K, LIM>(gp, sch, cnt);
    side_stats<K, LIM>(vm, sch, cnt);
  }
}

/* Decision statistics of the faces of one axis (both split sides of every field in FP64 and
   certified form), counted into A.stats; A.P holds the full primitives. */
template <int NV, int K, int LIM, int AXIS>
__global__ void __launch_bounds__(FaceTile<NV, K, AXIS>::THREADS, FACE_CTAS_PER_SM_STATS)
stats_kernel(const FaceArgs A) {
  using T = FaceTile<NV, K, AXIS>;
  constexpr int H = T::H, D = NV - 2;
  extern __shared__ double sm[];
  const int tid = threadIdx.x;
  const int na = A.n[AXIS];
  const int f0 = blockIdx.y * T::FACES;
  int x0 = 0, o1 = 0, o2 = 0;
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
  int st = 0;
  for (int p = tid; p < T::NP; p += T::THREADS) {
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
    double u[NV], vel[D];
#pragma unroll
    for (int q = 0; q < NV; ++q) u[q] = __ldg(A.U + q * A.ncell + cell);
#pragma unroll
    for (int d = 0; d < D; ++d) vel[d] = __ldg(A.P + d * A.ncell + cell);
    stage_point_from<NV, AXIS>(u, vel, __ldg(A.P + D * A.ncell + cell), __ldg(A.P + (D + 2) * A.ncell + cell),
                               __ldg(A.P + (D + 1) * A.ncell + cell), __ldg(A.P + (D + 3) * A.ncell + cell), sm, T::NP,
                               p);
  }
  __syncthreads();
  const int lane = (AXIS == 0) ? 0 : (tid % T::LANES);
  const int jf = (AXIS == 0) ? tid : (tid / T::LANES);
  unsigned cnt[SC_COUNT];
#pragma unroll
  for (int q = 0; q < SC_COUNT; ++q) cnt[q] = 0u;
  if (f0 + jf <= na && (AXIS == 0 || x0 + lane < A.n[0])) {
    face_stats<NV, K, LIM, AXIS, T::LANES>(sm, T::NP, jf, lane, A.gamma, A.sch, cnt, st);
  }
  /* warp sums, one 64-bit atomic per counter and warp */
#pragma unroll
  for (int q = 0; q < SC_COUNT; ++q) {
    const unsigned w = __reduce_add_sync(0xffffffffu, cnt[q]);
    if ((tid & 31) == 0 && w) atomicAdd(A.stats + q, (unsigned long long)w);
  }
  if (st) atomicOr(A.status, st);
}

}  // namespace tenom
