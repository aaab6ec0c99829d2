/* Frozen-branch adjoint of the operator: Z = L'(U)^T w, every branch taken from the forward pass
 * (Sections 2-4 of arXiv 2010.13289).
 *
 * TENO-M assembles the candidates with constant weights w_k = d_k (Section 3.3), so once the
 * cutoff flags and the limiter's selections are fixed, each reconstruction is a LINEAR
 * function of the K stencil values, and R L = I turns the face flux into
 *   F = Fc + sum_s r_s f'_s,   Fc = sum_q c_q F(U_q),
 *   f'_s = sum_q sigma'_q G_q + (alpha_s/2) sum_q delta_q W_q,   G = l_s.F, W = l_s.U,
 * with sigma'_q = (op_q + om_{K-1-q})/2 - c_q, delta_q = op_q - om_{K-1-q} (op, om: the frozen
 * weights of f+ and f- on its mirrored stencil).  f'_s vanishes identically where all
 * candidates of both sides are smooth.  So the adjoint is
 *   adj_central_kernel: the transposed central fluxes of every cell and axis, a stencil of w and
 *     one flux Jacobian per cell and axis, and
 *   adj_fields_kernel: per axis, the faces that have a field with f'_s != 0 (few in smooth flow),
 *     with the fields' weights from the recorded linearisation or rebuilt from the flags.
 * Reversing the whole characteristic decomposition of every face instead took 550-610 FP64
 * operations a face.  Per stage of the 2D 512^2 TENO6 workload (55 % of the faces listed, two
 * fields each): two sweeps of 317 us before, 47 us central and 2 x 260 us now, FP64 pipe 80 %
 * busy; with the flags on 256^2 TENO8 waves (13 % listed) two of 480 us before, 26 + 223 + 113 now. */
#pragma once
#include "tenom_face.cuh"

namespace tenom {

struct AdjArgs {
  const double* U;       /* state the operator was applied to [NV][ncell] */
  const uint8_t* flags;  /* forward flags of this axis [nface][NV][2], or null */
  const double* lin;     /* recorded linearisation of this axis [NV][2K+2][nface], or null */
  const double* P;       /* cell primitives of U [NV + 2][ncell] (velocity, p, c, H, sqrt rho) */
  const double* w;       /* cell adjoint [NV][ncell] */
  double* Z;             /* L'^T w [NV][ncell] */
  int n[3];
  int bc[3];
  long long ncell;
  long long nface;       /* faces of this axis */
  double rdx[3];
  double gamma;
  SchemeDev sch;
  int whole;             /* 1: no field is ever central (d_k of the caller's), so the fields carry the whole flux
                            (sigma instead of sigma') and there is no central part */
};

/* omegaW of a recorded field whose correction vanishes: -0.0 (sum_q delta_q W_q = 0), which a
   recorded sum never is */
__host__ __device__ constexpr unsigned long long kCentralMark = 0x8000000000000000ull;

/* Weight with which cell i enters the central flux of face f on an axis of n cells (zero-gradient
   ghosts fold onto the edge cells). */
template <int K>
__device__ __forceinline__ double central_entry(const double (&cw)[K], int f, int i, int n) {
  double x = 0.0;
#pragma unroll
  for (int q = 0; q < K; ++q) {
    int j = f - K / 2 + q;
    j = j < 0 ? 0 : (j >= n ? n - 1 : j);
    if (j == i) x += cw[q];
  }
  return x;
}

/* Z = sum over axes of the transposed central fluxes: with Fbar_f = (w_f - w_{f-1})/dx (w = 0 outside
   the grid), the adjoint of F_a(U_i) is sum_f c_{q(f,i)} Fbar_f = sum_m E_m (w_{i+m} - w_{i-m})/dx,
   E_m = c_{K/2-m} - c_{K/2-m-1}, and Z_i gains its Jacobian's transpose times that. */
template <int NV, int K>
__global__ void __launch_bounds__(256) adj_central_kernel(const AdjArgs A) {
  constexpr int D = NV - 2, H = K / 2;
  double cw[K], Em[H];
  central_weights<K>(cw);
#pragma unroll
  for (int m = 1; m <= H; ++m) Em[m - 1] = cw[H - m] - (m < H ? cw[H - m - 1] : 0.0);
  const long long nc = A.ncell;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < nc; c += (long long)gridDim.x * blockDim.x) {
    int ix[3];
    {
      const unsigned r = (unsigned)(c / A.n[0]);
      ix[0] = (int)(c - (long long)r * A.n[0]);
      ix[1] = (int)(r % (unsigned)A.n[1]);
      ix[2] = (int)(r / (unsigned)A.n[1]);
    }
    double u[D], z[NV], q2 = 0.0;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      u[d] = __ldg(A.P + d * nc + c);
      q2 = fma(u[d], u[d], q2);
    }
    const double Hh = __ldg(A.P + (D + 2) * nc + c), gm1 = A.gamma - 1.0;
#pragma unroll
    for (int v = 0; v < NV; ++v) z[v] = 0.0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const int n = A.n[a], i = ix[a];
      const long long sa = a == 0 ? 1 : (a == 1 ? (long long)A.n[0] : (long long)A.n[0] * A.n[1]);
      const long long line = c - sa * i;
      double g[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) g[v] = 0.0;
      if (A.bc[a] == 0 || (i >= H && i + H < n)) {
#pragma unroll
        for (int m = 1; m <= H; ++m) {
          int ip = i + m, im = i - m;
          if (A.bc[a] == 0) {
            ip = ip >= n ? ip - n : ip;
            im = im < 0 ? im + n : im;
          }
#pragma unroll
          for (int v = 0; v < NV; ++v)
            g[v] = fma(Em[m - 1], __ldg(A.w + v * nc + line + sa * ip) - __ldg(A.w + v * nc + line + sa * im), g[v]);
        }
      } else {
#pragma unroll 1
        for (int f = i - H; f <= i + H; ++f) {
          if (f < 0 || f > n) continue;
          const double e = central_entry<K>(cw, f, i, n);
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            const double wr = f < n ? __ldg(A.w + v * nc + line + sa * f) : 0.0;
            const double wl = f >= 1 ? __ldg(A.w + v * nc + line + sa * (f - 1)) : 0.0;
            g[v] = fma(e, wr - wl, g[v]);
          }
        }
      }
      /* J_a^T g: F = (m_n, m u_n + p e_n, (E + p) u_n) */
      double un = 0.0, gn = 0.0, t = fma(Hh, g[NV - 1], g[0]);
#pragma unroll
      for (int d = 0; d < D; ++d) {
        t = fma(u[d], g[1 + d], t);
        if (d == a) {
          un = u[d];
          gn = g[1 + d];
        }
      }
      const double gE = g[NV - 1], eb = gm1 * fma(un, gE, gn), r = A.rdx[a];
      z[0] = fma(r, fma(un, g[0] - t, 0.5 * q2 * eb), z[0]);
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const double x = fma(un, g[1 + d], fma(-u[d], eb, d == a ? t : 0.0));
        z[1 + d] = fma(r, x, z[1 + d]);
      }
      z[NV - 1] = fma(r, fma(un, gE, eb), z[NV - 1]);
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) A.Z[v * nc + c] = z[v];
  }
}

/* Reverse of the point quantities (stage_point_from): adjoints of the physical flux F_AXIS (Fb),
   of the velocity (velb), sound speed (cb), enthalpy (Hb) and sqrt(rho) (sb) of one point
   -> adjoint of its conserved state, added to Ub. */
template <int NV, int AXIS>
__device__ __forceinline__ void point_vjp(const double* sm, int NP, int p, double gamma, const double (&Fb)[NV],
                                          double (&velb)[NV - 2], double cb, double Hb, double sb, double (&Ub)[NV]) {
  using L = PointLayout<NV>;
  constexpr int D = NV - 2;
  const double rho = sm[L::cU * NP + p], E = sm[(L::cU + NV - 1) * NP + p];
  double m[D], vel[D], ke = 0.0;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    m[d] = sm[(L::cU + 1 + d) * NP + p];
    vel[d] = sm[(L::cV + d) * NP + p];
    ke += m[d] * vel[d];
  }
  const double pr = (gamma - 1.0) * (E - 0.5 * ke);
  const double H = sm[L::cH * NP + p], c = sm[L::cC * NP + p];
  const double un = vel[AXIS];
  const double rinv = rcp_nr(rho);
  double rhob = 0.0, Eb = 0.0, pb = 0.0, mb[D];
#pragma unroll
  for (int d = 0; d < D; ++d) mb[d] = 0.0;
  /* physical flux F = (rho un, m un + p e_a, (E + p) un) */
  double unb = rho * Fb[0];
  rhob += un * Fb[0];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    mb[d] += un * Fb[1 + d];
    unb += m[d] * Fb[1 + d];
  }
  pb += Fb[1 + AXIS];
  Eb += un * Fb[NV - 1];
  pb += un * Fb[NV - 1];
  unb += (E + pr) * Fb[NV - 1];
  velb[AXIS] += unb;
  /* H = (E + p)/rho */
  Eb += Hb * rinv;
  pb += Hb * rinv;
  rhob -= H * Hb * rinv;
  /* c = sqrt(gamma p / rho) */
  if (cb != 0.0) {
    const double k = cb * rcp_nr(2.0 * c * rho);
    pb += gamma * k;
    rhob -= c * c * k;
  }
  /* sqrt(rho) */
  if (sb != 0.0) rhob += sb * rcp_nr(2.0 * sm[L::cS * NP + p]);
  /* p = (gamma - 1)(E - ke/2), ke = sum m_d vel_d */
  Eb += (gamma - 1.0) * pb;
  const double keb = -0.5 * (gamma - 1.0) * pb;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    mb[d] += vel[d] * keb;
    velb[d] += m[d] * keb;
  }
  /* vel_d = m_d / rho */
#pragma unroll
  for (int d = 0; d < D; ++d) {
    mb[d] += velb[d] * rinv;
    rhob -= vel[d] * velb[d] * rinv;
  }
  Ub[0] += rhob;
#pragma unroll
  for (int d = 0; d < D; ++d) Ub[1 + d] += mb[d];
  Ub[NV - 1] += Eb;
}

__device__ __forceinline__ double dsign(double x) { return ipos(x) ? 1.0 : (ineg(x) ? -1.0 : 0.0); }

/* Tile of adj_fields_kernel (one thread per face) and its shared memory: the tile's points, per point
   the adjoints of U (NV), F (NV) and |lambda| (3), per face the Roe-state adjoints of its two centre
   points.  Along x 128 faces of a row; y/z 16 x columns by YZ faces: 16, or 8 on grids whose tiles
   would leave SMs without one (1.9 staged points per face instead of 1.4, but a full tile is 256
   faces of FP64 on one SM: 32^2 TENO6 102 -> 84 us a call, 1024^2 1516 -> 1547). */
template <int NV, int K, int AXIS, int YZ>
struct AdjTile {
  static constexpr int H = K / 2, LANES = AXIS == 0 ? 1 : 16;
  static constexpr int FACES = AXIS == 0 ? 128 : YZ;
  static constexpr int THREADS = FACES * LANES, NP = (FACES + K - 1) * LANES;
  static constexpr int NA = 2 * NV + 3, NR = 2 * NV;
  static constexpr size_t SMEM = sizeof(double) * ((size_t)(PointLayout<NV>::NC + NA) * NP + (size_t)NR * THREADS);
};

/* Adds the reverse of sum_s r_s f'_s of the axis's faces to Z.  A CTA finds its tile's faces with such
   a field and gives each to a thread (dense warps; a tile without any ends at once).  Per field: f'_s =
   l_s . (S_F + alpha/2 S_U) with S_F = sum_q sigma'_q F_q, S_U = sum_q delta_q U_q, so the adjoint of l_s
   is fbar (S_F + alpha/2 S_U) and point q receives fbar sigma'_q l_s (flux) and fbar (alpha/2) delta_q
   l_s (state).  Point adjoints are summed in shared memory in K phases (in phase q every face adds to
   its q-th point, all distinct); the reverse of the point quantities then runs once per touched point.
   From the tape all fields of a face are taken together, point by point, in the basis that the
   eigenvectors share; from the flags, where a field's weights have to be rebuilt first, one field after
   the other (faces with most fields first, so that a step fills whole warps).  One field at a time
   from the tape too cost a set of phases per field: 64x56x48 TENO6 with most faces listed 1007 us
   against 883 (965 with every face reversed whole), with d_k of the caller's 1607 against 1048 (964). */
template <int NV, int K, int LIM, int AXIS, bool TAPE, int YZ>
__global__ void __launch_bounds__(AdjTile<NV, K, AXIS, YZ>::THREADS, (TAPE ? 512 : 256) / AdjTile<NV, K, AXIS, YZ>::THREADS)
    adj_fields_kernel(const AdjArgs A) {
  using T = AdjTile<NV, K, AXIS, YZ>;
  using L = PointLayout<NV>;
  constexpr int H = T::H, D = NV - 2, TH = T::THREADS, NP = T::NP, LANES = T::LANES, W = TH / 32;
  constexpr int NA = T::NA, NR = T::NR, RS = 2 * K + 2;
  constexpr int aU = 0, aF = NV, aM = 2 * NV;  /* aM + 0 (u-c), 1 (u), 2 (u+c) */
  constexpr unsigned allk = (1u << (K - 2)) - 1u;
  extern __shared__ double sm[];
  double* const acc = sm + L::NC * NP;
  double* const roe = acc + NA * NP;
  __shared__ unsigned short s_list[TH];
  __shared__ int s_wc[NV][W];
  const int tid = threadIdx.x;
  const int na = A.n[AXIS];
  int x0 = 0, o1 = 0, o2 = 0;
  const int f0 = blockIdx.y * T::FACES;
  if (AXIS == 0) {
    o1 = blockIdx.x % A.n[1];
    o2 = blockIdx.x / A.n[1];
  } else {
    x0 = blockIdx.x * LANES;
    o2 = blockIdx.z;
  }
  const long long sy = A.n[0], sz = (long long)A.n[0] * A.n[1];
  const long long sa = (AXIS == 0) ? 1 : (AXIS == 1 ? sy : sz);
  /* cell with axis coordinate 0 of the line at x column xg; linear index of a face */
  auto line = [&](int xg) -> long long {
    if (AXIS == 0) return sy * o1 + sz * o2;
    return xg + (AXIS == 1 ? sz * o2 : sy * o2);
  };
  auto face_index = [&](int f, int xg) -> long long {
    if (AXIS == 0) return f + (long long)(A.n[0] + 1) * (o1 + (long long)A.n[1] * o2);
    if (AXIS == 1) return xg + (long long)A.n[0] * (f + (long long)(A.n[1] + 1) * o2);
    return xg + (long long)A.n[0] * (o2 + (long long)A.n[1] * f);
  };
  auto fields_of = [&](long long fi) -> unsigned {  /* the fields with f'_s != 0 */
    unsigned m = 0u;
#pragma unroll
    for (int s = 0; s < NV; ++s) {
      bool central;
      if constexpr (TAPE) {
        central = (unsigned long long)dbits(__ldg(A.lin + (long long)(s * RS + 1) * A.nface + fi)) == kCentralMark;
      } else {
        const uint8_t* b = A.flags + fi * NV * 2 + 2 * s;
        central = A.sch.default_d && (b[0] & allk) == allk && (b[1] & allk) == allk;
      }
      m |= central ? 0u : 1u << s;
    }
    return m;
  };
  auto jf_of = [&](int slot) { return AXIS == 0 ? slot : slot / LANES; };
  auto lane_of = [&](int slot) { return AXIS == 0 ? 0 : slot % LANES; };

  /* ---- the tile's faces with a field to reverse ---- */
  unsigned mask = 0u;
  {
    const int f = f0 + jf_of(tid), xg = x0 + lane_of(tid);
    if (f <= na && (AXIS == 0 || xg < A.n[0])) mask = fields_of(face_index(f, xg));
  }
  /* the list holds the faces with the most fields first, so that a step's faces fill whole warps */
  const int mine = __popc(mask);
  unsigned bal[NV];
#pragma unroll
  for (int b = 0; b < NV; ++b) {
    bal[b] = __ballot_sync(0xffffffffu, mine == NV - b);
    if ((tid & 31) == 0) s_wc[b][tid >> 5] = __popc(bal[b]);
  }
  __syncthreads();
  int before = 0, count = 0, steps = 0;
#pragma unroll
  for (int b = 0; b < NV; ++b) {
    int sum = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      if (mine == NV - b && w == (tid >> 5)) before = count + sum + __popc(bal[b] & ((1u << (tid & 31)) - 1u));
      sum += s_wc[b][w];
    }
    steps = steps == 0 && sum > 0 ? NV - b : steps;
    count += sum;
  }
  if (count == 0) return;
  if (mask) s_list[before] = (unsigned short)tid;

  /* ---- points, zeroed adjoints ---- */
  auto point_cell = [&](int p) -> long long {
    const int j = bc_wrap(f0 - H + jf_of(p), na, A.bc[AXIS]);
    int xg = x0 + lane_of(p);
    if (AXIS != 0) xg = xg < A.n[0] ? xg : A.n[0] - 1;
    return line(xg) + sa * j;
  };
  for (int p = tid; p < NP; p += TH) {
    const long long cell = point_cell(p);
    double u[NV], vel[D];
#pragma unroll
    for (int q = 0; q < NV; ++q) u[q] = __ldg(A.U + q * A.ncell + cell);
#pragma unroll
    for (int d = 0; d < D; ++d) vel[d] = __ldg(A.P + d * A.ncell + cell);
    stage_point_from<NV, AXIS>(u, vel, __ldg(A.P + D * A.ncell + cell), __ldg(A.P + (D + 2) * A.ncell + cell),
                               __ldg(A.P + (D + 1) * A.ncell + cell), __ldg(A.P + (D + 3) * A.ncell + cell), sm, NP, p);
  }
  for (int i = tid; i < NA * NP; i += TH) acc[i] = 0.0;
  for (int i = tid; i < NR * TH; i += TH) roe[i] = 0.0;
  __syncthreads();

  /* ---- one face per thread ---- */
  const bool has = tid < count;
  const int slot = has ? s_list[tid] : 0, jf = jf_of(slot), lane = lane_of(slot);
  const int f = f0 + jf, xg = x0 + lane;
  const long long fi = face_index(f, xg);
  auto P = [&](int comp, int q) -> double { return sm[comp * NP + (jf + q) * LANES + lane]; };
  const double gm1 = A.gamma - 1.0;
  double cw[K];
  central_weights<K>(cw);
  double ut[D], q2 = 0.0, Ht = 0.0, c2 = 1.0, cinv = 1.0, ct = 1.0, b1 = 0.0, b2 = 0.0, sL = 0.0, sR = 0.0, wsum = 0.0;
  double am[3] = {0.0, 0.0, 0.0}, Fb[NV];
  int im[3] = {-1, -1, -1};
  double utb[D], Htb = 0.0, ctb = 0.0, ab[NV], bb0 = 0.0, bb1 = 0.0;
#pragma unroll
  for (int d = 0; d < D; ++d) ut[d] = utb[d] = 0.0;
#pragma unroll
  for (int v = 0; v < NV; ++v) ab[v] = Fb[v] = 0.0;
  unsigned todo = 0u;
  if (has) {
    todo = fields_of(fi);
    sL = P(L::cS, H - 1);
    sR = P(L::cS, H);
    wsum = rcp_nr(sL + sR);
#pragma unroll
    for (int d = 0; d < D; ++d) {
      ut[d] = (sL * P(L::cV + d, H - 1) + sR * P(L::cV + d, H)) * wsum;
      q2 += ut[d] * ut[d];
    }
    Ht = (sL * P(L::cH, H - 1) + sR * P(L::cH, H)) * wsum;
    c2 = gm1 * (Ht - 0.5 * q2);
    cinv = rsqrt_nr(c2);
    ct = c2 * cinv;
    b1 = gm1 * (cinv * cinv);
    b2 = 0.5 * q2 * b1;
    /* LLF alpha with its argmax */
#pragma unroll
    for (int q = 0; q < K; ++q) {
      const double x[3] = {P(L::cLm, q), iabs(P(L::cV + AXIS, q)), P(L::cLp, q)};
#pragma unroll
      for (int i = 0; i < 3; ++i)
        if (dbits(am[i]) < dbits(x[i])) {
          am[i] = x[i];
          im[i] = q;
        }
    }
    /* Fbar = (w_f - w_{f-1})/dx (cells outside the grid contribute nothing) */
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const double* w = A.w + v * A.ncell + line(xg);
      Fb[v] = ((f < na ? __ldg(w + sa * f) : 0.0) - (f >= 1 ? __ldg(w + sa * (f - 1)) : 0.0)) * A.rdx[AXIS];
    }
  }
  const double una = ut[AXIS];
  double tb[D];  /* adjoint of -u_t in l_shear */
#pragma unroll
  for (int d = 0; d < D; ++d) tb[d] = 0.0;
  if constexpr (TAPE) {
    /* all fields at once: the adjoints of a point's F and U are combined in the basis (e_0, a, b, e_t)
       that the eigenvectors share before they are expanded, one set of phases for the face */
    const double* const lin = A.lin + fi;
    double kG[NV], kW[NV], Fc[NV], fp[NV], alb[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int s = 0; s < NV; ++s) {
      kG[s] = kW[s] = fp[s] = Fc[s] = 0.0;
      if (todo >> s & 1u) {
        const int fam = s == 0 ? 0 : (s == NV - 1 ? 2 : 1);
        double k = 0.0, hf = 1.0;  /* adjoint of f'_s; the 1/2 of l_{u-+c} = (a +- b)/2 */
        if (s == 0 || s == NV - 1) {
          const double sr = s == 0 ? -1.0 : 1.0;
          k = fma(Ht + sr * una * ct, Fb[NV - 1], Fb[0]);
#pragma unroll
          for (int d = 0; d < D; ++d) k = fma(ut[d] + (d == AXIS ? sr * ct : 0.0), Fb[1 + d], k);
          hf = 0.5;
        } else if (s == 1) {
          k = fma(0.5 * q2, Fb[NV - 1], Fb[0]);
#pragma unroll
          for (int d = 0; d < D; ++d) k = fma(ut[d], Fb[1 + d], k);
        } else {
          const int dt = (s - 2) < AXIS ? (s - 2) : (s - 1);
          k = fma(ut[dt], Fb[NV - 1], Fb[1 + dt]);
        }
        fp[s] = __ldg(lin + (long long)(s * RS) * A.nface);
        alb[fam] = fma(0.5 * k, __ldg(lin + (long long)(s * RS + 1) * A.nface), alb[fam]);
        kG[s] = hf * k;
        kW[s] = kG[s] * (0.5 * am[fam]);
      }
    }
    const double b0v = una * cinv;
#pragma unroll
    for (int q = 0; q < K; ++q) {
      double xu[NV], xf[NV];
      if (has) {
        double cU[NV], cF[NV];
        const double cs = A.whole ? 0.0 : 0.5 * (cw[q] + cw[K - 1 - q]);
#pragma unroll
        for (int s = 0; s < NV; ++s) {
          cF[s] = cU[s] = 0.0;
          if (todo >> s & 1u) {
            cF[s] = kG[s] * (__ldg(lin + (long long)(s * RS + 2 + q) * A.nface) - cs);
            cU[s] = kW[s] * __ldg(lin + (long long)(s * RS + 2 + K + q) * A.nface);
          }
        }
        const double AU = cU[0] + cU[NV - 1] - cU[1], BU = cU[0] - cU[NV - 1];
        const double AF = cF[0] + cF[NV - 1] - cF[1], BF = cF[0] - cF[NV - 1];
        double RU = cU[1], RF = cF[1];
#pragma unroll
        for (int s = 2; s < NV - 1; ++s) {
          const int dt = (s - 2) < AXIS ? (s - 2) : (s - 1);
          RU = fma(-ut[dt], cU[s], RU);
          RF = fma(-ut[dt], cF[s], RF);
        }
        xu[0] = fma(AU, b2, fma(BU, b0v, RU));
        xf[0] = fma(AF, b2, fma(BF, b0v, RF));
#pragma unroll
        for (int d = 0; d < D; ++d) {
          const int s = d < AXIS ? d + 2 : d + 1;  /* shear field of tangential axis d */
          xu[1 + d] = fma(-AU * b1, ut[d], d == AXIS ? -BU * cinv : cU[s]);
          xf[1 + d] = fma(-AF * b1, ut[d], d == AXIS ? -BF * cinv : cF[s]);
        }
        xu[NV - 1] = AU * b1;
        xf[NV - 1] = AF * b1;
        /* adjoints of the entries of a (all components), b (rho, m_n) and l_shear; Fc */
        const double U0 = P(L::cU, q), F0 = P(L::cF, q);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const double Fv = v == 0 ? F0 : P(L::cF + v, q), Uv = v == 0 ? U0 : P(L::cU + v, q);
          ab[v] = fma(AU, Uv, fma(AF, Fv, ab[v]));
          Fc[v] = fma(cs, Fv, Fc[v]);
        }
        bb0 = fma(BU, U0, fma(BF, F0, bb0));
        bb1 = fma(BU, P(L::cU + 1 + AXIS, q), fma(BF, P(L::cF + 1 + AXIS, q), bb1));
#pragma unroll
        for (int d = 0; d < D; ++d) {
          if (d == AXIS) continue;
          const int s = d < AXIS ? d + 2 : d + 1;
          tb[d] = fma(cU[s], U0, fma(cF[s], F0, tb[d]));
        }
      }
      __syncthreads();  /* the previous phase's additions are complete */
      if (has) {
        const int pq = (jf + q) * LANES + lane;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          acc[(aU + v) * NP + pq] += xu[v];
          acc[(aF + v) * NP + pq] += xf[v];
        }
#pragma unroll
        for (int i = 0; i < 3; ++i)
          if (im[i] == q) acc[(aM + i) * NP + pq] += alb[i];
      }
    }
    if (has) {  /* f'_s = fs - l_s . Fc, and the adjoints of r_s (= f'_s Fbar) */
      double uF = 0.0;
#pragma unroll
      for (int d = 0; d < D; ++d) uF = fma(ut[d], Fc[1 + d], uF);
      const double a = fma(b2, Fc[0], b1 * (Fc[NV - 1] - uF)), b = cinv * fma(una, Fc[0], -Fc[1 + AXIS]);
      const double FE = Fb[NV - 1];
#pragma unroll
      for (int s = 0; s < NV; ++s) {
        if (!(todo >> s & 1u)) continue;
        if (s == 0 || s == NV - 1) {
          const double sr = s == 0 ? -1.0 : 1.0, f1 = fp[s] - 0.5 * (a - sr * b);
#pragma unroll
          for (int d = 0; d < D; ++d) utb[d] = fma(f1, Fb[1 + d], utb[d]);
          ctb = fma(sr * f1, fma(una, FE, Fb[1 + AXIS]), ctb);
          Htb = fma(f1, FE, Htb);
          utb[AXIS] = fma(sr * ct * f1, FE, utb[AXIS]);
        } else if (s == 1) {
          const double f1 = fp[s] - (Fc[0] - a);
#pragma unroll
          for (int d = 0; d < D; ++d) utb[d] = fma(f1, fma(ut[d], FE, Fb[1 + d]), utb[d]);
        } else {
          const int dt = (s - 2) < AXIS ? (s - 2) : (s - 1);
          const double f1 = fp[s] - fma(-ut[dt], Fc[0], Fc[1 + dt]);
          utb[dt] = fma(f1, FE, utb[dt]);
        }
      }
#pragma unroll
      for (int d = 0; d < D; ++d)
        if (d != AXIS) utb[d] -= tb[d];
    }
  } else {
#pragma unroll 1
  for (int step = 0; step < steps; ++step) {
    const bool on = todo != 0u;
    double l[NV], sg[K], dl[K], kf = 0.0, kw = 0.0, alb = 0.0;
    int fam = 1, imax = -1;
    if (on) {
      const int s = __ffs(todo) - 1;
      todo &= todo - 1u;
      const bool acoustic = s == 0 || s == NV - 1;
      const double sgn = s == 0 ? 1.0 : -1.0;             /* l: +1 for u-c, -1 for u+c */
      const int dt = (s - 2) < AXIS ? (s - 2) : (s - 1);  /* shear fields: tangential axes in increasing order */
      fam = s == 0 ? 0 : (s == NV - 1 ? 2 : 1);
      const double al = fam == 0 ? am[0] : (fam == 2 ? am[2] : am[1]);
      imax = fam == 0 ? im[0] : (fam == 2 ? im[2] : im[1]);
      if (acoustic) {
        l[0] = 0.5 * (b2 + sgn * una * cinv);
#pragma unroll
        for (int d = 0; d < D; ++d) l[1 + d] = 0.5 * (-b1 * ut[d] - (d == AXIS ? sgn * cinv : 0.0));
        l[NV - 1] = 0.5 * b1;
      } else if (s == 1) {
        l[0] = 1.0 - b2;
#pragma unroll
        for (int d = 0; d < D; ++d) l[1 + d] = b1 * ut[d];
        l[NV - 1] = -b1;
      } else {
        double utt = 0.0;
#pragma unroll
        for (int d = 0; d < D; ++d) utt = (d == dt) ? ut[d] : utt;
        l[0] = -utt;
#pragma unroll
        for (int d = 0; d < D; ++d) l[1 + d] = (d == dt) ? 1.0 : 0.0;
        l[NV - 1] = 0.0;
      }
      {
        double Wv[K], Gv[K];
#pragma unroll
        for (int q = 0; q < K; ++q) {
          double x = 0.0, y = 0.0;
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            x = fma(l[v], P(L::cU + v, q), x);
            y = fma(l[v], P(L::cF + v, q), y);
          }
          Wv[q] = x;
          Gv[q] = y;
        }
        const uint8_t* fl = A.flags + fi * NV * 2 + 2 * s;
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {
          const double ha = side ? -0.5 * al : 0.5 * al;
          double v[K], om[K];
#pragma unroll
          for (int q = 0; q < K; ++q) v[q] = side ? fma(ha, Wv[K - 1 - q], 0.5 * Gv[K - 1 - q]) : fma(ha, Wv[q], 0.5 * Gv[q]);
          teno_general<K, LIM, true>(v, A.sch, fl[side] & allk, om);
#pragma unroll
          for (int q = 0; q < K; ++q) {
            if (side) {
              dl[q] = sg[q] - om[K - 1 - q];
              sg[q] = 0.5 * (sg[q] + om[K - 1 - q]) - (A.whole ? 0.0 : 0.5 * (cw[q] + cw[K - 1 - q]));
            } else {
              sg[q] = om[q];
            }
          }
        }
      }
      double SF[NV], SU[NV], oW = 0.0, fv = 0.0;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        SF[v] = 0.0;
        SU[v] = 0.0;
#pragma unroll
        for (int q = 0; q < K; ++q) {
          SF[v] = fma(sg[q], P(L::cF + v, q), SF[v]);
          SU[v] = fma(dl[q], P(L::cU + v, q), SU[v]);
        }
        oW = fma(l[v], SU[v], oW);
        fv = fma(l[v], SF[v], fv);
      }
      fv = fma(0.5 * al, oW, fv);  /* f'_s */
      /* adjoint of f'_s, and of r_s (= f'_s Fbar) */
      const double FE = Fb[NV - 1];
      if (acoustic) {
        const double sr = -sgn;  /* r: -c for u-c, +c for u+c */
        kf = fma(Ht + sr * una * ct, FE, Fb[0]);
#pragma unroll
        for (int d = 0; d < D; ++d) {
          kf = fma(ut[d] + (d == AXIS ? sr * ct : 0.0), Fb[1 + d], kf);
          utb[d] = fma(fv, Fb[1 + d], utb[d]);
        }
        ctb = fma(sr * fv, fma(una, FE, Fb[1 + AXIS]), ctb);
        Htb = fma(fv, FE, Htb);
        utb[AXIS] = fma(sr * ct * fv, FE, utb[AXIS]);
      } else if (s == 1) {
        kf = fma(0.5 * q2, FE, Fb[0]);
#pragma unroll
        for (int d = 0; d < D; ++d) {
          kf = fma(ut[d], Fb[1 + d], kf);
          utb[d] = fma(fv, fma(ut[d], FE, Fb[1 + d]), utb[d]);
        }
      } else {
#pragma unroll
        for (int d = 0; d < D; ++d)
          if (d == dt) {
            kf = fma(ut[d], FE, Fb[1 + d]);
            utb[d] = fma(fv, FE, utb[d]);
          }
      }
      /* adjoint of l_s: l_{u-+c} = (a +- b)/2, l_entropy = e_0 - a, l_shear = e_t - u_t e_0 with
         a = (b2, -b1 u, b1), b = (u_n, -e_n, 0)/c */
      const double ka = acoustic ? 0.5 * kf : -kf;
      if (acoustic || s == 1) {
#pragma unroll
        for (int v = 0; v < NV; ++v) ab[v] = fma(ka, fma(0.5 * al, SU[v], SF[v]), ab[v]);
        if (acoustic) {
          bb0 = fma(sgn * ka, fma(0.5 * al, SU[0], SF[0]), bb0);
          bb1 = fma(sgn * ka, fma(0.5 * al, SU[1 + AXIS], SF[1 + AXIS]), bb1);
        }
      } else {
#pragma unroll
        for (int d = 0; d < D; ++d)
          if (d == dt) utb[d] = fma(-kf, fma(0.5 * al, SU[0], SF[0]), utb[d]);
      }
      kw = 0.5 * al * kf;
      alb = 0.5 * kf * oW;
    }
#pragma unroll
    for (int q = 0; q < K; ++q) {
      __syncthreads();  /* the previous phase's additions are complete */
      if (on) {
        const int pq = (jf + q) * LANES + lane;
        const double xf = kf * sg[q], xu = kw * dl[q];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          acc[(aU + v) * NP + pq] = fma(xu, l[v], acc[(aU + v) * NP + pq]);
          acc[(aF + v) * NP + pq] = fma(xf, l[v], acc[(aF + v) * NP + pq]);
        }
        if (imax == q) acc[(aM + fam) * NP + pq] += alb;
      }
    }
  }
  }

  /* ---- eigenvector adjoints -> Roe average -> the two centre points ---- */
  if (has) {
    double b2b = ab[0], b1b = ab[NV - 1];
#pragma unroll
    for (int d = 0; d < D; ++d) {
      b1b -= ut[d] * ab[1 + d];
      utb[d] -= b1 * ab[1 + d];
    }
    utb[AXIS] += cinv * bb0;
    double cinvb = una * bb0 - bb1;
    double q2b = 0.5 * b1 * b2b;
    b1b += 0.5 * q2 * b2b;
    cinvb += 2.0 * gm1 * cinv * b1b;
    double c2b = cinv * ctb;
    cinvb += c2 * ctb;
    c2b -= 0.5 * cinv * cinv * cinv * cinvb;
    Htb += gm1 * c2b;
    q2b -= 0.5 * gm1 * c2b;
    double sLb = 0.0, sRb = 0.0;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const double u_b = (utb[d] + 2.0 * ut[d] * q2b) * wsum;
      roe[d * TH + slot] = sL * u_b;
      roe[(D + 2 + d) * TH + slot] = sR * u_b;
      sLb += (P(L::cV + d, H - 1) - ut[d]) * u_b;
      sRb += (P(L::cV + d, H) - ut[d]) * u_b;
    }
    const double hb = Htb * wsum;
    roe[D * TH + slot] = sL * hb;
    roe[(2 * D + 2) * TH + slot] = sR * hb;
    roe[(D + 1) * TH + slot] = sLb + (P(L::cH, H - 1) - Ht) * hb;
    roe[(2 * D + 3) * TH + slot] = sRb + (P(L::cH, H) - Ht) * hb;
  }
  __syncthreads();

  /* ---- per point: gather, reverse of the point quantities, add to Z ---- */
  for (int p = tid; p < NP; p += TH) {
    const int row = jf_of(p), lanep = lane_of(p);
    double ub[NV], Fq[NV], velb[D], Hb = 0.0, sb = 0.0;
    long long any = 0;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      ub[v] = acc[(aU + v) * NP + p];
      Fq[v] = acc[(aF + v) * NP + p];
      any |= dbits(ub[v]) | dbits(Fq[v]);
    }
    double xm[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      xm[i] = acc[(aM + i) * NP + p];
      any |= dbits(xm[i]);
    }
#pragma unroll
    for (int d = 0; d < D; ++d) velb[d] = 0.0;
#pragma unroll
    for (int e = 0; e < 2; ++e) {  /* the faces whose left (e = 0) / right centre point this is */
      const int j = row - (H - 1 + e);
      if (j < 0 || j >= T::FACES) continue;
      const double* r = roe + (e * (D + 2)) * TH + (j * LANES + lanep);
#pragma unroll
      for (int d = 0; d < D; ++d) velb[d] += r[d * TH];
      Hb += r[D * TH];
      sb += r[(D + 1) * TH];
    }
#pragma unroll
    for (int d = 0; d < D; ++d) any |= dbits(velb[d]);
    any |= dbits(Hb) | dbits(sb);
    if ((any & 0x7fffffffffffffffll) == 0) continue;  /* no face of the list touches this point */
    /* alpha = max |lambda| with the argmax frozen: lambda = u_n - c, u_n, u_n + c */
    const double un = sm[(L::cV + AXIS) * NP + p], c = sm[L::cC * NP + p];
    const double ym = xm[0] * dsign(un - c), y0 = xm[1] * dsign(un), yp = xm[2] * dsign(un + c);
    velb[AXIS] += ym + y0 + yp;
    point_vjp<NV, AXIS>(sm, NP, p, A.gamma, Fq, velb, yp - ym, Hb, sb, ub);
    const long long cell = point_cell(p);
#pragma unroll
    for (int v = 0; v < NV; ++v)
      if (ub[v] != 0.0) atomicAdd(A.Z + v * A.ncell + cell, ub[v]);
  }
}

}  // namespace tenom
