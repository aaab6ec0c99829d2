/* Face fluxes of a tile of a 1D line inside one CTA: the same two halves as the grid sweeps
 * (tenom_screen.cuh, tenom_nonlinear.cuh) on the tile's points in shared memory, without lists
 * or buffers in device memory.  Used where a line is too short to fill the GPU (line_kernel) and by
 * the batched launch (batch_stage_kernel: 512 Riemann tubes TENO6, 0.84 -> 0.20 ms a stage against the
 * unscreened FP64 flux of every face, now FP64 pipe 75 % busy with the points' primitives, the
 * central fluxes and the cell updates). */
#pragma once
#include "tenom_screen.cuh"
#include "tenom_nonlinear.cuh"
#include "tenom_positivity.cuh"

namespace tenom {

/* shared memory of a tile of at most FACES faces (TILE threads) */
template <int K, int TILE, int FACES = TILE>
struct LineTile {
  static constexpr int NV = 3, NP = FACES + K - 1, W = TILE / 32;
  /* FP64 point data, component c of point p at c * NP + p */
  static constexpr int rho = 0, m = 1, E = 2, un = 3, pr = 4, cs = 5, F1 = 6, F2 = 7, NC = 8;
  double pt[NC * NP];
  double F[NV * TILE];               /* the face fluxes */
  double row[NlRow<NV>::N * TILE];   /* uncertified faces: Roe state and LLF speeds */
  double fs[2 * NV * TILE];          /* their fields' f+ (first half) and f- */
  float sf[ScreenLayout<NV>::NF * NP];
  unsigned cm[2 * TILE];             /* fields central on the f+ side, on the f- side */
  unsigned short item[NV * TILE];    /* (face, field) pairs */
  int wc[NV * W + 1];
};

/* face_rows' view of face jf of the tile */
template <class T, int K>
struct LineFace {
  const double* pt;
  const float* sf;
  int jf;
  __device__ __forceinline__ void centre(int e, double& r, double& c, double (&v)[1]) const {
    const int p = jf + K / 2 - 1 + e;
    r = pt[T::rho * T::NP + p];
    c = pt[T::cs * T::NP + p];
    v[0] = pt[T::un * T::NP + p];
  }
  __device__ __forceinline__ void speed(int q, double& u, double& c) const {
    u = pt[T::un * T::NP + jf + q];
    c = pt[T::cs * T::NP + jf + q];
  }
  __device__ __forceinline__ void speed32(int q, double, double, float& uf, float& cf) const {
    using L = ScreenLayout<3>;
    uf = sf[(L::hi + L::V) * T::NP + jf + q];
    cf = sf[(L::hi + L::C) * T::NP + jf + q];
  }
};

/* Stages the points of faces f0 .. f0 + nf - 1 (nf <= FACES) of a line of n cells at U (component v
   at v * stride; read through L2, other CTAs of a cluster may have written it).  All threads of the
   CTA call it.  Returns the largest |u| + c of the tile's nf - 1 own cells seen by this thread.
   cfl: the CFL maximum is taken here, and a state that is not positive reported as the grid's signal
   speed kernel does (point_prims' integer tests let a NaN pass). */
template <int K, int TILE, int FACES>
__device__ __forceinline__ double line_stage(LineTile<K, TILE, FACES>& S, const double* U, long long stride, int n, int bc,
                                             int f0, int nf, double gamma, int& st, bool cfl = false) {
  using T = LineTile<K, TILE, FACES>;
  constexpr int NV = 3, H = K / 2, NP = T::NP;
  const int tid = threadIdx.x;
  double smax = 0.0;
  const int np = nf + K - 1;
  for (int p = tid; p < np; p += TILE) {
    const int j = bc_wrap(f0 - H + p, n, bc);
    double u[NV], vel[1], pr, cs;
#pragma unroll
    for (int v = 0; v < NV; ++v) u[v] = __ldcg(U + v * stride + j);
    point_prims<NV>(u, gamma, vel, pr, cs, st);
    S.pt[T::rho * NP + p] = u[0];
    S.pt[T::m * NP + p] = u[1];
    S.pt[T::E * NP + p] = u[2];
    S.pt[T::un * NP + p] = vel[0];
    S.pt[T::pr * NP + p] = pr;
    S.pt[T::cs * NP + p] = cs;
    S.pt[T::F1 * NP + p] = fma(u[1], vel[0], pr);
    /* no contraction of u + pr into pr's product, which the grid sweeps load: the same bits */
    S.pt[T::F2 * NP + p] = __dmul_rn(__dadd_rn(u[2], pr), vel[0]);
    stage_screen_point<NV>(u, vel, pr, cs, S.sf, NP, p);
    if (cfl) {
      if (!(u[0] > 0.0)) st |= ST_RHO;
      if (!(pr > 0.0)) st |= ST_P;
    }
    const double s = fabs(vel[0]) + cs;
    if (p >= H && p < H + nf - 1 && f0 - H + p < n && s > smax) smax = s;
  }
  __syncthreads();
  for (int p = tid; p < np - 1; p += TILE) stage_screen_differences<NV>(S.sf, NP, p, 1);
  __syncthreads();
  return smax;
}

/* Fluxes of the staged tile's nf faces (those <= n) into S.F, limited for a stage with mu = 2 dt/dx
   when PP.  ALL: the scheme is not screened (sch.screen = 0).  All threads of the CTA call it; S.F is
   complete on return. */
template <int K, int LIM, int TILE, bool PP, bool ALL = false, int FACES>
__device__ __forceinline__ void line_fluxes(LineTile<K, TILE, FACES>& S, int n, int f0, int nf, double gamma, double rgm1,
                                            const SchemeDev& sch, double mu, int& st) {
  using T = LineTile<K, TILE, FACES>;
  constexpr int NV = 3, H = K / 2, NP = T::NP, W = T::W;
  constexpr unsigned allk = (1u << (K - 2)) - 1u, allf = 7u;
  const int tid = threadIdx.x, wid = tid >> 5, ln = tid & 31;
  const double gm1 = gamma - 1.0;

  /* central flux and certificate, one face per thread; the Roe state where a field is left */
  const bool active = tid < nf && f0 + tid <= n;
  unsigned bad = 0u;
  double Fh[NV];
  if (active) {
    double cw[K];
    central_weights<K>(cw);
    const int comp[NV] = {T::m, T::F1, T::F2};
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const double* s = S.pt + comp[v] * NP + tid;
      Fh[v] = cw[0] * s[0];
#pragma unroll
      for (int q = 1; q < K; ++q) Fh[v] = fma(cw[q], s[q], Fh[v]);
    }
    bad = allf;
    if constexpr (!ALL)
      if (sch.screen) bad = screen_face<NV, K, 0, 1>(S.sf, NP, tid, (float)gm1, sch, false);
    if (bad) {
      const LineFace<T, K> src{S.pt, S.sf, tid};
      face_rows<NV, K, TILE>(src, S.row + tid, gm1, rgm1, st);
    }
  }
  S.cm[tid] = S.cm[TILE + tid] = sch.default_d ? (allf & ~bad) : 0u;
#pragma unroll
  for (int s = 0; s < NV; ++s) {
    const unsigned b = __ballot_sync(0xffffffffu, bad >> s & 1u);
    if (ln == 0) S.wc[s * W + wid] = __popc(b);
  }
  __syncthreads();
  int before[NV], nitem = 0;
#pragma unroll
  for (int s = 0; s < NV; ++s)
#pragma unroll
    for (int w = 0; w < W; ++w) {
      if (w == wid) before[s] = nitem;
      nitem += S.wc[s * W + w];
    }
#pragma unroll
  for (int s = 0; s < NV; ++s) {
    const unsigned b = __ballot_sync(0xffffffffu, bad >> s & 1u);
    if (bad >> s & 1u) S.item[before[s] + __popc(b & ((1u << ln) - 1u))] = (unsigned short)(tid | (s << 9));
  }
  if (nitem) {  /* uniform over the CTA */
    __syncthreads();
    auto project = [&](const double (&l)[NV], int p, double& w, double& hg) {  /* W and G/2 of tile point p */
      const double un = S.pt[T::un * NP + p];
      w = l[0] * S.pt[T::rho * NP + p];
      w = fma(l[1], S.pt[T::m * NP + p], w);
      w = fma(l[2], S.pt[T::E * NP + p], w);
      hg = 0.5 * fma(S.pt[T::pr * NP + p], fma(un, l[2], l[1]), un * w);
    };
    auto reconstruct = [&](const double (&v)[K], int side, int s, int fc) {
      unsigned b = 0u;
      int e = 7;
      if (!teno_decide_fast<K, false>(v, sch, b, e)) teno_decide_fp64<K>(v, sch, b, e, st);
      S.fs[(side * NV + s) * TILE + fc] = teno_general<K, LIM>(v, sch, b);
      if (b == allk && sch.default_d) atomicOr(&S.cm[side * TILE + fc], 1u << s);
    };
    if constexpr (ALL) {
      /* every field of every face: both sides from one projection */
#pragma unroll 1
      for (int it = tid; it < nitem; it += TILE) {
        const int item = S.item[it], fc = item & 511, s = item >> 9;
        double l[NV], w[K], hg[K];
        const double ha = left_vector<NV, TILE>(S.row + fc, s, l);
#pragma unroll
        for (int q = 0; q < K; ++q) project(l, fc + q, w[q], hg[q]);
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {
          double v[K];
#pragma unroll
          for (int q = 0; q < K; ++q) v[q] = side ? fma(-ha, w[K - 1 - q], hg[K - 1 - q]) : fma(ha, w[q], hg[q]);
          reconstruct(v, side, s, fc);
        }
      }
    } else {
      /* one (face, field, side) per thread: a short line is all latency, and projecting a second
         time costs less of it than two sides one after the other */
#pragma unroll 1
      for (int it = tid; it < 2 * nitem; it += TILE) {
        const int side = it >= nitem ? 1 : 0, item = S.item[it - (side ? nitem : 0)], fc = item & 511, s = item >> 9;
        double l[NV], v[K];
        const double ha = left_vector<NV, TILE>(S.row + fc, s, l);
#pragma unroll
        for (int q = 0; q < K; ++q) {
          double w, hg;
          project(l, fc + (side ? K - 1 - q : q), w, hg);  /* f- on the mirrored stencil */
          v[q] = fma(side ? -ha : ha, w, hg);
        }
        reconstruct(v, side, s, fc);
      }
    }
    __syncthreads();
    if (bad) {
      const unsigned cm = S.cm[tid] & S.cm[TILE + tid];
      if (cm != allf) {
#pragma unroll
        for (int s = 0; s < NV; ++s) S.fs[s * TILE + tid] += S.fs[(NV + s) * TILE + tid];
        compose<NV, TILE>(S.row + tid, S.fs + tid, cm, allf & ~cm, Fh);
      }
    }
  }
  if (active) {
    if constexpr (PP) {
      /* positivity limiter on the face between points tid + H - 1 and tid + H; a face computed
         by two tiles is limited identically by both */
      double Ua[NV], Ub[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        Ua[v] = S.pt[(T::rho + v) * NP + tid + H - 1];
        Ub[v] = S.pt[(T::rho + v) * NP + tid + H];
      }
      positivity_face<NV, 0>(Ua, Ub, Fh, mu, gamma, f32_rz(mu), f32_rz(gm1));
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) S.F[v * TILE + tid] = Fh[v];
  }
  __syncthreads();
}

/* ---------------------------------------------------------------- short 1D grids */

struct LineArgs {
  double* U;
  double* W1;           /* stage buffers, [3][n] */
  double* W2;
  const double* dt;     /* one step of this length, or null: CFL steps */
  double* t;            /* time, advanced in place (CFL steps) */
  double t_end, cfl, rdx, gamma, rgm1;
  int n, bc, nsteps;
  int* status;
  SchemeDev sch;
};

/* threads of a CTA of line_kernel (it stages as many points, one round) and CTAs of the cluster
   that covers the line, each an equal share of the cells */
constexpr int LINE_TILE = 128;
constexpr int LINE_CLUSTER = 16;
inline int line_cells_max(int K) { return LINE_CLUSTER * (LINE_TILE - K); }
/* CTAs for a line of n cells: four cells each until the cluster is full */
inline int line_ctas(int n) { return n < 4 * LINE_CLUSTER ? (n + 3) / 4 : LINE_CLUSTER; }
/* Whether a grid advances in line_kernel.  clusters: how many clusters of line_ctas CTAs the device can
   hold at once, as the runtime reports it (16 CTAs are above the portable 8, and a partition of the
   GPU may have no such group of SMs); none: the grid sweeps, which give the same bits. */
inline bool use_line(int nv, long long ncell, int K, int clusters) {
  return nv == 3 && ncell <= line_cells_max(K) && clusters > 0;
}

/* nsteps SSP-RK3 steps of a 1D grid of at most line_cells_max cells in one launch of one cluster,
   and the clusters that fit on the current device (asked once per device and size)
   (tenom_line_k6.cu, tenom_line_k8.cu) */
cudaError_t launch_line_k6(const LineArgs& a, int lim, bool pp, cudaStream_t st);
cudaError_t launch_line_k8(const LineArgs& a, int lim, bool pp, cudaStream_t st);
int line_clusters_k6(int n, int lim, bool pp);
int line_clusters_k8(int n, int lim, bool pp);

}  // namespace tenom
