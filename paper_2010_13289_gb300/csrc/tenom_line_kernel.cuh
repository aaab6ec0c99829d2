/* SSP-RK3 steps of a short 1D grid in one launch (instances in tenom_line_k6.cu, _k8.cu).
 *
 * A line of a few hundred cells is all latency: twelve launches a step, each a few
 * microseconds of start-up and cold instruction fetch around as much work.  Here one cluster of
 * up to LINE_CLUSTER CTAs keeps the line: a CTA per share of the cells computes the fluxes
 * (line_fluxes) and updates its cells, stage states go through L2, and the stages are separated
 * by the hardware's cluster barrier.  The CFL maximum is exchanged through distributed shared
 * memory.  What is left is the FP64 chain of the few nonlinear faces (an FP64 instruction takes a
 * warp 64 cycles): the cells are split evenly so that as many SMs as possible share them.
 * Measured per step: 256-cell Riemann tube TENO6 190 us (the launches), 127 (screened sweeps), 99
 * (clusters of full tiles), 58 here; 900-cell Le Blanc with the limiter 290, 183, 130, 117.  The
 * line stays in one cluster up to LINE_CLUSTER shares (1920-1952 cells: 75-130 us against 125-185
 * for the launches); with two rounds of tiles per CTA the launches win. */
#pragma once
#include <cooperative_groups.h>
#include "tenom_launch.cuh"
#include "tenom_line.cuh"

namespace tenom {

template <int K, int LIM, bool PP>
__global__ void __launch_bounds__(LINE_TILE) line_kernel(const LineArgs A) {
  namespace cg = cooperative_groups;
  constexpr int TILE = LINE_TILE;
  using T = LineTile<K, TILE, TILE - K + 1>;
  extern __shared__ double dyn[];
  T& S = *reinterpret_cast<T*>(dyn);
  __shared__ double s_warp[TILE / 32];
  __shared__ double s_speed[LINE_CLUSTER];
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank(), tid = threadIdx.x;
  const int n = A.n, share = (n + C - 1) / C;  /* <= TILE - K */
  const int f0 = rank * share, cells = n - f0 < share ? n - f0 : share, nf = cells > 0 ? cells + 1 : 0;
  const int c = f0 + tid;
  int st = 0;
  double t = A.dt ? 0.0 : *A.t;
  cl.sync();  /* every CTA runs before its shared memory is written from another */
#pragma unroll 1
  for (int step = 0; step < A.nsteps; ++step) {
    /* the CFL maximum comes with the first stage's points */
    double dt, m = nf ? line_stage(S, A.U, n, n, A.bc, f0, nf, A.gamma, st, !A.dt) * A.rdx : 0.0;
    if (A.dt) {
      dt = *A.dt;
    } else {  /* dt = min(cfl / max (|u| + c)/dx, t_end - t), 0 once t reaches t_end */
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double x = __shfl_xor_sync(0xffffffffu, m, o);
        m = x > m ? x : m;
      }
      if ((tid & 31) == 0) s_warp[tid >> 5] = m;
      __syncthreads();
      if (tid < C) {
#pragma unroll
        for (int w = 0; w < TILE / 32; ++w) m = s_warp[w] > m ? s_warp[w] : m;
        *cl.map_shared_rank(&s_speed[rank], tid) = m;
      }
      cl.sync();
      m = 0.0;
      for (int r = 0; r < C; ++r) m = s_speed[r] > m ? s_speed[r] : m;
      dt = A.cfl / m;
      const double rem = A.t_end - t;
      dt = rem < dt ? rem : dt;
      if (!(rem > 0.0)) dt = 0.0;
    }
#pragma unroll 1
    for (int stage = 0; stage < 3; ++stage) {
      const double* Us = stage == 0 ? A.U : (stage == 1 ? A.W1 : A.W2);
      double* out = stage == 0 ? A.W1 : (stage == 1 ? A.W2 : A.U);
      const double cA = stage == 1 ? 0.75 : 1.0 / 3.0, cB = stage == 1 ? 0.25 : 2.0 / 3.0;
      if (nf) {
        if (stage > 0) line_stage(S, Us, n, n, A.bc, f0, nf, A.gamma, st);
        line_fluxes<K, LIM, TILE, PP>(S, n, f0, nf, A.gamma, A.rgm1, A.sch, 2.0 * dt * A.rdx, st);
        if (tid < cells && dt != 0.0) {
#pragma unroll
          for (int v = 0; v < 3; ++v) {
            const long long g = (long long)v * n + c;
            const double r = 0.0 - (S.F[v * TILE + tid + 1] - S.F[v * TILE + tid]) * A.rdx;
            const double t1 = __ldcg(Us + g) + dt * r;
            /* rounded as stage_kernel's cA U0 + cB t1 is: a step has the bits of the grid sweeps' */
            __stcg(out + g, stage == 0 ? t1 : fma(cA, __ldcg(A.U + g), __dmul_rn(cB, t1)));
          }
        }
      }
      if (dt == 0.0) break;
      cl.sync();  /* the stage's state is complete, and S free */
    }
    /* nothing moves, now or in a later step (the same on every CTA); the fluxes of the state were
       formed once for what they report */
    if (dt == 0.0) break;
    t = t + dt;
  }
  cl.sync();  /* no CTA leaves while another may still write its shared memory */
  if (!A.dt && rank == 0 && tid == 0) *A.t = t;
  if (st) atomicOr(A.status, st);
}

template <int K, int LIM, bool PP>
struct LineLaunch {
  static constexpr size_t smem = sizeof(LineTile<K, LINE_TILE, LINE_TILE - K + 1>);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  LineLaunch(int n, cudaStream_t st) {
    cfg.gridDim = dim3((unsigned)line_ctas(n));
    cfg.blockDim = dim3(LINE_TILE);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cfg.gridDim.x;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
  static cudaError_t prepare() {
    static AttrOnce attr;
    return ensure_smem_attr(line_kernel<K, LIM, PP>, attr, smem, true);
  }
  static cudaError_t launch(const LineArgs& a, cudaStream_t st) {
    const cudaError_t e = prepare();
    if (e != cudaSuccess) return e;
    const LineLaunch l(a.n, st);
    return cudaLaunchKernelEx(&l.cfg, line_kernel<K, LIM, PP>, a);
  }
  static int clusters(int n) {
    static std::atomic<signed char> known[AttrOnce::kMaxDevices][LINE_CLUSTER + 1];  /* 0: not asked, else 1 + clusters (0 or 1) */
    int dev = -1, fit = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= AttrOnce::kMaxDevices) return 0;
    std::atomic<signed char>& k = known[dev][line_ctas(n)];
    if (const signed char v = k.load(std::memory_order_relaxed)) return v - 1;
    const LineLaunch l(n, nullptr);
    cudaError_t e = prepare();
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&fit, line_kernel<K, LIM, PP>, &l.cfg);
    if (e != cudaSuccess) {
      (void)cudaGetLastError();
      fit = 0;
    }
    k.store((signed char)(fit > 0 ? 2 : 1), std::memory_order_relaxed);
    return fit > 0 ? 1 : 0;
  }
};

struct LineOps {
  cudaError_t (*launch)(const LineArgs&, cudaStream_t);
  int (*clusters)(int);
};
template <int K, int LIM>
static LineOps line_ops(bool pp) {
  if (pp) return {LineLaunch<K, LIM, true>::launch, LineLaunch<K, LIM, true>::clusters};
  return {LineLaunch<K, LIM, false>::launch, LineLaunch<K, LIM, false>::clusters};
}
template <int K>
static LineOps line_ops_k(int lim, bool pp) {
  if (lim == LIM_MP) return line_ops<K, LIM_MP>(pp);
  if (lim == LIM_TVD5) return line_ops<K, LIM_TVD5>(pp);
  return line_ops<K, LIM_VA>(pp);
}

}  // namespace tenom
