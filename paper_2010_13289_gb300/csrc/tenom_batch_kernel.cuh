/* The batched SSP-RK3 stage kernel (see tenom_batch.cu), shared by the translation units
   that instantiate it: tenom_batch.cu (without the positivity limiter) and
   tenom_batch_pp.cu (with it). */
#pragma once
#include "tenom_internal.h"
#include "tenom_line.cuh"

namespace tenom {

struct BatchArgs {
  const int* n;
  const long long* off;
  const double* dx;
  const int* bc;
  const double* dt;
  const int2* items;
  int nitems;
  int* counter;
  int* status;
  long long total;
  double gamma;
  double rgm1;  /* 1 / (gamma - 1) */
  SchemeDev sch;
};

/* stage: 1 -> out = Us + dt L(Us); 2,3 -> out = cA U0 + cB (Us + dt L(Us)).  Compiled for
   512 resident threads per SM (128 registers a thread), so that the autotuner's CTA counts
   can reach 16 warps per SM.  ALL: schemes without a screen (FP64 decisions, d_k of the caller's): 512 tubes
   TENO6 with FP64 decisions 2.25 ms a step when projected once a side as the screened tiles are,
   1.97 with every face by itself. */
template <int K, int LIM, int TILE, bool PP, bool ALL>
__global__ void __launch_bounds__(TILE, 512 / TILE)
batch_stage_kernel(const BatchArgs A, const double* __restrict__ Us, const double* __restrict__ U0, double* out,
                   int mode, double cA, double cB) {
  constexpr int NV = 3;
  extern __shared__ double dyn[];
  LineTile<K, TILE>& S = *reinterpret_cast<LineTile<K, TILE>*>(dyn);
  __shared__ int s_item;
  const int tid = threadIdx.x;
  int st = 0;
  for (;;) {
    if (tid == 0) s_item = atomicAdd(A.counter, 1);
    __syncthreads();
    const int it = s_item;
    __syncthreads();
    if (it >= A.nitems) break;
    const int2 w = A.items[it];
    const int j = w.x, f0 = w.y;
    const double dt = A.dt[j];
    if (dt == 0.0) continue;  /* finished problem (uniform across the CTA) */
    const int n = A.n[j];
    const long long off = A.off[j];
    const double rdx = 1.0 / A.dx[j];
    line_stage(S, Us + off, A.total, n, A.bc[j], f0, TILE, A.gamma, st);
    line_fluxes<K, LIM, TILE, PP, ALL>(S, n, f0, TILE, A.gamma, A.rgm1, A.sch, 2.0 * dt * rdx, st);
    const int c = f0 + tid;
    if (tid < TILE - 1 && c < n) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const double r = 0.0 - (S.F[v * TILE + tid + 1] - S.F[v * TILE + tid]) * rdx;
        const long long g = v * A.total + off + c;
        const double t1 = Us[g] + dt * r;
        out[g] = (mode == 1) ? t1 : cA * U0[g] + cB * t1;
      }
    }
    __syncthreads();
  }
  if (st) atomicOr(A.status, st);
}

using StageFn = void (*)(const BatchArgs, const double*, const double*, double*, int, double, double);

/* the stage kernel of K in {6, 8}, LIM in {MP, TVD5}, TILE in {64, 128, 256}; null for other combinations */
template <bool PP, bool ALL>
static StageFn pick_stage_of(int K, int lim, int tile) {
#define TENOM_PICK(KK, LL, TT) if (K == KK && lim == LL && tile == TT) return batch_stage_kernel<KK, LL, TT, PP, ALL>;
  TENOM_PICK(6, LIM_MP, 64) TENOM_PICK(6, LIM_MP, 128) TENOM_PICK(6, LIM_MP, 256)
  TENOM_PICK(6, LIM_TVD5, 64) TENOM_PICK(6, LIM_TVD5, 128) TENOM_PICK(6, LIM_TVD5, 256)
  TENOM_PICK(8, LIM_MP, 64) TENOM_PICK(8, LIM_MP, 128) TENOM_PICK(8, LIM_MP, 256)
  TENOM_PICK(8, LIM_TVD5, 64) TENOM_PICK(8, LIM_TVD5, 128) TENOM_PICK(8, LIM_TVD5, 256)
#undef TENOM_PICK
  return nullptr;
}
/* the same with the positivity limiter (tenom_batch_pp.cu) */
StageFn pick_stage_pp(int K, int lim, int tile, bool all);

}  // namespace tenom
