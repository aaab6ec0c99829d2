/* Adjoint instantiations for nvar = 3 (flags and linearisation tape). */
#include "tenom_launch.cuh"

namespace tenom {

cudaError_t launch_adj_nv3(const AdjArgs& a, int axis, int K, int lim, cudaStream_t st) {
  return launch_adj_nv<3>(a, axis, K, lim, st);
}

}  // namespace tenom
