/* Recording nonlinear-kernel instantiations for nvar = 3 (1D Euler): the listed faces'
 * fluxes plus their fields' frozen-branch linearisation. */
#include "tenom_launch.cuh"

namespace tenom {

cudaError_t launch_nonlinear_rec_nv3(const NonlinArgs& a, int K, int lim, cudaStream_t st) {
  return launch_nonlinear_nv<3, true>(a, K, lim, st);
}

}  // namespace tenom
