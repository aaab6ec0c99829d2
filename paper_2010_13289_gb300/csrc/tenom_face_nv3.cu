/* Screen and nonlinear face-sweep instantiations for nvar = 3 (1D Euler). */
#include "tenom_launch.cuh"

namespace tenom {

cudaError_t launch_screen_nv3(const FaceArgs& a, int axis, int K, cudaStream_t st) {
  return launch_screen_nv<3>(a, axis, K, st);
}

cudaError_t launch_nonlinear_nv3(const NonlinArgs& a, int K, int lim, cudaStream_t st) {
  return launch_nonlinear_nv<3, false>(a, K, lim, st);
}

}  // namespace tenom
