/* Screen and nonlinear face-sweep instantiations for nvar = 4 (2D Euler). */
#include "tenom_launch.cuh"

namespace tenom {

cudaError_t launch_screen_nv4(const FaceArgs& a, int axis, int K, cudaStream_t st) {
  return launch_screen_nv<4>(a, axis, K, st);
}

cudaError_t launch_nonlinear_nv4(const NonlinArgs& a, int K, int lim, cudaStream_t st) {
  return launch_nonlinear_nv<4, false>(a, K, lim, st);
}

}  // namespace tenom
