/* Short-line instantiations for the 8-point stencil. */
#include "tenom_line_kernel.cuh"

namespace tenom {

cudaError_t launch_line_k8(const LineArgs& a, int lim, bool pp, cudaStream_t st) { return launch_line_k<8>(a, lim, pp, st); }

}  // namespace tenom
