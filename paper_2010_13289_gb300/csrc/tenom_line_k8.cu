/* Short-line instantiations for the 8-point stencil. */
#include "tenom_line_kernel.cuh"

namespace tenom {

cudaError_t launch_line_k8(const LineArgs& a, int lim, bool pp, cudaStream_t st) {
  return line_ops_k<8>(lim, pp).launch(a, st);
}
int line_clusters_k8(int n, int lim, bool pp) { return line_ops_k<8>(lim, pp).clusters(n); }

}  // namespace tenom
