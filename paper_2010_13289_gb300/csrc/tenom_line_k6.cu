/* Short-line instantiations for the 6-point stencil. */
#include "tenom_line_kernel.cuh"

namespace tenom {

cudaError_t launch_line_k6(const LineArgs& a, int lim, bool pp, cudaStream_t st) {
  return line_ops_k<6>(lim, pp).launch(a, st);
}
int line_clusters_k6(int n, int lim, bool pp) { return line_ops_k<6>(lim, pp).clusters(n); }

}  // namespace tenom
