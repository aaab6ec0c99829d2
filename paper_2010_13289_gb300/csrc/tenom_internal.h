/* Internal declarations shared by the library's translation units. */
#pragma once
#include <cuda_runtime.h>
#include "tenom_face.cuh"

namespace tenom {

struct NonlinArgs;
/* The screen of one axis (K = 6 or 8), also recording the linearisation when a.lin is set. */
cudaError_t launch_screen_nv3(const FaceArgs& a, int axis, int K, cudaStream_t st);
cudaError_t launch_screen_nv4(const FaceArgs& a, int axis, int K, cudaStream_t st);
cudaError_t launch_screen_nv5(const FaceArgs& a, int axis, int K, cudaStream_t st);
/* The faces the screens listed, every axis in one launch (K, limiter). */
cudaError_t launch_nonlinear_nv3(const NonlinArgs& a, int K, int lim, cudaStream_t st);
cudaError_t launch_nonlinear_nv4(const NonlinArgs& a, int K, int lim, cudaStream_t st);
cudaError_t launch_nonlinear_nv5(const NonlinArgs& a, int K, int lim, cudaStream_t st);
/* The same, also writing the linearisation of the listed fields to a.lin (record kernels). */
cudaError_t launch_nonlinear_rec_nv3(const NonlinArgs& a, int K, int lim, cudaStream_t st);
cudaError_t launch_nonlinear_rec_nv4(const NonlinArgs& a, int K, int lim, cudaStream_t st);
cudaError_t launch_nonlinear_rec_nv5(const NonlinArgs& a, int K, int lim, cudaStream_t st);
/* Decision statistics (tenom_stats.cuh) added to a.stats; no fluxes. */
cudaError_t launch_stats_nv3(const FaceArgs& a, int axis, int K, int lim, cudaStream_t st);
cudaError_t launch_stats_nv4(const FaceArgs& a, int axis, int K, int lim, cudaStream_t st);
cudaError_t launch_stats_nv5(const FaceArgs& a, int axis, int K, int lim, cudaStream_t st);

/* Launch geometry of a face sweep (kept in one place for the tests of the host logic):
   tiles over the n_a + 1 faces of a line, or over n_a faces (wrapped: the screen of a
   periodic axis, whose face n_a is face 0's copy); fwd_tile: the screen's tiles (fx_faces(K, nv)
   along x; FWD_LANES x columns in y/z), else FX_FACES along x and 32 x columns x ft_faces(K). */
inline void face_grid(int nv, int axis, const int* n, int K, dim3* grid, dim3* block, bool wrapped = false,
                      bool fwd_tile = false) {
  const int nf = n[axis] + (wrapped ? 0 : 1);
  if (axis == 0) {
    const int fx = fwd_tile ? fx_faces(K, nv) : FX_FACES;
    *block = dim3(fx);
    *grid = dim3((unsigned)(n[1] * n[2]), (unsigned)((nf + fx - 1) / fx));
  } else {
    const int other = (axis == 1) ? n[2] : n[1];
    const int lanes = fwd_tile ? FWD_LANES : 32;
    const int ft = fwd_tile ? fx_faces(K, nv) / FWD_LANES : ft_faces(K);
    *block = dim3(lanes * ft);
    *grid = dim3((unsigned)((n[0] + lanes - 1) / lanes), (unsigned)((nf + ft - 1) / ft), (unsigned)other);
  }
}

}  // namespace tenom

#include <string>
#include "tenom.h"

namespace tenom {
/* Argument checks of tenom_create, usable without a context. */
tenom_status check_grid_scheme(const tenom_grid* g, const tenom_scheme* s, std::string* msg);
/* Device copy of a scheme (all-zero d_k replaced by the maximal-order weights). */
SchemeDev scheme_for_device(const tenom_scheme& s);
/* The forward sweeps' cell primitives of U (velocity, p, c: [nv][ncell]) into P; clears the three
   list lengths at count. */
cudaError_t launch_primitives(int nv, const double* U, long long ncell, double gamma, double* P, unsigned* count,
                              int* status, cudaStream_t st);
/* dUdt = -sum_a (F_a[f+1] - F_a[f]) / dx_a from face buffers F[a] ([nv][nface_a]). */
cudaError_t launch_rhs_divergence(int nv, double* const F[3], const int n[3], const double dx[3], long long ncell,
                                  const long long nface[3], double* out, cudaStream_t st);
}  // namespace tenom

namespace tenom {
struct AdjArgs;
/* Adjoint launches: axis < 0 writes the central part of L'(U)^T w (all axes) to a.Z; axis >= 0 adds the
   axis's nonlinear fields, from a.lin (the recorded linearisation) when set, else from a.flags. */
cudaError_t launch_adj_nv3(const AdjArgs& a, int axis, int K, int lim, cudaStream_t st);
cudaError_t launch_adj_nv4(const AdjArgs& a, int axis, int K, int lim, cudaStream_t st);
cudaError_t launch_adj_nv5(const AdjArgs& a, int axis, int K, int lim, cudaStream_t st);
}  // namespace tenom
