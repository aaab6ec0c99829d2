/* Host-side launchers of the face sweeps and their adjoints, templated on the Euler system (NV = 3, 4, 5 for
 * 1D, 2D, 3D); each tenom_*_nvN.cu file instantiates one NV so the kernels compile in
 * parallel.  Dynamic shared memory above 48 KB is opted into once per kernel and device:
 * the attribute belongs to the device's context, so a process that launches on a second
 * GPU sets it there too. */
#pragma once
#include <atomic>
#include <mutex>
#include "tenom_internal.h"
#include "tenom_screen.cuh"
#include "tenom_nonlinear.cuh"
#include "tenom_adjoint.cuh"

namespace tenom {

/* Per kernel: whether its shared-memory attribute has been set on each device.  Readers
   take the flag without the lock; the first launch on a device sets the attribute under
   the lock and only then publishes the flag. */
struct AttrOnce {
  static constexpr int kMaxDevices = 64;
  std::atomic<bool> done[kMaxDevices];
  std::mutex mu;
  AttrOnce() {
    for (auto& d : done) d.store(false, std::memory_order_relaxed);
  }
};

template <class Kern>
static cudaError_t ensure_smem_attr(Kern kern, AttrOnce& attr, size_t smem, bool wide_cluster = false) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= AttrOnce::kMaxDevices) return cudaErrorInvalidDevice;
  if (attr.done[dev].load(std::memory_order_acquire)) return cudaSuccess;
  std::lock_guard<std::mutex> lock(attr.mu);
  if (attr.done[dev].load(std::memory_order_relaxed)) return cudaSuccess;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess && wide_cluster) /* clusters of more than 8 CTAs */
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  attr.done[dev].store(true, std::memory_order_release);
  return cudaSuccess;
}

template <class Kern>
static cudaError_t launch_tile(Kern kern, AttrOnce& attr, size_t smem, int nv, int axis, const int* n, int K,
                               cudaStream_t st, const void* args_ptr, bool wrapped = false,
                               bool fwd_tile = false) {
  cudaError_t e = ensure_smem_attr(kern, attr, smem);
  if (e != cudaSuccess) return e;
  dim3 grid, block;
  face_grid(nv, axis, n, K, &grid, &block, wrapped, fwd_tile);
  void* argv[1] = {const_cast<void*>(args_ptr)};
  return cudaLaunchKernel((const void*)kern, grid, block, argv, smem, st);
}

/* screen of one axis (REC: also record the linearisation of the certified fields) */
template <int NV, int K, int AXIS, bool REC>
static cudaError_t launch_screen_one(const FaceArgs& a, cudaStream_t st) {
  static AttrOnce attr;
  return launch_tile(screen_kernel<NV, K, AXIS, REC>, attr, screen_smem<NV, K, AXIS>(), NV, AXIS, a.n, K, st, &a,
                     a.bc[AXIS] == 0, true);
}

template <int NV, int K, bool REC>
static cudaError_t launch_screen_k(const FaceArgs& a, int axis, cudaStream_t st) {
  if (axis == 0) return launch_screen_one<NV, K, 0, REC>(a, st);
  if constexpr (NV >= 4)
    if (axis == 1) return launch_screen_one<NV, K, 1, REC>(a, st);
  if constexpr (NV >= 5)
    if (axis == 2) return launch_screen_one<NV, K, 2, REC>(a, st);
  return cudaErrorNotSupported;
}

template <int NV>
static cudaError_t launch_screen_nv(const FaceArgs& a, int axis, int K, cudaStream_t st) {
  if (K == 6) return a.lin ? launch_screen_k<NV, 6, true>(a, axis, st) : launch_screen_k<NV, 6, false>(a, axis, st);
  return a.lin ? launch_screen_k<NV, 8, true>(a, axis, st) : launch_screen_k<NV, 8, false>(a, axis, st);
}

/* the listed faces of every axis */
template <int NV, int K, int LIM, bool REC, bool FIX>
static cudaError_t launch_nonlinear_one(const NonlinArgs& a, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  nonlinear_kernel<NV, K, LIM, REC, FIX><<<sms * NL_CTAS_PER_SM, NL_THREADS, 0, st>>>(a);
  return cudaGetLastError();
}

template <int NV, int K, bool REC>
static cudaError_t launch_nonlinear_k(const NonlinArgs& a, int lim, cudaStream_t st) {
  if constexpr (NV > 3) {  /* a line's few listed faces are latency-bound: 45 us a launch in fixed point, 30 in FP64 */
    if (a.sch.fixed) {
      if (lim == LIM_MP) return launch_nonlinear_one<NV, K, LIM_MP, REC, true>(a, st);
      if (lim == LIM_TVD5) return launch_nonlinear_one<NV, K, LIM_TVD5, REC, true>(a, st);
    }
  }
  if constexpr (!REC) {
    /* Van Albada: forward only (no frozen linear form to record) */
    if (lim == LIM_VA) return launch_nonlinear_one<NV, K, LIM_VA, false, false>(a, st);
  }
  if (lim == LIM_MP) return launch_nonlinear_one<NV, K, LIM_MP, REC, false>(a, st);
  if (lim == LIM_TVD5) return launch_nonlinear_one<NV, K, LIM_TVD5, REC, false>(a, st);
  return cudaErrorNotSupported;
}

template <int NV, bool REC>
static cudaError_t launch_nonlinear_nv(const NonlinArgs& a, int K, int lim, cudaStream_t st) {
  if (K == 6) return launch_nonlinear_k<NV, 6, REC>(a, lim, st);
  if (K == 8) return launch_nonlinear_k<NV, 8, REC>(a, lim, st);
  return cudaErrorNotSupported;
}

/* decision statistics */
template <int NV, int K, int LIM, int AXIS>
static cudaError_t launch_stats_one(const FaceArgs& a, cudaStream_t st) {
  static AttrOnce attr;
  return launch_tile(stats_kernel<NV, K, LIM, AXIS>, attr, FaceTile<NV, K, AXIS>::SMEM, NV, AXIS, a.n, K, st, &a);
}

template <int NV, int AXIS>
static cudaError_t launch_stats_axis(const FaceArgs& a, int K, int lim, cudaStream_t st) {
  if (K == 6) {
    if (lim == LIM_MP) return launch_stats_one<NV, 6, LIM_MP, AXIS>(a, st);
    if (lim == LIM_TVD5) return launch_stats_one<NV, 6, LIM_TVD5, AXIS>(a, st);
    if (lim == LIM_VA) return launch_stats_one<NV, 6, LIM_VA, AXIS>(a, st);
  } else if (K == 8) {
    if (lim == LIM_MP) return launch_stats_one<NV, 8, LIM_MP, AXIS>(a, st);
    if (lim == LIM_TVD5) return launch_stats_one<NV, 8, LIM_TVD5, AXIS>(a, st);
    if (lim == LIM_VA) return launch_stats_one<NV, 8, LIM_VA, AXIS>(a, st);
  }
  return cudaErrorNotSupported;
}

template <int NV>
static cudaError_t launch_stats_nv(const FaceArgs& a, int axis, int K, int lim, cudaStream_t st) {
  if (axis == 0) return launch_stats_axis<NV, 0>(a, K, lim, st);
  if constexpr (NV >= 4)
    if (axis == 1) return launch_stats_axis<NV, 1>(a, K, lim, st);
  if constexpr (NV >= 5)
    if (axis == 2) return launch_stats_axis<NV, 2>(a, K, lim, st);
  return cudaErrorNotSupported;
}

/* reverse of the axis's nonlinear fields (from a.lin, else from a.flags) */
template <int NV, int K, int LIM, int AXIS, bool TAPE, int YZ>
static cudaError_t launch_adj_fields_tile(const AdjArgs& a, cudaStream_t st) {
  using T = AdjTile<NV, K, AXIS, YZ>;
  static AttrOnce attr;
  const cudaError_t e = ensure_smem_attr(adj_fields_kernel<NV, K, LIM, AXIS, TAPE, YZ>, attr, T::SMEM);
  if (e != cudaSuccess) return e;
  const unsigned tiles = (unsigned)((a.n[AXIS] + T::FACES) / T::FACES);  /* n_a + 1 faces */
  const dim3 grid = AXIS == 0 ? dim3((unsigned)(a.n[1] * a.n[2]), tiles)
                              : dim3((unsigned)((a.n[0] + T::LANES - 1) / T::LANES), tiles, (unsigned)(AXIS == 1 ? a.n[2] : a.n[1]));
  adj_fields_kernel<NV, K, LIM, AXIS, TAPE, YZ><<<grid, T::THREADS, T::SMEM, st>>>(a);
  return cudaGetLastError();
}
template <int NV, int K, int LIM, int AXIS, bool TAPE>
static cudaError_t launch_adj_fields_one(const AdjArgs& a, cudaStream_t st) {
  if constexpr (TAPE && AXIS > 0) {  /* fewer tiles of 256 faces than two a SM: tiles of 128 */
    if (a.nface < 2ll * 152 * 256) return launch_adj_fields_tile<NV, K, LIM, AXIS, TAPE, 8>(a, st);
  }
  return launch_adj_fields_tile<NV, K, LIM, AXIS, TAPE, 16>(a, st);
}

template <int NV, int K, int AXIS>
static cudaError_t launch_adj_fields_k(const AdjArgs& a, int lim, cudaStream_t st) {
  if (a.lin) return launch_adj_fields_one<NV, K, LIM_MP, AXIS, true>(a, st);  /* no limiter dependence */
  if (lim == LIM_MP) return launch_adj_fields_one<NV, K, LIM_MP, AXIS, false>(a, st);
  if (lim == LIM_TVD5) return launch_adj_fields_one<NV, K, LIM_TVD5, AXIS, false>(a, st);
  return cudaErrorNotSupported;
}

template <int NV, int AXIS>
static cudaError_t launch_adj_axis(const AdjArgs& a, int K, int lim, cudaStream_t st) {
  return K == 6 ? launch_adj_fields_k<NV, 6, AXIS>(a, lim, st) : launch_adj_fields_k<NV, 8, AXIS>(a, lim, st);
}

/* axis < 0: the central part (all axes), which writes a.Z; else the axis's fields added to it */
template <int NV>
static cudaError_t launch_adj_nv(const AdjArgs& a, int axis, int K, int lim, cudaStream_t st) {
  if (axis < 0) {
    const long long b = (a.ncell + 255) / 256;
    const unsigned grid = (unsigned)(b < 152 * 64 ? b : 152 * 64);
    if (K == 6) adj_central_kernel<NV, 6><<<grid, 256, 0, st>>>(a);
    else adj_central_kernel<NV, 8><<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
  }
  if (axis == 0) return launch_adj_axis<NV, 0>(a, K, lim, st);
  if constexpr (NV >= 4)
    if (axis == 1) return launch_adj_axis<NV, 1>(a, K, lim, st);
  if constexpr (NV >= 5)
    if (axis == 2) return launch_adj_axis<NV, 2>(a, K, lim, st);
  return cudaErrorNotSupported;
}

}  // namespace tenom
