/* tenom_rhs_noalloc: the operator dU/dt = L(U) of tenom_rhs for callers that cannot
 * allocate device memory (see include/tenom.h).  Its scratch -- the face-flux buffers of
 * every axis and a status word -- lives in one file-scope device array, so a call needs no
 * context and performs no allocation.  Every GPU that loads this library holds the array
 * (TENOM_NOALLOC_SCRATCH_BYTES) until the process exits. */
#include <cstdio>
#include <mutex>
#include <string>

#include "tenom.h"
#include "tenom_internal.h"
#include "tenom_nonlinear.cuh"

namespace tenom {

/* first 256 bytes: status word, list lengths; then the face buffers, axis after axis; after
   TENOM_NOALLOC_SCRATCH_BYTES the face lists of the nonlinear kernel (5 bytes per face, at most
   (16 MiB / 8) / 3 faces in 1D, 3.4 MiB).  The cell primitives, nvar values per cell, need no room of
   their own: dUdt has their size and is written last, by a kernel that reads faces only. */
static constexpr size_t kListBytes = 4u << 20;
static __device__ __align__(256) double g_noalloc_scratch[(TENOM_NOALLOC_SCRATCH_BYTES + kListBytes) / sizeof(double)];
static_assert(5 * (TENOM_NOALLOC_SCRATCH_BYTES / sizeof(double) / 3 + 1) + 64 <= kListBytes, "face lists fit");

static constexpr long long kStatusDoubles = 256 / sizeof(double);
static constexpr int kMaxDevices = 64;
static std::mutex g_setup_mu;
static double* g_scratch_dev[kMaxDevices];  /* device address of the array, per device */

/* Once per device, with that device current: look up the array's device address.  In
 * host code the symbol g_noalloc_scratch is only a host-side stand-in and must never be
 * handed to a kernel. */
static cudaError_t scratch_for_current_device(double** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_setup_mu);
  if (!g_scratch_dev[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_dev[dev] = static_cast<double*>(p);
  }
  *out = g_scratch_dev[dev];
  return cudaSuccess;
}

}  // namespace tenom

using namespace tenom;

extern "C" tenom_status tenom_rhs_noalloc(const tenom_grid* grid, const tenom_scheme* scheme, const double* U,
                                          double* dUdt, int* status_dev, void* stream) {
  std::string msg;
  tenom_status v = check_grid_scheme(grid, scheme, &msg);
  if (v != TENOM_OK) {
    fprintf(stderr, "tenom_rhs_noalloc: %s\n", msg.c_str());
    return v;
  }
  if (!U || !dUdt || ((uintptr_t)U & 7) || ((uintptr_t)dUdt & 7) || U == dUdt ||
      ((uintptr_t)status_dev & 3)) {
    fprintf(stderr, "tenom_rhs_noalloc: bad pointers\n");
    return TENOM_E_INVALID;
  }
  const int nv = grid->dim + 2;
  const long long ncell = (long long)grid->n[0] * grid->n[1] * grid->n[2];
  long long nface[3] = {0, 0, 0};
  long long need = kStatusDoubles;
  for (int a = 0; a < grid->dim; ++a) {
    nface[a] = ncell / grid->n[a] * (grid->n[a] + 1);
    need += nv * nface[a];
  }
  const long long cap = (long long)(TENOM_NOALLOC_SCRATCH_BYTES / sizeof(double));
  if (need > cap) {
    fprintf(stderr,
            "tenom_rhs_noalloc: grid needs %lld bytes of face scratch, the static scratch holds %lld "
            "(use tenom_create/tenom_rhs for this grid)\n",
            need * (long long)sizeof(double), cap * (long long)sizeof(double));
    return TENOM_E_INVALID;
  }
  double* scratch = nullptr;
  cudaError_t e = scratch_for_current_device(&scratch);
  if (e != cudaSuccess) {
    fprintf(stderr, "tenom_rhs_noalloc: cudaGetSymbolAddress: %s\n", cudaGetErrorString(e));
    return TENOM_E_CUDA;
  }
  cudaStream_t st = (cudaStream_t)stream;
  int* status = status_dev ? status_dev : reinterpret_cast<int*>(scratch);
  unsigned* count = reinterpret_cast<unsigned*>(scratch) + 16;
  if (!status_dev) {
    e = cudaMemsetAsync(status, 0, sizeof(int), st);  /* the shared word keeps the last call's bits */
    if (e != cudaSuccess) return TENOM_E_CUDA;
  }
  double* const P = dUdt;
  double* F[3] = {nullptr, nullptr, nullptr};
  long long off = kStatusDoubles;
  for (int a = 0; a < grid->dim; ++a) {
    F[a] = scratch + off;
    off += nv * nface[a];
  }
  FaceArgs fa;
  memset(&fa, 0, sizeof(fa));
  fa.U = U;
  fa.P = P;
  fa.flags = nullptr;
  fa.status = status;
  for (int d = 0; d < 3; ++d) {
    fa.n[d] = grid->n[d];
    fa.bc[d] = grid->bc[d];
  }
  fa.ncell = ncell;
  fa.gamma = grid->gamma;
  fa.sch = scheme_for_device(*scheme);
  e = launch_primitives(nv, U, ncell, grid->gamma, P, count, status, st);  /* clears the list lengths */
  NonlinArgs na;
  memset(&na, 0, sizeof(na));
  unsigned* list = reinterpret_cast<unsigned*>(scratch + cap);
  uint8_t* mask = reinterpret_cast<uint8_t*>(list + nface[0] + nface[1] + nface[2]);
  for (int a = 0; a < grid->dim && e == cudaSuccess; ++a) {
    fa.Fhat = F[a];
    fa.nface = nface[a];
    fa.list = list;
    fa.mask = mask;
    fa.count = count + a;
    list += nface[a];
    mask += nface[a];
    if (nv == 3) e = launch_screen_nv3(fa, a, scheme->K, st);
    else if (nv == 4) e = launch_screen_nv4(fa, a, scheme->K, st);
    else e = launch_screen_nv5(fa, a, scheme->K, st);
    na.Fhat[a] = F[a];
    na.list[a] = fa.list;
    na.mask[a] = fa.mask;
  }
  na.U = U;
  na.P = P;
  na.count = count;
  na.status = status;
  for (int d = 0; d < 3; ++d) {
    na.n[d] = fa.n[d];
    na.bc[d] = fa.bc[d];
    na.nface[d] = nface[d];
  }
  na.ncell = ncell;
  na.gamma = fa.gamma;
  na.rgm1 = 1.0 / (fa.gamma - 1.0);
  na.dim = grid->dim;
  na.sch = fa.sch;
  if (e == cudaSuccess) {
    if (nv == 3) e = launch_nonlinear_nv3(na, scheme->K, scheme->limiter, st);
    else if (nv == 4) e = launch_nonlinear_nv4(na, scheme->K, scheme->limiter, st);
    else e = launch_nonlinear_nv5(na, scheme->K, scheme->limiter, st);
  }
  if (e == cudaSuccess) e = launch_rhs_divergence(nv, F, grid->n, grid->dx, ncell, nface, dUdt, st);
  if (e != cudaSuccess) {
    fprintf(stderr, "tenom_rhs_noalloc: %s\n", cudaGetErrorString(e));
    return TENOM_E_CUDA;
  }
  return TENOM_OK;
}
