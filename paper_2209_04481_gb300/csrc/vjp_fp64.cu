// vjp_fp64.cu -- FP64 instantiation of the residual VJP.
#include "vjp_launch.cuh"

namespace crn {
cudaError_t launch_vjp_fp64(crn_grid* g, const double* U, const double* Rb, double* Ub, double* Brb,
                            cudaStream_t st, int* nl) {
  return vjp_t<double>(g, U, Rb, Ub, Brb, st, nl);
}
// The scratch of the slope/face/cell passes, if this grid runs them, at its first
// VJP.  1.15 kB per FP64 cell, where the kernels that formed the slopes at the
// faces took 0.94: a shell that fitted then and does not now runs the tiled VJP,
// until a later call outside a stream capture finds the room.
cudaError_t vjp_ensure_scratch(crn_grid* g, cudaStream_t st) {
  if (g->vjp_buf || !vjp_uses_scratch(g)) return cudaSuccess;
  const bool fp64 = g->d.precision == CRN_FP64;
  const size_t bytes = vjp_scratch_elems(g->shape, fp64) * (fp64 ? 8 : 4);
  if (fp64) {
    const char* limit = std::getenv("CRN_VJP_SCRATCH_LIMIT");
    if (limit && bytes > std::strtoull(limit, nullptr, 10)) {
      g->vjp_no_room = true;
      return cudaSuccess;
    }
    if (g->vjp_no_room) {
      cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
      const cudaError_t e = cudaStreamIsCapturing(st, &cap);
      if (e != cudaSuccess || cap != cudaStreamCaptureStatusNone) return e;
    }
  }
  const cudaError_t e = cudaMalloc(&g->vjp_buf, bytes);
  g->vjp_no_room = e == cudaErrorMemoryAllocation && fp64;
  if (!g->vjp_no_room) return e;
  cudaGetLastError();
  g->vjp_buf = nullptr;
  return cudaSuccess;
}
}  // namespace crn
