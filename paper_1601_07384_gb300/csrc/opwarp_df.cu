// Warp-per-tet operator kernels, binary64-accurate products from binary32 (hi, lo) planes.
#include "opwarp.cuh"

namespace stdg {

cudaError_t warp_prepare_df(stdg_solver* s) { return warp_prepare_t<WDF>(s, &s->wdB, &s->wdA); }

cudaError_t warp_launch_df(stdg_solver* s, const double* x, double* y, int pinned, int kron, double scale,
                             double pin_diag) {
  return launch_warp<WDF>(s, s->wdB, s->wdA, x, y, pinned, kron, scale, pin_diag);
}

}  // namespace stdg
