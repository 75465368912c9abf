// FP64 Brillouin stencil.
#include "bri_split.cuh"

namespace bri {
int launch_bri_f64(const Geom& g, double* y, const double* x, const double2* W, const double* cl, double diag, int nrhs,
                   int dagger, cudaStream_t s, const ShiftDot<double>* sd, int* sd_blocks) {
  return launch_split<double, double2>(g, y, x, W, cl, diag, nrhs, dagger, s, sd, sd_blocks);
}
}  // namespace bri
