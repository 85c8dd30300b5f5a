// The FP32 2D shared-slice variant for long slices (more than eight points per thread, in
// batches four), m <= 32.  Compiled on its own so the variants build in parallel.
#include "gmres_kernel.cuh"

namespace mlg {

cudaError_t launch_gmres_f2sl32(const KParams& kp, int grid, cudaStream_t s) {
  return launch_t<float, 2, kSmallM, 256, kVSharedL>(kp, grid, s);
}

}  // namespace mlg
