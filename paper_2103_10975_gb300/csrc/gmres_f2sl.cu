// The FP32 2D shared-slice variant for long slices (more than two points per
// thread), m <= 64.  Compiled on its own so the variants build in parallel.
#include "gmres_kernel.cuh"

namespace mlg {

cudaError_t launch_gmres_f2sl(const KParams& kp, int grid, cudaStream_t s) {
  return launch_t<float, 2, kMaxM, 256, kVSharedL>(kp, grid, s);
}

}  // namespace mlg
