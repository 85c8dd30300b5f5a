// The 3D shared-slice variant, FP64, for m <= 64: V slices in shared memory
// (single solves whose slices fit; batches of 3D systems stream V).  Compiled on
// its own so the variants build in parallel.
#include "gmres_kernel.cuh"

namespace mlg {

cudaError_t launch_gmres_d3s(const KParams& kp, int grid, cudaStream_t s) {
  return launch_t<double, 3, kMaxM, 256, kVShared>(kp, grid, s);
}

}  // namespace mlg
