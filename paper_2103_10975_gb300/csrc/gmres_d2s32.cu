// The FP64 shared-slice variant (2D, V slices in shared memory) instantiated
// for restart lengths m <= 32: a smaller shared state (R and the Hessenberg
// matrix take 17 KB instead of 66 KB), so larger slices of V fit, and half the
// buckets of j.  Compiled on its own so the variants build in parallel.
#include "gmres_kernel.cuh"

namespace mlg {

cudaError_t launch_gmres_d2s32(const KParams& kp, int grid, cudaStream_t s) {
  return launch_t<double, 2, kSmallM, 256, kVShared>(kp, grid, s);
}

}  // namespace mlg
