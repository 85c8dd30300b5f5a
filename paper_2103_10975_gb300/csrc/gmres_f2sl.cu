// The FP32 2D shared-slice variant for long slices (more than eight points per thread, in
// batches four), m <= 64.  Compiled on its own so the variants build in parallel.
// Reached by batches of m = 33 to about 40 (slices of at most 1 250 points): two systems
// of 101^2, m = 36, on 18 CTAs 13.1 ms, with the one-point passes 13.8.
#include "gmres_kernel.cuh"

namespace mlg {

cudaError_t launch_gmres_f2sl(const KParams& kp, int grid, cudaStream_t s) {
  return launch_t<float, 2, kMaxM, 256, kVSharedL>(kp, grid, s);
}

}  // namespace mlg
