#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace mlg {
cudaError_t launch_sumsq(const double* b, int N, double* out, cudaStream_t s);
// u = b / rms(b); *sumsq receives the sum of squares, part is scratch for
// kNormParts doubles.
constexpr int kNormParts = 152;
cudaError_t launch_normalise(const double* b, int N, double* part, double* sumsq, float* u,
                             cudaStream_t s);
cudaError_t launch_denormalise(const float* y, int N, const double* sumsq, double scale,
                               double* x, cudaStream_t s);
// `sweeps` damped-Jacobi sweeps on x, with tmp as the other buffer; *result is
// the one of the two that holds the outcome.
cudaError_t launch_jacobi(int dim, int n, const float* kappa, const double* b, double* x,
                          double* tmp, double omega, int sweeps, double** result,
                          cudaStream_t s);
cudaError_t launch_store_pair(const double* b, const double* x, int N, const double* sumsq,
                              float* u, float* t, cudaStream_t s);
cudaError_t launch_spread_dots(const double* x, const float* ring, long long stride,
                               const int* slots, int count, int N, double* out, cudaStream_t s);
}  // namespace mlg
