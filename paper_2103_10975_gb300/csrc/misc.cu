// Small vector kernels around the solver: the input normalisation of the
// learned guess (s = rms(b), u = b/s, x0 = s y), replay-ring stores and the
// dot products of the spread check (Sec. 2.2).
#include <atomic>

#include "misc.h"

namespace mlg {

static std::atomic<long long> g_launches{0};
void note_launches(long long k) { g_launches.fetch_add(k, std::memory_order_relaxed); }
long long launches_so_far() { return g_launches.load(std::memory_order_relaxed); }

// sum of squares of b into *out (one CTA, fixed order: deterministic).
__global__ void sumsq_kernel(const double* __restrict__ b, int N, double* out) {
  __shared__ double red[32];
  double s = 0.0;
  for (int i = threadIdx.x; i < N; i += blockDim.x) s += b[i] * b[i];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = threadIdx.x < (int)(blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
    s = warp_sum(s);
    if (threadIdx.x == 0) *out = s;
  }
}

// Partial sums of squares, one per CTA (fixed order: deterministic).
__global__ void __launch_bounds__(256) sumsq_part_kernel(const double* __restrict__ b, int N,
                                                         double* __restrict__ part) {
  __shared__ double red[8];
  double s = 0.0;
  for (int i = blockIdx.x * 256 + threadIdx.x; i < N; i += gridDim.x * 256) s += b[i] * b[i];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; w++) s += red[w];
    part[blockIdx.x] = s;
  }
}

// u = b / s with s = sqrt(sumsq / N) (s = 1 when b = 0); sumsq is the sum of the
// nparts partials, which every CTA adds up for itself (the same tree in each) and
// the first one stores.  (One CTA over all of b took 20 us at 256^2.)
__global__ void __launch_bounds__(256) normalise_kernel(const double* __restrict__ b, int N,
                                                        const double* __restrict__ part,
                                                        int nparts, double* __restrict__ sumsq,
                                                        float* __restrict__ u) {
  __shared__ double sh;
  if (threadIdx.x < 32) {
    double v = 0.0;
    for (int k = threadIdx.x; k < nparts; k += 32) v += part[k];
    v = warp_sum(v);
    if (threadIdx.x == 0) {
      if (blockIdx.x == 0) *sumsq = v;
      sh = sqrt(v / N);
    }
  }
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  double s = sh;
  if (!(s > 0.0)) s = 1.0;
  u[i] = (float)(b[i] / s);
}

// x = scale s y
__global__ void denormalise_kernel(const float* __restrict__ y, int N, const double* sumsq,
                                   double scale, double* __restrict__ x) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  double s = sqrt(*sumsq / N);
  if (!(s > 0.0)) s = 1.0;
  x[i] = scale * s * (double)y[i];
}

// Damped Jacobi on the 2D operator: out = in + omega/d (b - A in), d = 4/h^2 the
// diagonal of A.  s2 = 1/h^2 and f = omega/(4 s2) come from the host (the same
// IEEE divisions, once per launch instead of three FP64 divisions per point on a
// GPU whose FP64 pipe is narrow).  By differences from the neighbours: on a smooth
// iterate they are nearly exact, so a sweep adds little but the rounding of its last
// addition (32 sweeps at 256^2 against extended precision: 6e-17 of the iterate's norm).  A
// weighted sum of the five points takes five operations instead of nine (the guess
// 186 us instead of 218) and rounds to 9e-17: not used.
//
// One sweep, a thread per point.
__global__ void jacobi_kernel(int n, const double* __restrict__ b, const double* __restrict__ xin,
                              double* __restrict__ xout, double s2, double f) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n * n) return;
  const int ix = i % n, iy = i / n;
  const double c = xin[i];
  const double l = ix > 0 ? xin[i - 1] : 0.0;
  const double r = ix < n - 1 ? xin[i + 1] : 0.0;
  const double d = iy > 0 ? xin[i - n] : 0.0;
  const double t = iy < n - 1 ? xin[i + n] : 0.0;
  const double ax = s2 * (((c - l) + (c - r)) + ((c - d) + (c - t)));
  xout[i] = c + f * (b[i] - ax);
}

// Up to S damped-Jacobi sweeps of the 2D operator in one launch: a CTA loads its
// TW x TH tile with a halo of S points (x and b) into shared memory and sweeps
// there, the valid region shrinking by one point per sweep, so no sweep waits for
// another CTA and the tile goes through L2 once per S sweeps.  The same FP64
// operations per point whatever the tile or the number of sweeps per launch.  The halo
// is computed redundantly ((TW + 2 (S - s)) (TH + 2 (S - s)) points in sweep s: 1.4 x
// the tile at 32 x 16, S = 4).  32 sweeps at 256^2: 32 launches of one sweep 147 us, 8
// of four 112 (the whole guess 310 -> 276, and 218 with what its other kernels gained).
template <int TW, int TH, int S>
__global__ void __launch_bounds__(256) jacobi_tile_kernel(int n, const double* __restrict__ b,
                                                          const double* __restrict__ xin,
                                                          double* __restrict__ xout, double s2,
                                                          double f, int sweeps) {
  constexpr int RW = TW + 2 * S, RH = TH + 2 * S;
  __shared__ double sb[RH * RW], sx[2][RH * RW];
  const int gx0 = (int)blockIdx.x * TW - S, gy0 = (int)blockIdx.y * TH - S;
  for (int p = threadIdx.x; p < RH * RW; p += 256) {
    const int x = gx0 + p % RW, y = gy0 + p / RW;
    const bool in = x >= 0 && x < n && y >= 0 && y < n;
    const long long g = (long long)y * n + x;
    sb[p] = in ? b[g] : 0.0;
    sx[0][p] = in ? xin[g] : 0.0;
    sx[1][p] = 0.0;  // (points outside the grid stay 0 in both buffers)
  }
#pragma unroll
  for (int s = 1; s <= S; s++) {
    if (s > sweeps) break;
    __syncthreads();
    const double* __restrict__ u = sx[(s - 1) & 1];
    double* __restrict__ v = sx[s & 1];
    const int w = RW - 2 * s, cnt = w * (RH - 2 * s);
    for (int p = threadIdx.x; p < cnt; p += 256) {
      const int lx = s + p % w, ly = s + p / w;
      const int x = gx0 + lx, y = gy0 + ly;
      if (x < 0 || x >= n || y < 0 || y >= n) continue;
      const int q = ly * RW + lx;
      const double c = u[q], l = u[q - 1], r = u[q + 1], d = u[q - RW], t = u[q + RW];
      const double ax = s2 * (((c - l) + (c - r)) + ((c - d) + (c - t)));
      v[q] = c + f * (sb[q] - ax);
    }
  }
  __syncthreads();
  const double* __restrict__ u = sx[min(sweeps, S) & 1];
  for (int p = threadIdx.x; p < TW * TH; p += 256) {
    const int lx = S + p % TW, ly = S + p / TW;
    const int x = gx0 + lx, y = gy0 + ly;
    if (x < n && y < n) xout[(long long)y * n + x] = u[ly * RW + lx];
  }
}

// 3D: A u = (1/h^2) sum_faces k_f (u_c - u_nb), k_f the harmonic mean of the
// two cells' kappa (kappa_c on a wall face, u = 0 beyond it; kappa = NULL
// means 1); the diagonal is (1/h^2) sum_faces k_f.  s2 = 1/h^2 from the host.
__global__ void jacobi3d_kernel(int n, const float* __restrict__ kappa,
                                const double* __restrict__ b, const double* __restrict__ xin,
                                double* __restrict__ xout, double omega, double s2) {
  const long long N = (long long)n * n * n;
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int ix = (int)(i % n), iy = (int)((i / n) % n), iz = (int)(i / ((long long)n * n));
  const long long nn = (long long)n * n;
  const long long off[6] = {-1, 1, -(long long)n, (long long)n, -nn, nn};
  const bool has[6] = {ix > 0, ix < n - 1, iy > 0, iy < n - 1, iz > 0, iz < n - 1};
  const double c = xin[i];
  const double kc = kappa ? (double)kappa[i] : 1.0;
  double au = 0.0, diag = 0.0;
  for (int f = 0; f < 6; f++) {
    double kf = kc, unb = 0.0;
    if (has[f]) {
      const double kn = kappa ? (double)kappa[i + off[f]] : 1.0;
      kf = 2.0 * kc * kn / (kc + kn);
      unb = xin[i + off[f]];
    }
    au += kf * (c - unb);
    diag += kf;
  }
  xout[i] = c + omega * (b[i] - s2 * au) / (s2 * diag);
}

// ring pair: u = b/s, t = x/s
__global__ void store_pair_kernel(const double* __restrict__ b, const double* __restrict__ x,
                                  int N, const double* sumsq, float* __restrict__ u,
                                  float* __restrict__ t) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  double s = sqrt(*sumsq / N);
  if (!(s > 0.0)) s = 1.0;
  u[i] = (float)(b[i] / s);
  t[i] = (float)(x[i] / s);
}

// out[2c] = <x, t_c>, out[2c+1] = <t_c, t_c> for the listed ring slots;
// out[2*count] = <x, x>.  One CTA per slot (+1 for ||x||), fixed order.
__global__ void spread_dots_kernel(const double* __restrict__ x, const float* __restrict__ ring,
                                   long long stride, const int* __restrict__ slots, int count,
                                   int N, double* out) {
  __shared__ double red[2][32];
  const int c = blockIdx.x;
  double a = 0.0, bb = 0.0;
  if (c < count) {
    const float* tc = ring + (long long)slots[c] * stride;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
      const double tv = tc[i];
      a += x[i] * tv;
      bb += tv * tv;
    }
  } else {
    for (int i = threadIdx.x; i < N; i += blockDim.x) a += x[i] * x[i];
  }
  a = warp_sum(a);
  bb = warp_sum(bb);
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = a;
    red[1][threadIdx.x >> 5] = bb;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const bool in = threadIdx.x < (int)(blockDim.x >> 5);
    a = warp_sum(in ? red[0][threadIdx.x] : 0.0);
    bb = warp_sum(in ? red[1][threadIdx.x] : 0.0);
    if (threadIdx.x == 0) {
      if (c < count) {
        out[2 * c] = a;
        out[2 * c + 1] = bb;
      } else {
        out[2 * count] = a;
      }
    }
  }
}

static unsigned blocks_for(int N) { return (unsigned)((N + 255) / 256); }

cudaError_t launch_sumsq(const double* b, int N, double* out, cudaStream_t s) {
  sumsq_kernel<<<1, 1024, 0, s>>>(b, N, out);
  note_launches(1);
  return cudaGetLastError();
}
cudaError_t launch_normalise(const double* b, int N, double* part, double* sumsq, float* u,
                             cudaStream_t s) {
  // about four elements per thread and partial
  const int np = N < 1024 * kNormParts ? (N + 1023) / 1024 : kNormParts;
  sumsq_part_kernel<<<np, 256, 0, s>>>(b, N, part);
  normalise_kernel<<<blocks_for(N), 256, 0, s>>>(b, N, part, np, sumsq, u);
  note_launches(2);
  return cudaGetLastError();
}
cudaError_t launch_jacobi(int dim, int n, const float* kappa, const double* b, double* x,
                          double* tmp, double omega, int sweeps, double** result,
                          cudaStream_t s) {
  const double h = 2.0 / (n + 1);
  const double s2 = 1.0 / (h * h);
  // Four sweeps per launch where that saves more than the halos' FP64 work costs: up to
  // two tiles per SM (32 sweeps, us, one per launch / four: 128^2 145 / 65, 256^2 147 /
  // 112, 384^2 212 / 163; past that 416^2 213 / 227, 512^2 278 / 279, 1024^2 727 / 854),
  // and not for one or two sweeps (256^2 21 / 24 and 23 / 25).
  constexpr int S = 4, kMostTiles = 2 * 152;
  const long long tiles = (long long)((n + 31) / 32) * ((n + 15) / 16);
  const double f = omega / (4.0 * s2);
  double *cur = x, *oth = tmp;
  for (int k = 0; k < sweeps;) {
    const int left = sweeps - k;
    if (dim == 3) {
      jacobi3d_kernel<<<blocks_for(n * n * n), 256, 0, s>>>(n, kappa, b, cur, oth, omega, s2);
      k++;
    } else if (left < 3 || tiles > kMostTiles) {
      jacobi_kernel<<<blocks_for(n * n), 256, 0, s>>>(n, b, cur, oth, s2, f);
      k++;
    } else {
      const int c = left < S ? left : S;
      // 32 x 16 tiles where they fill the GPU, else 16 x 8 (a sweep of a tile is
      // a serial FP64 chain per point; more CTAs shorten it)
      if (tiles >= 100)
        jacobi_tile_kernel<32, 16, S><<<dim3((n + 31) / 32, (n + 15) / 16), 256, 0, s>>>(
            n, b, cur, oth, s2, f, c);
      else
        jacobi_tile_kernel<16, 8, S><<<dim3((n + 15) / 16, (n + 7) / 8), 256, 0, s>>>(
            n, b, cur, oth, s2, f, c);
      k += c;
    }
    note_launches(1);
    double* t = cur;
    cur = oth;
    oth = t;
  }
  *result = cur;
  return cudaGetLastError();
}
cudaError_t launch_denormalise(const float* y, int N, const double* sumsq, double scale,
                               double* x, cudaStream_t s) {
  denormalise_kernel<<<blocks_for(N), 256, 0, s>>>(y, N, sumsq, scale, x);
  note_launches(1);
  return cudaGetLastError();
}
cudaError_t launch_store_pair(const double* b, const double* x, int N, const double* sumsq,
                              float* u, float* t, cudaStream_t s) {
  store_pair_kernel<<<blocks_for(N), 256, 0, s>>>(b, x, N, sumsq, u, t);
  note_launches(1);
  return cudaGetLastError();
}
cudaError_t launch_spread_dots(const double* x, const float* ring, long long stride,
                               const int* slots, int count, int N, double* out, cudaStream_t s) {
  spread_dots_kernel<<<count + 1, 512, 0, s>>>(x, ring, stride, slots, count, N, out);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace mlg
