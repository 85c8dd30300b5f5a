// Initial-guess network N(b): forward, backward and Adam on the GPU.
// Architecture and parameter order are documented in nn.h; activations are
// NHWC with 32 channels in BF16, accumulation in FP32.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "nn.h"

namespace mlg {

namespace {

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ void store32(bf16* p, const float* v) {
  uint4* q = reinterpret_cast<uint4*>(p);
#pragma unroll
  for (int i = 0; i < 4; i++) {
    uint4 u;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&u);
#pragma unroll
    for (int j = 0; j < 4; j++) h[j] = __floats2bfloat162_rn(v[i * 8 + 2 * j], v[i * 8 + 2 * j + 1]);
    q[i] = u;
  }
}

// --------------------------------------------------------------- geometry --
// Grid points of a cubic grid of side n: p = ((b n + z) n + y) n + x in 3D,
// (b n + y) n + x in 2D.  Tap t of a 3^D stencil: kz = t / 9 (3D), ky = (t / 3) % 3,
// kx = t % 3, offsets k - 1 (times the dilation).
template <int D>
struct Geo {
  static constexpr int T = D == 3 ? 27 : 9;
  // Point indices stay below 2^31 (net_create checks 32 B_max n^D), so the
  // arithmetic is 32-bit: a 64-bit division is a long software sequence.
  __device__ static void decode(long long p, int n, int& b, int& z, int& y, int& x) {
    const unsigned un = (unsigned)n;
    unsigned r = (unsigned)p;
    x = (int)(r % un);
    r /= un;
    y = (int)(r % un);
    r /= un;
    if (D == 3) {
      z = (int)(r % un);
      r /= un;
    } else {
      z = 0;
    }
    b = (int)r;
  }
  // index of (b, z + dz, y + dy, x + dx), or -1 outside the grid
  __device__ static long long nb(int b, int z, int y, int x, int dz, int dy, int dx, int n) {
    const int zz = z + dz, yy = y + dy, xx = x + dx;
    if (yy < 0 || yy >= n || xx < 0 || xx >= n) return -1;
    if (D == 3 && (zz < 0 || zz >= n)) return -1;
    return D == 3 ? (long long)(((b * n + zz) * n + yy) * n + xx) : (long long)((b * n + yy) * n + xx);
  }
  __device__ static void tap(int t, int& dz, int& dy, int& dx) {
    dz = D == 3 ? t / 9 - 1 : 0;
    dy = (t / 3) % 3 - 1;
    dx = t % 3 - 1;
  }
  __host__ __device__ static long long pts(int n) {
    return D == 3 ? (long long)n * n * n : (long long)n * n;
  }
};

// ---------------------------------------------------------------- forward --

// a0[p][c] = relu(b[c] + sum_tap w[c][tap] u[p + off_tap])
template <int D>
__global__ void conv_in_fwd(int B, int n, const float* __restrict__ u,
                            const float* __restrict__ w, const float* __restrict__ bias,
                            bf16* __restrict__ a0) {
  constexpr int T = Geo<D>::T;
  __shared__ float ws[kC * T + kC];
  for (int i = threadIdx.x; i < kC * T; i += blockDim.x) ws[i] = w[i];
  for (int i = threadIdx.x; i < kC; i += blockDim.x) ws[kC * T + i] = bias[i];
  __syncthreads();
  const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p >= B * Geo<D>::pts(n)) return;
  int b, z, y, x;
  Geo<D>::decode(p, n, b, z, y, x);
  float tp[T];
#pragma unroll
  for (int t = 0; t < T; t++) {
    int dz, dy, dx;
    Geo<D>::tap(t, dz, dy, dx);
    const long long q = Geo<D>::nb(b, z, y, x, dz, dy, dx, n);
    tp[t] = q >= 0 ? u[q] : 0.f;
  }
  float v[kC];
#pragma unroll
  for (int c = 0; c < kC; c++) {
    float acc = ws[kC * T + c];
#pragma unroll
    for (int t = 0; t < T; t++) acc += ws[c * T + t] * tp[t];
    v[c] = fmaxf(acc, 0.f);
  }
  store32(a0 + p * kC, v);
}

// Up to kPoolDepth levels of the average-pool pyramid in one launch: out_l = mean
// of each 2^D block of level l - 1 (side s -> s/2), channels last, BF16.  A CTA
// owns a block of 2^kPoolDepth points per axis of the finest level, whose
// descendants depend on nothing else: level 1 comes from global memory, the
// others from the level before in shared memory (as rounded to BF16).
template <int D>
struct PoolFwd {
  static constexpr int kDepth = D == 3 ? 3 : 5;
  int nlev;                 // levels written
  int side[kDepth + 1];     // side[0]: of `in`
  const bf16* in;
  bf16* out[kDepth + 1];    // out[1 .. nlev]
};

template <int D>
__global__ void __launch_bounds__(256) pool_chain_fwd(PoolFwd<D> pf) {
  constexpr int kDepth = PoolFwd<D>::kDepth;
  constexpr int kHalf = 1 << (kDepth - 1);  // level-1 points of a block per axis
  constexpr int kPts1 = D == 3 ? kHalf * kHalf * kHalf : kHalf * kHalf;
  __shared__ __align__(16) bf16 buf[2][kPts1 * kC];
  // block coordinates (x fastest) and batch
  const int bps = (pf.side[1] + kHalf - 1) / kHalf;
  int r = blockIdx.x;
  const int bx = r % bps;
  r /= bps;
  const int by = r % bps;
  r /= bps;
  const int bz = D == 3 ? r % bps : 0;
  const int b = D == 3 ? r / bps : r;
  for (int l = 1; l <= pf.nlev; l++) {
    const int w = kHalf >> (l - 1);  // the block's points of level l per axis
    const int so = pf.side[l], si = pf.side[l - 1];
    const int pts = D == 3 ? w * w * w : w * w;
    const bf16* __restrict__ prev = buf[(l - 1) & 1];
    bf16* __restrict__ mine = buf[l & 1];
    for (int i = threadIdx.x; i < pts * 4; i += 256) {
      const int q = (i & 3) * 8, p = i >> 2;
      const int lx = p % w, ly = (p / w) % w, lz = D == 3 ? p / (w * w) : 0;
      const int x = bx * w + lx, y = by * w + ly, z = bz * w + lz;
      if (x >= so || y >= so || (D == 3 && z >= so)) continue;
      float v[8];
#pragma unroll
      for (int e = 0; e < 8; e++) v[e] = 0.f;
#pragma unroll
      for (int k = 0; k < (1 << D); k++) {
        const int dz = (k >> 2) & 1, dy = (k >> 1) & 1, dx = k & 1;
        uint4 u;
        if (l == 1) {
          const int f = D == 3 ? ((b * si + 2 * z + dz) * si + 2 * y + dy) * si + 2 * x + dx
                               : (b * si + 2 * y + dy) * si + 2 * x + dx;
          u = *reinterpret_cast<const uint4*>(pf.in + (long long)f * kC + q);
        } else {
          const int f = ((2 * lz + dz) * 2 * w + 2 * ly + dy) * 2 * w + 2 * lx + dx;
          u = *reinterpret_cast<const uint4*>(prev + f * kC + q);
        }
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
        for (int e = 0; e < 4; e++) {
          const float2 t = __bfloat1622float2(h[e]);
          v[2 * e] += t.x;
          v[2 * e + 1] += t.y;
        }
      }
      uint4 o;
      __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&o);
      constexpr float sc = 1.f / (1 << D);
#pragma unroll
      for (int e = 0; e < 4; e++)
        h[e] = __floats2bfloat162_rn(v[2 * e] * sc, v[2 * e + 1] * sc);
      const int f = D == 3 ? ((b * so + z) * so + y) * so + x : (b * so + y) * so + x;
      *reinterpret_cast<uint4*>(pf.out[l] + (long long)f * kC + q) = o;
      *reinterpret_cast<uint4*>(mine + p * kC + q) = o;
    }
    __syncthreads();
  }
}

struct Levels {
  const bf16* z[kMaxLevels];
  const float2* tab[kMaxLevels];  // half-pixel source of each fine index: (weight of i0 + 1, i0)
  int side[kMaxLevels];
  int L;
};

// s[p][c] = sum_l upsample(z_l)[p][c]  (bilinear in 2D, trilinear in 3D);
// four threads per point, eight channels (16 bytes) each; the source positions
// come from the levels' tables (an IEEE division per axis, level and thread
// otherwise)
template <int D>
__global__ void upsum_fwd(int B, int n, Levels lv, bf16* __restrict__ s) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= B * Geo<D>::pts(n) * 4) return;
  const int cg = (int)(i & 3);
  const long long p = i >> 2;
  int b, z, y, x;
  Geo<D>::decode(p, n, b, z, y, x);
  float acc[8];
  {
    const uint4 v = *reinterpret_cast<const uint4*>(lv.z[0] + p * kC + cg * 8);
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const float2 f = __bfloat1622float2(h[q]);
      acc[2 * q] = f.x;
      acc[2 * q + 1] = f.y;
    }
  }
  for (int l = 1; l < lv.L; l++) {
    const int m = lv.side[l];
    const float2* __restrict__ tab = lv.tab[l];
    const float2 tz = D == 3 ? __ldg(tab + z) : make_float2(0.f, 0.f);
    const float2 ty = __ldg(tab + y), tx = __ldg(tab + x);
    const float lz = tz.x, ly = ty.x, lx = tx.x;
    const int z0 = __float_as_int(tz.y), y0 = __float_as_int(ty.y), x0 = __float_as_int(tx.y);
    const int z1 = min(z0 + 1, m - 1), y1 = min(y0 + 1, m - 1), x1 = min(x0 + 1, m - 1);
#pragma unroll
    for (int k = 0; k < (1 << D); k++) {
      const int zz = (k >> 2) & 1 ? z1 : z0, yy = (k >> 1) & 1 ? y1 : y0, xx = k & 1 ? x1 : x0;
      const float wz = D == 3 ? ((k >> 2) & 1 ? lz : 1.f - lz) : 1.f;
      const float w = wz * ((k >> 1) & 1 ? ly : 1.f - ly) * (k & 1 ? lx : 1.f - lx);
      const long long q = Geo<D>::nb(b, zz, yy, xx, 0, 0, 0, m);
      const uint4 v = *reinterpret_cast<const uint4*>(lv.z[l] + q * kC + cg * 8);
      const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
      for (int qq = 0; qq < 4; qq++) {
        const float2 f = __bfloat1622float2(h[qq]);
        acc[2 * qq] += w * f.x;
        acc[2 * qq + 1] += w * f.y;
      }
    }
  }
  uint4 o;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
  for (int q = 0; q < 4; q++) h[q] = __floats2bfloat162_rn(acc[2 * q], acc[2 * q + 1]);
  *reinterpret_cast<uint4*>(s + p * kC + cg * 8) = o;
}

// y[p] = b + sum_tap sum_c w[c][tap] t[p + off_tap][c].  A CTA owns a tile of the grid
// (32 x 8 points, 3D 8 x 8 x 4) and stages its rows and their halo in shared memory
// once, so each row is read by coalesced accesses and once per tile instead of by
// every tap of its neighbours (reads a thread per point made 64 bytes apart, bound by
// L1: 50 us at 256^2 x 8 and 59 at 48^3 x 2, now 26 and 32).  Rows are 80 bytes apart in shared memory: a warp's 16-byte
// reads of 32 rows meet no bank conflict.  The weights are staged [tap][c], so that
// four channels' come in one 16-byte read.
template <int D>
struct OutTile {
  static constexpr int X = D == 2 ? 32 : 8, Y = 8, Z = D == 2 ? 1 : 4;  // 256 points
  static constexpr int PX = X + 2, PY = Y + 2, PZ = D == 2 ? 1 : Z + 2;
  static constexpr int kRows = PX * PY * PZ;
  static constexpr int kSmem = kRows * 80 + Geo<D>::T * kC * (int)sizeof(float);
};
template <int D>
__global__ void __launch_bounds__(256) conv_out_fwd(int n, const bf16* __restrict__ t,
                                                    const float* __restrict__ w,
                                                    const float* __restrict__ bias,
                                                    float* __restrict__ y) {
  using O = OutTile<D>;
  constexpr int T = Geo<D>::T;
  extern __shared__ __align__(16) uint4 tile[];  // [kRows][5], the fifth word unused
  float* ws = reinterpret_cast<float*>(tile + O::kRows * 5);
  const int tx = (n + O::X - 1) / O::X, ty = (n + O::Y - 1) / O::Y;
  const int tz = D == 3 ? (n + O::Z - 1) / O::Z : 1;
  int id = blockIdx.x;
  const int x0 = id % tx * O::X;
  id /= tx;
  const int y0 = id % ty * O::Y;
  id /= ty;
  const int z0 = id % tz * O::Z, b = id / tz;
  for (int i = threadIdx.x; i < kC * T; i += 256) ws[(i % T) * kC + i / T] = w[i];
#pragma unroll 6
  for (int i = threadIdx.x; i < O::kRows * 4; i += 256) {
    const int r = i >> 2, q = i & 3;
    const int x = x0 + r % O::PX - 1, yy = y0 + r / O::PX % O::PY - 1;
    const int z = D == 3 ? z0 + r / (O::PX * O::PY) - 1 : 0;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (x >= 0 && x < n && yy >= 0 && yy < n && z >= 0 && z < n) {
      const long long p = ((D == 3 ? (long long)b * n + z : (long long)b) * n + yy) * n + x;
      v = reinterpret_cast<const uint4*>(t + p * kC)[q];
    }
    tile[r * 5 + q] = v;
  }
  __syncthreads();
  const int lx = threadIdx.x % O::X, ly = threadIdx.x / O::X % O::Y;
  const int lz = threadIdx.x / (O::X * O::Y);
  const int x = x0 + lx, yy = y0 + ly, z = z0 + lz;
  if (x >= n || yy >= n || (D == 3 && z >= n)) return;
  float acc = bias[0];
#pragma unroll 1
  for (int dz = D == 3 ? -1 : 0; dz <= (D == 3 ? 1 : 0); dz++) {
    if (z + dz < 0 || z + dz >= n) continue;
    const int t0 = D == 3 ? 9 * (dz + 1) : 0;
    const uint4* row = tile + (((D == 3 ? lz + 1 + dz : 0) * O::PY + ly + 1) * O::PX + lx + 1) * 5;
#pragma unroll
    for (int k = 0; k < 9; k++) {
      const int dy = k / 3 - 1, dx = k % 3 - 1;
      if (yy + dy < 0 || yy + dy >= n || x + dx < 0 || x + dx >= n) continue;
      const uint4* r = row + (dy * O::PX + dx) * 5;
      const float4* wt = reinterpret_cast<const float4*>(ws + (t0 + k) * kC);
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const uint4 v = r[i];
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
        for (int q = 0; q < 2; q++) {
          const float4 wv = wt[2 * i + q];
          const float2 f0 = __bfloat1622float2(h[2 * q]), f1 = __bfloat1622float2(h[2 * q + 1]);
          acc += wv.x * f0.x;
          acc += wv.y * f0.y;
          acc += wv.z * f1.x;
          acc += wv.w * f1.y;
        }
      }
    }
  }
  y[((D == 3 ? (long long)b * n + z : (long long)b) * n + yy) * n + x] = acc;
}

// --------------------------------------------------------------- backward --

// gy = 2 (y - ts t) / (B N); per-CTA partial sums of (y - ts t)^2 (ts from
// tsp when given: the target scale of a training phase, in device memory)
__global__ void mse_grad(long long total, float scale, float ts, const float* __restrict__ tsp,
                         const float* __restrict__ y, const float* __restrict__ t,
                         float* __restrict__ gy, float* __restrict__ part) {
  __shared__ float red[32];
  if (tsp) ts = *tsp;
  float acc = 0.f;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const float d = y[i] - ts * t[i];
    gy[i] = 2.f * d * scale;
    acc += d * d;
  }
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    acc = threadIdx.x < (int)(blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
    acc = warp_sum(acc);
    if (threadIdx.x == 0) part[blockIdx.x] = acc;
  }
}

// loss = scale * sum of the CTA partials (FP64, a fixed tree over 256 threads: one
// thread adding them in turn took 20 us of dependent FP64 additions)
__global__ void __launch_bounds__(256) loss_finish(const float* __restrict__ part, int nparts,
                                                   float scale, float* __restrict__ loss) {
  __shared__ double red[8];
  double v = 0.0;
  for (int i = threadIdx.x; i < nparts; i += 256) v += part[i];
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; w++) v += red[w];
    *loss = (float)(v * scale);
  }
}

// Segments of the 1-channel <-> 32-channel kernels: R rows x W points of one
// (b, z) plane (W = min(n, 256), R = max(1, 256 / n)), with the 1-channel field
// of the segment and its one-point halo staged in shared memory, zero outside
// the grid, so each tap is one shared-memory read at a fixed offset.
constexpr int kSeg = 256;
constexpr int kW1Threads = 256;

template <int D>
__host__ __device__ constexpr int w1_planes() { return D == 3 ? 3 : 1; }

__host__ __device__ inline int w1_w(int n) { return n < kSeg ? n : kSeg; }
__host__ __device__ inline int w1_r(int n) { return n < kSeg ? kSeg / n : 1; }

template <int D>
int w1_stage_floats(int n) { return w1_planes<D>() * (w1_r(n) + 2) * (w1_w(n) + 2); }

// sf[pz][r][cx] = f at (plane pl + pz - 1 (3D), row y0 + r - 1, column x0 + cx - 1)
template <int D, int NT>
__device__ __forceinline__ void w1_stage(float* sf, const float* __restrict__ f, int n, int pl,
                                         int y0, int x0, int W, int R) {
  const int TW = W + 2, TP = (R + 2) * TW;
  for (int i = threadIdx.x; i < w1_planes<D>() * TP; i += NT) {
    const int pz = D == 3 ? i / TP : 1, r = (i % TP) / TW, cx = (i % TP) % TW;
    const int gy = y0 + r - 1, gx = x0 + cx - 1;
    bool ok = gy >= 0 && gy < n && gx >= 0 && gx < n;
    int gpl = pl;
    if (D == 3) {
      const int gz = pl % n + pz - 1;
      ok = ok && gz >= 0 && gz < n;
      gpl = pl + pz - 1;
    }
    sf[i] = ok ? f[((long long)gpl * n + gy) * n + gx] : 0.f;
  }
}

// The 3^D neighbourhood of a point in a staged segment, kept in registers while a
// warp walks along x: each step reads the new column only (3 or 9 shared-memory
// reads instead of 9 or 27).  With the points' loads issued ahead (below) the
// network's forward and backward at 256^2 x 8 went from 1367 to 1246 us, at 48^3 x 2
// from 2365 to 2224.
template <int D>
struct Window {
  float v[w1_planes<D>()][3][3];  // [dz + 1][dy + 1][dx + 1] (2D: [0][dy + 1][dx + 1])
  __device__ __forceinline__ void column(const float* sf, int base, int TP, int TW, int dx) {
#pragma unroll
    for (int a = 0; a < w1_planes<D>(); a++)
#pragma unroll
      for (int b = 0; b < 3; b++)
        v[a][b][dx + 1] = sf[base + (D == 3 ? (a - 1) * TP : 0) + (b - 1) * TW + dx];
  }
  // at the point `base`; next: the window was at base - 1
  __device__ __forceinline__ void move(const float* sf, int base, int TP, int TW, bool next) {
    if (next) {
#pragma unroll
      for (int a = 0; a < w1_planes<D>(); a++)
#pragma unroll
        for (int b = 0; b < 3; b++) {
          v[a][b][0] = v[a][b][1];
          v[a][b][1] = v[a][b][2];
        }
    } else {
      column(sf, base, TP, TW, -1);
      column(sf, base, TP, TW, 0);
    }
    column(sf, base, TP, TW, 1);
  }
  // the value at + off (sgn = 1) or - off (sgn = -1) of tap t
  template <int SGN>
  __device__ __forceinline__ float at(int t) const {
    int dz, dy, dx;
    Geo<D>::tap(t, dz, dy, dx);
    return v[D == 3 ? SGN * dz + 1 : 0][SGN * dy + 1][SGN * dx + 1];
  }
};

// A lane of the kernels below holds kLaneCh channels of a point (2D 4, 3D 2: what its
// taps' weights or sums leave of the registers), 32 / kLaneCh lanes a point: a point's
// window is read from shared memory once for all of them, and a warp's access to a
// 32-channel field covers 4 (2) points at 16 and 8 (8 and 4) bytes per lane.  One
// channel per lane left these kernels bound by instructions and 2- and 4-byte accesses
// (us, one channel / now, 256^2 x 8 and 48^3 x 2; floors by bytes 19, 5, 15 and 8, 2,
// 6): conv_out_bwd_data 68 / 42, 50 / 38; conv1_wgrad<0> 46 / 30, 37 / 29;
// conv1_wgrad<1> 61 / 47, 45 / 36.
template <int D>
constexpr int kLaneCh = D == 2 ? 4 : 2;
template <int C>
struct LaneVec;
template <>
struct LaneVec<4> {
  using B = uint2;   // bf16 values
  using F = float4;  // float values
};
template <>
struct LaneVec<2> {
  using B = unsigned;
  using F = float2;
};
template <int C>
__device__ __forceinline__ void lane_floats(float (&v)[C], typename LaneVec<C>::B b) {
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&b);
#pragma unroll
  for (int q = 0; q < C / 2; q++) {
    const float2 t = __bfloat1622float2(h[q]);
    v[2 * q] = t.x;
    v[2 * q + 1] = t.y;
  }
}
template <int C>
__device__ __forceinline__ typename LaneVec<C>::B lane_bf(const float (&v)[C]) {
  typename LaneVec<C>::B b;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&b);
#pragma unroll
  for (int q = 0; q < C / 2; q++) h[q] = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
  return b;
}

// gt[p][c] = sum_tap w[c][tap] gy[p - off_tap] (transpose of the 32 -> 1 output
// conv) and, when gbf is given, gbf[p][c] = bf16(mask[p][c] > 0 ? gt : 0) for
// the masked consumer that follows.  Segments as above (gy staged), each group of
// lanes U points of the segment in a row.
template <int D>
__global__ void __launch_bounds__(kW1Threads, 2) conv_out_bwd_data(
    int B, int n, const float* __restrict__ gy, const float* __restrict__ w,
    float* __restrict__ gt, const bf16* __restrict__ mask, bf16* __restrict__ gbf) {
  constexpr int T = Geo<D>::T;
  constexpr int C = kLaneCh<D>, LP = kC / C;  // channels per lane, lanes per point
  constexpr int U = kSeg / (kW1Threads / LP);
  constexpr int CH = 8;
  using BV = typename LaneVec<C>::B;
  using FV = typename LaneVec<C>::F;
  extern __shared__ float sf[];
  const int W = w1_w(n), R = w1_r(n);
  const int TW = W + 2, TP = (R + 2) * TW;
  const int xsegs = (n + W - 1) / W, ysegs = (n + R - 1) / R;
  const int nseg = B * (D == 3 ? n : 1) * ysegs * xsegs;
  const int c = threadIdx.x % LP * C, wp = threadIdx.x / LP;
  float wc[C][T];
#pragma unroll
  for (int d = 0; d < C; d++)
#pragma unroll
    for (int tp = 0; tp < T; tp++) wc[d][tp] = w[(c + d) * T + tp];
  const int ry0 = (wp * U) / W, xl0 = (wp * U) % W;
  const int center = D == 3 ? TP : 0;
  for (int sg = blockIdx.x; sg < nseg; sg += gridDim.x) {
    const int xs = sg % xsegs, t2 = sg / xsegs;
    const int ys = t2 % ysegs, pl = t2 / ysegs;
    const int x0 = xs * W, y0 = ys * R;
    int ry = ry0, xl = xl0, lry = ry0, lxl = xl0;  // next point to compute, to load
    // CH points' masks in flight together, the first ones' during the staging
    BV mk[CH];
    auto load = [&]() {
#pragma unroll
      for (int k = 0; k < CH; k++) {
        const int y = y0 + lry, x = x0 + lxl;
        mk[k] = BV{};
        if (gbf && lry < R && y < n && x < n)
          mk[k] = *reinterpret_cast<const BV*>(mask + ((pl * n + y) * n + x) * kC + c);
        if (++lxl == W) {
          lxl = 0;
          ++lry;
        }
      }
    };
    load();
    __syncthreads();
    w1_stage<D, kW1Threads>(sf, gy, n, pl, y0, x0, W, R);
    __syncthreads();
    Window<D> win;
    bool next = false;
#pragma unroll 1
    for (int k0 = 0; k0 < U; k0 += CH) {
      if (k0) load();
#pragma unroll
      for (int k = 0; k < CH; k++) {
        const int y = y0 + ry, x = x0 + xl;
        if (ry < R) {
          win.move(sf, center + (ry + 1) * TW + xl + 1, TP, TW, next);
          next = true;
          if (y < n && x < n) {
            float acc[C];
#pragma unroll
            for (int d = 0; d < C; d++) {
              acc[d] = 0.f;
#pragma unroll
              for (int tp = 0; tp < T; tp++) acc[d] += wc[d][tp] * win.template at<-1>(tp);
            }
            const int e = ((pl * n + y) * n + x) * kC + c;  // (below 2^31: network size check)
            FV o;
            memcpy(&o, acc, sizeof(o));
            *reinterpret_cast<FV*>(gt + e) = o;
            if (gbf) {
              float m[C];
              lane_floats<C>(m, mk[k]);
#pragma unroll
              for (int d = 0; d < C; d++) m[d] = m[d] > 0.f ? acc[d] : 0.f;
              *reinterpret_cast<BV*>(gbf + e) = lane_bf<C>(m);
            }
          }
        }
        if (++xl == W) {
          xl = 0;
          ++ry;
          next = false;
        }
      }
    }
  }
}

// Per-CTA partial weight gradients of a 1-channel <-> 32-channel 3^D conv:
//   part[cta][c*T + tap] and the biases at part[cta][32 T + c].
// MODE 0 (output conv):  dW[c][tap] = sum_p gy[p] t[p + off][c]
//                                   = sum_q t[q][c] gy[q - off],  db = sum_q gy[q]
// MODE 1 (input conv):   dW[c][tap] = sum_p g32[p][c] u[p + off], db[c] = sum_p g32[p][c],
//                        with g32 taken as 0 where m32 <= 0 (the ReLU of a0), plus
//                        2^-D of the pooled level's gradient gc (null: no such level)
// The grid is cut into segments of R rows x W points of one (b, z) plane
// (W = min(n, 256), R = max(1, 256 / n)).  Every 32-channel row is read once,
// coalesced, CH rows per group of lanes in flight; the 1-channel field (gy or u) of
// the segment and its halo is staged in shared memory, zero outside the grid, so each
// tap is one shared-memory read at a fixed offset.  The sums of a warp's groups
// of lanes, then of the warps, are added in a fixed order.
template <int D>
int conv1_wgrad_smem(int n) {
  constexpr int T = Geo<D>::T;
  const int stage = w1_stage_floats<D>(n);
  const int red = (kW1Threads / 32) * 32 * (T + 1);
  return (int)sizeof(float) * (stage > red ? stage : red);
}

template <int MODE, int D>
__global__ void __launch_bounds__(kW1Threads, 2) conv1_wgrad(
    int B, int n, const float* __restrict__ g1, const bf16* __restrict__ x32,
    const float* __restrict__ g32, const float* __restrict__ gc, const bf16* __restrict__ m32,
    const float* __restrict__ u, float* __restrict__ part, int stride) {
  constexpr int T = Geo<D>::T;
  constexpr int NW = kW1Threads / 32;
  constexpr int C = kLaneCh<D>, LP = kC / C;      // channels per lane, lanes per point
  constexpr int U = kSeg / (kW1Threads / LP);     // points per group of lanes and segment
  constexpr int CH = MODE == 1 || D == 3 ? 4 : 8; // points whose loads are in flight together
  using BV = typename LaneVec<C>::B;
  using FV = typename LaneVec<C>::F;
  constexpr int sgn = MODE == 0 ? -1 : 1;  // MODE 0 reads gy at q - off, MODE 1 u at p + off
  extern __shared__ float sf[];
  const int W = w1_w(n), R = w1_r(n);
  const int TW = W + 2, TP = (R + 2) * TW;
  const int xsegs = (n + W - 1) / W, ysegs = (n + R - 1) / R;
  const int nplanes = B * (D == 3 ? n : 1);  // (b, z) planes
  const int nseg = nplanes * ysegs * xsegs;
  const int c = threadIdx.x % LP * C, gw = threadIdx.x / LP;
  const float* __restrict__ f = MODE == 0 ? g1 : u;
  float acc[C][T], accb[C];
#pragma unroll
  for (int d = 0; d < C; d++) {
    accb[d] = 0.f;
#pragma unroll
    for (int t = 0; t < T; t++) acc[d][t] = 0.f;
  }
  for (int sg = blockIdx.x; sg < nseg; sg += gridDim.x) {
    const int xs = sg % xsegs, t2 = sg / xsegs;
    const int ys = t2 % ysegs, pl = t2 / ysegs;  // pl = b (2D) or b n + z (3D)
    const int x0 = xs * W, y0 = ys * R;
    // the group's U points run along x from (ry, xl), wrapping to the next row;
    // CH at a time, the next ones' loads in flight while these are used (the
    // first ones' during the staging).  All loads of a point are unconditional:
    // behind its mask, each would wait for the one before it.
    int ry = (gw * U) / W, xl = (gw * U) % W;
    int lry = ry, lxl = xl;  // of the next point to load
    const int center = D == 3 ? TP : 0;
    const int so = n / 2, pz = pl % n;
    const int cp = D == 3 ? (pl / n) * so + pz / 2 : pl;
    const bool cok = MODE == 1 && gc && (D == 2 || pz / 2 < so);
    BV rm[CH];
    FV rg[CH], rc[CH];
    auto load = [&]() {
#pragma unroll
      for (int k = 0; k < CH; k++) {
        const int x = x0 + lxl, y = y0 + lry;
        const bool ok = lry < R && y < n && x < n;
        const int e = ((pl * n + y) * n + x) * kC + c;  // (below 2^31: network size check)
        rm[k] = BV{};
        if (ok) rm[k] = *reinterpret_cast<const BV*>((MODE == 0 ? x32 : m32) + e);
        if constexpr (MODE == 1) {
          rg[k] = FV{};
          rc[k] = FV{};
          if (ok) rg[k] = *reinterpret_cast<const FV*>(g32 + e);
          // the pooled level's share (odd sides: the last point has none)
          if (ok && cok && y / 2 < so && x / 2 < so)
            rc[k] = *reinterpret_cast<const FV*>(gc + ((cp * so + y / 2) * so + x / 2) * kC + c);
        }
        if (++lxl == W) {
          lxl = 0;
          ++lry;
        }
      }
    };
    load();
    __syncthreads();  // the previous segment's readers are done with sf
    w1_stage<D, kW1Threads>(sf, f, n, pl, y0, x0, W, R);
    __syncthreads();
    Window<D> win;
    bool next = false;
#pragma unroll 1
    for (int k0 = 0; k0 < U; k0 += CH) {
      float val[CH][C];
#pragma unroll
      for (int k = 0; k < CH; k++) {
        lane_floats<C>(val[k], rm[k]);
        if constexpr (MODE == 1) {
          float a[C], b[C];
          memcpy(a, &rg[k], sizeof(a));
          memcpy(b, &rc[k], sizeof(b));
#pragma unroll
          for (int d = 0; d < C; d++)
            val[k][d] = val[k][d] > 0.f ? a[d] + (1.f / (1 << D)) * b[d] : 0.f;
        }
      }
      if (k0 + CH < U) load();
#pragma unroll
      for (int k = 0; k < CH; k++) {
        if (ry < R) {
          win.move(sf, center + (ry + 1) * TW + xl + 1, TP, TW, next);
          next = true;
          // (a ragged segment's points past the grid's edge are no terms of the sums: 0
          // times a neighbour that is not finite would be one)
          if (y0 + ry < n && x0 + xl < n) {
#pragma unroll
            for (int d = 0; d < C; d++) {
#pragma unroll
              for (int t = 0; t < T; t++) acc[d][t] += val[k][d] * win.template at<sgn>(t);
              if (MODE == 1) accb[d] += val[k][d];
            }
            if (MODE == 0) accb[0] += win.template at<1>(T / 2);
          }
        }
        if (++xl == W) {
          xl = 0;
          ++ry;
          next = false;
        }
      }
    }
  }
  // fixed-order sum of the groups' partials within a warp, then of the warps'
  __syncthreads();
  float* red = sf + (threadIdx.x >> 5) * 32 * (T + 1);  // [NW][32 (T + 1)]
#pragma unroll
  for (int d = 0; d < C; d++)
#pragma unroll
    for (int t = 0; t < T + 1; t++) {
      float v = t < T ? acc[d][t < T ? t : 0] : accb[d];
#pragma unroll
      for (int off = LP; off < 32; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
      if ((threadIdx.x & 31) < LP) red[(c + d) * (T + 1) + t] = v;
    }
  red = sf;
  __syncthreads();
  for (int t = threadIdx.x; t < kC * T + kC; t += kW1Threads) {
    // t < 32 T: weight c*T + tap; t >= 32 T: bias of channel t - 32 T (MODE 0: one bias)
    const int cc = t < kC * T ? t / T : t - kC * T;
    const int k = t < kC * T ? t % T : T;
    float v = 0.f;
    if (!(MODE == 0 && k == T && cc != 0))
      for (int ww = 0; ww < NW; ww++) v += red[ww * 32 * (T + 1) + cc * (T + 1) + k];
    part[(long long)blockIdx.x * stride + t] = v;
  }
}

// out = bf16(g * (mask > 0)), eight elements per thread (count is a multiple
// of 32: whole channel rows; the buffers are 32-byte aligned)
__global__ void mask_to_bf16(long long count, const float* __restrict__ g,
                             const bf16* __restrict__ mask, bf16* __restrict__ out) {
  const long long i = (blockIdx.x * (long long)blockDim.x + threadIdx.x) * 8;
  if (i >= count) return;
  const float4 a = *reinterpret_cast<const float4*>(g + i);
  const float4 b = *reinterpret_cast<const float4*>(g + i + 4);
  const uint4 mv = *reinterpret_cast<const uint4*>(mask + i);
  const bf16* m = reinterpret_cast<const bf16*>(&mv);
  const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  uint4 o;
  bf16* ob = reinterpret_cast<bf16*>(&o);
#pragma unroll
  for (int k = 0; k < 8; k++) ob[k] = __float2bfloat16(__bfloat162float(m[k]) > 0.f ? v[k] : 0.f);
  *reinterpret_cast<uint4*>(out + i) = o;
}

// grad[dst_w[i]] = sum over CTAs of part[cta][i] for the weight layout used by
// the partial kernels; the mapping to the parameter layout [o][k][tap] is done
// here so the parameters keep the documented order (T taps).
//   kind 0 (32->32): part index (tap*32 + k)*32 + o  -> param (o*32 + k)*T + tap; bias 1024 T + o
//   kind 1/2 (1-ch): part index c*T + tap (+ 32 T + c bias) -> same order
// One launch for all convolutions of the network: job k's outputs on the CTAs
// first[k] .. first[k+1]-1 (one launch per convolution cost 5 us each, mostly
// latency; with the coarse levels' convolutions and the pooling levels in shared
// launches, and the upsampling's tables: 1245 -> 1120 us at 256^2 x 8, the learned
// guess at 256^2 272 -> 221 us).
struct ReduceJob {
  const float* part;
  float *gw, *gb;
  int nparts, stride, kind;
};
struct ReduceJobs {
  static constexpr int kMost = kMaxLevels + kMaxExtra + 3;
  int n;
  int first[kMost + 1];
  ReduceJob job[kMost];
};

__global__ void __launch_bounds__(256) reduce_wgrad(const __grid_constant__ ReduceJobs jobs,
                                                    int T) {
  int jb = 0;
  while (jb + 1 < jobs.n && (int)blockIdx.x >= jobs.first[jb + 1]) jb++;
  const float* __restrict__ part = jobs.job[jb].part;
  float* __restrict__ gw = jobs.job[jb].gw;
  float* __restrict__ gb = jobs.job[jb].gb;
  const int nparts = jobs.job[jb].nparts, stride = jobs.job[jb].stride;
  const int kind = jobs.job[jb].kind;
  // 32 outputs per CTA (lane = output), the CTA partials split over the 8 warps
  // (coalesced rows), four independent sums per lane so that four loads are in
  // flight, all added in a fixed order (FP32: the FP64 pipe of this GPU is slow)
  __shared__ float red[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = ((int)blockIdx.x - jobs.first[jb]) * 32 + lane;
  const int nw = kind == 0 ? T * kC * kC : T * kC;
  const int nb = kind == 0 ? kC : (kind == 1 ? kC : 1);
  float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
  if (i < nw + nb) {
    int c = w;
    for (; c + 24 < nparts; c += 32) {
      s0 += part[(long long)c * stride + i];
      s1 += part[(long long)(c + 8) * stride + i];
      s2 += part[(long long)(c + 16) * stride + i];
      s3 += part[(long long)(c + 24) * stride + i];
    }
    for (; c < nparts; c += 8) s0 += part[(long long)c * stride + i];
  }
  red[w][lane] = (s0 + s1) + (s2 + s3);
  __syncthreads();
  if (w != 0 || i >= nw + nb) return;
  float t = 0.f;
#pragma unroll
  for (int k = 0; k < 8; k++) t += red[k][lane];
  if (i < nw) {
    if (kind == 0) {
      const int tp = i / (kC * kC), k = (i / kC) % kC, o = i % kC;
      gw[(o * kC + k) * T + tp] = (float)t;
    } else {
      gw[i] = (float)t;
    }
  } else {
    gb[i - nw] = (float)t;
  }
}

// Transpose of the linear upsampling from m to n along one axis of a tensor
// viewed as (outer, n, inner) -> (outer, m, inner):
//   out[o][j][c] = sum_x U[x][j] in[o][x][c],  U[x][j] = the weight of coarse j
// in fine x's half-pixel interpolation, read from the level's sparse rows
// (built once on the host with the arithmetic of the forward tables).  The
// D-dimensional transpose is D such passes, one per axis.

// One axis of one level; the levels' x-axis passes where a fine row is too long
// to stage (upsample_bwd_x_levels otherwise).
__global__ void upsample_bwd_axis(long long outer, int n, int m, long long inner,
                                  const int* __restrict__ ptr, const int* __restrict__ idx,
                                  const float* __restrict__ wt, const float* __restrict__ in,
                                  float* __restrict__ out) {
  const long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (id >= outer * m * inner) return;
  // element indices stay below 2^31 (network size check): 32-bit division
  const unsigned ui = (unsigned)id, uin = (unsigned)inner;
  const unsigned c = ui % uin;
  const unsigned p = ui / uin;
  const int j = (int)(p % (unsigned)m);
  const unsigned o = p / (unsigned)m;
  float acc = 0.f;
  for (int k = ptr[j]; k < ptr[j + 1]; k++)
    acc += wt[k] * in[((long long)o * n + idx[k]) * inner + c];
  out[id] = acc;
}

// Sum of wt[k] * src[k * stride] over k < cnt for four channels, in the order of
// k, eight loads in flight.
__device__ __forceinline__ float4 row_sum4(const float* __restrict__ src, long long stride,
                                           const float* __restrict__ wt, int cnt) {
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  auto add = [&](float w, const float4& v) {
    acc.x += w * v.x;
    acc.y += w * v.y;
    acc.z += w * v.z;
    acc.w += w * v.w;
  };
  int k = 0;
  for (; k + 8 <= cnt; k += 8) {
    float4 v[8];
    float w[8];
#pragma unroll
    for (int u = 0; u < 8; u++) {
      v[u] = *reinterpret_cast<const float4*>(src + (k + u) * stride);
      w[u] = wt[k + u];
    }
#pragma unroll
    for (int u = 0; u < 8; u++) add(w[u], v[u]);
  }
  for (; k < cnt; k++) add(wt[k], *reinterpret_cast<const float4*>(src + k * stride));
  return acc;
}

// The x-axis pass of every coarse level's transposed upsampling at once:
//   out_l[r][j][c] = sum_x U_l[x][j] in[r][x][c]   (levels l = 1 .. L-1)
// for each row r of the fine grid (x is the innermost axis in 2D and 3D).  One
// CTA per row: its n x 32 values are read from HBM once and from shared memory
// for every level.  A thread forms four channels of one coarse point (16-byte
// reads, a quarter of the instructions of one channel per lane; the fine points
// of a coarse one are consecutive, so only the first index is read).  Same
// sums, in the same order, as upsample_bwd_axis.  The staging also writes the
// masked BF16 gradient of the finest level, maskbf = bf16(mask > 0 ? in : 0), which
// would read the row from HBM once more in a launch of its own (256^2 x 8: 65 + 21 us
// in two launches, 79 in one).
struct UpLevels {
  int nlev;                     // levels 1 .. nlev-1
  int m[kMaxLevels];
  const int* ptr[kMaxLevels];
  const int* idx[kMaxLevels];
  const float* wt[kMaxLevels];
  long long in_off[kMaxLevels], out_off[kMaxLevels];
  unsigned first[kMaxLevels + 1];  // first CTA of each level (axis kernel)
  long long outer[kMaxLevels], inner[kMaxLevels];
  const bf16* mask[kMaxLevels];    // last axis: the ReLU mask of the level's output
};

constexpr int kXLevelsMaxN = 384;  // the staged row (n x 32 floats) stays within 48 KB

__global__ void __launch_bounds__(256) upsample_bwd_x_levels(int n, UpLevels lv,
                                                             const float* __restrict__ in,
                                                             float* __restrict__ out,
                                                             const bf16* __restrict__ mask,
                                                             bf16* __restrict__ maskbf) {
  extern __shared__ float row[];  // the fine row, n x 32
  const long long r = blockIdx.x;
  const int c4 = (threadIdx.x & 7) * 4, g = threadIdx.x >> 3;
  {
    const float4* src = reinterpret_cast<const float4*>(in + r * n * kC);
    const uint2* mk = reinterpret_cast<const uint2*>(mask + r * n * kC);
    uint2* mo = reinterpret_cast<uint2*>(maskbf + r * n * kC);
    float4* dst = reinterpret_cast<float4*>(row);
#pragma unroll 4
    for (int i = threadIdx.x; i < n * kC / 4; i += 256) {
      const float4 v = src[i];
      float m[4];
      lane_floats<4>(m, mk[i]);
      dst[i] = v;
      const float o[4] = {m[0] > 0.f ? v.x : 0.f, m[1] > 0.f ? v.y : 0.f, m[2] > 0.f ? v.z : 0.f,
                          m[3] > 0.f ? v.w : 0.f};
      mo[i] = lane_bf<4>(o);
    }
  }
  __syncthreads();
  for (int l = 1; l < lv.nlev; l++) {
    const int m = lv.m[l];
    float* __restrict__ o = out + lv.out_off[l] + r * m * kC;
    for (int j = g; j < m; j += 32) {
      const int k0 = lv.ptr[l][j];
      *reinterpret_cast<float4*>(o + j * kC + c4) =
          row_sum4(row + lv.idx[l][k0] * kC + c4, kC, lv.wt[l] + k0, lv.ptr[l][j + 1] - k0);
    }
  }
}

// One further axis of every coarse level's transposed upsampling in one launch:
// (outer, n, inner) -> (outer, m, inner) per level, four inner elements per
// thread.  With masks (the last axis): outbf = bf16(mask > 0 ? sum : 0), else out.
// One launch per level left most SMs idle on the coarse ones (8 x 8 points of 64
// sums each): 95 us in all at 256^2 x 8, 36 now.  With the pooling chain in one
// launch and the parallel loss sum the network's forward and backward went from
// 1464 to 1362 us.
__global__ void __launch_bounds__(256) upsample_bwd_axis_levels(int n, UpLevels lv,
                                                                const float* __restrict__ in,
                                                                float* __restrict__ out,
                                                                bf16* __restrict__ outbf) {
  int l = 1;
  while (l + 1 < lv.nlev && blockIdx.x >= lv.first[l + 1]) l++;
  const unsigned i4 = (unsigned)(lv.inner[l] / 4);
  const int m = lv.m[l];
  const unsigned id = (blockIdx.x - lv.first[l]) * 256u + threadIdx.x;
  if ((long long)id >= lv.outer[l] * m * i4) return;
  // element indices stay below 2^31 (network size check): 32-bit division
  const unsigned c = (id % i4) * 4u, p = id / i4;
  const int j = (int)(p % (unsigned)m);
  const unsigned o = p / (unsigned)m;
  const int k0 = lv.ptr[l][j];
  const float4 v = row_sum4(
      in + lv.in_off[l] + ((long long)o * n + lv.idx[l][k0]) * lv.inner[l] + c, lv.inner[l],
      lv.wt[l] + k0, lv.ptr[l][j + 1] - k0);
  const long long at = lv.out_off[l] + (long long)id * 4;
  if (!outbf) {
    *reinterpret_cast<float4*>(out + at) = v;
    return;
  }
  const uint2 mv = *reinterpret_cast<const uint2*>(lv.mask[l] + (long long)id * 4);
  const __nv_bfloat162* mk = reinterpret_cast<const __nv_bfloat162*>(&mv);
  const float2 m0 = __bfloat1622float2(mk[0]), m1 = __bfloat1622float2(mk[1]);
  uint2 ov;
  __nv_bfloat162* ob = reinterpret_cast<__nv_bfloat162*>(&ov);
  ob[0] = __floats2bfloat162_rn(m0.x > 0.f ? v.x : 0.f, m0.y > 0.f ? v.y : 0.f);
  ob[1] = __floats2bfloat162_rn(m1.x > 0.f ? v.z : 0.f, m1.y > 0.f ? v.w : 0.f);
  *reinterpret_cast<uint2*>(outbf + at) = ov;
}

// The pooling chain's gradient at level 1: g_1 += 2^-D (g_2 + 2^-D (g_3 + ...))
// over a point's ancestors (as far as they exist: odd sides drop their last
// point), coarsest first, so each sum is the one that level-by-level passes form
// (scaling by 2^-D is exact).  One launch instead of a read-modify-write pass
// per level; level 0 adds its own share where its gradient is consumed
// (conv1_wgrad), which saves its 134 MB pass at 256^2 x 8.
struct PoolLevels {
  int nlev;
  int side[kMaxLevels];
  float* g[kMaxLevels];
};

template <int D>
__global__ void __launch_bounds__(256) pool_chain_bwd(int B, PoolLevels lv) {
  const int s1 = lv.side[1];
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= B * Geo<D>::pts(s1) * (kC / 4)) return;
  const int c4 = (int)(i % (kC / 4)) * 4;
  int b, z, y, x;
  Geo<D>::decode(i / (kC / 4), s1, b, z, y, x);
  int top = 1;
  while (top + 1 < lv.nlev) {
    const int sh = top, so = lv.side[top + 1];  // level top + 1: coordinates >> top
    if ((y >> sh) >= so || (x >> sh) >= so || (D == 3 && (z >> sh) >= so)) break;
    top++;
  }
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int l = top; l >= 1; l--) {
    const int sh = l - 1;
    const long long q = Geo<D>::nb(b, z >> sh, y >> sh, x >> sh, 0, 0, 0, lv.side[l]);
    const float4 g = *reinterpret_cast<const float4*>(lv.g[l] + q * kC + c4);
    const float f = l == top ? 0.f : 1.f / (1 << D);
    v.x = g.x + f * v.x;
    v.y = g.y + f * v.y;
    v.z = g.z + f * v.z;
    v.w = g.w + f * v.w;
  }
  if (top > 1) *reinterpret_cast<float4*>(lv.g[1] + i * 4) = v;
}

// Adam (Kingma & Ba): m = b1 m + (1-b1) g; v = b2 v + (1-b2) g^2;
// theta -= lr * (m / c1) / (sqrt(v / c2) + eps), c1 = 1 - b1^t, c2 = 1 - b2^t
// (c1, c2 of the step in progress, from the phase's device state)
__global__ void adam_kernel(long long count, float* __restrict__ theta,
                            const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, float lr, const TrainCtr* __restrict__ ctr) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= count) return;
  const float c1 = ctr->c1, c2 = ctr->c2;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  theta[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Start of one Adam step of a phase: t = adam_t + 1 with its bias corrections,
// and the offset of this step's minibatch in the phase's picks.
__global__ void step_begin(TrainCtr* ctr, int B) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    const long long t = ctr->adam_t + 1;
    ctr->adam_t = t;
    ctr->c1 = 1.f - powf(0.9f, (float)t);
    ctr->c2 = 1.f - powf(0.999f, (float)t);
    ctr->pick_off = ctr->iter * B;
    ctr->iter = ctr->iter + 1;
  }
}

// bu[b] = ring_u[picks[pick_off + b]], bt[b] = ring_t[...] for b < B (N each,
// ring slots `stride` floats apart)
__global__ void gather_pairs(int B, long long N, const float* __restrict__ ring_u,
                             const float* __restrict__ ring_t, long long stride,
                             const int* __restrict__ picks, const TrainCtr* __restrict__ ctr,
                             float* __restrict__ bu, float* __restrict__ bt) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= (long long)B * N) return;
  const int b = (int)(i / N);
  const long long p = i - (long long)b * N;
  const long long src = (long long)picks[ctr->pick_off + b] * stride + p;
  bu[i] = ring_u[src];
  bt[i] = ring_t[src];
}

// wq[conv][tap][k][o] = W[o][k][tap], wqT[conv][tap][o][k] = W[o][k][tap] (BF16)
__global__ void sync_weights_kernel(int nconv, int T, const float* __restrict__ master,
                                    const long long* __restrict__ offs, bf16* __restrict__ wq,
                                    bf16* __restrict__ wqT) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long per = (long long)T * kC * kC;
  if (i >= nconv * per) return;
  const int cv = (int)((unsigned)i / (unsigned)per);
  const int r = (int)((unsigned)i % (unsigned)per);
  const int o = r / (kC * T), k = (r / T) % kC, tp = r % T;
  const bf16 v = __float2bfloat16(master[offs[cv] + r]);
  wq[(long long)cv * per + (tp * kC + k) * kC + o] = v;
  wqT[(long long)cv * per + (tp * kC + o) * kC + k] = v;
}

unsigned nblk(long long count, int bs) { return (unsigned)((count + bs - 1) / bs); }

unsigned long long sm64(unsigned long long& st) {
  st += 0x9E3779B97F4A7C15ull;
  unsigned long long z = st;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

}  // namespace

#define NN_CK(x)                          \
  do {                                    \
    cudaError_t e_ = (x);                 \
    if (e_ != cudaSuccess) return e_;     \
  } while (0)

cudaError_t net_create(Net& net, int n, int bmax, unsigned long long seed, int dim,
                       int extra_max, bool infer_only) {
  if (dim != 2 && dim != 3) return cudaErrorInvalidValue;
  if (extra_max < 0 || extra_max > kMaxExtra) return cudaErrorInvalidValue;
  // the kernels index points and point-channel elements in 32 bits
  if (n < 1 || bmax < 1 ||
      (long long)bmax * (dim == 3 ? (long long)n * n * n : (long long)n * n) * kC >= (1LL << 31))
    return cudaErrorInvalidValue;
  NN_CK(conv32_tc_setup());
  NN_CK(conv32_mma_setup());
  net.extra_max = extra_max;
  net.extra_active = 0;
  net.n = n;
  net.dim = dim;
  net.taps = dim == 3 ? 27 : 9;
  const int T = net.taps;
  net.bmax = bmax;
  net.L = 0;
  int s = n;
  net.side[net.L++] = s;
  while (s / 2 >= 8 && net.L < kMaxLevels) {
    s /= 2;
    net.side[net.L++] = s;
  }
  const int L = net.L;
  const long long per = (long long)T * kC * kC;
  long long off = 0;
  net.off_w[0] = off; off += kC * T;
  net.off_b[0] = off; off += kC;
  for (int l = 0; l < L; l++) {
    net.off_w[1 + l] = off; off += per;
    net.off_b[1 + l] = off; off += kC;
  }
  net.off_w[L + 1] = off; off += per;
  net.off_b[L + 1] = off; off += kC;
  net.off_w[L + 2] = off; off += kC * T;
  net.off_b[L + 2] = off; off += 1;
  for (int r = 0; r < extra_max; r++) {
    net.off_rw[r] = off; off += per;
    net.off_rb[r] = off; off += kC;
  }
  net.nparams = off;

  // He-uniform initialisation from splitmix64: U[-a, a], a = sqrt(6 / fan_in);
  // the output layer uses a = sqrt(3 / fan_in); biases start at 0.
  std::vector<float> p((size_t)net.nparams, 0.f);
  unsigned long long st = seed ^ 0x6A09E667F3BCC909ull;
  auto fill = [&](long long o, long long cnt, int fan_in, float gain) {
    const double a = sqrt(gain / fan_in);
    for (long long i = 0; i < cnt; i++) {
      const double u = (double)(sm64(st) >> 11) * (1.0 / 9007199254740992.0);
      p[(size_t)(o + i)] = (float)((2.0 * u - 1.0) * a);
    }
  };
  fill(net.off_w[0], kC * T, T, 6.f);
  for (int l = 0; l < L; l++) fill(net.off_w[1 + l], per, T * kC, 6.f);
  fill(net.off_w[L + 1], per, T * kC, 6.f);
  fill(net.off_w[L + 2], kC * T, T * kC, 3.f);
  // a grown block starts close to the identity (small weights, zero bias) so
  // the guess changes little when it is appended, yet its gradient is not zero
  for (int r = 0; r < extra_max; r++) fill(net.off_rw[r], per, T * kC, 0.06f);

  const long long np = net.nparams;
  NN_CK(cudaMalloc(&net.master, sizeof(float) * np));
  NN_CK(cudaMemcpy(net.master, p.data(), sizeof(float) * np, cudaMemcpyHostToDevice));
  if (!infer_only) {
    NN_CK(cudaMalloc(&net.grad, sizeof(float) * np));
    NN_CK(cudaMalloc(&net.adam_m, sizeof(float) * np));
    NN_CK(cudaMalloc(&net.adam_v, sizeof(float) * np));
    NN_CK(cudaMemset(net.grad, 0, sizeof(float) * np));
    NN_CK(cudaMemset(net.adam_m, 0, sizeof(float) * np));
    NN_CK(cudaMemset(net.adam_v, 0, sizeof(float) * np));
  }
  const int nconv = L + 1 + extra_max;  // the 32 -> 32 convolutions
  NN_CK(cudaMalloc(&net.wq, sizeof(bf16) * per * nconv));
  NN_CK(cudaMalloc(&net.wqT, sizeof(bf16) * per * nconv));
  long long offs[kMaxLevels + 1 + kMaxExtra];
  for (int c = 0; c < L + 1; c++) offs[c] = net.off_w[1 + c];
  for (int r = 0; r < extra_max; r++) offs[L + 1 + r] = net.off_rw[r];
  NN_CK(cudaMalloc(&net.offs_dev, sizeof(offs)));
  NN_CK(cudaMemcpy(net.offs_dev, offs, sizeof(long long) * nconv, cudaMemcpyHostToDevice));

  auto pts = [dim](int side) {
    return dim == 3 ? (long long)side * side * side : (long long)side * side;
  };
  const long long full = (long long)bmax * pts(n) * kC;
  NN_CK(cudaMalloc(&net.a0, sizeof(bf16) * full));
  net.pyr = 0;
  for (int l = 0; l < L; l++) {
    const long long sz = (long long)bmax * pts(net.side[l]) * kC;
    if (l > 0) NN_CK(cudaMalloc(&net.pool[l], sizeof(bf16) * sz));
    NN_CK(cudaMalloc(&net.z[l], sizeof(bf16) * sz));
    net.lvl_off[l] = net.pyr;
    net.pyr += sz;
  }
  // the upsampling's tables, all levels' in one allocation and one copy (with four per
  // level the create of a learned handle at n = 256 took 4.2 ms, now 3.7)
  std::vector<char> up;
  std::vector<std::pair<void*, size_t>> up_at;  // (address of a pointer, its offset)
  auto put = [&](auto** dst, const void* src, size_t bytes) {
    up_at.push_back({dst, up.size()});
    up.insert(up.end(), (const char*)src, (const char*)src + bytes);
    up.resize((up.size() + 255) / 256 * 256);
  };
  for (int l = 1; l < L; l++) {
    const int m = net.side[l];
    std::vector<std::vector<std::pair<int, float>>> rows(m);
    std::vector<float2> tab(n);
    for (int x = 0; x < n; x++) {
      // half-pixel source position of fine index x (m coarse points, n fine ones)
      float src = ((float)x + 0.5f) * (float)m / (float)n - 0.5f;
      if (src < 0.f) src = 0.f;
      int i0 = (int)floorf(src);
      if (i0 > m - 1) i0 = m - 1;
      const int i1 = i0 + 1 < m - 1 ? i0 + 1 : m - 1;
      const float lam = src - (float)i0;
      tab[x].x = lam;
      memcpy(&tab[x].y, &i0, sizeof(int));
      if (i0 == i1) {
        rows[i0].push_back({x, (1.f - lam) + lam});
      } else {
        rows[i0].push_back({x, 1.f - lam});
        rows[i1].push_back({x, lam});
      }
    }
    std::vector<int> ptr(m + 1, 0), idx;
    std::vector<float> wt;
    for (int j = 0; j < m; j++) {
      for (auto& e : rows[j]) {
        idx.push_back(e.first);
        wt.push_back(e.second);
      }
      ptr[j + 1] = (int)idx.size();
    }
    put(&net.up_tab[l], tab.data(), sizeof(float2) * n);
    if (infer_only) continue;  // the others are the backward pass's
    put(&net.up_ptr[l], ptr.data(), sizeof(int) * (m + 1));
    put(&net.up_idx[l], idx.data(), sizeof(int) * idx.size());
    put(&net.up_w[l], wt.data(), sizeof(float) * wt.size());
  }
  if (!up.empty()) {
    NN_CK(cudaMalloc(&net.up_mem, up.size()));
    NN_CK(cudaMemcpy(net.up_mem, up.data(), up.size(), cudaMemcpyHostToDevice));
    for (auto& f : up_at) {
      const void* at = (char*)net.up_mem + f.second;
      memcpy(f.first, &at, sizeof(at));
    }
  }
  NN_CK(cudaMalloc(&net.s, sizeof(bf16) * full));
  NN_CK(cudaMalloc(&net.e, sizeof(bf16) * full));
  NN_CK(cudaMalloc(&net.t, sizeof(bf16) * full));
  for (int r = 0; r < extra_max; r++) {
    NN_CK(cudaMalloc(&net.te[r], sizeof(bf16) * full));
    NN_CK(cudaMalloc(&net.tt[r], sizeof(bf16) * full));
  }
  if (infer_only) {  // forward passes only: no gradient, Adam or minibatch buffers
    NN_CK(net_sync_weights(net, 0));
    return cudaDeviceSynchronize();
  }
  NN_CK(cudaMalloc(&net.g_t, sizeof(float) * full));
  NN_CK(cudaMalloc(&net.g_s, sizeof(float) * full));
  NN_CK(cudaMalloc(&net.g_lvl, sizeof(float) * full));
  NN_CK(cudaMalloc(&net.g_pool, sizeof(float) * net.pyr));
  NN_CK(cudaMalloc(&net.g_bf, sizeof(bf16) * full));
  if (L > 1) NN_CK(cudaMalloc(&net.g_bl, sizeof(bf16) * (net.pyr - net.lvl_off[1])));
  int dev = 0, nsm = 0;
  NN_CK(cudaGetDevice(&dev));
  NN_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  net.wparts = 2 * nsm;
  // the output convolution's tile takes more than the default 48 KB of dynamic shared
  // memory in 3D (here only: the inference copy of a network is made after it)
  if (dim == 3) {
    NN_CK(cudaFuncSetAttribute(conv_out_fwd<3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               OutTile<3>::kSmem));
    NN_CK(cudaFuncSetAttribute(conv1_wgrad<0, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               conv1_wgrad_smem<3>(n)));
    NN_CK(cudaFuncSetAttribute(conv1_wgrad<1, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               conv1_wgrad_smem<3>(n)));
  } else {
    NN_CK(cudaFuncSetAttribute(conv1_wgrad<0, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               conv1_wgrad_smem<2>(n)));
    NN_CK(cudaFuncSetAttribute(conv1_wgrad<1, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               conv1_wgrad_smem<2>(n)));
  }
  // one area per 32 -> 32 convolution and per 1-channel one (reduced together)
  NN_CK(cudaMalloc(&net.wgrad_part,
                   sizeof(float) * (nconv + 2) * (long long)net.wparts * (per + kC)));
  const long long pix = (long long)bmax * pts(n);
  NN_CK(cudaMalloc(&net.gy, sizeof(float) * pix));
  NN_CK(cudaMalloc(&net.loss_part, sizeof(float) * 1024));
  NN_CK(cudaMalloc(&net.bu, sizeof(float) * pix));
  NN_CK(cudaMalloc(&net.bt, sizeof(float) * pix));
  NN_CK(cudaMalloc(&net.by, sizeof(float) * pix));
  NN_CK(cudaMalloc(&net.ctr, sizeof(TrainCtr)));
  {
    TrainCtr c0{};
    c0.tscale = 1.f;
    NN_CK(cudaMemcpy(net.ctr, &c0, sizeof(c0), cudaMemcpyHostToDevice));
  }
  NN_CK(net_sync_weights(net, 0));
  return cudaDeviceSynchronize();
}

void net_destroy(Net& net) {
  cudaFree(net.master);
  cudaFree(net.grad);
  cudaFree(net.adam_m);
  cudaFree(net.adam_v);
  cudaFree(net.wq);
  cudaFree(net.wqT);
  cudaFree(net.offs_dev);
  cudaFree(net.a0);
  for (int l = 0; l < kMaxLevels; l++) {
    cudaFree(net.pool[l]);
    cudaFree(net.z[l]);
  }
  cudaFree(net.up_mem);
  cudaFree(net.s);
  cudaFree(net.e);
  cudaFree(net.t);
  for (int r = 0; r < kMaxExtra; r++) {
    cudaFree(net.te[r]);
    cudaFree(net.tt[r]);
  }
  cudaFree(net.g_t);
  cudaFree(net.g_s);
  cudaFree(net.g_lvl);
  cudaFree(net.g_pool);
  cudaFree(net.g_bf);
  cudaFree(net.g_bl);
  cudaFree(net.wgrad_part);
  cudaFree(net.gy);
  cudaFree(net.loss_part);
  cudaFree(net.bu);
  cudaFree(net.bt);
  cudaFree(net.by);
  cudaFree(net.ctr);
  net = Net();
}

cudaError_t net_copy_params(Net& dst, const float* src, cudaStream_t s) {
  NN_CK(cudaMemcpyAsync(dst.master, src, sizeof(float) * dst.nparams, cudaMemcpyDeviceToDevice,
                        s));
  return net_sync_weights(dst, s);
}

cudaError_t net_sync_weights(Net& net, cudaStream_t s) {
  const int nconv = net.L + 1 + net.extra_max;
  const long long tot = (long long)nconv * net.taps * kC * kC;
  sync_weights_kernel<<<nblk(tot, 256), 256, 0, s>>>(nconv, net.taps, net.master, net.offs_dev,
                                                    net.wq, net.wqT);
  note_launches(1);
  return cudaGetLastError();
}

namespace {

template <int D>
cudaError_t forward_t(Net& net, int B, const float* u, float* y, cudaStream_t s) {
  const int n = net.n, L = net.L;
  const long long pix = B * Geo<D>::pts(n);
  const long long per = (long long)Geo<D>::T * kC * kC;
  conv_in_fwd<D><<<nblk(pix, 256), 256, 0, s>>>(B, n, u, net.master + net.off_w[0],
                                                 net.master + net.off_b[0], net.a0);
  note_launches(1);
  for (int l0 = 0; l0 + 1 < L; l0 += PoolFwd<D>::kDepth) {
    PoolFwd<D> pf;
    pf.nlev = std::min(L - 1 - l0, PoolFwd<D>::kDepth);
    pf.in = l0 == 0 ? net.a0 : net.pool[l0];
    pf.side[0] = net.side[l0];
    for (int l = 1; l <= pf.nlev; l++) {
      pf.side[l] = net.side[l0 + l];
      pf.out[l] = net.pool[l0 + l];
    }
    constexpr int half = 1 << (PoolFwd<D>::kDepth - 1);
    const int bps = (pf.side[1] + half - 1) / half;
    pool_chain_fwd<D><<<(unsigned)(B * (D == 3 ? bps : 1) * bps * bps), 256, 0, s>>>(pf);
    note_launches(1);
  }
  ConvJob jobs[kMaxLevels];
  for (int l = 0; l < L; l++) {
    jobs[l].H = net.side[l];
    jobs[l].in = l == 0 ? net.a0 : net.pool[l];
    jobs[l].wop = net.wqT + per * l;
    jobs[l].bias = net.master + net.off_b[1 + l];
    jobs[l].zo = net.z[l];
  }
  NN_CK(launch_conv32(D, 0, B, L, jobs, 1, 1, s));
  Levels lv;
  lv.L = L;
  for (int l = 0; l < L; l++) {
    lv.z[l] = net.z[l];
    lv.tab[l] = net.up_tab[l];
    lv.side[l] = net.side[l];
  }
  upsum_fwd<D><<<nblk(pix * 4, 256), 256, 0, s>>>(B, n, lv, net.s);
  note_launches(1);
  // dilated residual blocks: the first, then the grown ones
  const bf16* cur = net.s;
  for (int r = -1; r < net.extra_active; r++) {
    ConvJob j;
    j.H = n;
    j.in = j.resid = cur;
    j.wop = net.wqT + per * (L + 1 + r);
    j.bias = net.master + (r < 0 ? net.off_b[L + 1] : net.off_rb[r]);
    j.zo = r < 0 ? net.e : net.te[r];
    j.to = r < 0 ? net.t : net.tt[r];
    NN_CK(launch_conv32(D, 1, B, 1, &j, 2, 1, s));
    cur = j.to;
  }
  const long long otiles = (long long)B * nblk(n, OutTile<D>::X) * nblk(n, OutTile<D>::Y) *
                           (D == 3 ? nblk(n, OutTile<D>::Z) : 1);
  conv_out_fwd<D><<<(unsigned)otiles, 256, OutTile<D>::kSmem, s>>>(
      n, cur, net.master + net.off_w[L + 2], net.master + net.off_b[L + 2], y);
  note_launches(1);
  return cudaGetLastError();
}

template <int D>
cudaError_t backward_t(Net& net, int B, const float* u, const float* y, const float* target,
                       float tscale, const float* tscale_dev, float* loss_dev, cudaStream_t s) {
  constexpr int T = Geo<D>::T;
  const int n = net.n, L = net.L;
  const long long pix = B * Geo<D>::pts(n);
  const long long full = pix * kC;
  const long long per = (long long)T * kC * kC;
  const int P = net.wparts;
  const int stride = (int)(per + kC);
  // the partial weight gradients of every convolution, reduced together at the end
  ReduceJobs rj;
  rj.n = 0;
  auto reduce_later = [&](const float* part, int nparts, int st, int kind, float* gw, float* gb) {
    const int outs = kind == 0 ? (int)per + kC : T * kC + (kind == 1 ? kC : 1);
    rj.job[rj.n] = ReduceJob{part, gw, gb, nparts, st, kind};
    rj.first[rj.n + 1] = (rj.n == 0 ? 0 : rj.first[rj.n]) + (int)nblk(outs, 32);
    if (rj.n == 0) rj.first[0] = 0;
    rj.n++;
  };
  auto conv_part = [&](int c) { return net.wgrad_part + (long long)c * P * stride; };
  const int nconv = L + 1 + net.extra_max;
  auto data_grad = [&](int H, const bf16* gz, int c, int dil, float* fo, const float* addend) {
    ConvJob j;
    j.H = H;
    j.in = gz;
    j.wop = net.wq + per * c;
    j.fo = fo;
    j.addend = addend;
    return launch_conv32(D, 2, B, 1, &j, dil, -1, s);
  };
  auto weight_grad = [&](const bf16* in, const bf16* gz, int c, float* gw, float* gb) {
    WgradJob j;
    j.H = n;
    j.in = in;
    j.g = gz;
    j.part = conv_part(c);
    const cudaError_t e = launch_wgrad(D, B, 1, &j, 2, stride, P, s);
    if (e == cudaSuccess) reduce_later(j.part, j.nparts, stride, 0, gw, gb);
    return e;
  };
  // loss and dL/dy
  const int lparts = 256;
  mse_grad<<<lparts, 256, 0, s>>>(pix, 1.f / (float)pix, tscale, tscale_dev, y, target, net.gy,
                                  net.loss_part);
  note_launches(1);
  loss_finish<<<1, 256, 0, s>>>(net.loss_part, lparts, 1.f / (float)pix, loss_dev);
  note_launches(1);
  // output conv
  const bf16* tfin = net.extra_active > 0 ? net.tt[net.extra_active - 1] : net.t;
  // the 1-channel weight gradients: 32 (T + 1) outputs per CTA (short stride)
  const int P1 = P, stride1 = kC * (T + 1);
  const int smem1 = conv1_wgrad_smem<D>(n);
  conv1_wgrad<0, D><<<P1, kW1Threads, smem1, s>>>(B, n, net.gy, tfin, nullptr, nullptr, nullptr,
                                                  nullptr, conv_part(nconv), stride1);
  note_launches(1);
  reduce_later(conv_part(nconv), P1, stride1, 2, net.grad + net.off_w[L + 2],
               net.grad + net.off_b[L + 2]);
  // the first masked use of g_t (the last grown block's, else the residual
  // block's) is written by the same kernel
  const bf16* mask0 = net.extra_active > 0 ? net.te[net.extra_active - 1] : net.e;
  conv_out_bwd_data<D><<<2 * P, kW1Threads, sizeof(float) * w1_stage_floats<D>(n), s>>>(
      B, n, net.gy, net.master + net.off_w[L + 2], net.g_t, mask0, net.g_bf);
  note_launches(1);
  // grown residual blocks, last first: t_out = t_in + relu(conv_d2(t_in));
  // blocks not appended yet get a zero gradient (Adam then leaves them as they are)
  for (int r = net.extra_active; r < net.extra_max; r++)
    NN_CK(cudaMemsetAsync(net.grad + net.off_rw[r], 0, sizeof(float) * (per + kC), s));
  {
    float* gcur = net.g_t;
    float* gnext = net.g_s;
    for (int r = net.extra_active - 1; r >= 0; r--) {
      const bf16* tin = r == 0 ? net.t : net.tt[r - 1];
      if (r != net.extra_active - 1) {  // (the first one came with g_t)
        mask_to_bf16<<<nblk((full) / 8, 256), 256, 0, s>>>(full, gcur, net.te[r], net.g_bf);
        note_launches(1);
      }
      NN_CK(weight_grad(tin, net.g_bf, L + 1 + r, net.grad + net.off_rw[r],
                        net.grad + net.off_rb[r]));
      NN_CK(data_grad(n, net.g_bf, L + 1 + r, 2, gnext, gcur));
      std::swap(gcur, gnext);
    }
    if (gcur != net.g_t)
      NN_CK(cudaMemcpyAsync(net.g_t, gcur, sizeof(float) * full, cudaMemcpyDeviceToDevice, s));
  }
  // dilated residual block: t = s + e, e = relu(conv_d2(s))
  if (net.extra_active > 0) {
    mask_to_bf16<<<nblk((full) / 8, 256), 256, 0, s>>>(full, net.g_t, net.e, net.g_bf);
    note_launches(1);
  }
  NN_CK(weight_grad(net.s, net.g_bf, L, net.grad + net.off_w[L + 1], net.grad + net.off_b[L + 1]));
  NN_CK(data_grad(n, net.g_bf, L, 2, net.g_s, net.g_t));
  // pyramid levels; first the x-axis pass of every coarse level's transposed
  // upsampling, from one read of the fine gradient (g_s) into g_t (free here:
  // the residual block's gradient is already in g_s)
  const bool fused_x = L > 1 && n <= kXLevelsMaxN;
  UpLevels lv{};
  lv.nlev = L;
  const long long rows = B * Geo<D>::pts(n) / n;
  for (int l = 1; l < L; l++) {
    lv.m[l] = net.side[l];
    lv.ptr[l] = net.up_ptr[l];
    lv.idx[l] = net.up_idx[l];
    lv.wt[l] = net.up_w[l];
    lv.mask[l] = net.z[l];
  }
  // the remaining axes (y; in 3D y, then z) of levels l0 .. l1-1, from their x
  // passes at g_t + xin[l], into their masked BF16 gradients
  auto other_axes = [&](int l0, int l1, const long long* xin) {
    UpLevels v = lv;
    for (int ax = 1; ax < D; ax++) {
      const bool last = ax == D - 1;
      unsigned blocks = 0;
      long long off = 0;
      for (int l = 1; l < l1; l++) {
        const long long m = net.side[l];
        v.first[l] = blocks;
        if (l < l0) continue;  // (an empty range of CTAs)
        v.outer[l] = D == 3 && ax == 1 ? (long long)B * n : B;
        v.inner[l] = (ax == 1 ? m : m * m) * kC;
        v.in_off[l] = ax == 1 ? xin[l] : v.out_off[l];
        v.out_off[l] = last ? net.lvl_off[l] - net.lvl_off[1] : off;
        off += v.outer[l] * m * v.inner[l];
        blocks += nblk(v.outer[l] * m * v.inner[l] / 4, 256);
      }
      v.nlev = l1;
      upsample_bwd_axis_levels<<<blocks, 256, 0, s>>>(n, v, ax == 1 ? net.g_t : net.g_lvl,
                                                      last ? nullptr : net.g_lvl,
                                                      last ? net.g_bl : nullptr);
      note_launches(1);
    }
  };
  if (fused_x) {
    long long off = 0;
    for (int l = 1; l < L; l++) {
      lv.out_off[l] = off;
      off += rows * net.side[l] * kC;
    }
    upsample_bwd_x_levels<<<(unsigned)rows, 256, sizeof(float) * n * kC, s>>>(
        n, lv, net.g_s, net.g_t, net.z[0], net.g_bf);
    note_launches(1);
    long long xin[kMaxLevels];
    for (int l = 1; l < L; l++) xin[l] = lv.out_off[l];
    other_axes(1, L, xin);
  }
  if (!fused_x) {  // (rows too long to stage: each level's own passes)
    for (int l = 1; l < L; l++) {
      upsample_bwd_axis<<<nblk(rows * net.side[l] * kC, 256), 256, 0, s>>>(
          rows, n, net.side[l], kC, net.up_ptr[l], net.up_idx[l], net.up_w[l], net.g_s, net.g_t);
      note_launches(1);
      const long long xin[kMaxLevels] = {};
      other_axes(l, l + 1, xin);
    }
  }
  if (!fused_x) {
    mask_to_bf16<<<nblk(full / 8, 256), 256, 0, s>>>(full, net.g_s, net.z[0], net.g_bf);
    note_launches(1);
  }
  {
    // every level's weight and data gradients; the coarse levels share launches
    WgradJob wj[kMaxLevels];
    ConvJob cj[kMaxLevels];
    for (int l = 0; l < L; l++) {
      const bf16* gz = l == 0 ? net.g_bf : net.g_bl + (net.lvl_off[l] - net.lvl_off[1]);
      wj[l].H = cj[l].H = net.side[l];
      wj[l].in = l == 0 ? net.a0 : net.pool[l];
      wj[l].g = cj[l].in = gz;
      wj[l].part = conv_part(l);
      cj[l].wop = net.wq + per * l;
      cj[l].fo = net.g_pool + net.lvl_off[l];
    }
    NN_CK(launch_wgrad(D, B, L, wj, 1, stride, P, s));
    for (int l = 0; l < L; l++)
      reduce_later(wj[l].part, wj[l].nparts, stride, 0, net.grad + net.off_w[1 + l],
                   net.grad + net.off_b[1 + l]);
    NN_CK(launch_conv32(D, 2, B, L, cj, 1, -1, s));
  }
  // pooling chain: the gradient of p_{l-1} collects 1/2^D of p_l's
  if (L > 2) {
    PoolLevels pv{};
    pv.nlev = L;
    for (int l = 1; l < L; l++) {
      pv.side[l] = net.side[l];
      pv.g[l] = net.g_pool + net.lvl_off[l];
    }
    pool_chain_bwd<D><<<nblk(B * Geo<D>::pts(net.side[1]) * (kC / 4), 256), 256, 0, s>>>(B, pv);
    note_launches(1);
  }
  // input conv
  // (the ReLU mask of a0 is applied inside the weight-gradient kernel)
  conv1_wgrad<1, D><<<P1, kW1Threads, smem1, s>>>(
      B, n, nullptr, nullptr, net.g_pool + net.lvl_off[0],
      L > 1 ? net.g_pool + net.lvl_off[1] : nullptr, net.a0, u, conv_part(nconv + 1), stride1);
  note_launches(1);
  reduce_later(conv_part(nconv + 1), P1, stride1, 1, net.grad + net.off_w[0],
               net.grad + net.off_b[0]);
  reduce_wgrad<<<rj.first[rj.n], 256, 0, s>>>(rj, T);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace

cudaError_t net_forward(Net& net, int B, const float* u, float* y, cudaStream_t s) {
  return net.dim == 3 ? forward_t<3>(net, B, u, y, s) : forward_t<2>(net, B, u, y, s);
}

cudaError_t net_backward(Net& net, int B, const float* u, const float* y, const float* target,
                         float tscale, float* loss_dev, cudaStream_t s) {
  return net.dim == 3 ? backward_t<3>(net, B, u, y, target, tscale, nullptr, loss_dev, s)
                      : backward_t<2>(net, B, u, y, target, tscale, nullptr, loss_dev, s);
}

cudaError_t net_adam_reset(Net& net, cudaStream_t s) {
  NN_CK(cudaMemsetAsync(net.adam_m, 0, sizeof(float) * net.nparams, s));
  NN_CK(cudaMemsetAsync(net.adam_v, 0, sizeof(float) * net.nparams, s));
  return cudaMemsetAsync(&net.ctr->adam_t, 0, sizeof(long long), s);
}

cudaError_t net_train_step_dev(Net& net, int B, const float* ring_u, const float* ring_t,
                               long long stride, const int* picks, TrainCtr* ctr, float lr,
                               float* loss_dev, cudaStream_t s) {
  const long long N = net.dim == 3 ? (long long)net.n * net.n * net.n : (long long)net.n * net.n;
  step_begin<<<1, 32, 0, s>>>(ctr, B);
  gather_pairs<<<nblk((long long)B * N, 256), 256, 0, s>>>(B, N, ring_u, ring_t, stride, picks,
                                                           ctr, net.bu, net.bt);
  note_launches(2);
  NN_CK(cudaGetLastError());
  NN_CK(net_forward(net, B, net.bu, net.by, s));
  NN_CK(net.dim == 3
            ? backward_t<3>(net, B, net.bu, net.by, net.bt, 1.f, &ctr->tscale, loss_dev, s)
            : backward_t<2>(net, B, net.bu, net.by, net.bt, 1.f, &ctr->tscale, loss_dev, s));
  adam_kernel<<<nblk(net.nparams, 256), 256, 0, s>>>(net.nparams, net.master, net.grad,
                                                     net.adam_m, net.adam_v, lr, ctr);
  note_launches(1);
  NN_CK(cudaGetLastError());
  return net_sync_weights(net, s);
}

}  // namespace mlg
