// photometry.cu -- the photometric-accuracy and binning experiments (Sect.
// 4.2, 4.3): median binning of consecutive frames, fake companion injection
// into raw frames, aperture photometry of the reduced image.
//
//  * bin_median_kernel<W, V>: one thread per group and V pixels; the group's
//    B <= W values are loaded (coalesced along the pixels, all loads in
//    flight) and the two middle ones of W slots taken by an odd-even merge
//    network pruned to them, in registers (all indices compile-time).
//    HBM-bound: T x n^2 x 4 B read, ceil(T/B) x n^2 x 4 B written.
//    1000 frames of 512 x 512 by 10: 0.167 ms = 6.9 TB/s, the copy rate
//    (0.60 with a 16-key bitonic sort of total-order keys).  Loading two
//    pixels per thread with every load ahead of the first comparison, in a
//    branch of its own for full bins, is what brings it there: with the
//    slot tests between the loads it ran at 4.7 TB/s.
//    Groups of more than 64 frames go to the median collapse kernel, one
//    launch per group; the collapse of at most 64 frames comes here as one
//    group.
//  * inject_kernel: one block per frame; companions in turn (a barrier
//    between them, so overlapping windows never race), each over its window
//    of (2 half + 1)^2 pixels; positions and windows come from the FP64 host
//    plan, the Moffat profile is evaluated in FP32.
//  * aperture_kernel: one block per aperture over the bounding box of the
//    disc, FP64 block sum.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "graphic_internal.h"
#include "select_common.cuh"

namespace graphic {
namespace {

constexpr int BIN_THREADS = 128;

// V pixels per thread (V = 2: 8-byte loads) and W value slots per pixel, W
// even and at least the group's m values.  The W - m free slots are padded
// with -inf and +inf so that the middle values of the m sit in the middle of
// the W: (W - m) / 2 of them, rounded down, below (an odd m leaves one more
// above).  All loads are issued before the first comparison.
template <int W, int V>
__global__ void __launch_bounds__(BIN_THREADS) bin_median_kernel(const float *__restrict__ in, float *__restrict__ out,
                                                                 long long T, long long nn, long long fs, int B,
                                                                 unsigned blocks_per_group, int *status) {
  const long long g = blockIdx.x / blocks_per_group;
  const long long p = ((long long)(blockIdx.x % blocks_per_group) * BIN_THREADS + threadIdx.x) * V;
  if (p >= nn) return;
  const long long f0 = g * B;
  const int m = (int)((T - f0) < B ? (T - f0) : B);
  const float *src = in + f0 * fs + p;
  float v[V][W];
  float acc = 0.f;   // 0 while every value is finite: v * 0 is NaN for NaN and infinities
  auto load = [&](int i, bool there, float pad) {
    if constexpr (V == 2) {
      const float2 x = there ? __ldcs(reinterpret_cast<const float2 *>(src + (long long)i * fs)) : make_float2(pad, pad);
      v[0][i] = x.x;
      v[V - 1][i] = x.y;
    } else {
      v[0][i] = there ? __ldcs(src + (long long)i * fs) : pad;
    }
  };
  if (m == W) {   // a full bin of the network's own width: no slot to test
#pragma unroll
    for (int i = 0; i < W; i++) load(i, true, 0.f);
#pragma unroll
    for (int i = 0; i < W; i++)
#pragma unroll
      for (int u = 0; u < V; u++) acc = fmaf(v[u][i], 0.f, acc);
  } else if constexpr (V == 1) {
#pragma unroll
    for (int i = 0; i < W; i++) load(i, i < m, ((i - m) & 1) ? -INFINITY : INFINITY);
#pragma unroll
    for (int i = 0; i < W; i++) acc = i < m ? fmaf(v[0][i], 0.f, acc) : acc;
  } else {
    // a branch per slot, after which a load is counted at once: with two pixels
    // a thread 11 frames a bin take 208 us so and 227 as above, 18 244 and 267,
    // 9 268 and 232; one pixel and 40 to 64 slots 1310 us for 55, 352 as above
#pragma unroll
    for (int i = 0; i < W; i++) {
      if (i < m) {
        load(i, true, 0.f);
#pragma unroll
        for (int u = 0; u < V; u++) acc = fmaf(v[u][i], 0.f, acc);
      } else {
#pragma unroll
        for (int u = 0; u < V; u++) v[u][i] = ((i - m) & 1) ? -INFINITY : INFINITY;
      }
    }
  }
  if (!(acc == 0.f)) atomicOr(status, STATUS_NONFINITE);
  float med[V];
#pragma unroll
  for (int u = 0; u < V; u++) {
    middle_pair<W>(v[u]);
    const float lo = v[u][W / 2 - 1], hi = v[u][W / 2];
    med[u] = (m & 1) ? lo : (lo + hi) * 0.5f;
  }
  if constexpr (V == 2)
    *reinterpret_cast<float2 *>(out + g * nn + p) = make_float2(med[0], med[V - 1]);
  else
    out[g * nn + p] = med[0];
}

__global__ void inject_kernel(float *cube, long long T, int n, int n_comp, const double *__restrict__ pos,
                              const int *__restrict__ win, const float *__restrict__ amp,
                              const float *__restrict__ shape, int half) {
  const long long t = blockIdx.x;
  float *fr = cube + t * (long long)n * n;
  const int side = 2 * half + 1;
  const float ia2 = shape[2 * t], beta = shape[2 * t + 1];
  for (int j = 0; j < n_comp; j++) {
    const long long q = t * n_comp + j;
    const double xp = pos[2 * q], yp = pos[2 * q + 1];
    const int cr = win[2 * q], cc = win[2 * q + 1];
    const float A = amp[q];
    for (int i = threadIdx.x; i < side * side; i += blockDim.x) {
      const int row = cr - half + i / side, col = cc - half + i % side;
      if (row < 0 || row >= n || col < 0 || col >= n) continue;
      const double dx = (double)col - xp, dy = (double)row - yp;
      const float rho2 = (float)(dx * dx + dy * dy);
      const float u = 1.0f + rho2 * ia2;
      const float m = A * exp2f(-beta * log2f(u));
      float *px = fr + (long long)row * n + col;
      *px = *px + m;
    }
    __syncthreads();   // the next companion's window may overlap this one
  }
}

__global__ void aperture_kernel(const float *__restrict__ img, int n, const double *__restrict__ xy, double radius,
                                double *out) {
  __shared__ double part[32];
  const int k = blockIdx.x;
  const double x = xy[2 * k], y = xy[2 * k + 1], r2 = radius * radius;
  const int r0 = max(0, (int)floor(y - radius) - 1), r1 = min(n - 1, (int)ceil(y + radius) + 1);
  const int c0 = max(0, (int)floor(x - radius) - 1), c1 = min(n - 1, (int)ceil(x + radius) + 1);
  double s = 0.0;
  if (r0 <= r1 && c0 <= c1) {
    const int W = c1 - c0 + 1, H = r1 - r0 + 1;
    for (int i = threadIdx.x; i < W * H; i += blockDim.x) {
      const int row = r0 + i / W, col = c0 + i % W;
      const double dx = (double)col - x, dy = (double)row - y;
      if (dx * dx + dy * dy <= r2) s += (double)img[(long long)row * n + col];
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += part[w];
    out[k] = t;
  }
}

template <int W, int V>
cudaError_t bin_launch(const float *in, float *out, long long T, long long nn, long long fs, int B, int *status,
                       cudaStream_t st) {
  const long long G = (T + B - 1) / B;
  const long long bpg = (nn + BIN_THREADS * V - 1) / (BIN_THREADS * V);
  // one block per (bin, 128 or 256 pixels); the limit of the one-pixel form holds for both
  if (G * ((nn + BIN_THREADS - 1) / BIN_THREADS) > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  bin_median_kernel<W, V><<<(unsigned)(G * bpg), BIN_THREADS, 0, st>>>(in, out, T, nn, fs, B, (unsigned)bpg, status);
  return cudaGetLastError();
}

}  // namespace

// Medians of groups of B <= 64 frames, fs elements apart.
cudaError_t launch_median_network(const float *in, float *out, long long T, int n, long long fs, int B, int *status,
                                  cudaStream_t st) {
  const long long nn = (long long)n * n;
  if (B > 64) return cudaErrorInvalidValue;
  // two pixels per thread (8-byte loads) up to 32 values: 1000 frames of 512 x
  // 512 in 165 us against 195 for B = 10, 185 / 194 for 32; from 40 on their
  // registers cost more (B = 50: 240 us with one pixel, 260 with two)
  return with_median_width(B, [&](auto w) {
    constexpr int W = decltype(w)::value;
    return bin_launch<W, W <= 32 ? 2 : 1>(in, out, T, nn, fs, B, status, st);
  });
}

cudaError_t launch_bin_median(const float *in, float *out, long long T, int n, int B, int *status, cudaStream_t st,
                              int *launched) {
  if (launched) *launched = 0;
  if (T <= 0) return cudaSuccess;
  const long long nn = (long long)n * n;
  const long long G = (T + B - 1) / B;
  cudaError_t e;
  if (B <= 64) e = launch_median_network(in, out, T, n, nn, B, status, st);
  else {
    for (long long g = 0; g < G; g++) {
      CollapseArgs a{};
      a.in = in + g * B * nn;
      a.out = out + g * nn;
      a.status = status;
      a.T = (T - g * B) < B ? (T - g * B) : B;
      a.n = n;
      if ((e = launch_collapse(a, st)) != cudaSuccess) return e;
    }
    if (launched) *launched = (int)G;
    return cudaSuccess;
  }
  if (launched && e == cudaSuccess) *launched = 1;
  return e;
}

cudaError_t launch_inject(float *cube, long long T, int n, int n_comp, const double *pos, const int *win,
                          const float *amp, const float *shape, int half, cudaStream_t st) {
  if (T <= 0 || n_comp <= 0) return cudaSuccess;
  inject_kernel<<<(unsigned)T, 256, 0, st>>>(cube, T, n, n_comp, pos, win, amp, shape, half);
  return cudaGetLastError();
}

cudaError_t launch_aperture(const float *img, int n, int n_ap, const double *xy, double radius, double *out,
                            cudaStream_t st) {
  if (n_ap <= 0) return cudaSuccess;
  aperture_kernel<<<(unsigned)n_ap, 256, 0, st>>>(img, n, xy, radius, out);
  return cudaGetLastError();
}

}  // namespace graphic
