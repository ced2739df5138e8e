// prep.cu -- image-quality pre-processing (Sect. 3.2): sky subtraction with
// the master sky closest in time, the sigma-clip bad pixel map (radix
// histograms of total-order keys, FP64 frame sums, the map), and the
// neighbour-median bad pixel correction.  The master sky itself is the
// masked variant of the median collapse (median.cu).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "graphic_internal.h"

namespace graphic {
namespace {

// IEEE total-order key of a float: a larger key is a larger value, -0 < +0.
__device__ __forceinline__ uint32_t key_of(float x) {
  const uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// out[t] = in[t] - skies[sky_of_frame[t]], four floats per thread.
__global__ void sky_subtract_kernel(const float4 *__restrict__ in, float4 *__restrict__ out, long long T,
                                    long long nn4, const float4 *__restrict__ skies,
                                    const int *__restrict__ sky_of_frame) {
  const long long total = T * nn4;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const long long t = i / nn4, q = i - t * nn4;
    const float4 a = in[i];
    const float4 b = skies[(long long)__ldg(&sky_of_frame[t]) * nn4 + q];
    out[i] = make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
  }
}

// Bad pixel map (Sect. 3.2) in four launches on one stream: the exact median
// by three radix digits (11, 11 and 10 bits) of the total-order keys, the FP64
// sum riding on the first digit's pass and the squared deviations on the
// second's; every block works the digits chosen so far out of the finished
// global histograms by itself.  The frame stays in the L2 between the passes
// (4 MB at n = 1024), so launches are what is left: 35 us of kernels at
// n = 512, against 57 us in twelve kernels with ten host round trips between
// them (the host picked each 8-bit digit of each of the two middle ranks),
// 250 us in all.
constexpr int MAP_THREADS = 512;
constexpr int MAP_BINS = 2048;
// Count: 32 bits, 64 for frames of 2^32 pixels and more (64 bits everywhere
// cost 5 us a call, in clearing and in reading twice the bytes per block).
template <class Count>
struct MapWs {
  double sums[2];               // sum, sum of squared deviations
  Count hist[3][2][MAP_BINS];   // [digit][lower, upper median]
};

// Bin of rank k in a histogram of MAP_BINS global counts and the counts
// before it, found by the whole block (each thread sums MAP_BINS /
// MAP_THREADS bins, then a block scan); every thread gets the result.
template <class Count>
__device__ __forceinline__ void map_find(const Count *hist, unsigned long long k, int &bin,
                                         unsigned long long &before) {
  __shared__ Count wsum[MAP_THREADS / 32];
  __shared__ int bin_s;
  __shared__ Count before_s;
  constexpr int PER = MAP_BINS / MAP_THREADS;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  Count h[PER], s = 0;
#pragma unroll
  for (int b = 0; b < PER; b++) {
    h[b] = hist[threadIdx.x * PER + b];
    s += h[b];
  }
  Count inc = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const Count t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  __syncthreads();   // the shared words of an earlier call have been read
  if (lane == 31) wsum[w] = inc;
  __syncthreads();
  Count acc = inc - s;
  for (int q = 0; q < w; q++) acc += wsum[q];
#pragma unroll
  for (int b = 0; b < PER; b++) {
    if (k >= acc && k < (unsigned long long)acc + h[b]) {
      bin_s = threadIdx.x * PER + b;
      before_s = acc;
    }
    acc += h[b];
  }
  __syncthreads();
  bin = bin_s;
  before = before_s;
}

// The key prefixes (aligned to bit 31) of the lower and upper median after
// DIGITS digits, and the ranks left within them.
template <int DIGITS, class Count>
__device__ __forceinline__ void map_prefix(const MapWs<Count> *ws, long long n, uint32_t (&prefix)[2]) {
  unsigned long long k[2] = {(unsigned long long)((n - 1) / 2), (unsigned long long)(n / 2)};
  prefix[0] = prefix[1] = 0u;
#pragma unroll
  for (int d = 0; d < DIGITS; d++) {
    const int shift = d == 0 ? 21 : d == 1 ? 10 : 0;
#pragma unroll
    for (int q = 0; q < 2; q++) {
      int bin;
      unsigned long long before;
      // both medians share the first digit's histogram
      map_find(ws->hist[d][d == 0 ? 0 : q], k[q], bin, before);
      prefix[q] |= (uint32_t)bin << shift;
      k[q] -= before;
    }
  }
}

__device__ __forceinline__ void block_add(double acc, double *dst) {
  __shared__ double part[MAP_THREADS / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < MAP_THREADS / 32; w++) s += part[w];
    atomicAdd(dst, s);
  }
}

// Digit DIGIT's histograms of the keys that match the digits before it; with
// the sum (DIGIT 0) or the squared deviations from the mean (DIGIT 1).
template <int DIGIT, class Count>
__global__ void __launch_bounds__(MAP_THREADS) map_digit_kernel(const float *__restrict__ v, long long n,
                                                                MapWs<Count> *ws) {
  __shared__ unsigned int h[2][MAP_BINS];
  for (int b = threadIdx.x; b < 2 * MAP_BINS; b += MAP_THREADS) h[b / MAP_BINS][b % MAP_BINS] = 0u;
  uint32_t prefix[2];
  map_prefix<DIGIT>(ws, n, prefix);
  __syncthreads();
  constexpr uint32_t PMASK = DIGIT == 0 ? 0u : DIGIT == 1 ? 0xffe00000u : 0xfffffc00u;
  constexpr int SHIFT = DIGIT == 0 ? 21 : DIGIT == 1 ? 10 : 0;
  constexpr uint32_t DMASK = DIGIT == 2 ? 1023u : 2047u;
  const double mu = DIGIT == 1 ? ws->sums[0] / (double)n : 0.0;
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)MAP_THREADS + threadIdx.x; i < n; i += (long long)gridDim.x * MAP_THREADS) {
    const float x = v[i];
    const uint32_t k = key_of(x);
    if constexpr (DIGIT == 0) {
      acc += (double)x;
      atomicAdd(&h[0][k >> SHIFT], 1u);
    } else {
      if constexpr (DIGIT == 1) acc += ((double)x - mu) * ((double)x - mu);
      const uint32_t d = (k >> SHIFT) & DMASK;
      if ((k & PMASK) == prefix[0]) atomicAdd(&h[0][d], 1u);
      if ((k & PMASK) == prefix[1]) atomicAdd(&h[1][d], 1u);
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < 2 * MAP_BINS; b += MAP_THREADS) {
    const unsigned int c = h[b / MAP_BINS][b % MAP_BINS];
    if (c) atomicAdd(&ws->hist[DIGIT][b / MAP_BINS][b % MAP_BINS], (Count)c);
  }
  if constexpr (DIGIT < 2) block_add(acc, &ws->sums[DIGIT]);
}

// map[p] = |ref[p] - median| > C sigma (FP64 comparison; the median FP32: the
// lower middle value, or the mean of the two for an even count).  A frame
// whose sum is not finite is refused by the caller: its map stays as it is.
template <class Count>
__global__ void __launch_bounds__(MAP_THREADS) bad_map_kernel(const float *__restrict__ ref, long long n, double C,
                                                              const MapWs<Count> *ws, uint8_t *map) {
  if (!isfinite(ws->sums[0])) return;
  uint32_t key[2];
  map_prefix<3>(ws, n, key);
  auto val = [](uint32_t k) { return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k); };
  const float lo = val(key[0]);
  const double m = (double)((n & 1) ? lo : (lo + val(key[1])) * 0.5f);
  const double th = C * sqrt(ws->sums[1] / (double)n);
  for (long long i = blockIdx.x * (long long)MAP_THREADS + threadIdx.x; i < n; i += (long long)gridDim.x * MAP_THREADS)
    map[i] = fabs((double)ref[i] - m) > th ? 1 : 0;
}

__device__ __forceinline__ void count_block(unsigned long long mine, unsigned long long *dst) {
  __shared__ unsigned long long part[8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = mine;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long s = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) s += part[w];
    if (s) atomicAdd(dst, s);
  }
  __syncthreads();   // part is reused by the next call
}

// Flagged and non-finite pixels become NaN, are counted per frame and, up to
// `cap` a frame, listed: pixel p of frame f as list[f nn + j], j from the
// frame's counter (any order).  Without lists (cap 0) the count only says
// whether there is one: a frame may hold 2^32 pixels.  One block per (chunk of
// MARK_CHUNK pixels, frame): four values and four map bytes per load where
// frames and map are aligned for it (VEC), no division per value; a warp's
// marked pixels take their places with one step of the counter (a step per
// pixel: 200 frames of 512 x 512 with 5 % bad 1526 us a call, 220 so).
// HBM-bound where little is marked: 200 frames of 512 x 512 in 52 us = 4.0
// TB/s, against 207 us with a 64-bit modulo and 4-byte accesses per value.
constexpr int MARK_THREADS = 256;
constexpr int MARK_CHUNK = MARK_THREADS * 16;
template <bool VEC>
__global__ void __launch_bounds__(MARK_THREADS) bad_mark_kernel(float *__restrict__ cube, long long T,
                                                                long long nn, long long chunks, uint32_t cap,
                                                                const uint8_t *__restrict__ map,
                                                                uint32_t *__restrict__ list, uint32_t *counts) {
  const float NANF = __uint_as_float(0x7fc00000u);
  const long long items = T * chunks;
  const int lane = threadIdx.x & 31;
  for (long long it = blockIdx.x; it < items; it += gridDim.x) {
    const long long f = it / chunks;
    const long long c0 = (it - f * chunks) * MARK_CHUNK;
    float *fr = cube + f * nn;
    uint32_t *lf = list + f * nn, *cnt = counts + f;
    // count and list the warp's marked pixels: bit b of a lane's m is pixel at(b)
    auto add = [&](uint32_t m, auto at) {
      if (!__any_sync(0xffffffffu, m != 0u)) return;
      const uint32_t mine = __popc(m);
      uint32_t end = mine, j = 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, end, o);
        if (lane >= o) end += t;
      }
      if (lane == 31) j = cap > 0 ? atomicAdd(cnt, end) : atomicOr(cnt, 1u);
      j = __shfl_sync(0xffffffffu, j, 31) + end - mine;
      for (; m && j < cap; m &= m - 1, j++) lf[j] = (uint32_t)at(__ffs(m) - 1);
    };
    if constexpr (VEC) {
      float4 v[4];
      uint32_t b[4];
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const long long p = c0 + 4 * (threadIdx.x + k * MARK_THREADS);
        v[k] = p < nn ? __ldcs(reinterpret_cast<const float4 *>(fr + p)) : make_float4(0.f, 0.f, 0.f, 0.f);
        b[k] = p < nn && map ? __ldg(reinterpret_cast<const uint32_t *>(map + p)) : 0u;
      }
      uint32_t m = 0u;
#pragma unroll
      for (int k = 0; k < 4; k++) {
        float q[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
        uint32_t mk = 0u;
#pragma unroll
        for (int l = 0; l < 4; l++)
          if (!isfinite(q[l]) || ((b[k] >> (8 * l)) & 255u)) {
            q[l] = NANF;
            mk |= 1u << l;
          }
        if (mk)
          *reinterpret_cast<float4 *>(fr + c0 + 4 * (threadIdx.x + k * MARK_THREADS)) =
              make_float4(q[0], q[1], q[2], q[3]);
        m |= mk << (4 * k);
      }
      add(m, [&](int i) { return c0 + 4 * (threadIdx.x + (i >> 2) * MARK_THREADS) + (i & 3); });
    } else {
      for (long long q0 = c0; q0 < min(nn, c0 + MARK_CHUNK); q0 += MARK_THREADS) {
        const long long p = q0 + threadIdx.x;
        const bool bad = p < nn && (!isfinite(fr[p]) || (map && map[p]));
        if (bad) fr[p] = NANF;
        add(bad ? 1u : 0u, [&](int) { return p; });
      }
    }
  }
}

// Median of the finite 8-neighbours of pixel (r, c) of a frame of side n (two
// middle values averaged for an even count, FP32); false when it has none.
__device__ __forceinline__ bool neighbour_median(const float *fr, int n, int r, int c, float &med) {
  uint32_t k[8];
  int m = 0;
#pragma unroll
  for (int dr = -1; dr <= 1; dr++)
#pragma unroll
    for (int dc = -1; dc <= 1; dc++) {
      if (!dr && !dc) continue;
      const int rr = r + dr, cc = c + dc;
      if (rr < 0 || rr >= n || cc < 0 || cc >= n) continue;
      const float w = fr[(long long)rr * n + cc];
      if (!isnan(w)) k[m++] = key_of(w);
    }
  if (m == 0) return false;
  // insertion sort of at most 8 keys
  for (int a = 1; a < m; a++) {
    const uint32_t x = k[a];
    int b = a - 1;
    while (b >= 0 && k[b] > x) {
      k[b + 1] = k[b];
      b--;
    }
    k[b + 1] = x;
  }
  auto val = [](uint32_t key) { return __uint_as_float((key & 0x80000000u) ? (key & 0x7fffffffu) : ~key); };
  const float lo = val(k[(m - 1) / 2]);
  med = (m & 1) ? lo : (lo + val(k[m / 2])) * 0.5f;
  return true;
}

// Most pixels a frame's list may hold where D frames hold more than a short
// list (D = 1).  A pass over a list costs its frame a round of one block per
// 1024 pixels left, whatever the other frames do; a dense pass costs every
// pixel of the D frames, but all blocks share it.  Calls with 1024 threads a
// frame, listed and dense (calls in dense passes only): one frame of 512 x 512
// with 1310 bad pixels 46 us (75), with 2621 57 (79); of 1024 x 1024 with 5243 70
// (83), with 10 486 93 (85); eight of 512 x 512 with 13 107 each 98 (119), with
// 26 214 156 (121); 50 of 1024 x 1024 with 104 858 702 (922), with 209 715 1184
// (1060); 200 of 512 x 512 with 104 858 890 (1411).  Lists of up to half a frame,
// whatever D: one frame of 1024 x 1024 with 40 % bad 5441 us, 107 so.
// List and fill values share a frame's n x n words, pixel numbers have 32 bits.
__host__ __device__ inline uint32_t list_cap(long long D, long long nn) {
  if (nn >= (1ll << 32)) return 0u;
  const long long half = nn / 2, c = 4096 + D * nn / 320;
  return (uint32_t)(c < half ? c : half);
}

// One block per frame fills the frame's listed pixels pass by pass: every
// pixel of a pass reads the values of the pass before (a pass keeps its fills
// in vals and writes them after a barrier), filled pixels leave the list,
// until it is empty or a pass fills nothing.  A pass costs the pixels left,
// not the frame.  Frames with too many pixels for that are listed in
// counts[2 + T ...] and left to the dense passes.  `cap`: the lists' room.
template <int FILL_THREADS>
__global__ void __launch_bounds__(FILL_THREADS) bad_fill_kernel(float *cube, long long T, int n, uint32_t cap,
                                                                uint32_t *lists, uint32_t *counts) {
  const long long nn = (long long)n * n;
  const float NANF = __uint_as_float(0x7fc00000u);
  const uint32_t few = list_cap(1, nn);
  __shared__ uint32_t kept_s;
  for (long long f = blockIdx.x; f < T; f += gridDim.x) {
    float *fr = cube + f * nn;
    uint32_t *list = lists + f * nn;
    float *vals = reinterpret_cast<float *>(list + cap);   // cap + cap <= nn
    uint32_t left = counts[2 + f];
    if (left > few) {
      // count the frames that would share the dense passes, from this one on
      // and only until they allow the list (to the end with at most 160 such
      // frames: list_cap has then reached half of a frame)
      bool dense = left > cap;
      long long many = 0;
      for (long long i = 0; !dense && left > list_cap(many, nn); i += FILL_THREADS) {
        const long long t = i + threadIdx.x, u = f + t < T ? f + t : f + t - T;
        many += __syncthreads_count(t < T && counts[2 + u] > few);
        dense = i + FILL_THREADS >= T && left > list_cap(many, nn);
      }
      if (dense) {
        if (threadIdx.x == 0) counts[2 + T + atomicAdd(&counts[0], 1u)] = (uint32_t)f;
        continue;
      }
    }
    while (left > 0) {
      for (uint32_t j = threadIdx.x; j < left; j += FILL_THREADS) {
        const uint32_t p = list[j], r = p / (uint32_t)n;
        float med;
        vals[j] = neighbour_median(fr, n, (int)r, (int)(p - r * (uint32_t)n), med) ? med : NANF;
      }
      if (threadIdx.x == 0) kept_s = 0u;
      __syncthreads();
      // write the fills and close the list up, a block's worth of entries at
      // a time: entries move to slots already read
      for (uint32_t j0 = 0; j0 < left; j0 += FILL_THREADS) {
        const uint32_t j = j0 + threadIdx.x;
        bool keep = false;
        uint32_t p = 0;
        if (j < left) {
          p = list[j];
          const float v = vals[j];
          keep = isnan(v);
          if (!keep) fr[p] = v;
        }
        __syncthreads();
        if (keep) list[atomicAdd(&kept_s, 1u)] = p;
        __syncthreads();
      }
      const uint32_t now = kept_s;
      __syncthreads();
      if (now == left) {   // nothing was filled: no finite pixel to fill from
        if (threadIdx.x == 0) atomicAdd(&counts[1], left);
        break;
      }
      left = now;
    }
  }
}

// One pass over the D frames listed in `frames` (null: frames 0 .. D - 1): every NaN pixel with a finite
// 8-neighbour in src takes the median of those neighbours (two middle values
// averaged for an even count, FP32), the others are copied; counts[0] += NaN
// pixels left, counts[1] += pixels filled.  Blocks (pixels, frame).
constexpr int PASS_THREADS = 256;
__global__ void __launch_bounds__(PASS_THREADS) bad_pass_kernel(const float *__restrict__ src,
                                                                float *__restrict__ dst, uint32_t D, int n,
                                                                const uint32_t *__restrict__ frames,
                                                                unsigned long long *counts) {
  unsigned long long left = 0, filled = 0;
  const long long nn = (long long)n * n;
  for (uint32_t k = blockIdx.y; k < D; k += gridDim.y) {
    const long long f = frames ? __ldg(&frames[k]) : k;
    const float *s = src + f * nn;
    float *d = dst + f * nn;
    for (long long p = blockIdx.x * PASS_THREADS + threadIdx.x; p < nn; p += gridDim.x * PASS_THREADS) {
      const float v = s[p];
      if (!isnan(v)) {
        d[p] = v;
        continue;
      }
      const int r = (int)(p / n);
      float med;
      if (!neighbour_median(s, n, r, (int)(p - (long long)r * n), med)) {
        d[p] = v;
        left++;
        continue;
      }
      d[p] = med;
      filled++;
    }
  }
  count_block(left, &counts[0]);
  count_block(filled, &counts[1]);
}

unsigned grid_for(long long work, int threads) {
  long long g = (work + threads - 1) / threads;
  if (g > 152 * 16) g = 152 * 16;
  if (g < 1) g = 1;
  return (unsigned)g;
}

template <class Count>
cudaError_t bad_map(const float *ref, long long n_vals, double C, uint8_t *map, void *ws, cudaStream_t st) {
  MapWs<Count> *w = static_cast<MapWs<Count> *>(ws);
  cudaError_t e = cudaMemsetAsync(w, 0, sizeof(*w), st);
  if (e != cudaSuccess) return e;
  // at most one block per SM: each flushes its own histograms
  long long grid = (n_vals + MAP_THREADS - 1) / MAP_THREADS;
  if (grid > 152) grid = 152;
  map_digit_kernel<0><<<(unsigned)grid, MAP_THREADS, 0, st>>>(ref, n_vals, w);
  map_digit_kernel<1><<<(unsigned)grid, MAP_THREADS, 0, st>>>(ref, n_vals, w);
  map_digit_kernel<2><<<(unsigned)grid, MAP_THREADS, 0, st>>>(ref, n_vals, w);
  bad_map_kernel<<<(unsigned)grid, MAP_THREADS, 0, st>>>(ref, n_vals, C, w, map);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_sky_subtract(const float *in, float *out, long long T, int n, const float *skies,
                                const int *sky_of_frame, cudaStream_t st) {
  const long long nn4 = (long long)n * n / 4;
  if (T <= 0) return cudaSuccess;
  sky_subtract_kernel<<<grid_for(T * nn4, 256), 256, 0, st>>>(reinterpret_cast<const float4 *>(in),
                                                              reinterpret_cast<float4 *>(out), T, nn4,
                                                              reinterpret_cast<const float4 *>(skies), sky_of_frame);
  return cudaGetLastError();
}

size_t bad_map_bytes() { return sizeof(MapWs<unsigned long long>); }

cudaError_t launch_bad_map(const float *ref, long long n_vals, double C, uint8_t *map, void *ws, cudaStream_t st) {
  return n_vals < (1ll << 32) ? bad_map<unsigned int>(ref, n_vals, C, map, ws, st)
                              : bad_map<unsigned long long>(ref, n_vals, C, map, ws, st);
}

size_t fix_count_words(long long T) { return 2 + 2 * (size_t)T; }

cudaError_t launch_bad_fill(float *cube, long long T, int n, const uint8_t *map, uint32_t *ws, uint32_t *counts,
                            cudaStream_t st) {
  const long long nn = (long long)n * n;
  const long long chunks = (nn + MARK_CHUNK - 1) / MARK_CHUNK;
  const uint32_t cap = list_cap(T, nn);
  cudaError_t e = cudaMemsetAsync(counts, 0, (2 + (size_t)T) * sizeof(uint32_t), st);
  if (e != cudaSuccess) return e;
  const long long items = T * chunks;
  const unsigned grid = (unsigned)std::min<long long>(items, 152ll * 64);
  const bool vec = ((uintptr_t)cube & 15) == 0 && ((uintptr_t)map & 3) == 0 && (nn & 3) == 0;
  if (vec) bad_mark_kernel<true><<<grid, MARK_THREADS, 0, st>>>(cube, T, nn, chunks, cap, map, ws, counts + 2);
  else bad_mark_kernel<false><<<grid, MARK_THREADS, 0, st>>>(cube, T, nn, chunks, cap, map, ws, counts + 2);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // the widest blocks, that is the shortest chain per frame, of which every
  // frame has one resident (2048 threads an SM); with more frames, which fill
  // the chip by their number, 256 threads (2000 of 256 x 256 with 0.1 % bad 132
  // us, 160 with 1024 threads; 310 of 1024 x 1024 with 40 % 8257, 5210 with 512)
  const unsigned fills = (unsigned)std::min<long long>(T, 1 << 20);
  if (T <= 304) bad_fill_kernel<1024><<<fills, 1024, 0, st>>>(cube, T, n, cap, ws, counts);
  else if (T <= 608) bad_fill_kernel<512><<<fills, 512, 0, st>>>(cube, T, n, cap, ws, counts);
  else bad_fill_kernel<256><<<fills, 256, 0, st>>>(cube, T, n, cap, ws, counts);
  return cudaGetLastError();
}

cudaError_t launch_bad_pass(const float *src, float *dst, uint32_t D, int n, const uint32_t *frames,
                            unsigned long long *counts, cudaStream_t st) {
  const long long nn = (long long)n * n;
  // the chip's blocks twice over, at least one a frame
  const unsigned gy = std::min(D, 65535u);
  const unsigned gx = (unsigned)std::min<long long>((nn + PASS_THREADS - 1) / PASS_THREADS, (152 * 16 + gy - 1) / gy);
  bad_pass_kernel<<<dim3(gx, gy), PASS_THREADS, 0, st>>>(src, dst, D, n, frames, counts);
  return cudaGetLastError();
}

}  // namespace graphic
