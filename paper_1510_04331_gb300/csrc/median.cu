// median.cu -- median collapse (Sect. 3.4) and master sky (Sect. 3.2) on
// sm_103a.
//
// Collapse.  The paper's "spatial" data-parallel scheme: a CTA owns 4
// consecutive pixels of every frame (a 16-byte row per frame), one warp per
// pixel.  Values are compared as 32-bit IEEE total-order keys (negative: all
// bits flipped, positive: sign bit set), so selection is exact and
// bit-reproducible.  Per pixel, a value-linear histogram over a sampled range
// locates the two middle ranks, read off a short candidate list
// (collapse2_kernel); radix selects (8-bit digits) are its exact fallback and
// the masked (master sky) and long-cube form (collapse_kernel).  Up to 64
// frames both take register networks (launch_median_network, sky_net_kernel).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "graphic_internal.h"
#include "select_common.cuh"

namespace graphic {
namespace {

// ---------------------------------------------------------------------------
// Median collapse
// ---------------------------------------------------------------------------

// One warp per pixel, COL_PPC pixels per CTA.  Keys in shared memory are
// frame-major with an odd row stride (COL_KS words), so a warp reading its
// pixel's keys of 32 consecutive frames hits 32 distinct banks.  Radix
// select of the lower median: 8-bit digits, most significant first, digits
// constant over the pixel's keys skipped, histograms by shared-memory
// reductions.
constexpr int COL_PPC = 4;
constexpr int COL_KS = 5;
// collapse2_kernel: words per frame row (one 16-byte copy per frame; a
// warp's column reads meet 4-way bank conflicts, cheaper here than four
// 4-byte copies per frame)
constexpr int C2_KS = 4;

// Whether frame t's star mask covers pixel (col, row): (col - mask_x)^2 +
// (row - mask_y)^2 < mask_r2 in FP64.  The same sum in FP32 decides unless it
// lies within its own error of the bound (f.z = 4 E with E = 2^-23 (|mask_x|,
// |mask_y| max + n) bounds the error of either difference, the rest is the
// rounding of the squares, their sum and mask_r2); a mask too far off or not
// finite has f.z = inf and always takes the FP64 sum.  GB300's FP64 pipe is
// 1/64 of its FP32 one: the FP64 test of every value was most of the master
// sky's time (290 us for 50 frames of 512 x 512, 262144 x 50 x 4 FP64
// operations at about 2 per SM and cycle being 90 us of it).
__device__ __forceinline__ bool mask_filter(const float4 f, int col, int row, float r2, bool &sure) {
  const float dx = (float)col - f.x, dy = (float)row - f.y;
  const float d2 = fmaf(dx, dx, dy * dy);
  const float tol = f.z * (fabsf(dx) + fabsf(dy) + 1.0f) + 4.8e-7f * (d2 + r2);
  sure = fabsf(d2 - r2) > tol;
  return d2 < r2;
}
__device__ __forceinline__ bool mask_exact(const CollapseArgs &a, long long t, int col, int row) {
  const double ex = (double)col - a.mask_x[t], ey = (double)row - a.mask_y[t];
  return ex * ex + ey * ey < a.mask_r2;
}
__device__ __forceinline__ bool mask_covers(const CollapseArgs &a, long long t, const float4 f, int col, int row) {
  bool sure;
  const bool in = mask_filter(f, col, row, (float)a.mask_r2, sure);
  return sure ? in : mask_exact(a, t, col, row);
}

// MASKED (master sky, Sect. 3.2): values that are not finite or fall in the
// frame's star mask are left out -- they get the largest key, so they rank
// after every value kept -- and the median is taken over the m values kept
// (NaN when m = 0).  STARS: there are star masks (the test compiled in but not
// used: 300 frames of 512 x 512 452 us instead of 423).
template <bool SMEM, bool MASKED = false, bool STARS = false>
__global__ void __launch_bounds__(32 * COL_PPC) collapse_kernel(const CollapseArgs a) {
  extern __shared__ uint32_t csm[];
  uint32_t *hist_all = csm;                       // [COL_PPC][256]
  uint32_t *keys_all = csm + COL_PPC * 256;       // [T][COL_KS] (SMEM only)
  const long long T = a.T;
  const long long NN = a.fs ? a.fs : (long long)a.n * a.n;   // frame stride
  const long long p0 = (long long)blockIdx.x * COL_PPC;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;

  bool bad = false;
  if constexpr (SMEM) {
    for (long long j = threadIdx.x; j < COL_PPC * T; j += 32 * COL_PPC) {
      const long long t = j / COL_PPC;
      const int q = (int)(j - t * COL_PPC);
      cp_async4(keys_all + t * COL_KS + q, a.in + t * NN + p0 + q);
    }
    cp_async_wait_all();
    __syncthreads();
  }
  uint32_t *hist = hist_all + w * 256;
  const long long p = p0 + w;
  const int row = (int)((unsigned)p / (unsigned)a.n), col = (int)((unsigned)p - (unsigned)row * (unsigned)a.n);
  // masked-out values (MASKED) get the largest key
  auto key_of = [&](long long t, float v) -> uint32_t {
    if constexpr (MASKED) {
      bool keep = isfinite(v);
      if constexpr (STARS) {
        if (a.mask_x) keep &= !mask_covers(a, t, __ldg(&a.maskf[t]), (int)(p % a.n), (int)(p / a.n));
      }
      return keep ? f2key(v) : 0xffffffffu;
    } else {
      return f2key(v);
    }
  };
  auto key_at = [&](long long t) -> uint32_t {
    if constexpr (SMEM) return keys_all[t * COL_KS + w];
    else return key_of(t, a.in[t * NN + p]);
  };
  // keys in place (each warp converts its own pixel), finiteness, and the
  // digits shared by every key
  uint32_t orv = 0, andv = 0xffffffffu;
  int kept = 0;
  if constexpr (SMEM && STARS) {
    // four frames a step: their masks are loaded together, and the FP64 test at
    // a rim is out of the way (300 frames of 512 x 512 622 us; a frame at a time
    // 670, FP64 tests only 978)
    const float r2 = (float)a.mask_r2;
    for (long long t0 = lane; t0 - lane < T; t0 += 128) {
      bool in[4], sure[4], all = true;
      float4 f[4];
#pragma unroll
      for (int u = 0; u < 4; u++) f[u] = __ldg(&a.maskf[t0 + 32 * u < T ? t0 + 32 * u : T - 1]);
#pragma unroll
      for (int u = 0; u < 4; u++) {
        in[u] = mask_filter(f[u], col, row, r2, sure[u]);
        all &= sure[u] || t0 + 32 * u >= T;
      }
      if (!all) {
#pragma unroll
        for (int u = 0; u < 4; u++)
          if (!sure[u] && t0 + 32 * u < T) in[u] = mask_exact(a, t0 + 32 * u, col, row);
      }
#pragma unroll
      for (int u = 0; u < 4; u++) {
        if (t0 + 32 * u >= T) continue;
        uint32_t *at = &keys_all[(t0 + 32 * u) * COL_KS + w];
        const float v = __uint_as_float(*at);
        const uint32_t key = isfinite(v) && !in[u] ? f2key(v) : 0xffffffffu;
        kept += key != 0xffffffffu ? 1 : 0;
        *at = key;
        orv |= key;
        andv &= key;
      }
    }
  } else {
    for (long long t = lane; t < T; t += 32) {
      float v;
      if constexpr (SMEM) v = __uint_as_float(keys_all[t * COL_KS + w]);
      else v = a.in[t * NN + p];
      const uint32_t key = key_of(t, v);
      if constexpr (MASKED) kept += (key != 0xffffffffu) ? 1 : 0;
      else bad |= !isfinite(v);
      if constexpr (SMEM) keys_all[t * COL_KS + w] = key;
      orv |= key;
      andv &= key;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    orv |= __shfl_xor_sync(FULL, orv, o);
    andv &= __shfl_xor_sync(FULL, andv, o);
  }
  const bool anybad = __any_sync(FULL, bad);
  if (anybad && lane == 0) atomicOr(a.status, STATUS_NONFINITE);
  __syncwarp();
  const uint32_t varying = orv ^ andv;

  long long m = T;
  if constexpr (MASKED) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) kept += __shfl_xor_sync(FULL, kept, o);
    m = kept;
    if (m == 0) {
      if (lane == 0) a.out[p] = __uint_as_float(0x7fc00000u);   // no value left: NaN
      return;
    }
  }
  const uint32_t k = (uint32_t)((m - 1) / 2);
  uint32_t prefix = 0, pmask = 0, krem = k, cnt = (uint32_t)T;
  // Candidate list: the pass in which at most `cap` keys still match the
  // prefix also copies them (in frame order) into the row padding words
  // (word COL_KS - 1 of rows [w cap, (w + 1) cap), which no key uses), and
  // the later passes read only the list.
  const int cap = SMEM ? (int)(T / COL_PPC < 128 ? T / COL_PPC : 128) : 0;
  uint32_t *cbuf = keys_all + (long long)w * cap * COL_KS + (COL_KS - 1);   // element j at cbuf[j * COL_KS]
  int nc = -1;                                                            // list length, -1: none yet
  const unsigned lt = (1u << lane) - 1u;
  for (int pass = 0; pass < 4; pass++) {
    const int shift = 24 - 8 * pass;
    if (((varying >> shift) & 255u) == 0) {   // every key has this digit
      prefix |= andv & (0xffu << shift);
      pmask |= 0xffu << shift;
      continue;
    }
#pragma unroll
    for (int b = 0; b < 8; b++) hist[lane * 8 + b] = 0;
    __syncwarp();
    if (nc >= 0) {
      for (int j = lane; j < nc; j += 32) {
        const uint32_t key = cbuf[j * COL_KS];
        if ((key & pmask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
      }
    } else if (cnt <= (uint32_t)cap) {
      int len = 0;
      for (long long t0 = 0; t0 < T; t0 += 32) {
        const long long t = t0 + lane;
        const uint32_t key = t < T ? key_at(t) : 0u;
        const bool match = t < T && (key & pmask) == prefix;
        const unsigned mm = __ballot_sync(FULL, match);
        if (match) {
          cbuf[(len + __popc(mm & lt)) * COL_KS] = key;
          atomicAdd(&hist[(key >> shift) & 255u], 1u);
        }
        len += __popc(mm);
      }
      nc = len;
    } else {
#pragma unroll 4
      for (long long t = lane; t < T; t += 32) {
        const uint32_t key = key_at(t);
        if ((key & pmask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
      }
    }
    __syncwarp();
    uint32_t d, below;
    hist_find(hist, krem, lane, d, below, cnt);
    prefix |= d << shift;
    pmask |= 0xffu << shift;
    krem -= below;
    __syncwarp();
  }
  const float lo = key2f(prefix);
  float med = lo;
  if ((m & 1) == 0) {
    uint32_t hi = prefix;
    if (krem + 1 >= cnt) {
      // smallest key greater than the lower median: from the candidate list
      // when it holds one (the list's bucket is a contiguous key range, so a
      // larger key inside it beats every key above it), else from all keys
      uint32_t mn = 0xffffffffu;
      if (nc >= 0) {
        for (int j = lane; j < nc; j += 32) {
          const uint32_t key = cbuf[j * COL_KS];
          if (key > prefix && key < mn) mn = key;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mn = min(mn, __shfl_xor_sync(FULL, mn, o));
      }
      if (nc < 0 || mn == 0xffffffffu) {
        mn = 0xffffffffu;
        for (long long t = lane; t < T; t += 32) {
          const uint32_t key = key_at(t);
          if (key > prefix && key < mn) mn = key;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mn = min(mn, __shfl_xor_sync(FULL, mn, o));
      }
      hi = mn;
    }
    med = (lo + key2f(hi)) * 0.5f;
  }
  if (lane == 0) a.out[p] = med;
}

// Master sky of at most W frames (W <= 64): one thread per pixel, the values
// in registers, the two middle ones by the pruned odd-even merge network
// (middle_pair).  A value left out, like a slot beyond the last frame, is
// replaced by +inf and -inf in turn, +inf first: the kept values stay in the
// middle of the W slots (kept values are finite).  Reads every value once,
// with all of a pixel's loads independent.  Bound by the instruction stream
// (mask and finiteness tests and 612 of the 806 min / max of 403 comparators
// per 50 values): 50 frames of 512 x 512 with masks in 30 us = 1.7 TB/s, where
// the radix select with an FP64 mask test per value took 290 us.
template <int W>
__global__ void __launch_bounds__(128) sky_net_kernel(const CollapseArgs a) {
  const int NN = a.n * a.n, T = (int)a.T;
  const int p = blockIdx.x * 128 + threadIdx.x;
  const int row = p / a.n, col = p - row * a.n;
  float v[W];
#pragma unroll
  for (int i = 0; i < W; i++) v[i] = i < T ? __ldcs(a.in + (long long)i * NN + p) : INFINITY;
  float pad = INFINITY;
  int m = 0;
#pragma unroll
  for (int i = 0; i < W; i++) {
    bool keep = i < T && isfinite(v[i]);
    if (i < T && a.mask_x) {
      // a warp's pixels share their row: most masks stay clear of it
      const float4 f = __ldg(&a.maskf[i]);
      if (fabsf((float)row - f.y) <= f.w) keep &= !mask_covers(a, i, f, col, row);
    }
    m += keep ? 1 : 0;
    v[i] = keep ? v[i] : pad;
    pad = keep ? pad : -pad;
  }
  middle_pair<W>(v);
  const float lo = v[W / 2 - 1], hi = v[W / 2];
  const float med = (m & 1) ? lo : (lo + hi) * 0.5f;
  a.out[p] = m > 0 ? med : __uint_as_float(0x7fc00000u);   // no value left: NaN
}

// Median collapse of unmasked cubes that fit shared memory.  Per pixel
// (one warp): the values in shared memory, one 16-byte row of the CTA's 4
// pixels per frame.
// A 256-bin histogram linear in value over the interquartile range of 32
// sampled frames (values outside it counted below or ignored above), filled
// in one pass over the raw values, locates the bins of the two middle
// ranks; a second pass copies the total-order keys of those bins (a few
// values) into the warp's second 256 histogram words, and the middle ranks
// are read off by counting within that list.  A middle rank outside the
// range, a list longer than 256 keys (many equal values) or a non-finite
// value falls back to exact radix selects of the two middle ranks over all
// keys.
// Registers for twelve CTAs per SM (40, no spills): 250 frames of 512 x 512 254
// -> 229 us, 65 frames 165 -> 151; 2000 frames, five CTAs by shared memory, 1608
// and 1618.
__global__ void __launch_bounds__(32 * COL_PPC, 12) collapse2_kernel(const CollapseArgs a) {
  extern __shared__ uint32_t csm[];
  uint32_t *hist_all = csm;                       // [COL_PPC][512]
  uint32_t *keys_all = csm + COL_PPC * 512;       // [T][C2_KS]
  const int T = (int)a.T;
  const long long NN = a.fs ? a.fs : (long long)a.n * a.n;   // frame stride
  const long long p0 = (long long)blockIdx.x * COL_PPC;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int t = threadIdx.x; t < T; t += 32 * COL_PPC) cp_async16(keys_all + t * C2_KS, a.in + (long long)t * NN + p0);
  cp_async_wait_all();
  __syncthreads();
  uint32_t *hist = hist_all + w * 512;
  uint32_t *kw = keys_all + w;   // value (then key) of frame t: kw[t * C2_KS]
  const uint32_t k0 = (uint32_t)((T - 1) / 2);
  const bool even = (T & 1) == 0;
  const uint32_t k1 = even ? k0 + 1 : k0;
  // histogram range: the interquartile range of 32 frames sampled evenly in
  // time (bitonic sort across the warp; the min and max of the sample when
  // the quartiles coincide).  The median lies between the sample's quartiles
  // unless fewer than 9 or more than 23 of the 32 sampled values fall below
  // it (well under 1 % of pixels when frames vary independently); then, as
  // for a range the sample missed, the exact path below takes over.
  float lo = 0.f, scale = 0.f;
  if (T >= 32) {
    float x = __uint_as_float(kw[(int)(((long long)lane * T) >> 5) * C2_KS]);
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
      for (int d = k >> 1; d > 0; d >>= 1) {
        const float y = __shfl_xor_sync(FULL, x, d);
        const bool up = (lane & k) == 0, low = (lane & d) == 0;
        x = (up == low) ? fminf(x, y) : fmaxf(x, y);
      }
    }
    float qlo = __shfl_sync(FULL, x, 8), qhi = __shfl_sync(FULL, x, 23);
    if (!(qhi > qlo)) {
      qlo = __shfl_sync(FULL, x, 0);
      qhi = __shfl_sync(FULL, x, 31);
    }
    const float sc = 256.f / (qhi - qlo);
    if (qhi > qlo && sc <= 3.4e38f) {   // finite range and scale
      lo = qlo;
      scale = sc;
    }
  }
  // one pass over the raw values: x = (v - lo) scale is monotone in v;
  // x < 0 counts below the range, [0, 256) takes bin (int) x, the rest is
  // above.  (scale = 0 puts every finite value in bin 0.)  The finiteness
  // check rides along.
#pragma unroll
  for (int b = 0; b < 8; b++) hist[lane * 8 + b] = 0u;
  __syncwarp();
  bool bad = false;
  uint32_t nb = 0;
#pragma unroll 4
  for (int t = lane; t < T; t += 32) {
    const float v = __uint_as_float(kw[t * C2_KS]);
    bad |= !isfinite(v);
    const float xv = (v - lo) * scale;
    if (xv < 0.f) nb++;
    else if (xv < 256.f) atomicAdd(&hist[(int)xv], 1u);
  }
  const bool anybad = __any_sync(FULL, bad);
  if (anybad && lane == 0) atomicOr(a.status, STATUS_NONFINITE);
  const uint32_t nbelow = __reduce_add_sync(FULL, nb);
  __syncwarp();
  uint32_t h[8], hs = 0;
#pragma unroll
  for (int b = 0; b < 8; b++) {
    h[b] = hist[lane * 8 + b];
    hs += h[b];
  }
  uint32_t inc = hs;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t tt = __shfl_up_sync(FULL, inc, o);
    if (lane >= o) inc += tt;
  }
  const uint32_t inside = __shfl_sync(FULL, inc, 31);
  // bins of ranks k0 and k1 (ranks within the range: k - nbelow) and the
  // values below them; a rank outside the range takes the exact path
  const bool in_range = k0 >= nbelow && k1 - nbelow < inside;
  int bin[2] = {0, 0};
  uint32_t bel[2] = {0u, 0u};
  if (in_range) {
#pragma unroll
    for (int q = 0; q < 2; q++) {
      const uint32_t r = (q ? k1 : k0) - nbelow;
      const unsigned ball = __ballot_sync(FULL, inc > r);
      const int L = __ffs(ball) - 1;
      int bb = 0;
      uint32_t be = 0;
      if (lane == L) {
        uint32_t acc = inc - hs;
        bool done = false;
#pragma unroll
        for (int b = 0; b < 8; b++) {
          if (!done && acc + h[b] > r) {
            bb = lane * 8 + b;
            be = acc;
            done = true;
          }
          acc += h[b];
        }
      }
      bin[q] = __shfl_sync(FULL, bb, L);
      bel[q] = __shfl_sync(FULL, be, L) + nbelow;
    }
  }
  const int nlist = in_range ? (int)(bel[1] + hist[bin[1]] - bel[0]) : 0x7fffffff;
  // the list lives in the warp's second 256 histogram words
  const int cap = min(T, 256);
  float med;
  if (!anybad && nlist <= cap) {
    uint32_t *cbuf = hist + 256;   // element j at cbuf[j] (the second histogram's words)
    const unsigned lt = (1u << lane) - 1u;
    int len = 0;
    // four 32-frame rounds per step: their loads and bins are independent;
    // the list holds total-order keys.  Bins bin0 .. bin1 of x >= 0 are the
    // x in [bin0, bin1 + 1) (truncation is the floor there; -0 is in bin 0).
    const float xlo = (float)bin[0], xhi = (float)(bin[1] + 1);
    for (int t0 = 0; t0 < T; t0 += 128) {
      float v[4];
      bool in[4];
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const int t = t0 + 32 * u + lane;
        v[u] = t < T ? __uint_as_float(kw[t * C2_KS]) : 0.f;
        const float xv = (v[u] - lo) * scale;
        in[u] = t < T && xv >= xlo && xv < xhi;
      }
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const unsigned mm = __ballot_sync(FULL, in[u]);
        if (in[u]) cbuf[len + __popc(mm & lt)] = f2key(v[u]);
        len += __popc(mm);
      }
    }
    __syncwarp();
    // ranks r0, r1 within the list: the key with (#smaller) <= r < (#smaller or equal)
    const uint32_t r0 = k0 - bel[0], r1 = k1 - bel[0];
    uint32_t f0 = 0xffffffffu, f1 = 0xffffffffu;
    for (int j = lane; j < len; j += 32) {
      const uint32_t kj = cbuf[j];
      uint32_t nlt = 0, nle = 0;
      for (int x = 0; x < len; x++) {
        const uint32_t kx = cbuf[x];
        nlt += kx < kj ? 1u : 0u;
        nle += kx <= kj ? 1u : 0u;
      }
      if (nlt <= r0 && r0 < nle) f0 = kj;
      if (nlt <= r1 && r1 < nle) f1 = kj;
    }
    f0 = __reduce_min_sync(FULL, f0);
    f1 = __reduce_min_sync(FULL, f1);
    med = even ? (key2f(f0) + key2f(f1)) * 0.5f : key2f(f0);
  } else {
    // exact: keys in place, then radix selects of the two middle ranks
    uint32_t orv = 0u, andv = 0xffffffffu;
    for (int t = lane; t < T; t += 32) {
      const uint32_t k = f2key(__uint_as_float(kw[t * C2_KS]));
      kw[t * C2_KS] = k;
      orv |= k;
      andv &= k;
    }
    orv = __reduce_or_sync(FULL, orv);
    andv = __reduce_and_sync(FULL, andv);
    __syncwarp();
    uint32_t Klo, Khi, clo, chi;
    band_select2([&](int t) { return kw[t * C2_KS]; }, T, k0, k1, orv ^ andv, andv, hist, hist + 256, lane, Klo, clo, Khi, chi);
    med = even ? (key2f(Klo) + key2f(Khi)) * 0.5f : key2f(Klo);
  }
  if (lane == 0) a.out[p0 + w] = med;
}

}  // namespace

cudaError_t launch_collapse(const CollapseArgs &a, cudaStream_t st) {
  const long long NN = (long long)a.n * a.n;
  const unsigned grid = (unsigned)(NN / COL_PPC);
  const long long fs = a.fs ? a.fs : NN;
  const bool rows16 = ((uintptr_t)a.in & 15) == 0 && (fs & 3) == 0;   // 16-byte frame rows of 4 pixels
  // up to 64 frames: the register network of the binning, a thread per pixel
  // (pair), where a warp per pixel is mostly idle (20 frames of 1024 x 1024:
  // 541 -> 19 us; 32 of 128 x 128: 20 -> 7; 65 of 512 x 512 below: 165)
  if (a.T >= 1 && a.T <= 64 && (((uintptr_t)a.in | (uintptr_t)a.out) & 7) == 0 && (fs & 1) == 0)
    return launch_median_network(a.in, a.out, a.T, a.n, fs, (int)a.T, a.status, st);
  if (a.T <= 8192 && rows16) {
    const size_t smem = (size_t)(COL_PPC * 512 + C2_KS * a.T) * sizeof(uint32_t);
    cudaError_t e = cudaFuncSetAttribute(collapse2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    collapse2_kernel<<<grid, 32 * COL_PPC, smem, st>>>(a);
  } else if (a.T <= 8192) {
    const size_t smem = (size_t)(COL_PPC * 256 + COL_KS * a.T) * sizeof(uint32_t);
    cudaError_t e = cudaFuncSetAttribute(collapse_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    collapse_kernel<true><<<grid, 32 * COL_PPC, smem, st>>>(a);
  } else {
    const size_t smem = (size_t)(COL_PPC * 256) * sizeof(uint32_t);
    collapse_kernel<false><<<grid, 32 * COL_PPC, smem, st>>>(a);
  }
  return cudaGetLastError();
}

float4 sky_mask_filter(double mask_x, double mask_y, double mask_r, int n) {
  const double E = (std::max(fabs(mask_x), fabs(mask_y)) + n) * 0x1p-23;
  if (!(E < 0.5)) return make_float4(0.f, 0.f, INFINITY, INFINITY);
  return make_float4((float)mask_x, (float)mask_y, (float)(4.0 * E), (float)(mask_r * 1.000001 + 4.0 * E));
}

cudaError_t launch_sky_median(const CollapseArgs &a, cudaStream_t st) {
  const long long NN = (long long)a.n * a.n;
  // up to 64 frames: the network that holds them, one thread per pixel (n a
  // power of two from 64 on: whole blocks); longer stacks one warp per pixel
  if (a.T <= 64) {
    const unsigned blocks = (unsigned)(NN / 128);
    with_median_width((int)a.T, [&](auto w) { sky_net_kernel<decltype(w)::value><<<blocks, 128, 0, st>>>(a); });
    return cudaGetLastError();
  }
  const unsigned grid = (unsigned)(NN / COL_PPC);
  if (a.T <= 8192) {
    const size_t smem = (size_t)(COL_PPC * 256 + COL_KS * a.T) * sizeof(uint32_t);
    void (*const kernel)(CollapseArgs) = a.mask_x ? collapse_kernel<true, true, true> : collapse_kernel<true, true>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<grid, 32 * COL_PPC, smem, st>>>(a);
  } else {
    const size_t smem = (size_t)(COL_PPC * 256) * sizeof(uint32_t);
    if (a.mask_x) collapse_kernel<false, true, true><<<grid, 32 * COL_PPC, smem, st>>>(a);
    else collapse_kernel<false, true><<<grid, 32 * COL_PPC, smem, st>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace graphic
