// psf_general.cu -- general path of the angle-gated median PSF subtraction
// (Sect. 3.3) on sm_103a: the annuli without a rank band (psf_band.cu), i.e.
// bands wider than 1024 ranks, gates that move back and time-gated calls; and
// the rest of the 4-pixel groups that such annuli share with others.
//
// Notation.  Frames in angle order s = 0..T-1 (perm[s] = frame index).  The
// PSF of query i (the frame at angle position i) is the median of the pixel
// over its reference set S_i = [A_i, L_i) u [R_i, B_i) (host plan, FP64 gate;
// [A, B) = [0, T) without a time gate): the (|S_i|-1)/2-th member in the IEEE
// total order of the values, ties ordered by s, averaged in FP32 with the
// next member when |S_i| is even.  Frame s is in the set when it lies in the
// window and outside [L, R): the XOR of two range indicators, so moving any of
// the four boundaries toggles exactly the frames it passes over.
//
// Two kernels per chunk of units (32 pixels of ONE annulus: four segments of
// 8 adjacent pixels):
//   full_rank_kernel   one CTA of 8 warps per segment, one warp per pixel:
//     every frame's rank ("code") and the values in value order, written as
//     rows of the unit's 32 pixels;
//   psf_sweep_kernel   one warp per unit and chunk of consecutive queries, one
//     LANE per pixel.  The gates are the annulus' own, so the frames that
//     leave and enter are the same for the whole warp: their codes arrive as
//     one coalesced row, each lane flips its bit in its map over the ranks,
//     keeps the number of members below its pointer, and moves the pointer by
//     the few set bits that the median moved.  Values in and residuals out
//     move as whole sectors.
// Against one kernel with 8 pixels per CTA and one CTA per SM (a radix sort
// per pixel, then queries across the lanes, each lane meeting its events at
// other queries and walking its own words): 600 frames of 256 x 256 with a
// time gate 3.61 ms, so 1.14 (ranking 0.46, sweep 0.68).  Bound by instruction
// issue (65 %) and the codes' loads.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "graphic_internal.h"
#include "select_common.cuh"

namespace graphic {
namespace {

constexpr int SEG = 8;          // pixels of a segment (and warps of a ranking CTA)
constexpr int UNIT = 32;        // pixels (lanes) of a unit
constexpr int UNIT_SEGS = UNIT / SEG;
constexpr int RANK_THREADS = 32 * SEG;
constexpr int ANN_SHIFT = 18;   // unit word 0: segment | annulus << 18 (n <= 1024: 2^17 segments)

__host__ __device__ constexpr size_t al16(size_t x) { return (x + 15) & ~(size_t)15; }

// A unit's tables in the scratch, NB = T rounded up to whole map words: rows
// of 32 values in value order (row = rank), then rows of 32 ranks (row = frame
// in angle order).
__host__ __device__ inline int table_rows(int T) { return (T + 31) & ~31; }
__host__ __device__ inline size_t unit_codes_off(int NB) { return (size_t)NB * UNIT * 4; }
__host__ __device__ inline size_t unit_bytes(int T) { return unit_codes_off(table_rows(T)) + (size_t)table_rows(T) * UNIT * 2; }

struct GeneralArgs {
  AdiArgs a;
  const int *units;      // this launch's units, UNIT_SEGS ints each
  char *tables;          // their tables
  size_t table_bytes;    // of one unit
  int NB;                // table_rows(T)
  int C;                 // queries per chunk (psf_sweep_kernel)
};

// Annuli of a segment's 8 pixels and which of its two 4-pixel groups are the
// general path's: those with a pixel of an annulus without a band.
__device__ __forceinline__ bool group_general(const AdiArgs &a, long long p) {
  bool g = a.wmax == 0;   // no band path at all
  for (int q = 0; q < 4 && !g; q++) {
    const int an = annulus_of((p & ~3ll) + q, a.n, a.iedge2, a.n_ann);
    g = an >= 0 && __ldg(&a.band[4 * an + 2]) == 0;
  }
  return g;
}

__device__ __forceinline__ const float *frame_ptr(const AdiArgs &a, int s) {
  return a.in + (long long)(a.perm_id ? s : __ldg(&a.perm[s])) * a.in_fs;
}

// Bin of a value in a 256-bin histogram linear in value from v0 with `scale`
// bins per unit: monotone non-decreasing (every step is a monotone rounding).
// A scale of 0 (empty or overflowing range) puts every value in bin 0
// (x = 0, or NaN, which converts to 0).
__device__ __forceinline__ float vpos(float v, float v0, float scale) { return (v - v0) * scale; }
__device__ __forceinline__ int vbin(float x, int bins) { return (int)min((unsigned)(int)x, (unsigned)(bins - 1)); }

// ---------------------------------------------------------------------------
// full_rank_kernel: every frame's rank
// ---------------------------------------------------------------------------

// Shared memory per pixel (warp): kA[T], kB[T] u32, iA[T], iB[T] u16, and BINS
// u16 counters.  Bins linear in value between the extremes, the frames of a
// bin ordered by counting; a bin of more than FULL_BIN_MAX frames (outliers
// that stretch the range, many ties) sends the pixel to a stable radix sort
// (BINS >= 512: its 256 u32 counters fit).
constexpr int FULL_BIN_MAX = 48;
template <int BINS>
__host__ __device__ inline size_t full_pixel_bytes(int T) {
  return (size_t)T * 8 + al16((size_t)T * 4) + (size_t)BINS * 2;
}

template <int BINS>
__global__ void __launch_bounds__(RANK_THREADS) full_rank_kernel(const GeneralArgs g) {
  extern __shared__ __align__(16) unsigned char fsm[];
  __shared__ int ann_s[SEG];
  const AdiArgs &a = g.a;
  const int T = a.T;
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int unit = blockIdx.x / UNIT_SEGS, slot = blockIdx.x % UNIT_SEGS;
  const int *u = g.units + (size_t)unit * UNIT_SEGS;
  const int ann = u[0] >> ANN_SHIFT;
  const int seg = slot == 0 ? (u[0] & ((1 << ANN_SHIFT) - 1)) : u[slot];
  if (seg < 0) return;
  const long long p0 = (long long)seg * SEG;
  if (tid < SEG)
    ann_s[tid] = group_general(a, p0 + tid) ? annulus_of(p0 + tid, a.n, a.iedge2, a.n_ann) : -1;
  __syncthreads();
  const size_t pb = full_pixel_bytes<BINS>(T);
  auto kA_of = [&](int q) { return reinterpret_cast<uint32_t *>(fsm + q * pb); };
  auto iB_of = [&](int q) { return reinterpret_cast<uint16_t *>(fsm + q * pb + (size_t)T * 10); };
  {
    float acc[SEG];
#pragma unroll
    for (int q = 0; q < SEG; q++) acc[q] = 0.f;
    for (int s0 = tid; s0 < T; s0 += 2 * RANK_THREADS) {
      float4 v[2][2];
#pragma unroll
      for (int k = 0; k < 2; k++) {
        const int s = s0 + k * RANK_THREADS;
        if (s < T) {
          const float4 *src = reinterpret_cast<const float4 *>(frame_ptr(a, s) + p0);
          v[k][0] = src[0];
          v[k][1] = src[1];
        }
      }
#pragma unroll
      for (int k = 0; k < 2; k++) {
        const int s = s0 + k * RANK_THREADS;
        if (s < T) {
          const float x[SEG] = {v[k][0].x, v[k][0].y, v[k][0].z, v[k][0].w,
                                v[k][1].x, v[k][1].y, v[k][1].z, v[k][1].w};
#pragma unroll
          for (int q = 0; q < SEG; q++) {
            kA_of(q)[s] = f2key(x[q]);
            acc[q] = fmaf(x[q], 0.f, acc[q]);
          }
        }
      }
    }
    // the unit's own pixels, and those of the segment that no unit has (they
    // are set to zero, or are the band path's, after every unit): other
    // annuli's are their own units' to test, and in a call in place they may
    // hold residuals by now
    bool bad = false;
#pragma unroll
    for (int q = 0; q < SEG; q++) bad |= !(acc[q] == 0.f);
    if (__any_sync(FULL, bad)) {   // seldom: which pixels (asked at once, 9 us of 163 at 8 frames of 512 x 512)
      bad = false;
#pragma unroll
      for (int q = 0; q < SEG; q++) bad |= !(acc[q] == 0.f) && (ann_s[q] == ann || ann_s[q] < 0);
      if (__any_sync(FULL, bad) && lane == 0) atomicOr(a.status, STATUS_NONFINITE);
    }
  }
  __syncthreads();
  if (ann_s[w] == ann) {
    uint32_t *kA = kA_of(w), *kB = kA + T;
    uint16_t *iA = reinterpret_cast<uint16_t *>(kB + T), *iB = iA + T;
    uint32_t *hw = reinterpret_cast<uint32_t *>(fsm + w * pb + (size_t)T * 8 + al16((size_t)T * 4));   // BINS / 2 words
    uint32_t kmin = 0xffffffffu, kmax = 0u;
    for (int s = lane; s < T; s += 32) {
      kmin = min(kmin, kA[s]);
      kmax = max(kmax, kA[s]);
    }
    kmin = __reduce_min_sync(FULL, kmin);
    kmax = __reduce_max_sync(FULL, kmax);
    const float v0 = key2f(kmin);
    const float range = key2f(kmax) - v0;
    const float sc = (range > 0.f) ? (float)BINS / range : 0.f;
    constexpr int WPL = BINS / 64;   // counter words per lane
#pragma unroll
    for (int b = 0; b < WPL; b++) hw[b * 32 + lane] = 0u;
    __syncwarp();
    // counts per bin (two u16 counters a word), each frame's place in its bin
    int most = 0;
    for (int s = lane; s < T; s += 32) {
      const int b = vbin(vpos(key2f(kA[s]), v0, sc), BINS);
      const int sh = 16 * (b & 1);
      const int at = (int)((atomicAdd(&hw[b >> 1], 1u << sh) >> sh) & 0xffffu);
      iB[s] = (uint16_t)at;
      most = max(most, at);
    }
    most = __reduce_max_sync(FULL, most);
    __syncwarp();
    if (BINS < 512 || most < FULL_BIN_MAX) {
      // exclusive prefix over the bins: lane l holds words l WPL ..
      uint32_t h[WPL], sum = 0;
#pragma unroll
      for (int b = 0; b < WPL; b++) {
        h[b] = hw[lane * WPL + b];
        sum += (h[b] & 0xffffu) + (h[b] >> 16);
      }
      uint32_t inc = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += t;
      }
      uint32_t run = inc - sum;
#pragma unroll
      for (int b = 0; b < WPL; b++) {
        const uint32_t mid = run + (h[b] & 0xffffu);
        hw[lane * WPL + b] = run | (mid << 16);
        run = mid + (h[b] >> 16);
      }
      __syncwarp();
      const uint16_t *start = reinterpret_cast<const uint16_t *>(hw);
      for (int s = lane; s < T; s += 32) iA[start[vbin(vpos(key2f(kA[s]), v0, sc), BINS)] + iB[s]] = (uint16_t)s;
      __syncwarp();
      for (int s = lane; s < T; s += 32) {
        const uint32_t k = kA[s];
        const int b = vbin(vpos(key2f(k), v0, sc), BINS);
        const int st = start[b], en = b + 1 < BINS ? (int)start[b + 1] : T;
        int r = st;
        if (en - st > 1)
          for (int x = st; x < en; x++) {
            const int s2 = iA[x];
            const uint32_t k2 = kA[s2];
            r += (k2 < k || (k2 == k && s2 < s)) ? 1 : 0;
          }
        iB[s] = (uint16_t)r;
        kB[r] = k;
      }
    } else {
      // stable LSD radix sort of (key, frame): 8-bit digits, digits equal in
      // every key skipped; ends with the sorted keys in kB, ranks in iB
      const uint32_t varying = [&] {
        uint32_t orv = 0, andv = 0xffffffffu;
        for (int s = lane; s < T; s += 32) {
          orv |= kA[s];
          andv &= kA[s];
        }
        return __reduce_or_sync(FULL, orv) ^ __reduce_and_sync(FULL, andv);
      }();
      for (int s = lane; s < T; s += 32) iA[s] = (uint16_t)s;
      __syncwarp();
      uint32_t *sk = kA, *dk = kB;
      uint16_t *si = iA, *di = iB;
      const unsigned lt = (1u << lane) - 1u;
      constexpr uint32_t NOTAG = 0xffffffffu;
      for (int pass = 0; pass < 4; pass++) {
        const int shift = 8 * pass;
        if (((varying >> shift) & 255u) == 0) continue;
#pragma unroll
        for (int b = 0; b < 8; b++) hw[lane * 8 + b] = 0u;
        __syncwarp();
        for (int s = lane; s < T; s += 32) atomicAdd(&hw[(sk[s] >> shift) & 255u], 1u);
        __syncwarp();
        hist_exclusive_scan(hw, lane);
        __syncwarp();
        for (int base = 0; base < T; base += 32) {
          const int i = base + lane;
          uint32_t key = 0, tag = NOTAG;
          uint16_t fi = 0;
          if (i < T) {
            key = sk[i];
            fi = si[i];
            tag = (key >> shift) & 255u;
          }
          const unsigned peers = __match_any_sync(FULL, tag);
          uint32_t o = 0;
          if (tag != NOTAG) {
            o = hw[tag];
            const int pos = (int)o + __popc(peers & lt);
            dk[pos] = key;
            di[pos] = fi;
          }
          __syncwarp();
          if (tag != NOTAG && lane == __ffs(peers) - 1) hw[tag] = o + __popc(peers);
          __syncwarp();
        }
        uint32_t *const tk = sk;
        sk = dk;
        dk = tk;
        uint16_t *const ti = si;
        si = di;
        di = ti;
      }
      if (sk == kA) {
        for (int pos = lane; pos < T; pos += 32) kB[pos] = kA[pos];
      } else {
        for (int pos = lane; pos < T; pos += 32) iA[pos] = iB[pos];
      }
      __syncwarp();
      for (int pos = lane; pos < T; pos += 32) iB[iA[pos]] = (uint16_t)pos;
    }
  }
  __syncthreads();
  char *tab = g.tables + (size_t)unit * g.table_bytes;
  char *codes_g = tab + unit_codes_off(g.NB) + slot * SEG * 2;
  char *vals_g = tab + slot * SEG * 4;
  for (int s = tid; s < T; s += RANK_THREADS) {
    unsigned c[SEG];
    float v[SEG];
#pragma unroll
    for (int q = 0; q < SEG; q++) {
      c[q] = iB_of(q)[s];
      v[q] = key2f((kA_of(q) + T)[s]);
    }
    *reinterpret_cast<uint4 *>(codes_g + (size_t)s * UNIT * 2) =
        make_uint4(c[0] | c[1] << 16, c[2] | c[3] << 16, c[4] | c[5] << 16, c[6] | c[7] << 16);
    float4 *vg = reinterpret_cast<float4 *>(vals_g + (size_t)s * UNIT * 4);
    vg[0] = make_float4(v[0], v[1], v[2], v[3]);
    vg[1] = make_float4(v[4], v[5], v[6], v[7]);
  }
}

// ---------------------------------------------------------------------------
// psf_sweep_kernel
// ---------------------------------------------------------------------------

// One CTA per unit and group of warps, one warp per chunk of C queries (chunk
// blockIdx.y * warps + warp).  Shared memory: 512 bytes that nobody reads, then
// per warp the lanes' bit maps, word wd of lane l at wd 32 + l (every access
// of a warp meets every bank once, whatever words its lanes want), and two
// blocks of SWB value rows.  The medians are read from the value table through
// the L1: in shared memory they cost resident warps (600 x 256 x 256: 1.22
// against 1.58 ms).
// The warp stays together: lanes without a pixel of the annulus run along,
// loops whose trip counts differ between lanes turn on a vote, and nothing is
// loaded into a register ahead of its use (a copy of such a register waits for
// the load): values come through the rows in shared memory, the next block's
// codes are pulled into the L1 by copies of which only that side effect is
// wanted (600 x 256 x 256 with a time gate: 1.61 ms with registers two codes
// ahead, 1.20 so).
constexpr int SWB = 4;   // queries per block
__host__ __device__ constexpr size_t sweep_warp_bytes(int NW) { return (size_t)(NW + 1) * 128 + 2 * SWB * 128; }
constexpr size_t SWEEP_SINK = 512;

__device__ __forceinline__ void cp_async16_ca(void *smem_dst, const void *gmem_src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem_src) : "memory");
}

template <bool PERM>
__global__ void __launch_bounds__(512, 2) psf_sweep_kernel(const GeneralArgs g) {
  extern __shared__ __align__(16) uint32_t ssm[];
  const AdiArgs &a = g.a;
  const int T = a.T;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int *u = g.units + (size_t)blockIdx.x * UNIT_SEGS;
  const int ann = __ldg(&u[0]) >> ANN_SHIFT;
  const int NW = g.NB >> 5;   // map words per lane
  const char *tab = g.tables + (size_t)blockIdx.x * g.table_bytes;
  const float *sk = reinterpret_cast<const float *>(tab) + lane;
  uint32_t *sink = ssm;
  uint32_t *bm = sink + SWEEP_SINK / 4 + w * (int)(sweep_warp_bytes(NW) / 4);
  float *ring = reinterpret_cast<float *>(bm + (NW + 1) * 32);   // [2][SWB][32]
  bm += lane;
  const int16_t *rows = reinterpret_cast<const int16_t *>(tab + unit_codes_off(g.NB));
  const int16_t *codes = rows + lane;

  const int i0 = (blockIdx.y * (blockDim.x >> 5) + w) * g.C;
  const int i1 = min(T, i0 + g.C);
  if (i0 >= T) return;
  // lanes without a pixel of the annulus run along on the first segment's
  const int seg0 = __ldg(&u[0]) & ((1 << ANN_SHIFT) - 1);
  auto segment = [&](int q) {
    const int sgm = q == 0 ? seg0 : __ldg(&u[q]);
    return sgm < 0 ? seg0 : sgm;
  };
  const long long p = (long long)segment(lane / SEG) * SEG + (lane & (SEG - 1));
  const bool mine = (lane < SEG || __ldg(&u[lane / SEG]) >= 0) &&
                    annulus_of(p, a.n, a.iedge2, a.n_ann) == ann && group_general(a, p);

  auto code = [&](int s) { return (int)__ldg(&codes[s * UNIT]); };   // a signed load
  const int2 *LR = reinterpret_cast<const int2 *>(a.lr + (size_t)ann * T * 2);
  const int2 *AB = reinterpret_cast<const int2 *>(a.ab);
  auto frame = [&](int i) { return PERM ? (long long)__ldg(&a.perm[i]) : (long long)i; };
  // block b's value rows: lane (row, piece) copies 16 bytes
  const float *vsrc = a.in + (long long)segment((lane & 7) >> 1) * SEG + (lane & 1) * 4;
  auto fetch_values = [&](int b) {
    const int i = min(i0 + b * SWB + (lane >> 3), i1 - 1);
    cp_async16(ring + ((b & 1) * SWB + (lane >> 3)) * 32 + (lane & 7) * 4, vsrc + frame(i) * a.in_fs);
    cp_async_commit();
  };
  // code rows [P, P + 8) into the L1
  auto touch = [&](int P) {
    cp_async16_ca(sink + lane * 4, rows + min(P + (lane >> 2), T - 1) * UNIT + (lane & 3) * 8);
  };
  fetch_values(0);

  // ---- the first query's map: the members set, or, when they are the
  // majority, every rank set and the other frames cleared ------------------
  int L, R, A = 0, B = T;
  {
    const int2 gate = __ldg(&LR[i0]);
    L = gate.x;
    R = gate.y;
  }
  if (AB) {
    const int2 win = __ldg(&AB[i0]);
    A = win.x;
    B = win.y;
  }
  int nset = (L - A) + (B - R);
  const bool inv = 2 * nset > T;
  for (int wd = 0; wd < NW; wd++)
    bm[wd * 32] = !inv ? 0u : T >= wd * 32 + 32 ? FULL : (1u << (T - wd * 32)) - 1u;
  // (the codes of lanes without a pixel may be anything: theirs flip bits of
  // the word after the map's last one)
  auto word_of = [&](int c) { return &bm[min((unsigned)c >> 5, (unsigned)NW) * 32]; };
  auto flip = [&](int s0, int s1) {
    for (int s = s0; s < s1; s += 8) {
      int c[8];
#pragma unroll
      for (int q = 0; q < 8; q++) c[q] = code(min(s + q, T - 1));
#pragma unroll
      for (int q = 0; q < 8; q++)
        if (s + q < s1) *word_of(c[q]) ^= 1u << (c[q] & 31);
    }
  };
  if (inv) {
    flip(0, A);
    flip(L, R);
    flip(B, T);
  } else {
    flip(A, L);
    flip(R, B);
  }
  // the pointer pos at the k-th member; below = members before it
  int below = 0;
  int k = (nset - 1) >> 1;
  int pos = -1;
  for (int wd = 0; wd < NW; wd++) {
    const uint32_t word = bm[wd * 32];
    const int pc = __popc(word);
    if (pos < 0) {
      if (below + pc > k) {
        pos = wd * 32 + nth_set(word, k - below);
        below = k;
      } else {
        below += pc;
      }
    }
  }
  // act: this lane still follows its pixel's median.  Whatever the codes
  // hold, a map has bits of ranks below 32 NW only, and the value table has
  // that many rows.
  bool act = mine && pos >= 0;
  bool fail = mine && !act;
  pos = act ? pos : 0;
  __syncwarp();

  // ---- sweep ---------------------------------------------------------------
  // frame s leaves or enters, as its bit says
  auto toggle = [&](int s) {
    const int c = code(s);
    uint32_t *wp = word_of(c);
    const uint32_t bit = 1u << (c & 31);
    const uint32_t nw = *wp ^ bit;
    *wp = nw;
    if (c < pos) below += (nw & bit) ? 1 : -1;
  };
  auto pass_to = [&](int &P, int to) {
#pragma unroll 1
    while (__any_sync(FULL, P < to)) toggle(P++);
#pragma unroll 1
    while (__any_sync(FULL, P > to)) toggle(--P);
  };
  float *op = a.out + p + (PERM ? 0 : i0 * a.out_fs);
  const int nblk = (i1 - i0 + SWB - 1) / SWB;
#pragma unroll 1
  for (int b = 0; b < nblk; b++) {
    cp_async_wait_group<0>();
    __syncwarp();
    if (b + 1 < nblk) {
      fetch_values(b + 1);
      const int2 far = __ldg(&LR[min(i0 + (b + 1) * SWB, T - 1)]);
      touch(far.y);
      touch(far.x);
    }
    const float *vrow = ring + (b & 1) * SWB * 32 + lane;
    const int ie = min(i1, i0 + (b + 1) * SWB);
#pragma unroll 1
    for (int i = i0 + b * SWB; i < ie; i++, vrow += 32) {
      const int2 gt = __ldg(&LR[i]);
      pass_to(R, gt.y);
      pass_to(L, gt.x);
      if (AB) {
        const int2 wn = __ldg(&AB[i]);
        pass_to(A, wn.x);
        pass_to(B, wn.y);
      }
      nset = (L - A) + (B - R);
      k = (nset - 1) >> 1;
      // to the k-th member, one set bit at a time (one or two at most where
      // one frame leaves and one enters): down while more than k members lie
      // below, else up past members and cleared bits; the next word when this
      // one has no more (seldom one further)
      uint32_t cw = bm[(pos >> 5) * 32];
      bool here = (cw >> (pos & 31)) & 1u;
#pragma unroll 1
      while (__any_sync(FULL, act && (below != k || !here))) {
        const bool go = act && (below != k || !here), down = below > k;
        uint32_t m = cw & (down ? (1u << (pos & 31)) - 1u : 0xfffffffeu << (pos & 31));
        int wd = pos >> 5;
#pragma unroll 1
        while (__any_sync(FULL, go && act && m == 0u)) {
          if (go && act && m == 0u) {
            wd += down ? -1 : 1;
            act = (unsigned)wd < (unsigned)NW;
            if (act) m = cw = bm[wd * 32];
          }
        }
        if (go) {
          below += down ? -1 : here ? 1 : 0;
          pos = act ? wd * 32 + 31 - __clz(down ? m : m & (0u - m)) : 0;
          here = true;
        }
      }
      float med = __ldg(&sk[pos * 32]);
      if (__any_sync(FULL, (nset & 1) == 0)) {
        uint32_t m = cw & (0xfffffffeu << (pos & 31));
        int wd = pos >> 5;
#pragma unroll 1
        while (__any_sync(FULL, act && m == 0u)) {
          if (act && m == 0u) {
            wd++;
            act = wd < NW;
            if (act) m = bm[wd * 32];
          }
        }
        med = (med + __ldg(&sk[(act ? wd * 32 + __ffs(m) - 1 : 0) * 32])) * 0.5f;
      }
      fail |= mine && !act;
      if (PERM) op = a.out + p + frame(i) * a.out_fs;
      if (act) __stcs(op, *vrow - med);
      if (!PERM) op += a.out_fs;
    }
    __syncwarp();   // this block's rows are read before the next fetch lands in them
  }
  cp_async_wait_all();
  if (fail) atomicOr(a.status, STATUS_INTERNAL);
}

// Pixels of no annulus in the general path's 4-pixel groups: residual 0 in
// every frame, after the units, whose ranking tests these pixels' input (a
// call may be in place).  One CTA per listed segment.
__global__ void __launch_bounds__(128) general_zero_kernel(const AdiArgs a) {
  const long long p = (long long)__ldg(&a.zero[blockIdx.x]) * SEG + (threadIdx.x & (SEG - 1));
  if (annulus_of(p, a.n, a.iedge2, a.n_ann) >= 0 || !group_general(a, p)) return;
  for (int t = threadIdx.x / SEG; t < a.T; t += 128 / SEG) a.out[(long long)t * a.out_fs + p] = 0.f;
}

// Unit lists of a frame geometry, cached: the computation visits every pixel
// once, the plan of a repeated call is the same.
struct UnitKey {
  int n;
  std::vector<double> edge2;
  std::vector<int> banded;   // per annulus: has a band
  bool operator<(const UnitKey &o) const { return std::tie(n, edge2, banded) < std::tie(o.n, o.edge2, o.banded); }
};
struct UnitLists {
  std::vector<int> units, zero;
};
std::mutex g_unit_mu;
std::map<UnitKey, UnitLists> g_unit_cache;

}  // namespace

int plan_general_path(AdiPlanHost &ap, int64_t T, int32_t n) {
  (void)T;
  const int A = (int)ap.edge2.size() - 1;
  UnitKey key{n, ap.edge2, {}};
  bool any_band = false, all_band = true;
  for (int an = 0; an < A; an++) {
    key.banded.push_back(ap.band[4 * an + 2] > 0);
    any_band |= key.banded[an] != 0;
    all_band &= key.banded[an] != 0;
  }
  ap.units.clear();
  ap.zero.clear();
  if (all_band) return GRAPHIC_OK;
  {
    std::lock_guard<std::mutex> lk(g_unit_mu);
    auto it = g_unit_cache.find(key);
    if (it != g_unit_cache.end()) {
      ap.units = it->second.units;
      ap.zero = it->second.zero;
      return GRAPHIC_OK;
    }
  }
  // per annulus the segments with a pixel of it in a general 4-pixel group
  std::vector<std::vector<int>> segs(A);
  for (int s = 0; s < n * n / SEG; s++) {
    int an[SEG];
    for (int q = 0; q < SEG; q++) {
      const int p = s * SEG + q;
      const int64_t x = p % n - n / 2, y = p / n - n / 2;
      const double rho2 = (double)(x * x + y * y);
      const int k = (int)(std::upper_bound(ap.edge2.begin(), ap.edge2.end(), rho2) - ap.edge2.begin()) - 1;
      an[q] = k >= 0 && k < A ? k : -1;
    }
    bool zero = false;
    for (int h = 0; h < SEG; h += 4) {
      bool general = !any_band;
      for (int q = h; q < h + 4; q++) general |= an[q] >= 0 && !key.banded[an[q]];
      if (!general) continue;
      for (int q = h; q < h + 4; q++) {
        if (an[q] < 0) zero = true;
        else if (segs[an[q]].empty() || segs[an[q]].back() != s) segs[an[q]].push_back(s);
      }
    }
    if (zero) ap.zero.push_back(s);
  }
  for (int a = 0; a < A; a++)
    for (size_t k = 0; k < segs[a].size(); k += UNIT_SEGS)
      for (int q = 0; q < UNIT_SEGS; q++) {
        const int s = k + q < segs[a].size() ? segs[a][k + q] : -1;
        ap.units.push_back(q == 0 ? (s | a << ANN_SHIFT) : s);
      }
  std::lock_guard<std::mutex> lk(g_unit_mu);
  if (g_unit_cache.size() > 16) g_unit_cache.clear();
  g_unit_cache[key] = {ap.units, ap.zero};
  return GRAPHIC_OK;
}

size_t general_scratch_bytes(const AdiPlanHost &ap, int64_t T) {
  const size_t units = ap.units.size() / UNIT_SEGS, one = unit_bytes((int)T);
  return units == 0 ? 0 : std::max(one, std::min(units * one, kBandScratchMax));
}

namespace {

constexpr size_t kPlainSmem = 47 * 1024;   // dynamic shared memory that needs no attribute (48 KB with the static)

cudaError_t launch_adi_general(const AdiArgs &a, cudaStream_t st, int &nl) {
  const int T = a.T;
  cudaError_t e;
  auto zero = [&]() {
    if (a.n_zero == 0) return cudaSuccess;
    general_zero_kernel<<<(unsigned)a.n_zero, 128, 0, st>>>(a);
    nl++;
    return cudaGetLastError();
  };
  if (a.n_units == 0) return zero();
  int dev = 0, sms = 0, per_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  GeneralArgs g{};
  g.a = a;
  g.NB = table_rows(T);
  g.tables = a.band_scratch;
  g.table_bytes = unit_bytes(T);
  const int per = (int)std::min<size_t>((size_t)a.n_units, a.band_scratch_cap / g.table_bytes);
  if (per < 1) return cudaErrorInvalidValue;
  // counters: 1024 from 257 frames on, 512 from 129 (512 and 256 alike on plain
  // noise; one bright frame, which leaves all others in one bin: ranking 256
  // frames of 512 x 512 4392 us with 256 counters, without the radix sort, 2018
  // with 512 and the sort, 130 frames 1542 and 1136), 256 below (64 frames 246
  // us, 265 with 512; one bright frame 456 and 695)
  void (*rank)(GeneralArgs) = T <= 128 ? full_rank_kernel<256> : T <= 256 ? full_rank_kernel<512> : full_rank_kernel<1024>;
  const size_t rsmem = SEG * (T <= 128   ? full_pixel_bytes<256>(T)
                              : T <= 256 ? full_pixel_bytes<512>(T)
                                         : full_pixel_bytes<1024>(T));
  if (rsmem > kPlainSmem &&
      (e = cudaFuncSetAttribute(rank, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rsmem)) != cudaSuccess)
    return e;
  // sweep: chunks of at least 32 queries; of 16, 8 or 4 warps a CTA the most
  // that leaves the most warps resident (32 by registers: 2000 frames, whose
  // maps take 9 KB a warp, 2.86 ms for 128 x 128 with 8 warps, 3.30 with 16)
  const size_t maps = sweep_warp_bytes(g.NB / 32);
  int warps = 16;
  auto resident = [&](int w) {
    return std::min<long long>(32 / w, per_sm / (long long)(w * maps + SWEEP_SINK + 1024)) * w;
  };
  while (warps > 4 && resident(warps / 2) > resident(warps)) warps /= 2;
  const int most = warps;
  warps = std::min(warps, std::max(1, T / 32));
  int cols = 1;
  while ((T + warps * cols - 1) / (warps * cols) > 128 ||
         ((long long)per * warps * cols < 16ll * sms && T / (warps * cols * 2) >= 32))
    cols *= 2;
  // few units leave SMs idle for as long as a chunk takes: chunks of down to 4
  // queries (each builds its own map first) until the SMs have 24 warps each.
  // Sweeps with chunks of 32 queries and 16 warps, then so: two annuli of 64 x
  // 64, 64 frames 38 -> 8 us, 1000 frames 315 -> 53; all of 64 x 64, 2048 frames
  // 1057 -> 772; the two inner annuli of 2000 x 512 x 512 125 -> 110 (16 warps
  // 103, 32 140; 64 x 64 x 1000 329, 197 and 198)
  const int chunks = (int)std::min<long long>((T + 3) / 4, (24ll * sms + per - 1) / per);
  if (chunks > warps * cols) {
    warps = std::min(most, chunks);
    cols = (chunks + warps - 1) / warps;
  }
  const size_t ssmem = SWEEP_SINK + warps * maps;
  g.C = (T + warps * cols - 1) / (warps * cols);
  void (*sweep)(GeneralArgs) = a.perm_id ? psf_sweep_kernel<false> : psf_sweep_kernel<true>;
  if (ssmem > kPlainSmem &&
      (e = cudaFuncSetAttribute(sweep, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ssmem)) != cudaSuccess)
    return e;
  for (int u0 = 0; u0 < a.n_units; u0 += per) {
    const unsigned nu = (unsigned)std::min(per, a.n_units - u0);
    g.units = a.units + (size_t)u0 * UNIT_SEGS;
    rank<<<nu * UNIT_SEGS, RANK_THREADS, rsmem, st>>>(g);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    sweep<<<dim3(nu, cols), 32 * warps, ssmem, st>>>(g);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    nl += 2;
  }
  return zero();
}

}  // namespace

cudaError_t launch_adi_median(const AdiArgs &a, cudaStream_t st, int *launched) {
  int dummy = 0;
  int &nl = launched ? *launched : dummy;
  nl = 0;
  // the two paths' 4-pixel groups are disjoint, also for calls in place
  if (a.n_zero > 0 || a.n_units > 0) {
    if (a.mark) a.mark(a.mark_user, 0, 1);
    const cudaError_t e = launch_adi_general(a, st, nl);
    if (a.mark) a.mark(a.mark_user, 0, 0);
    if (e != cudaSuccess) return e;
  }
  return a.wmax > 0 ? launch_adi_band(a, st, &nl) : cudaSuccess;
}

}  // namespace graphic
