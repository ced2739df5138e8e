// register.cu -- registration (Sect. 3.1): per frame the centroid of the
// patch of contiguous pixels above a threshold around the brightest pixel,
// then a Moffat fit by Levenberg-Marquardt started there; the centre gives
// the recentring shift, alpha and beta the FWHM.
//
// Two kernels.
//  * frame_argmax_kernel: the only pass over whole frames, HBM-bound.  One
//    block per (frame, chunk of REG_CHUNK pixels), 16-byte loads; each block
//    merges its maximum into the frame's 64-bit word by atomicMax on the
//    packed (total-order key of the value, ~index): the largest value wins,
//    the smallest index on a tie.  A non-finite value sets the word to all
//    ones (no finite value packs to it) and the status flag.
//  * register_fit_kernel: one block of four or two warps per frame.  The box of
//    half-size R around the seed and its 8-connected flood fill in shared
//    memory (sweeps until none changes: the fixpoint is the connected
//    component whatever the order of the updates), FP64 patch sums, then the
//    fit window in the same shared buffer and the Levenberg-Marquardt loop.
//    Warp 0 holds the parameters, solves the damped 6 x 6 system and takes
//    the decisions; the model and its derivatives are evaluated by every
//    warp, a pixel per thread, into shared memory, and the 28 sums of the
//    normal equations are then taken in four groups of seven.  Each sum is
//    taken in one fixed order (32 strided partials, then a butterfly over
//    them).  Start values, damping schedule and stopping rules are those of the
//    FP64 oracle.
//    Bound: the FP64 pipe (a warp instruction takes it 16 cycles; 14 000 of
//    them per fitted frame of the 256 x 256 workload) and, below a few frames
//    per SM, the latency of the chain evaluate - sum - solve.  With a frame on
//    one warp that chain was all there was; calls with one warp and with four,
//    same bits: one frame 612 and 315 us, 400 of 256 x 256 1259 and 774, 1600
//    2084 and 1849.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "graphic_internal.h"

namespace graphic {
namespace {

constexpr int ARG_THREADS = 256;
constexpr int ARG_VEC = 8;                                   // float4 loads per thread per chunk
constexpr long long REG_CHUNK = (long long)ARG_THREADS * ARG_VEC * 4;   // pixels per block
// Twelve warps an SM (register budget), as blocks of WARPS = 4 or 2, a frame
// each (launch_register_fit chooses).  The bits do not depend on it: warp w
// takes the groups w, w + WARPS, ... of the sums, each in its one order.
constexpr int FIT_SM_WARPS = 12;
constexpr int GROUPS = 4;
constexpr int FIT_TILE = 512;  // window pixels whose model values are in shared memory at a time
constexpr int FIT_Z = 6;       // values per pixel there: dI/dI0, dx0, dy0, dalpha, dbeta and the residual
constexpr double REG_PI = 3.14159265358979323846;
constexpr unsigned long long KEY_NONFINITE = ~0ull;

__device__ __forceinline__ uint32_t order_key(float x) {
  if (x == 0.0f) x = 0.0f;   // -0 and +0 compare equal: the index decides
  const uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__device__ __forceinline__ unsigned long long pack(float v, uint32_t idx) {
  return ((unsigned long long)order_key(v) << 32) | (unsigned long long)(~idx);
}

__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, x, o);
    x = y > x ? y : x;
  }
  return x;
}

__global__ void __launch_bounds__(ARG_THREADS) frame_argmax_kernel(const float *__restrict__ in, long long T,
                                                                   long long nn, long long chunks,
                                                                   unsigned long long *keys, int *status) {
  __shared__ unsigned long long part[ARG_THREADS / 32];
  __shared__ int part_bad[ARG_THREADS / 32];
  const long long items = T * chunks;
  const bool vec = (nn & 3) == 0;
  for (long long it = blockIdx.x; it < items; it += gridDim.x) {
    const long long f = it / chunks, c = it - f * chunks;
    const float *fr = in + f * nn;
    const long long s = c * REG_CHUNK, e = min(nn, s + REG_CHUNK);
    float best = -INFINITY;
    long long bi = -1;
    bool bad = false;
    if (vec) {
      const float4 *f4 = reinterpret_cast<const float4 *>(fr);
      const long long s4 = s >> 2, e4 = e >> 2;
      float4 v[ARG_VEC];
#pragma unroll
      for (int k = 0; k < ARG_VEC; k++) {
        const long long j = s4 + threadIdx.x + (long long)k * ARG_THREADS;
        v[k] = j < e4 ? __ldcs(&f4[j]) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      }
#pragma unroll
      for (int k = 0; k < ARG_VEC; k++) {
        const long long j = s4 + threadIdx.x + (long long)k * ARG_THREADS;
        const float q[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
        if (j < e4) {
#pragma unroll
          for (int l = 0; l < 4; l++) {
            bad |= !(fabsf(q[l]) <= 3.402823466e38f);
            if (q[l] > best || bi < 0) {
              best = q[l];
              bi = 4 * j + l;
            }
          }
        }
      }
    } else {
      for (long long j = s + threadIdx.x; j < e; j += ARG_THREADS) {
        const float x = fr[j];
        bad |= !(fabsf(x) <= 3.402823466e38f);
        if (x > best || bi < 0) {
          best = x;
          bi = j;
        }
      }
    }
    unsigned long long key = bi >= 0 ? pack(best, (uint32_t)bi) : 0ull;
    key = warp_max_u64(key);
    const int wbad = __any_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0) {
      part[threadIdx.x >> 5] = key;
      part_bad[threadIdx.x >> 5] = wbad;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned long long k = 0;
      int b = 0;
      for (int w = 0; w < ARG_THREADS / 32; w++) {
        k = part[w] > k ? part[w] : k;
        b |= part_bad[w];
      }
      if (b) {
        atomicMax(&keys[f], KEY_NONFINITE);
        atomicOr(status, STATUS_NONFINITE);
      } else {
        atomicMax(&keys[f], k);
      }
    }
    __syncthreads();
  }
}

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

__device__ __forceinline__ float warp_min(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fminf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}

// Moffat profile (Sect. 3.1) with parameters p = (I0, x0, y0, alpha, beta,
// Bg): the quotients that do not depend on the pixel, once per parameter set.
struct MoffatConst {
  double x0, y0, beta, bg, ia2, A, c0, c1, c3, c4, c5;
};

__device__ __forceinline__ MoffatConst moffat_const(const double *p) {
  constexpr double INV_PI = 0.318309886183790671537767526745;   // 1 / pi
  MoffatConst k;
  const double I0 = p[0], al = p[3], be = p[4];
  const double ia = 1.0 / al;                  // the one division of a parameter set
  k.x0 = p[1];
  k.y0 = p[2];
  k.beta = be;
  k.bg = p[5];
  k.ia2 = ia * ia;
  k.c0 = (be - 1.0) * k.ia2 * INV_PI;          // dI/dI0 = c0 P
  k.A = I0 * k.c0;                             // I0 (beta - 1) / (pi alpha^2)
  k.c1 = 2.0 * k.A * be * k.ia2;               // dI/dx0 = c1 P / u dx
  k.c3 = -2.0 * k.A * ia;                      // dI/dalpha = c3 P + c4 rho^2 P / u
  k.c4 = k.c1 * ia;
  k.c5 = I0 * k.ia2 * INV_PI;                  // dI/dbeta = c5 P - A ln(u) P
  return k;
}

// Damped 6 x 6 solve by Cholesky; false when the matrix is not positive
// definite.  The six pivots' reciprocals are taken once, so the
// factorisation and both substitutions run on multiplications (FP64
// divisions are long instruction sequences on this GPU).
__device__ bool chol6(const double *A, const double *b, double *x) {
  double L[21], inv[6];   // lower triangle, row i at i (i + 1) / 2; 1 / L[i][i]
#pragma unroll
  for (int i = 0; i < 6; i++)
#pragma unroll
    for (int j = 0; j <= i; j++) {
      double s = A[i * 6 + j];
#pragma unroll
      for (int k = 0; k < j; k++) s -= L[i * (i + 1) / 2 + k] * L[j * (j + 1) / 2 + k];
      if (i == j) {
        if (!(s > 0)) return false;
        const double d = sqrt(s);
        L[i * (i + 1) / 2 + i] = d;
        inv[i] = 1.0 / d;
      } else {
        L[i * (i + 1) / 2 + j] = s * inv[j];
      }
    }
  double y[6];
#pragma unroll
  for (int i = 0; i < 6; i++) {
    double s = b[i];
#pragma unroll
    for (int k = 0; k < i; k++) s -= L[i * (i + 1) / 2 + k] * y[k];
    y[i] = s * inv[i];
  }
#pragma unroll
  for (int i = 5; i >= 0; i--) {
    double s = y[i];
#pragma unroll
    for (int k = i + 1; k < 6; k++) s -= L[k * (k + 1) / 2 + i] * x[k];
    x[i] = s * inv[i];
  }
  return true;
}

// What the warps of a block share besides the window and the model values.
struct FitShared {
  double kc[11];      // MoffatConst of the parameters to evaluate
  float kf[11];       // the same in FP32
  double ne[28];      // the last evaluation's sums: J^T J lower triangle, J^T r, the squared error
  double ne_cur[28];  // those of the current parameters
  double patch[4];    // patch size, value sum and first moments
  int mode;           // what to evaluate next (EVAL_*)
  int touch;          // the patch touches the box's inner border
  long long frame;
};
enum { EVAL_DONE = 0, EVAL_F32 = 1, EVAL_F64 = 2 };

// Barrier of all the block's warps, for the places where warp 0 and the
// others wait at different instructions.
template <int WARPS>
__device__ __forceinline__ void fit_sync() {
  if constexpr (WARPS == 1) __syncwarp();
  else asm volatile("bar.sync 1, %0;" ::"n"(32 * WARPS) : "memory");
}

// Model values of one pixel at the parameters k: derivatives by I0, x0, y0,
// alpha, beta (the one by Bg is 1) and the residual.  Where a sum of two
// products leaves open which of them is rounded, the fused form is written
// out: alpha and beta are so correlated that a last bit here moves them by
// 1e-8, so the bits must not depend on how the compiler orders the code.
__device__ __forceinline__ void moffat_pixel(const MoffatConst &k, int col, int row, float val, double (&z)[FIT_Z]) {
  const double dx = (double)col - k.x0, dy = (double)row - k.y0;
  const double rho2 = fma(dy, dy, dx * dx);
  const double u = 1.0 + rho2 * k.ia2;
  const double lu = log(u);
  const double P = exp(-k.beta * lu);
  // 1 / u: the FP32 reciprocal refined by two Newton steps r <- r (2 - u r)
  // (relative error 1e-7 -> 1e-14 -> below FP64 rounding; u >= 1)
  double ru = (double)__frcp_rn((float)u);
  ru = ru * (2.0 - u * ru);
  ru = ru * (2.0 - u * ru);
  const double Pu = P * ru;
  z[5] = k.A * P + k.bg - (double)val;
  z[0] = k.c0 * P;
  z[1] = k.c1 * Pu * dx;
  z[2] = k.c1 * Pu * dy;
  z[3] = fma(k.c4 * rho2, Pu, k.c3 * P);
  z[4] = fma(k.c5, P, -(k.A * lu * P));
}

// The same in FP32: on GB300 the FP32 pipe is 64 times the FP64 one, and the
// first iterations only need to come close.
struct MoffatConst32 {
  float x0, y0, beta, bg, ia2, A, c0, c1, c3, c4, c5;
};

__device__ __forceinline__ void moffat_pixel(const MoffatConst32 &k, int col, int row, float val, float (&z)[FIT_Z]) {
  const float dx = (float)col - k.x0, dy = (float)row - k.y0;
  const float rho2 = fmaf(dy, dy, dx * dx);
  const float u = 1.0f + rho2 * k.ia2;
  const float l2 = log2f(u);
  const float P = exp2f(-k.beta * l2);
  const float Pu = P / u;
  z[5] = k.A * P + k.bg - val;
  z[0] = k.c0 * P;
  z[1] = k.c1 * Pu * dx;
  z[2] = k.c1 * Pu * dy;
  z[3] = fmaf(k.c3, P, k.c4 * rho2 * Pu);
  z[4] = fmaf(k.c5, P, -(k.A * (l2 * 0.69314718056f) * P));
}

// The seven sums of group G over the tile's pixels lane, lane + 32, ... (the
// 28 products of derivatives and residual; the derivative by Bg is 1):
//   0  residual x (five derivatives, 1, residual)
//   1  1 x (five derivatives, 1); dI0 dI0
//   2  dbeta x (five derivatives); dx0 x (dI0, dx0)
//   3  dalpha x (dI0, dx0, dy0, dalpha); dy0 x (dI0, dx0, dy0)
template <int G, class R>
__device__ __forceinline__ void group_sums(const R *z, int count, int lane, R (&acc)[8]) {
#pragma unroll 2
  for (int i = lane; i < count; i += 32) {
    R v[FIT_Z];
#pragma unroll
    for (int c = 0; c < FIT_Z; c++) v[c] = z[c * FIT_TILE + i];   // those unused are dropped
    if constexpr (G == 0) {
#pragma unroll
      for (int c = 0; c < 5; c++) acc[c] += v[c] * v[5];
      acc[5] += v[5];
      acc[6] += v[5] * v[5];
    } else if constexpr (G == 1) {
#pragma unroll
      for (int c = 0; c < 5; c++) acc[c] += v[c];
      acc[5] += (R)1;
      acc[6] += v[0] * v[0];
    } else if constexpr (G == 2) {
#pragma unroll
      for (int c = 0; c < 5; c++) acc[c] += v[4] * v[c];
      acc[5] += v[1] * v[0];
      acc[6] += v[1] * v[1];
    } else {
#pragma unroll
      for (int c = 0; c < 4; c++) acc[c] += v[3] * v[c];
#pragma unroll
      for (int c = 0; c < 3; c++) acc[4 + c] += v[2] * v[c];
    }
  }
}

// Place of sum j of group G among the 28 (row i of the triangle starts at
// i (i + 1) / 2).
template <int G>
__device__ __forceinline__ int group_place(int j) {
  if constexpr (G == 0) return 21 + j;
  else if constexpr (G == 1) return j < 6 ? 15 + j : 0;
  else if constexpr (G == 2) return j < 5 ? 10 + j : j - 4;
  else return j < 4 ? 6 + j : j - 1;
}

// Butterfly sums of acc[0..8) over the warp, halving what a lane holds at
// each of the first three levels (9 additions for 8 sums instead of 40; every
// addition adds the two operands that the full butterfly adds, so the bits
// are those of eight full ones): acc[0] ends as the sum of slot
// 4 (lane & 16) / 16 + 2 (lane & 8) / 8 + (lane & 4) / 4.
template <class R>
__device__ __forceinline__ void butterfly8(R (&acc)[8], int lane) {
#pragma unroll
  for (int o = 16, h = 4; o >= 4; o >>= 1, h >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int k = 0; k < h; k++) {
      const R send = up ? acc[k] : acc[k + h], keep = up ? acc[k + h] : acc[k];
      acc[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 2);
  acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
}

template <int G, class R>
__device__ __forceinline__ void group_finish(R (&acc)[8], int lane, double *ne) {
  butterfly8(acc, lane);
  const int j = (lane >> 2) & 7, slot = ((j & 4) ? 4 : 0) + ((j & 2) ? 2 : 0) + (j & 1);
  if ((lane & 3) == 0 && slot < 7) ne[group_place<G>(slot)] = (double)acc[0];
}

// One pass over the window at the shared parameters, by every warp of the
// block: the squared error of the model and the normal equations of its
// analytic Jacobian, in s.ne when the closing barrier has passed.  The oracle
// takes the two in separate passes; one pass serves both here because the
// normal equations of an accepted trial point are those of the next
// iteration.
template <int WARPS, class R, class K>
__device__ __forceinline__ void window_pass(const K &k, FitShared &s, R *z, const float *win, int WH, int WW, int wr0,
                                            int wc0) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int np = WH * WW;
  R acc[GROUPS / WARPS][8] = {};
  for (int t0 = 0; t0 < np; t0 += FIT_TILE) {
    const int count = min(FIT_TILE, np - t0);
    if (t0 > 0) fit_sync<WARPS>();   // the sums have read the tile before
    for (int i = threadIdx.x; i < count; i += 32 * WARPS) {
      const int r = (t0 + i) / WW, c = t0 + i - r * WW;
      R v[FIT_Z];
      moffat_pixel(k, c + wc0, r + wr0, win[t0 + i], v);
#pragma unroll
      for (int q = 0; q < FIT_Z; q++) z[q * FIT_TILE + i] = v[q];
    }
    fit_sync<WARPS>();
    if (wid == 0 % WARPS) group_sums<0>(z, count, lane, acc[0 / WARPS]);
    if (wid == 1 % WARPS) group_sums<1>(z, count, lane, acc[1 / WARPS]);
    if (wid == 2 % WARPS) group_sums<2>(z, count, lane, acc[2 / WARPS]);
    if (wid == 3 % WARPS) group_sums<3>(z, count, lane, acc[3 / WARPS]);
  }
  if (wid == 0 % WARPS) group_finish<0>(acc[0 / WARPS], lane, s.ne);
  if (wid == 1 % WARPS) group_finish<1>(acc[1 / WARPS], lane, s.ne);
  if (wid == 2 % WARPS) group_finish<2>(acc[2 / WARPS], lane, s.ne);
  if (wid == 3 % WARPS) group_finish<3>(acc[3 / WARPS], lane, s.ne);
  fit_sync<WARPS>();
}

// The parameters' quotients from shared memory, then the pass.
template <int WARPS>
__device__ __forceinline__ void window_pass_shared(int mode, FitShared &s, unsigned char *zb, const float *win, int WH,
                                                   int WW, int wr0, int wc0) {
  if (mode == EVAL_F32) {
    const MoffatConst32 k = {s.kf[0], s.kf[1], s.kf[2], s.kf[3], s.kf[4], s.kf[5],
                             s.kf[6], s.kf[7], s.kf[8], s.kf[9], s.kf[10]};
    window_pass<WARPS, float>(k, s, reinterpret_cast<float *>(zb), win, WH, WW, wr0, wc0);
  } else {
    const MoffatConst k = {s.kc[0], s.kc[1], s.kc[2], s.kc[3], s.kc[4], s.kc[5],
                           s.kc[6], s.kc[7], s.kc[8], s.kc[9], s.kc[10]};
    window_pass<WARPS, double>(k, s, reinterpret_cast<double *>(zb), win, WH, WW, wr0, wc0);
  }
}

// The damped step of the FP32 phase: the normal equations scaled by D =
// diag(J^T J)^(-1/2) (unit diagonal, so the damping lambda diag(J^T J)
// becomes lambda I), factorised and solved in FP32, the step scaled back.
// False when the scaled matrix is not positive definite.
__device__ bool step32(const double *ne, double lambda, double *d) {
  float dinv[6], L[21], inv[6], y[6];
#pragma unroll
  for (int i = 0; i < 6; i++) {
    const double a = ne[i * (i + 1) / 2 + i];
    dinv[i] = a > 0 ? rsqrtf((float)a) : 1.0f;
  }
#pragma unroll
  for (int i = 0; i < 6; i++)
#pragma unroll
    for (int j = 0; j <= i; j++) {
      float s = (float)ne[i * (i + 1) / 2 + j] * dinv[i] * dinv[j];
      if (i == j) {
        const double a = ne[i * (i + 1) / 2 + i];
        s += (float)(lambda * (a > 0 ? 1.0 : 1e-12));
      }
#pragma unroll
      for (int k = 0; k < j; k++) s -= L[i * (i + 1) / 2 + k] * L[j * (j + 1) / 2 + k];
      if (i == j) {
        if (!(s > 0.0f)) return false;
        const float dd = sqrtf(s);
        L[i * (i + 1) / 2 + i] = dd;
        inv[i] = 1.0f / dd;
      } else {
        L[i * (i + 1) / 2 + j] = s * inv[j];
      }
    }
#pragma unroll
  for (int i = 0; i < 6; i++) {
    float s = -(float)ne[21 + i] * dinv[i];
#pragma unroll
    for (int k = 0; k < i; k++) s -= L[i * (i + 1) / 2 + k] * y[k];
    y[i] = s * inv[i];
  }
  float x[6];
#pragma unroll
  for (int i = 5; i >= 0; i--) {
    float s = y[i];
#pragma unroll
    for (int k = i + 1; k < 6; k++) s -= L[k * (k + 1) / 2 + i] * x[k];
    x[i] = s * inv[i];
  }
#pragma unroll
  for (int i = 0; i < 6; i++) d[i] = (double)(x[i] * dinv[i]);
  return true;
}

// Evaluation at the parameters p, called by warp 0: hands the quotients to
// the block and takes part in the pass.  Returns the squared error (the other
// sums are in s.ne).
template <int WARPS, bool F32>
__device__ __forceinline__ double evaluate(const double *p, FitShared &s, unsigned char *zb, const float *win, int WH,
                                           int WW, int wr0, int wc0) {
  const int lane = threadIdx.x & 31;
  const MoffatConst k = moffat_const(p);
  __syncwarp();   // every lane has read the last evaluation's sums
  if (lane == 0) {
    const double v[11] = {k.x0, k.y0, k.beta, k.bg, k.ia2, k.A, k.c0, k.c1, k.c3, k.c4, k.c5};
#pragma unroll
    for (int q = 0; q < 11; q++) {
      if constexpr (F32) s.kf[q] = (float)v[q];
      else s.kc[q] = v[q];
    }
    s.mode = F32 ? EVAL_F32 : EVAL_F64;
  }
  fit_sync<WARPS>();
  window_pass_shared<WARPS>(F32 ? EVAL_F32 : EVAL_F64, s, zb, win, WH, WW, wr0, wc0);
  return s.ne[27];
}

// Levenberg-Marquardt iterations from p (the oracle's steps: damping lambda
// x diag(J^T J) from 1e-3, /10 (floor lam_floor) on an accepted step, x10 on
// a rejected one or one leaving alpha <= 0 or beta <= 1, at most 10 tries;
// stop when an accepted step lowers the squared error by at most stop_rel
// of it, when no try lowers it, or after 200 iterations).  F32 selects the
// FP32 evaluation.  Returns the iterations made; p and cost are updated.
template <int WARPS, bool F32>
__device__ __forceinline__ int lm_loop(double (&p)[6], double &cost, double lam_floor, double stop_rel, FitShared &s,
                                       unsigned char *zb, const float *buf, int WH, int WW, int wr0, int wc0) {
  const int lane = threadIdx.x & 31;
  const double *ne_cur = s.ne_cur;
  cost = evaluate<WARPS, F32>(p, s, zb, buf, WH, WW, wr0, wc0);
  // the normal equations at p
  if (lane < 27) s.ne_cur[lane] = s.ne[lane];
  __syncwarp();
  double lambda = 1e-3;
  int it;
  for (it = 0; it < 200; it++) {
    bool accepted = false;
    double newcost = cost;
    for (int tries = 0; tries < 10; tries++) {
      double d[6], q[6];
      bool ok;
      if constexpr (F32) {
        ok = step32(ne_cur, lambda, d);
      } else {
        double A[36], mg[6];
        int k = 0;
#pragma unroll
        for (int ii = 0; ii < 6; ii++)
#pragma unroll
          for (int jj = 0; jj <= ii; jj++) {
            A[ii * 6 + jj] = ne_cur[k];
            A[jj * 6 + ii] = ne_cur[k];
            k++;
          }
#pragma unroll
        for (int ii = 0; ii < 6; ii++) {
          const double di = A[ii * 6 + ii] > 0 ? A[ii * 6 + ii] : 1e-12;
          A[ii * 6 + ii] += lambda * di;
          mg[ii] = -ne_cur[21 + ii];
        }
        ok = chol6(A, mg, d);
      }
      if (!ok) {
        lambda *= 10.0;
        continue;
      }
#pragma unroll
      for (int ii = 0; ii < 6; ii++) q[ii] = p[ii] + d[ii];
      if (!(q[3] > 0) || !(q[4] > 1.0)) {
        lambda *= 10.0;
        continue;
      }
      newcost = evaluate<WARPS, F32>(q, s, zb, buf, WH, WW, wr0, wc0);
      if (newcost < cost) {
#pragma unroll
        for (int ii = 0; ii < 6; ii++) p[ii] = q[ii];
        __syncwarp();   // every lane has read ne_cur
        if (lane < 27) s.ne_cur[lane] = s.ne[lane];
        __syncwarp();
        lambda = fmax(lambda / 10.0, lam_floor);
        accepted = true;
        break;
      }
      lambda *= 10.0;
    }
    if (!accepted) break;
    const double drop = cost - newcost;
    cost = newcost;
    if (drop <= stop_rel * cost) {
      it++;
      break;
    }
  }
  return it;
}

// One frame on one block: seed from the argmax word, patch, centroid, fit.
// buf: side^2 floats (the box, then the window); lab: side^2 bytes (the
// patch), the same memory as the model values zb, which come after it.
template <int WARPS>
__device__ __forceinline__ void fit_frame(const RegArgs &a, unsigned long long key, long long f, float *buf,
                                          uint8_t *lab, unsigned char *zb, FitShared &s) {
  constexpr int THREADS = 32 * WARPS;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int n = a.n;
  const float *fr = a.in + f * (long long)n * n;
  double *out = a.out + f * 8;
  auto not_found = [&]() {
    if (tid < 8) out[tid] = 0.0;
    if (tid == 0 && a.iters) a.iters[f] = 0;
  };
  if (key == KEY_NONFINITE) {
    not_found();
    return;
  }
  const long long seed = (long long)(~(uint32_t)(key & 0xffffffffull));
  if (key == 0ull || seed >= (long long)n * n) {   // no maximum recorded: cannot happen for n >= 1
    if (tid == 0) atomicOr(a.status, STATUS_INTERNAL);
    not_found();
    return;
  }
  const int r0 = (int)(seed / n), c0 = (int)(seed - (long long)r0 * n), R = a.R;
  const int rlo = max(r0 - R, 0), rhi = min(r0 + R, n - 1), clo = max(c0 - R, 0), chi = min(c0 + R, n - 1);
  const int H = rhi - rlo + 1, W = chi - clo + 1;
  const double th = a.thresh;

  // ---- patch: flood fill of the pixels above the threshold ----------------
  // lab: 0 below the threshold, 2 above and not (yet) reached, 1 in the patch
  const int si = (r0 - rlo) * W + (c0 - clo);
  for (int i = tid; i < H * W; i += THREADS) {
    const int r = i / W, c = i - r * W;
    const float v = fr[(long long)(r + rlo) * n + (c + clo)];
    buf[i] = v;
    lab[i] = (double)v > th ? (i == si ? 1 : 2) : 0;
  }
  if (tid == 0) s.touch = 0;
  __syncthreads();
  if (lab[si] == 0) {   // the seed itself is not above the threshold
    not_found();
    return;
  }
  for (int sweep = 0; sweep <= H * W; sweep++) {
    int changed = 0;
    // 32 pixels a thread at a time: all found against the same labels, then
    // all marked
    for (int b = 0; b < H * W; b += 32 * THREADS) {
      uint32_t reached = 0;
      for (int i = b + tid, k = 0; k < 32 && i < H * W; i += THREADS, k++) {
        if (lab[i] != 2) continue;
        const int r = i / W, c = i - r * W;
        bool nb = false;
        for (int dr = -1; dr <= 1; dr++)
          for (int dc = -1; dc <= 1; dc++) {
            const int rr = r + dr, cc = c + dc;
            if ((dr || dc) && rr >= 0 && rr < H && cc >= 0 && cc < W && lab[rr * W + cc] == 1) nb = true;
          }
        if (nb) reached |= 1u << k;
      }
      __syncthreads();
      changed |= reached != 0;
      for (; reached; reached &= reached - 1) lab[b + tid + (__ffs(reached) - 1) * THREADS] = 1;
      __syncthreads();
    }
    if (!__syncthreads_or(changed)) break;
  }
  // the four sums, warp by warp (each in the order of 32 strided partials)
  for (int k = wid; k < 4; k += WARPS) {
    double acc = 0.0;
    bool touch = false;
    for (int i = lane; i < H * W; i += 32) {
      if (lab[i] != 1) continue;
      const int r = i / W, c = i - r * W;
      const double v = buf[i];
      if (k == 0) {
        acc += 1.0;
        touch |= (r == 0 && rlo > 0) || (r == H - 1 && rhi < n - 1) || (c == 0 && clo > 0) || (c == W - 1 && chi < n - 1);
      } else if (k == 1) {
        acc += v;
      } else {
        acc += v * (double)(k == 2 ? c + clo : r + rlo);
      }
    }
    acc = warp_sum(acc);
    if (lane == 0) s.patch[k] = acc;
    if (touch) s.touch = 1;
  }
  __syncthreads();
  const int size = (int)s.patch[0];
  if (s.touch || size < a.min_size || size > a.max_size) {
    not_found();
    return;
  }
  const double sv = s.patch[1];
  const double cx = s.patch[2] / sv, cy = s.patch[3] / sv;

  // ---- Moffat fit ---------------------------------------------------------
  // (a patch with values of either sign, from a threshold below zero, can have
  // its centroid anywhere: the window may then be empty)
  const int far = 1 << 30, w = a.w;
  const int rc = max(min((int)floor(cy + 0.5), far), -far), cc = max(min((int)floor(cx + 0.5), far), -far);
  const int wr0 = max(rc - w, 0), wr1 = min(rc + w, n - 1), wc0 = max(cc - w, 0), wc1 = min(cc + w, n - 1);
  const int WH = max(wr1 - wr0 + 1, 0), WW = max(wc1 - wc0 + 1, 0);
  // the box reads are done: the buffer now takes the window
  for (int i = tid; i < WH * WW; i += THREADS) {
    const int r = i / WW, c = i - r * WW;
    buf[i] = fr[(long long)(r + wr0) * n + (c + wc0)];
  }
  __syncthreads();
  if (wid > 0) {   // evaluate what warp 0 asks for
    for (;;) {
      fit_sync<WARPS>();
      const int mode = s.mode;
      if (mode == EVAL_DONE) return;
      window_pass_shared<WARPS>(mode, s, zb, buf, WH, WW, wr0, wc0);
    }
  }
  float lmin = INFINITY;
  for (int i = lane; i < WH * WW; i += 32) lmin = fminf(lmin, buf[i]);
  const double bg = warp_min(lmin);
  double i0 = 0.0;
  for (int i = lane; i < WH * WW; i += 32) i0 += (double)buf[i] - bg;
  i0 = warp_sum(i0);
  double p[6] = {i0, cx, cy, fmax(1.0, sqrt((double)size / REG_PI)), 2.5, bg};
  double cost;
  // Phase A: FP32 evaluation until the FP32 cost stops improving (its
  // rounding is about 1e-7 of it; a lambda floor of 1e-6 keeps the damped
  // system well away from the FP32 noise of J^T J).  Phase B: the FP64
  // iteration of the oracle from there, which converges in a few steps to
  // the same minimum.
  const int it_a = lm_loop<WARPS, true>(p, cost, 1e-6, 1e-7, s, zb, buf, WH, WW, wr0, wc0);
  const int it_b = lm_loop<WARPS, false>(p, cost, 1e-12, 1e-14, s, zb, buf, WH, WW, wr0, wc0);
  const int it = it_a + it_b;
  if (lane == 0) {
    s.mode = EVAL_DONE;
    out[0] = 1.0;
    out[1] = p[1];
    out[2] = p[2];
    out[3] = 2.0 * p[3] * sqrt(pow(2.0, 1.0 / p[4]) - 1.0);
    out[4] = p[0];
    out[5] = p[3];
    out[6] = p[4];
    out[7] = p[5];
    if (a.iters) a.iters[f] = it;
  }
  fit_sync<WARPS>();
}

// Shared memory of a block: side^2 floats, then the labels or the model values.
__host__ __device__ inline size_t fit_buf_bytes(int side) { return ((size_t)side * side * 4 + 15) & ~(size_t)15; }
__host__ __device__ inline size_t fit_smem_bytes(int side) {
  const size_t lab = ((size_t)side * side + 15) & ~(size_t)15, z = (size_t)FIT_TILE * FIT_Z * sizeof(double);
  return fit_buf_bytes(side) + (lab > z ? lab : z);
}

// Persistent blocks: each takes the next frame from the counter after the
// per-frame words (no waiting on other blocks).
template <int WARPS>
__global__ void __launch_bounds__(32 * WARPS, FIT_SM_WARPS / WARPS)
register_fit_kernel(const RegArgs a, unsigned long long *__restrict__ keys, int side) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ FitShared s;
  float *buf = reinterpret_cast<float *>(smem);
  unsigned char *zb = smem + fit_buf_bytes(side);
  unsigned long long *counter = keys + a.T;
  for (;;) {
    __syncthreads();   // the frame before is done with the shared memory
    if (threadIdx.x == 0) s.frame = (long long)atomicAdd(counter, 1ull);
    __syncthreads();
    const long long f = s.frame;
    if (f >= a.T) break;
    fit_frame<WARPS>(a, keys[f], f, buf, zb, zb, s);
  }
}

template <int WARPS>
cudaError_t launch_fit(const RegArgs &a, unsigned long long *keys, int sms, cudaStream_t st) {
  const int side = 2 * (a.R > a.w ? a.R : a.w) + 1;
  const size_t smem = fit_smem_bytes(side);
  auto kernel = register_fit_kernel<WARPS>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 32 * WARPS, smem)) != cudaSuccess) return e;
  long long grid = (long long)(per_sm > 0 ? per_sm : 1) * sms;
  if (grid > a.T) grid = a.T;
  kernel<<<(unsigned)grid, 32 * WARPS, smem, st>>>(a, keys, side);
  return cudaGetLastError();
}

}  // namespace

size_t register_keys_bytes(long long T) { return (size_t)(T + 1) * sizeof(unsigned long long); }

cudaError_t launch_register_argmax(const RegArgs &a, unsigned long long *keys, cudaStream_t st) {
  if (a.T <= 0) return cudaSuccess;
  const long long nn = (long long)a.n * a.n;
  cudaError_t e = cudaMemsetAsync(keys, 0, register_keys_bytes(a.T), st);
  if (e != cudaSuccess) return e;
  const long long chunks = (nn + REG_CHUNK - 1) / REG_CHUNK;
  const long long items = a.T * chunks;
  const unsigned grid = (unsigned)(items < 152LL * 64 ? items : 152LL * 64);
  frame_argmax_kernel<<<grid, ARG_THREADS, 0, st>>>(a.in, a.T, nn, chunks, keys, a.status);
  return cudaGetLastError();
}

cudaError_t launch_register_fit(const RegArgs &a, unsigned long long *keys, cudaStream_t st) {
  if (a.T <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  // Four warps a frame while about all frames are resident at once, and for
  // windows of more than one tile; else, where the solves on one warp are much
  // of the work, two, so that twice as many frames are solved at a time.  The
  // fewer the pixels, the sooner.  Calls on 100 x 100 frames (a tenth lost), two
  // and four warps, and one warp without shared sums: w = 4, 480 frames 1112,
  // 1026, 1430 us, 560 1162, 1434, 1436, 1000 1405, 1849, 1767, 4000 4768, 6255,
  // 4988; w = 8, 560 819, 778, 1175, 720 923, 975, 1222, 4000 3033, 3387, 3247; w
  // = 10, 608 949, 966, 1310, 912 1196, 1165, 1473, 1800 1838, 1937, 2139; w = 14,
  // 720 1708, 1618, 2238, 1800 3065, 2979, 3424.
  const long long pixels = (2ll * a.w + 1) * (2 * a.w + 1);
  const long long four = pixels <= 128 ? 7ll * sms / 2 : pixels <= 300 ? 4ll * sms : 10ll * sms;
  if (a.T <= four || pixels > FIT_TILE) return launch_fit<4>(a, keys, sms, st);
  return launch_fit<2>(a, keys, sms, st);
}

}  // namespace graphic
