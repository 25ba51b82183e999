// Prediction T = F W^T: the "small inner product" of Sec. 2,
// T_wall(n) ~= sum_i alpha_i p_i(n), for many feature rows and device models.
//
// FP64-accurate path: exact fixed-point arithmetic, for up to 32 columns on the tensor cores
// (predict_exact.cu, topk_exact.cu), here on the integer pipes: for 33 to 40 columns, and the
// top-k for few models (1e6 x 32 x 64 predictions: 2.08 ms here, 0.32 there).  Each
// model's weights become integers W = round(w * 2^E_m) with sum_i |W_i| <= 2^62 (so
// any int64 counts keep the sum below 2^126); every product F_ri W_mi is formed
// exactly and summed in 128 bits, then converted once.  Error <= 2^-(E_m+1)
// sum_i |F_ri| + 2^-56 |T|, i.e. at most 2^-62 (sum_i |w_i| / min_i |w_i|) + 2^-56 of
// sum_i |F_ri w_mi|: 4e-11 for weights spread like the paper's Table 2.
// (64-bit integer <-> float conversions, which would be needed per term by a float-float
// scheme, run on the FP64 pipe of this GPU.)
// The same products feed a per-model argmin over rows and a top-k per (group, model)
// (configuration selection, Sec. 6.1) without writing T.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "eval_common.cuh"
#include "kernels.h"
#include "pm.h"
#include "pm_internal.h"
#include "topk_list.cuh"
#include "trace.h"

namespace pmd {

constexpr int PR_ROWS = 32;     // rows per tile
constexpr int PR_WARPS = 8;     // each warp: 4 rows of the tile
constexpr int PR_MAXK = 40;
constexpr int PR_MAXM = 64;

struct PredictSmem {
  int64_t f[PR_ROWS][PR_MAXK + 1];
  int64_t w[PR_MAXK][PR_MAXM];
  int E[PR_MAXM];
};

__device__ void load_weights(PredictSmem &S, const double *W, int M, int k) {
  for (int m = threadIdx.x; m < PR_MAXM; m += blockDim.x) {
    const int E = m < M ? weight_exponent(W + (int64_t)m * k, k) : 0;
    for (int i = 0; i < PR_MAXK; i++) S.w[i][m] = (m < M && i < k) ? llrint(ldexp(W[(int64_t)m * k + i], E)) : 0;
    S.E[m] = E;
  }
}

__device__ void load_rows(PredictSmem &S, const int64_t *F, int64_t r0, int64_t R, int k) {
  for (int i = threadIdx.x; i < PR_ROWS * k; i += blockDim.x) {
    int r = i / k, c = i - r * k;
    S.f[r][c] = (r0 + r < R) ? F[(r0 + r) * k + c] : 0;
  }
}

// A += v W (mod 2^128), v and W signed 64-bit, A four 32-bit limbs: the unsigned
// product from three carry chains of 32-bit multiply-adds (limb products v0 W0, v0 W1,
// v1 W0, v1 W1), then the corrections of the signed operands (v = v_u - 2^64 when
// negative, likewise W), which subtract the other operand from the upper 64 bits.
__device__ __forceinline__ void acc_mad(uint32_t (&A)[4], int64_t v, int64_t W) {
  const uint32_t v0 = (uint32_t)v, v1 = (uint32_t)((uint64_t)v >> 32);
  const uint32_t w0 = (uint32_t)W, w1 = (uint32_t)((uint64_t)W >> 32);
  asm("mad.lo.cc.u32  %0, %4, %6, %0;\n\t"
      "madc.lo.cc.u32 %1, %4, %7, %1;\n\t"
      "madc.lo.cc.u32 %2, %5, %7, %2;\n\t"
      "madc.hi.u32    %3, %5, %7, %3;\n\t"
      "mad.hi.cc.u32  %1, %4, %6, %1;\n\t"
      "madc.hi.cc.u32 %2, %4, %7, %2;\n\t"
      "addc.u32       %3, %3, 0;\n\t"
      "mad.lo.cc.u32  %1, %5, %6, %1;\n\t"
      "madc.hi.cc.u32 %2, %5, %6, %2;\n\t"
      "addc.u32       %3, %3, 0;\n\t"
      : "+r"(A[0]), "+r"(A[1]), "+r"(A[2]), "+r"(A[3])
      : "r"(v0), "r"(v1), "r"(w0), "r"(w1));
  if (v < 0) asm("sub.cc.u32 %0, %0, %2;\n\tsubc.u32 %1, %1, %3;\n\t" : "+r"(A[2]), "+r"(A[3]) : "r"(w0), "r"(w1));
  if (W < 0) asm("sub.cc.u32 %0, %0, %2;\n\tsubc.u32 %1, %1, %3;\n\t" : "+r"(A[2]), "+r"(A[3]) : "r"(v0), "r"(v1));
}

// The same for 0 <= v < 2^32: four multiply-adds.
__device__ __forceinline__ void acc_mad_u32(uint32_t (&A)[4], uint32_t v, int64_t W) {
  const uint32_t w0 = (uint32_t)W, w1 = (uint32_t)((uint64_t)W >> 32);
  asm("mad.lo.cc.u32  %0, %4, %5, %0;\n\t"
      "madc.lo.cc.u32 %1, %4, %6, %1;\n\t"
      "madc.hi.cc.u32 %2, %4, %6, %2;\n\t"
      "addc.u32       %3, %3, 0;\n\t"
      "mad.hi.cc.u32  %1, %4, %5, %1;\n\t"
      "addc.cc.u32    %2, %2, 0;\n\t"
      "addc.u32       %3, %3, 0;\n\t"
      : "+r"(A[0]), "+r"(A[1]), "+r"(A[2]), "+r"(A[3])
      : "r"(v), "r"(w0), "r"(w1));
  if (W < 0) asm("sub.cc.u32 %0, %0, %2;\n\tsubc.u32 %1, %1, 0;\n\t" : "+r"(A[2]), "+r"(A[3]) : "r"(v));
}

// One feature of a warp's 32 rows, with every model's weight.  Most features are zero in all
// rows of a batch (a kernel has a few properties), many are below 2^32: what the whole warp
// can leave out, it does.
template <int MN>
__device__ __forceinline__ void acc_feature(uint32_t (&a)[MN][4], int64_t v, const int64_t *w) {
  if (__any_sync(0xffffffffu, v != 0)) {
    if (__any_sync(0xffffffffu, (uint64_t)v >> 32 != 0)) {
#pragma unroll
      for (int m = 0; m < MN; m++) acc_mad(a[m], v, w[m]);
    } else {
#pragma unroll
      for (int m = 0; m < MN; m++) acc_mad_u32(a[m], (uint32_t)v, w[m]);
    }
  }
}

// Each thread: rows warp + 8 q (q < 4), models lane + 32 j (j < 2).
__device__ __forceinline__ void tile_fixed(const PredictSmem &S, int k, Acc128 acc[4][2]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t a[4][2][4];
#pragma unroll
  for (int q = 0; q < 4; q++)
#pragma unroll
    for (int j = 0; j < 2; j++)
#pragma unroll
      for (int l = 0; l < 4; l++) a[q][j][l] = 0;
  for (int i = 0; i < k; i++) {
    const int64_t w0 = S.w[i][lane], w1 = S.w[i][lane + 32];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int64_t v = S.f[warp + 8 * q][i];
      acc_mad(a[q][0], v, w0);
      acc_mad(a[q][1], v, w1);
    }
  }
#pragma unroll
  for (int q = 0; q < 4; q++)
#pragma unroll
    for (int j = 0; j < 2; j++) {
      acc[q][j].lo = (uint64_t)a[q][j][0] | ((uint64_t)a[q][j][1] << 32);
      acc[q][j].hi = (uint64_t)a[q][j][2] | ((uint64_t)a[q][j][3] << 32);
    }
}

__global__ void __launch_bounds__(PR_WARPS * 32) k_predict_ff(const int64_t *__restrict__ F, int64_t R, int k,
                                                              const double *__restrict__ W, int M,
                                                              double *__restrict__ T) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  PredictSmem &S = *(PredictSmem *)smem_raw;
  load_weights(S, W, M, k);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t ntiles = (R + PR_ROWS - 1) / PR_ROWS;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t r0 = tile * PR_ROWS;
    __syncthreads();
    load_rows(S, F, r0, R, k);
    __syncthreads();
    Acc128 acc[4][2];
    tile_fixed(S, k, acc);
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int64_t r = r0 + warp + 8 * q;
      if (r >= R) continue;
#pragma unroll
      for (int j = 0; j < 2; j++) {
        const int m = lane + 32 * j;
        if (m < M) T[r * M + m] = key_value(acc_key(acc[q][j]), S.E[m]);
      }
    }
  }
}

// Plain double FMA (cross-check path).
__global__ void k_predict_f64(const int64_t *__restrict__ F, int64_t R, int k, const double *__restrict__ W, int M,
                              double *__restrict__ T) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= R * M) return;
  const int64_t r = i / M;
  const int m = (int)(i - r * M);
  double acc = 0;
  for (int c = 0; c < k; c++) acc = fma((double)F[r * k + c], W[(int64_t)m * k + c], acc);
  T[i] = acc;
}

static int g_num_sms = 0;
static int num_sms() {
  if (!g_num_sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (g_num_sms <= 0) g_num_sms = 148;
  }
  return g_num_sms;
}

cudaError_t launch_predict(const int64_t *F, int64_t R, int k, const double *W, int M, int precision, double *T,
                           int *status, cudaStream_t st) {
  if (R == 0) return cudaSuccess;
  if (precision == PM_PREC_NATIVE_FP64) {
    int64_t n = R * M;
    k_predict_f64<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(F, R, k, W, M, T);
    return cudaGetLastError();
  }
  if (k > PR_MAXK || M > PR_MAXM) return cudaErrorInvalidValue;
  if (exact_tc_ok(k, M)) return launch_predict_exact(F, R, k, W, M, T, status, num_sms(), st);
  size_t sm = sizeof(PredictSmem);
  cudaFuncSetAttribute(k_predict_ff, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  int64_t ntiles = (R + PR_ROWS - 1) / PR_ROWS;
  int grid = (int)std::min<int64_t>(ntiles, (int64_t)num_sms() * 8);
  k_predict_ff<<<grid, PR_WARPS * 32, sm, st>>>(F, R, k, W, M, T);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- argmin over rows per model

__global__ void __launch_bounds__(PR_WARPS * 32) k_predict_argmin_part(const int64_t *__restrict__ F, int64_t R,
                                                                       int k, const double *__restrict__ W, int M,
                                                                       ArgPart *__restrict__ part) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  PredictSmem &S = *(PredictSmem *)smem_raw;
  __shared__ ArgPart red[PR_WARPS][PR_MAXM];
  load_weights(S, W, M, k);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double bt[2] = {__longlong_as_double(0x7ff0000000000000ll), __longlong_as_double(0x7ff0000000000000ll)};
  int64_t br[2] = {INT64_MAX, INT64_MAX};
  const int64_t ntiles = (R + PR_ROWS - 1) / PR_ROWS;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t r0 = tile * PR_ROWS;
    __syncthreads();
    load_rows(S, F, r0, R, k);
    __syncthreads();
    Acc128 acc[4][2];
    tile_fixed(S, k, acc);
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int64_t r = r0 + warp + 8 * q;
      if (r >= R) continue;
#pragma unroll
      for (int j = 0; j < 2; j++) {
        const int m = lane + 32 * j;
        const double tv = key_value(acc_key(acc[q][j]), S.E[m]);
        if (arg_less(tv, r, bt[j], br[j])) { bt[j] = tv; br[j] = r; }
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 2; j++) red[warp][lane + 32 * j] = ArgPart{bt[j], br[j]};
  __syncthreads();
  for (int m = threadIdx.x; m < M; m += blockDim.x) {
    ArgPart b = red[0][m];
    for (int w = 1; w < PR_WARPS; w++)
      if (arg_less(red[w][m].t, red[w][m].r, b.t, b.r)) b = red[w][m];
    part[(int64_t)blockIdx.x * M + m] = b;
  }
}

// One CTA per model: strided scan of the partials, then a warp and a CTA reduction.
__global__ void __launch_bounds__(128) k_argmin_reduce(const ArgPart *__restrict__ part, int n_part, int M,
                                                       int64_t *arg, double *mn) {
  __shared__ double s_t[4];
  __shared__ int64_t s_r[4];
  const int m = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double bt = __longlong_as_double(0x7ff0000000000000ll);
  int64_t br = INT64_MAX;
  for (int p = threadIdx.x; p < n_part; p += blockDim.x) {
    const ArgPart x = part[(int64_t)p * M + m];
    if (arg_less(x.t, x.r, bt, br)) { bt = x.t; br = x.r; }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const double ot = __shfl_xor_sync(0xffffffffu, bt, o);
    const int64_t orr = __shfl_xor_sync(0xffffffffu, br, o);
    if (arg_less(ot, orr, bt, br)) { bt = ot; br = orr; }
  }
  if (lane == 0) { s_t[warp] = bt; s_r[warp] = br; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 4; w++)
      if (arg_less(s_t[w], s_r[w], bt, br)) { bt = s_t[w]; br = s_r[w]; }
    arg[m] = br == INT64_MAX ? -1 : br;
    mn[m] = bt;
  }
}

cudaError_t launch_argmin_reduce(const ArgPart *part, int n_part, int M, int64_t *arg, double *mn, cudaStream_t st) {
  k_argmin_reduce<<<M, 128, 0, st>>>(part, n_part, M, arg, mn);
  return cudaGetLastError();
}

int argmin_parts() { return num_sms() * 4; }
size_t argmin_scratch_bytes(int M, int n_part) { return (size_t)M * n_part * sizeof(ArgPart); }

static cudaError_t launch_argmin_parts(const int64_t *F, int64_t R, int k, const double *W, int M, void *scratch,
                                       int np, int64_t *arg, double *mn, int *status, cudaStream_t st) {
  if (exact_tc_ok(k, M)) {
    np = std::min(np, num_sms());   // one CTA per SM
    cudaError_t e = launch_argmin_exact(F, R, k, W, M, (ArgPart *)scratch, np, status, st);
    return e != cudaSuccess ? e : launch_argmin_reduce((const ArgPart *)scratch, np, M, arg, mn, st);
  }
  size_t sm = sizeof(PredictSmem);
  cudaFuncSetAttribute(k_predict_argmin_part, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k_predict_argmin_part<<<np, PR_WARPS * 32, sm, st>>>(F, R, k, W, M, (ArgPart *)scratch);
  return launch_argmin_reduce((const ArgPart *)scratch, np, M, arg, mn, st);
}

cudaError_t launch_predict_argmin(const int64_t *F, int64_t R, int k, const double *W, int M, int precision,
                                  void *scratch, int64_t *arg, double *mn, int *status, cudaStream_t st) {
  if (k > PR_MAXK || M > PR_MAXM || precision != PM_PREC_FP64) return cudaErrorInvalidValue;
  return launch_argmin_parts(F, R, k, W, M, scratch, argmin_parts(), arg, mn, status, st);
}

// ---------------------------------------------------------------- top-k rows per (group, model)

// Configuration selection over materialised features (Sec. 6.1): for every group of
// rows and every model, the topk rows with the smallest predicted time, ordered by
// (time, row).  The times are those k_predict_ff writes, bit for bit.  A warp keeps one
// sorted list per model it owns, entry i in lane i; a tile's 32 candidates are tested
// against the list's last entry and only the passing ones are inserted, smallest first.

constexpr int TK_MODELS_PER_WARP = PR_MAXM / PR_WARPS;   // 8

// the tile's times, [row][model] with one pad column, so that a warp reading one
// model's 32 rows hits 32 different banks
constexpr int TK_TSTRIDE = PR_MAXM + 1;
size_t predict_topk_smem() { return sizeof(PredictSmem) + sizeof(double) * PR_ROWS * TK_TSTRIDE + sizeof(int64_t) * PR_ROWS; }

__global__ void __launch_bounds__(PR_WARPS * 32) k_predict_topk(const int64_t *__restrict__ F, int64_t R, int k,
                                                                const double *__restrict__ W, int M,
                                                                const int64_t *__restrict__ rows,
                                                                const TopkUnit *__restrict__ units, int n_units,
                                                                int topk, double *__restrict__ part_t,
                                                                int64_t *__restrict__ part_r,
                                                                int64_t *__restrict__ top_idx,
                                                                double *__restrict__ top_t, int *status) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  PredictSmem &S = *(PredictSmem *)smem_raw;
  double(*tT)[TK_TSTRIDE] = (double(*)[TK_TSTRIDE])(smem_raw + sizeof(PredictSmem));
  int64_t *tR = (int64_t *)(smem_raw + sizeof(PredictSmem) + sizeof(double) * PR_ROWS * TK_TSTRIDE);
  load_weights(S, W, M, k);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int u = blockIdx.x; u < n_units; u += gridDim.x) {
    const TopkUnit U = units[u];
    double lt[TK_MODELS_PER_WARP];
    int64_t lr[TK_MODELS_PER_WARP];
#pragma unroll
    for (int j = 0; j < TK_MODELS_PER_WARP; j++) { lt[j] = TK_INF; lr[j] = INT64_MAX; }
    for (int64_t t0 = U.p0; t0 < U.p1; t0 += PR_ROWS) {
      __syncthreads();
      // rows of this tile: positions t0 .. t0+31 of the unit, through the row list if any
      for (int i = threadIdx.x; i < PR_ROWS * k; i += blockDim.x) {
        const int r = i / k, c = i - r * k;
        const int64_t pos = t0 + r;
        int64_t row = -1;
        if (pos < U.p1) {
          row = rows ? rows[pos] : pos;
          if (row < 0 || row >= R) {
            if (c == 0) atomicOr(status, ST_BAD_ROW);
            row = -1;
          }
        }
        S.f[r][c] = row >= 0 ? F[row * k + c] : 0;
        if (c == 0) tR[r] = row;
      }
      __syncthreads();
      Acc128 acc[4][2];
      tile_fixed(S, k, acc);
#pragma unroll
      for (int q = 0; q < 4; q++)
#pragma unroll
        for (int j = 0; j < 2; j++) {
          const int m = lane + 32 * j;
          tT[warp + 8 * q][m] = m < M ? key_value(acc_key(acc[q][j]), S.E[m]) : 0.0;
        }
      __syncthreads();
      const int64_t row = tR[lane];
#pragma unroll
      for (int j = 0; j < TK_MODELS_PER_WARP; j++) {
        const int m = warp + PR_WARPS * j;
        if (m < M) warp_list_merge(lt[j], lr[j], tT[lane][m], row, row >= 0, topk, lane);
      }
    }
#pragma unroll
    for (int j = 0; j < TK_MODELS_PER_WARP; j++) {
      const int m = warp + PR_WARPS * j;
      if (m >= M || lane >= topk) continue;
      if (U.part < 0) {
        const int64_t o = ((int64_t)U.g * M + m) * topk + lane;
        top_idx[o] = lr[j] == INT64_MAX ? -1 : lr[j];
        top_t[o] = lt[j];
      } else {
        const int64_t o = ((int64_t)U.part * M + m) * topk + lane;
        part_t[o] = lt[j];
        part_r[o] = lr[j];
      }
    }
  }
}

// The same top-k for few models (M <= 8): the 64-model tile above would leave most of
// its products and warps idle, so here each lane owns one row (a warp takes 32
// consecutive positions of the unit, the CTA 128) and computes its M exact sums; each
// warp keeps its own sorted lists per model, and at the end of the unit warp m merges
// the four warps' lists of model m.  Same products, same keys, same (time, row) order.
//
// STAGED (k even, 24 to 32, F 16-byte aligned): a warp copies its 32 rows to shared memory
// with 16-byte asynchronous copies, whole rows at a time, and each lane then reads its own
// row; the chunk index is XORed with the row's low bits, which keeps the 16-byte reads of
// eight lanes on distinct banks.  Lanes reading their rows straight from global memory touch
// 32 lines per instruction, and the kernel waited for L1 (1.02 ms for 4.5 M rows x 32, one
// model; with the copies the multiply-adds and the reads from HBM bound it).
constexpr int TR_WARPS = 4;
// the time of an exact sum, once in the code
static __device__ __noinline__ double time_of(Acc128 A, int E) { return key_value(acc_key(A), E); }

template <int MN, bool STAGED>
__global__ void __launch_bounds__(TR_WARPS * 32) k_predict_topk_rows(const int64_t *__restrict__ F, int64_t R, int k,
                                                                     const double *__restrict__ W, int M,
                                                                     const int64_t *__restrict__ rows,
                                                                     const TopkUnit *__restrict__ units, int n_units,
                                                                     int topk, double *__restrict__ part_t,
                                                                     int64_t *__restrict__ part_r,
                                                                     int64_t *__restrict__ top_idx,
                                                                     double *__restrict__ top_t, int *status) {
  __shared__ int64_t sw[PR_MAXK][MN];
  __shared__ int sE[MN];
  // the warps' lists, then the staged rows [warp][row][chunk ^ (row & 15)].  One buffer per
  // warp: with two, half the warps fit, and 12 warps per SM are slower (four models, 4,096
  // groups of 244 rows: 782 us).
  constexpr int LISTS = TR_WARPS * MN * 32;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  longlong2 *stage = (longlong2 *)smem_raw + LISTS;
  double(*st)[MN][32] = (double(*)[MN][32])smem_raw;
  int64_t(*sr)[MN][32] = (int64_t(*)[MN][32])((double *)smem_raw + LISTS);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < MN * k; i += TR_WARPS * 32) {
    const int m = i / k;
    sw[i - m * k][m] = m < M ? __double_as_longlong(W[i]) : 0;
  }
  __syncthreads();
  if (threadIdx.x < MN) {   // the serial loop of weight_exponent over the staged weights
    double w[PR_MAXK];
    for (int c = 0; c < k; c++) w[c] = __longlong_as_double(sw[c][threadIdx.x]);
    sE[threadIdx.x] = (int)threadIdx.x < M ? weight_exponent(w, k) : 0;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < MN * k; i += TR_WARPS * 32) {
    const int m = i / k, c = i - m * k;
    if (m < M) sw[c][m] = fixed_weight(__longlong_as_double(sw[c][m]), sE[m]);
  }
  __syncthreads();
  const int cpr = k / 2, inv = (65536 + cpr - 1) / max(cpr, 1);   // 16-byte chunks per row; x / cpr = x inv / 2^16 for x < 512
  for (int u = blockIdx.x; u < n_units; u += gridDim.x) {
    const TopkUnit U = units[u];
    // this warp's lists, one model's entry i in lane i
#pragma unroll
    for (int m = 0; m < MN; m++) { st[warp][m][lane] = TK_INF; sr[warp][m][lane] = INT64_MAX; }
    __syncwarp();
    for (int64_t t0 = U.p0 + 32 * warp; t0 < U.p1; t0 += 32 * TR_WARPS) {   // warp-uniform
      const int64_t pos = t0 + lane;
      int64_t row = -1;
      if (pos < U.p1) {
        row = rows ? rows[pos] : pos;
        if (row < 0 || row >= R) {
          atomicOr(status, ST_BAD_ROW);
          row = -1;
        }
      }
      uint32_t a[MN][4];
#pragma unroll
      for (int m = 0; m < MN; m++) a[m][0] = a[m][1] = a[m][2] = a[m][3] = 0;
      if (STAGED) {
        longlong2 *S = stage + warp * (32 * 16);
        __syncwarp();   // the batch before has been read
        for (int j = 0; j < cpr; j++) {
          const int x = lane + 32 * j, r = (x * inv) >> 16, c = x - r * cpr;
          const int64_t src = __shfl_sync(0xffffffffu, row, r);
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(
                           (unsigned)__cvta_generic_to_shared(S + r * 16 + (c ^ (r & 15)))),
                       "l"(F + (src >= 0 ? src : 0) * k + 2 * c), "r"(src >= 0 ? 16 : 0));
        }
        asm volatile("cp.async.wait_all;\n" ::);
        __syncwarp();
        for (int c = 0; c < cpr; c++) {
          const longlong2 v = S[lane * 16 + (c ^ (lane & 15))];
          acc_feature(a, v.x, sw[2 * c]);
          acc_feature(a, v.y, sw[2 * c + 1]);
        }
      } else {
        const int64_t *f = F + (row >= 0 ? row : 0) * k;
#pragma unroll 4
        for (int i = 0; i < k; i++) acc_feature(a, row >= 0 ? __ldg(f + i) : 0, sw[i]);
      }
      // one merge in the code for all models: unrolled, it outgrows the instruction cache (four
      // models: 8.5 of 15 stall cycles per instruction)
      double t[MN];
#pragma unroll
      for (int m = 0; m < MN; m++) {
        Acc128 A;
        A.lo = (uint64_t)a[m][0] | ((uint64_t)a[m][1] << 32);
        A.hi = (uint64_t)a[m][2] | ((uint64_t)a[m][3] << 32);
        t[m] = time_of(A, sE[m]);
      }
#pragma unroll 1
      for (int m = 0; m < M && m < MN; m++) {
        double x = t[0];
#pragma unroll
        for (int q = 1; q < MN; q++) x = m == q ? t[q] : x;
        double lt = st[warp][m][lane];
        int64_t lr = sr[warp][m][lane];
        warp_list_merge(lt, lr, x, row, row >= 0, topk, lane);
        st[warp][m][lane] = lt;
        sr[warp][m][lane] = lr;
      }
    }
    __syncthreads();
    for (int m = warp; m < M && m < MN; m += TR_WARPS) {
      double ft = TK_INF;
      int64_t fr = INT64_MAX;
      for (int w = 0; w < TR_WARPS; w++) {
        const double t = st[w][m][lane];
        const int64_t r = sr[w][m][lane];
        warp_list_merge(ft, fr, t, r, lane < topk && r != INT64_MAX, topk, lane);
      }
      if (lane < topk) {
        if (U.part < 0) {
          const int64_t o = ((int64_t)U.g * M + m) * topk + lane;
          top_idx[o] = fr == INT64_MAX ? -1 : fr;
          top_t[o] = ft;
        } else {
          const int64_t o = ((int64_t)U.part * M + m) * topk + lane;
          part_t[o] = ft;
          part_r[o] = fr;
        }
      }
    }
    __syncthreads();   // the lists have been read
  }
}

template <int MN, bool STAGED>
static void launch_topk_rows(const int64_t *F, int64_t R, int k, const double *W, int M, const int64_t *rows,
                             const TopkUnit *units, int n_units, int topk, double *part_t, int64_t *part_r,
                             int64_t *top_idx, double *top_t, int *status, cudaStream_t st) {
  const size_t sm = sizeof(longlong2) * (TR_WARPS * MN * 32 + (STAGED ? TR_WARPS * 32 * 16 : 0));
  int per_sm = 1;
  cudaFuncSetAttribute(k_predict_topk_rows<MN, STAGED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_predict_topk_rows<MN, STAGED>, TR_WARPS * 32, sm);
  const int grid = std::min(n_units, num_sms() * std::max(1, per_sm));
  k_predict_topk_rows<MN, STAGED><<<grid, TR_WARPS * 32, sm, st>>>(F, R, k, W, M, rows, units, n_units, topk, part_t, part_r,
                                                                  top_idx, top_t, status);
}

// Which kernel, and how large a unit may be.
//
// Up to eight models, 1e6 x 32, us, row-per-lane | tensor cores: one group 303 | 360 for 4 models,
// 440 | 388 for 5, 471 | 358 for 6, 501 | 402 for 7, 531 | 363 for 8; 10 groups 407 | 648, 439 | 587,
// 469 | 653, 497 | 574 for 5 to 8; 400 groups 535 | 791, 575 | 721, 614 | 804, 650 | 709; between them
// eight models are as fast on either (200 groups 615 | 573).  100,000 rows in one group 81 | 108,
// 86 | 108, 90 | 117, 96 | 112.  The end of a group costs the tensor-core kernel as much as many
// of its tiles: from 2^17 rows a group on it takes five to eight models.  Rows of 16 counts and
// fewer have at most half the products to do: 8 models x 12 in 10 groups 408 | 547.
//
// More than eight models take the tensor cores unless there are many short groups: each group
// fills M empty lists there, some 15 merges a model, where the integer tile's lists are its warps'
// own, but the integer tile pays for every product.  So the line is in a group's rows times what
// a row costs, k + M / 4, against the lists, 600 + 50 M.  100,000 rows, us, integer | tensor
// cores: 9 models x 12 columns 270 | 343 (64 rows a group), 268 | 245 (100); 64 models x 12
// 558 | 642 (100), 566 | 423 (256); 64 x 32 800 | 879 (64), 782 | 632 (100); 33 x 32 629 | 886
// (32), 650 | 577 (64).  One CTA per SM takes a group, so what counts is how many each SM takes in
// turn: one alone is faster on the tensor cores whatever its length (10 groups of 100 rows, 64 x
// 12: 140 | 110), and so are two (64 x 12, 50 rows: 201 | 198); with three the line lies at two
// thirds (37 x 12: 267 | 259 at 100 rows, 158 | 212 at 50), from four on where it is above.  Short
// rankings fill their lists sooner (64 x 32, 64 rows: the fastest row 435 | 376), and wide rows
// cost the integer tile more than their width (9 x 32, 30 rows: 207 | 173).
TopkPath topk_path(int k, int M, int topk, int64_t total, int64_t G) {
  if (M <= 4) return TopkPath::ROWS;
  if (M <= 8)
    return k <= 16 || !exact_tc_ok(k, M) || total < (int64_t(1) << 17) * G ? TopkPath::ROWS : TopkPath::TENSOR;
  if (!exact_tc_ok(k, M)) return TopkPath::INTEGER;
  const double turns = std::min(1.0, std::max(0.0, ((double)G / num_sms() - 1) / 3));
  const double row = (k + 0.25 * M) * std::max(1.0, k / 24.0), lists = (600 + 50.0 * M) * (0.75 + 0.25 * (topk - 1) / (TOPK_MAX - 1));
  return (double)total * row >= turns * G * lists ? TopkPath::TENSOR : TopkPath::INTEGER;
}
// The row-per-lane kernel's units fill its resident CTAs once (six per SM, four with eight
// models' lists): of 977 units of 1,024 positions on 912 CTAs the last 65 took as
// long as the rest (1e6 rows, 4 models).  At most 2,048 positions, so that larger problems
// balance over many units while the variants of one template and point stay one unit.  The
// tensor-core kernel keeps one list per CTA and unit: one unit per SM.
int64_t topk_chunk(int k, int M, int topk, int64_t total, int64_t G) {
  auto split = [&](int64_t ctas, int64_t grain, int64_t lo, int64_t hi) {
    const int64_t each = ((total + ctas - 1) / ctas + grain - 1) / grain * grain;
    return std::min(hi, std::max(lo, each));
  };
  const TopkPath path = topk_path(k, M, topk, total, G);
  if (path == TopkPath::ROWS) return split((int64_t)num_sms() * (M <= 2 ? 6 : M <= 4 ? 5 : 4), 32, 32 * TR_WARPS, 2048);
  if (path == TopkPath::INTEGER) return TOPK_CHUNK;
  return split(num_sms(), 128, TOPK_CHUNK, int64_t(1) << 20);
}

// Groups split over several units: one CTA per (group, model) merges the units' sorted lists
// of that model in rounds: the first entries of all lists, then the next ones, until no entry
// of a round is below the warps' shared bound (the lists are sorted, so later ones are not
// either).  Then warp 0 merges the eight warp lists.  A round is one entry of many lists or
// several of few, about four candidates a thread.  With every entry of 782 lists merged, one
// group of 100,000 rows x 32 took 79 us (one model, 16 entries), 46 now.
__global__ void __launch_bounds__(PR_WARPS * 32) k_topk_merge(const TopkMerge *__restrict__ merges, int M, int topk,
                                                              const double *__restrict__ part_t,
                                                              const int64_t *__restrict__ part_r,
                                                              int64_t *__restrict__ top_idx,
                                                              double *__restrict__ top_t) {
  __shared__ double st[PR_WARPS][32];
  __shared__ int64_t sr[PR_WARPS][32];
  const TopkMerge G = merges[blockIdx.x];
  const int m = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double lt = TK_INF;
  int64_t lr = INT64_MAX;
  __shared__ long long s_thr;   // no time above it is among the topk: the least of the warps' last entries
  const bool few = (int64_t)G.n_parts * topk <= 32 * PR_WARPS;   // one candidate a thread: no rounds
  if (few) {
    const int p = (int)threadIdx.x / topk, q = (int)threadIdx.x - p * topk;
    double t = TK_INF;
    int64_t r = INT64_MAX;
    if (p < G.n_parts) {
      const int64_t o = (((int64_t)G.part0 + p) * M + m) * topk + q;
      t = part_t[o];
      r = part_r[o];
    }
    warp_list_merge(lt, lr, t, r, r != INT64_MAX, topk, lane);
  } else {
    if (threadIdx.x == 0) s_thr = INT64_MAX;
    __syncthreads();
  }
  int sh = 0;   // 2^sh entries of a list per round
  while ((1 << sh) < topk && ((int64_t)G.n_parts << (sh + 1)) <= 4 * 32 * PR_WARPS) sh++;
  const int64_t n = (int64_t)G.n_parts << sh;
  for (int j = 0; j < topk && !few; j += 1 << sh) {
    bool some = false;
    for (int64_t c0 = 32 * warp; c0 < n; c0 += 4 * 32 * PR_WARPS) {   // warp-uniform
      double t[4];
      int64_t r[4];
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const int64_t c = c0 + u * 32 * PR_WARPS + lane, q = j + (c & ((1 << sh) - 1));
        t[u] = TK_INF;
        r[u] = INT64_MAX;
        if (c < n && q < topk) {
          const int64_t o = ((G.part0 + (c >> sh)) * M + m) * topk + q;
          t[u] = part_t[o];
          r[u] = part_r[o];
        }
      }
#pragma unroll 1
      for (int u = 0; u < 4; u++) {   // one copy of the merge's code
        const bool ok = r[0] != INT64_MAX && time_order(t[0]) <= *(volatile long long *)&s_thr;
        if (__any_sync(0xffffffffu, ok)) {
          some = true;
          warp_list_merge(lt, lr, t[0], r[0], ok, topk, lane);
          if (lane == topk - 1 && lr != INT64_MAX && time_order(lt) < *(volatile long long *)&s_thr)
            atomicMin(&s_thr, (long long)time_order(lt));
        }
        t[0] = t[1], t[1] = t[2], t[2] = t[3];
        r[0] = r[1], r[1] = r[2], r[2] = r[3], r[3] = INT64_MAX;
      }
    }
    if (j + (1 << sh) >= topk || !__syncthreads_or(some)) break;
  }
  st[warp][lane] = lt;
  sr[warp][lane] = lr;
  __syncthreads();
  if (warp == 0) {
    double ft = TK_INF;
    int64_t fr = INT64_MAX;
    for (int w = 0; w < PR_WARPS; w++) {
      const int64_t r = sr[w][lane];
      warp_list_merge(ft, fr, st[w][lane], r, lane < topk && r != INT64_MAX, topk, lane);
    }
    if (lane < topk) {
      const int64_t o = ((int64_t)G.g * M + m) * topk + lane;
      top_idx[o] = fr == INT64_MAX ? -1 : fr;
      top_t[o] = ft;
    }
  }
}

cudaError_t launch_predict_topk(const int64_t *F, int64_t R, int k, const double *W, int M, const int64_t *rows,
                                const TopkUnit *units, int n_units, const TopkMerge *merges, int n_merges, int topk,
                                double *part_t, int64_t *part_r, int64_t *top_idx, double *top_t, TopkPath path,
                                int *status, cudaStream_t st) {
  if (k > PR_MAXK || M > PR_MAXM || topk < 1 || topk > TOPK_MAX) return cudaErrorInvalidValue;
  if (n_units <= 0) return cudaSuccess;
  if (path == TopkPath::ROWS) {   // few models: one row per lane
    // rows of 12 counts are read well enough as they are (1e6 x 12, 4 models: staged 331 us)
    const bool staged = k % 2 == 0 && k >= 24 && k <= 32 && ((uintptr_t)F & 15) == 0;
    auto go = [&](auto mn) {
      constexpr int MN = decltype(mn)::value;
      if (staged) launch_topk_rows<MN, true>(F, R, k, W, M, rows, units, n_units, topk, part_t, part_r, top_idx, top_t, status, st);
      else launch_topk_rows<MN, false>(F, R, k, W, M, rows, units, n_units, topk, part_t, part_r, top_idx, top_t, status, st);
    };
    if (M == 1) go(std::integral_constant<int, 1>{});
    else if (M == 2) go(std::integral_constant<int, 2>{});
    else if (M <= 4) go(std::integral_constant<int, 4>{});
    else go(std::integral_constant<int, 8>{});
  } else if (path == TopkPath::TENSOR) {
    const cudaError_t x = launch_topk_exact(F, R, k, W, M, rows, units, n_units, topk, part_t, part_r, top_idx, top_t, status,
                                            num_sms(), st);
    if (x != cudaSuccess) return x;
  } else {
    const size_t sm = predict_topk_smem();
    cudaFuncSetAttribute(k_predict_topk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    const int grid = std::min(n_units, num_sms() * 2);
    k_predict_topk<<<grid, PR_WARPS * 32, sm, st>>>(F, R, k, W, M, rows, units, n_units, topk, part_t, part_r,
                                                    top_idx, top_t, status);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || n_merges == 0) return e;
  k_topk_merge<<<dim3((unsigned)n_merges, (unsigned)M), PR_WARPS * 32, 0, st>>>(merges, M, topk, part_t, part_r,
                                                                              top_idx, top_t);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- allocation-free argmin

// Partial results of pm_predict_argmin_static live in this fixed device array instead
// of memory from cudaMalloc.  Every GPU that loads the library holds it until exit.
constexpr size_t STATIC_ARGMIN_BYTES = size_t(1) << 20;
static __device__ __align__(256) unsigned char g_argmin_scratch[STATIC_ARGMIN_BYTES];

// Device address of g_argmin_scratch per device, looked up on the first call made
// with that device current (host code may not use the symbol itself as a pointer).
constexpr int STATIC_MAX_DEVICES = 64;
static std::atomic<void *> g_argmin_addr[STATIC_MAX_DEVICES];

}  // namespace pmd

extern "C" pm_status pm_predict_argmin_static(const int64_t *d_F, int64_t R, int32_t k, const double *d_W,
                                              int32_t M, int64_t *d_arg, double *d_min, void *stream) {
  PM_TRACE("pm_predict_argmin_static");
  using namespace pmd;
  if (R < 0 || k <= 0 || k > PR_MAXK || M <= 0 || M > PR_MAXM)
    return pm_set_error_c(PM_ERR_INVALID_ARG, "pm_predict_argmin_static: need R >= 0, 0 < k <= 40, 0 < M <= 64");
  if ((!d_F && R > 0) || !d_W || !d_arg || !d_min) return pm_set_error_c(PM_ERR_INVALID_ARG, "pm_predict_argmin_static: null pointer");
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= STATIC_MAX_DEVICES)
    return pm_set_error_c(PM_ERR_CUDA, "pm_predict_argmin_static: no usable current device");
  void *scratch = g_argmin_addr[dev].load();
  if (!scratch) {
    if (cudaGetSymbolAddress(&scratch, g_argmin_scratch) != cudaSuccess || !scratch)
      return pm_set_error_c(PM_ERR_CUDA, "pm_predict_argmin_static: cudaGetSymbolAddress of the scratch array failed");
    g_argmin_addr[dev].store(scratch);
  }
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
    return pm_set_error_c(PM_ERR_CUDA, "pm_predict_argmin_static: cannot read the SM count");
  // one partial result per (CTA, model); fewer CTAs if the fixed array would overflow
  const int cap = (int)(STATIC_ARGMIN_BYTES / ((size_t)M * sizeof(ArgPart)));
  const int np = std::min(4 * sms, cap);
  if (np < 1) return pm_set_error_c(PM_ERR_INVALID_ARG, "pm_predict_argmin_static: M too large for the scratch array");
  if (launch_argmin_parts(d_F, R, k, d_W, M, scratch, np, d_arg, d_min, nullptr, (cudaStream_t)stream) != cudaSuccess)
    return pm_set_error_c(PM_ERR_CUDA, "pm_predict_argmin_static: kernel launch failed");
  return PM_OK;
}
