// FP64-accurate prediction T = F W^T on the tensor cores, as times, per-model argmin or the
// residuals of the weight fit (Sec. 4.3), from
// exact digit products (exact_tc.cuh has the number scheme and the operand layouts).
//
// One CTA of 16 warps per SM, persistent over 128-row tiles.  Per tile: the counts' digits
// go to shared memory (the loads are issued before the previous tile's times are formed),
// one warp issues the MMAs of the groups of diagonals, and every thread gathers 16 exact
// sums limb by limb, turns them into times and hands them on.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "exact_tc.cuh"
#include "float_float.cuh"
#include "kernels.h"
#include "pm.h"
#include "topk_list.cuh"

namespace pmd {

// XP_TIMES: write T (fp64 [R][M]).  XP_ARGMIN: per-model minimum over the CTA's rows
// (smaller time, then smaller row) -> part[blockIdx.x][M].  The fit's residual passes, with
// measured times t and predictions p (FitResidual): XP_RESIDUAL writes the residuals for
// A^T r, relative (t - p) / t^2 or absolute t - p; XP_SUMS_REL and XP_SUMS_ABS add up the
// squares of the residual, and of t (absolute).
enum XpMode { XP_TIMES, XP_ARGMIN, XP_RESIDUAL, XP_SUMS_REL, XP_SUMS_ABS };

// what a thread carries over its rows, for its two models of a pass
template <int MODE> struct XpAcc {};
template <> struct XpAcc<XP_ARGMIN> {
  double t[2];
  int64_t r[2];
  __device__ XpAcc() { t[0] = t[1] = __longlong_as_double(0x7ff0000000000000ll); r[0] = r[1] = INT64_MAX; }
};
template <> struct XpAcc<XP_SUMS_REL> { float s[2] = {0, 0}, c[2] = {0, 0}; };
template <> struct XpAcc<XP_SUMS_ABS> { double r[2] = {0, 0}, b[2] = {0, 0}; };
// With two passes these wait in shared memory between tiles: in registers next to a pass's
// limbs they would spill.
template <class G, int MODE>
constexpr size_t xp_stash() {
  return G::PASSES > 1 && (MODE == XP_ARGMIN || MODE >= XP_SUMS_REL) ? 2 * 32 * XP_WARPS * sizeof(XpAcc<MODE>) : 0;
}

// HELD: the issuing warp leaves after its first tile and the waits are short, so that the
// working warps' waits for the second tile run out (pmx_predict_held).
template <class G, int MODE, bool HELD = false>
__global__ void __launch_bounds__(XP_THREADS, 1) k_predict_exact(const int64_t *__restrict__ F, int64_t R, int k,
                                                                 const double *__restrict__ W, int M,
                                                                 double *__restrict__ T, ArgPart *__restrict__ part,
                                                                 int *status, uint32_t m256, FitResidual res) {
  constexpr unsigned long long LIMIT = HELD ? XP_HELD_NS : MBAR_WAIT_NS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = smem_raw + ((128u - (xp_saddr(smem_raw) & 127u)) & 127u);
  __shared__ __align__(8) uint64_t full[XP_RING], empty[XP_RING], digits[2];   // sums ready / read, a tile's digits ready
  __shared__ __align__(16) int s_nd[4][XP_WARPS];   // by tile modulo 4: a slow warp may still read an older tile's
  __shared__ uint32_t tmem_base;
  __shared__ int s_E[XP_MAXM];
  __shared__ volatile int s_abort;
  uint8_t *sA = smem, *sB = smem + G::OFF_B;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform for the compiler: TMEM addresses stay in uniform registers
  const int quarter = warp & 3, slice = warp >> 2;
  const int64_t ntiles = (R + XP_ROWS - 1) / XP_ROWS;
  const bool vec = (k & 1) == 0 && ((uintptr_t)F & 15) == 0;
  const double *meas = MODE >= XP_RESIDUAL ? res.T : T;
  const bool vst = (M & 1) == 0 && ((uintptr_t)meas & 15) == 0;   // (measured) times move in pairs
  const int row = xp_row<G>();   // this thread's row of a tile when it loads counts

  if (tid == 0) {
    for (int b = 0; b < XP_RING; b++) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 2;\n" ::"r"(xp_saddr(&full[b])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(xp_saddr(&empty[b])), "n"(XP_WARPS));
    }
    for (int b = 0; b < 2; b++) asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(xp_saddr(&digits[b])), "n"(XP_WARPS));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
    s_abort = 0;
  }
  if (tid < 4 * XP_WARPS) s_nd[0][tid] = 1;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(xp_saddr(&tmem_base)),
                 "r"(G::TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  int64_t v[8];
  auto load = [&](int64_t tile) {
    const int64_t r = tile * XP_ROWS + row;
#pragma unroll
    for (int c = 0; c < 8; c++) v[c] = 0;
    if (tile < ntiles && row < XP_ROWS && r < R) xp_load_row<G>(F + r * k, k, vec, v);
  };
  load(blockIdx.x);
  xp_load_weights<G>(W, M, k, (double *)sA, sB, s_E);
  asm volatile("fence.proxy.async.shared::cta;\n" ::);
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();   // the staged weights in sA have been read
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
  const uint32_t tmem = xp_uniform(tmem_base), s0 = xp_uniform(xp_saddr(smem));
  uint32_t seq = 0;            // groups so far: columns seq % XP_RING, their (seq / XP_RING)-th use
  uint32_t it = 0;             // tiles so far
  bool ok = true;
  const bool active = warp < XP_WARPS && slice * 8 < G::NB;   // this warp has models
  XpAcc<MODE> acc;   // one pass: in registers throughout
  XpAcc<MODE> *stash = (XpAcc<MODE> *)(smem + G::SMEM - 128) + tid;   // [passes][working threads]
  constexpr bool STASH = xp_stash<G, MODE>() != 0;
  if (STASH && warp < XP_WARPS)
    for (int ps = 0; ps < 2; ps++) stash[ps * 32 * XP_WARPS] = XpAcc<MODE>();
  if (warp == XP_WARPS) {
    // this warp issues, ahead of the working warps as far as digits and columns allow
    for (int64_t tile = blockIdx.x; tile < ntiles && ok && !(HELD && it); tile += gridDim.x, it++) {
      if (!(ok = xp_wait(xp_saddr(&digits[it & 1]), (it >> 1) & 1, &s_abort, LIMIT))) break;
      const int nd = (int)xp_uniform((uint32_t)xp_tile_digits(s_nd[it & 3])), ng = xp_groups(nd);
      for (int n = 0; n < G::PASSES * ng && ok; n++, seq++) {
        const uint32_t b = seq % XP_RING;
        const int ps = n >= ng;
        if (seq >= XP_RING && !(ok = xp_wait(xp_saddr(&empty[b]), (seq / XP_RING - 1) & 1, &s_abort, LIMIT))) break;
        xp_issue<G>(s0, s0 + (it & 1) * G::A_BUF, s0 + G::OFF_B + ps * G::B_PASS, tmem + b * G::RANGE, n - ps * ng, nd,
                    xp_saddr(&full[b]));
      }
    }
    if (!ok) xp_drain(full, XP_RING, seq);   // (with `ok` unused after the loop the compiler's loop is slower: 1e6 x 32 x 64 by 1.2 us)
    __syncwarp();
  } else {
    const int c0 = slice * 8 + 2 * (lane & 3);   // this thread's models of a pass: c0, c0 + 1
    const uint32_t tread = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(slice * 8);
    // this warp's digits of the n-th tile are stored
    auto stored = [&](uint32_t n) {
      xp_store_digits<G>(v, sA + (n & 1) * G::A_BUF, s_nd[n & 3]);
      asm volatile("fence.proxy.async.shared::cta;\n" ::);
      __syncwarp();
      if (lane == 0) xp_arrive(xp_saddr(&digits[n & 1]));
    };
    auto wait = [&]() { return xp_wait(xp_saddr(&full[seq % XP_RING]), (seq / XP_RING) & 1, &s_abort, LIMIT); };
    auto done = [&]() {   // this warp has read its share of a group
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
      __syncwarp();
      if (lane == 0) xp_arrive(xp_saddr(&empty[seq % XP_RING]));
      seq++;
    };
    // the sums of one (tile, pass): four limbs, then the times
    auto pass = [&](int ps, int64_t tile, XpAcc<MODE> &acc) -> bool {
      uint32_t limb[4][8];
      uint32_t cy[8];
      if (!wait()) return false;
      const int ng = xp_groups(xp_tile_digits(s_nd[it & 3]));
      if (active) xp_limb<G, 0>(m256, tread + (seq % XP_RING) * G::RANGE, limb[0], cy);
      done();
      if (!wait()) return false;
      if (active) xp_limb<G, 1>(m256, tread + (seq % XP_RING) * G::RANGE, limb[1], cy);
      done();
      if (ng > 2) {
        if (!wait()) return false;
        if (active) xp_limb<G, 2>(m256, tread + (seq % XP_RING) * G::RANGE, limb[2], cy);
        done();
      } else {
#pragma unroll
        for (int o = 0; o < 8; o++) {
          limb[2][o] = cy[o] - XP_HI;
          cy[o] = (uint32_t)((int32_t)limb[2][o] >> 31) + XP_HI;
        }
      }
      if (ng > 3) {
        if (!wait()) return false;
        if (active) xp_limb<G, 3>(m256, tread + (seq % XP_RING) * G::RANGE, limb[3], cy);
        done();
      } else {
#pragma unroll
        for (int o = 0; o < 8; o++) limb[3][o] = cy[o] - XP_HI;
      }
      if (!active) return true;
      const int64_t r0 = tile * XP_ROWS + quarter * 32 + (lane >> 2);   // this thread's rows: r0 + 8 i, i < 4
      const int left = (int)min((int64_t)XP_ROWS, R - r0);               // row r0 + 8 i exists for 8 i < left
      const int m = 32 * ps + c0;
      double *out = MODE == XP_TIMES ? T + r0 * M + m : nullptr;
      const int x0[2] = {1150 - s_E[m], 1150 - s_E[m + 1]};
      const bool wide = min(x0[0], x0[1]) < XP_XMIN || max(x0[0], x0[1]) > XP_XMAX;   // times may leave the normal range
      // the residual passes' inputs, on their way while the times are formed
      double2 tm[4];
      float2 fh[4], fl[4];
      if constexpr (MODE >= XP_RESIDUAL) {
#pragma unroll
        for (int i = 0; i < 4; i++) {
          tm[i] = make_double2(0, 0);
          fh[i] = fl[i] = make_float2(0, 0);
          if (m < M && 8 * i < left) {
            const double *tin = res.T + (r0 + 8 * i) * M + m;
            if (vst) {
              tm[i] = __ldcs((const double2 *)tin);
            } else {
              tm[i].x = __ldcs(tin);
              if (m + 1 < M) tm[i].y = __ldcs(tin + 1);
            }
            if (MODE == XP_SUMS_REL || (MODE == XP_RESIDUAL && res.relative)) {
              fh[i] = *(const float2 *)(res.rfh + (r0 + 8 * i) * res.ld + m);
              fl[i] = *(const float2 *)(res.rfl + (r0 + 8 * i) * res.ld + m);
            }
          }
        }
      }
      auto emit = [&](auto neg) {
#pragma unroll
        for (int i = 0; i < 4; i++) {
          double t[2];
          bool bad = wide;
#pragma unroll
          for (int e = 0; e < 2; e++)
            t[e] = xp_value<decltype(neg)::value>(limb[0][2 * i + e], limb[1][2 * i + e], limb[2][2 * i + e], limb[3][2 * i + e], x0[e], bad);
          if (bad) {
#pragma unroll
            for (int e = 0; e < 2; e++)
              t[e] = xp_value_rare(limb[0][2 * i + e], limb[1][2 * i + e], limb[2][2 * i + e], limb[3][2 * i + e], 1150 - x0[e]);
          }
          if (8 * i < left) {
            if constexpr (MODE == XP_ARGMIN) {
#pragma unroll
              for (int e = 0; e < 2; e++)   // rows come in increasing order: only a smaller time improves
                if (time_order(t[e]) < time_order(acc.t[e])) { acc.t[e] = t[e]; acc.r[e] = r0 + 8 * i; }
            } else if constexpr (MODE != XP_TIMES) {
              if (m < M) {
                if constexpr (MODE == XP_SUMS_ABS) {
#pragma unroll
                  for (int e = 0; e < 2; e++) {
                    const double b = e ? tm[i].y : tm[i].x, r = b - t[e];
                    acc.r[e] = fma(r, r, acc.r[e]);
                    acc.b[e] = fma(b, b, acc.b[e]);
                  }
                } else {
                  // t - p in FP64 (exact while p is within a factor 2 of t), then float-float
                  float2 d[2] = {ff_of_double(tm[i].x - t[0]), ff_of_double(tm[i].y - t[1])};
                  if (MODE == XP_SUMS_REL || res.relative) {
                    d[0] = ff_mul(d[0].x, d[0].y, fh[i].x, fl[i].x);
                    d[1] = ff_mul(d[1].x, d[1].y, fh[i].y, fl[i].y);
                    if constexpr (MODE == XP_SUMS_REL) {
                      ff_acc(acc.s[0], acc.c[0], ff_mul(d[0].x, d[0].y, d[0].x, d[0].y));
                      ff_acc(acc.s[1], acc.c[1], ff_mul(d[1].x, d[1].y, d[1].x, d[1].y));
                    } else {
                      d[0] = ff_mul(d[0].x, d[0].y, fh[i].x, fl[i].x);
                      d[1] = ff_mul(d[1].x, d[1].y, fh[i].y, fl[i].y);
                    }
                  }
                  if constexpr (MODE == XP_RESIDUAL) {
                    const int64_t q = (r0 + 8 * i) * res.ld + m;
                    *(float2 *)(res.Qh + q) = make_float2(d[0].x, d[1].x);
                    *(float2 *)(res.Ql + q) = make_float2(d[0].y, d[1].y);
                  }
                }
              }
            } else if (vst) {
              if (m < M) __stcs((double2 *)out, make_double2(t[0], t[1]));
            } else {
              if (m < M) __stcs(out, t[0]);
              if (m + 1 < M) __stcs(out + 1, t[1]);
            }
          }
          if (MODE == XP_TIMES) out += 8 * M;
        }
      };
      uint32_t sg = 0;
#pragma unroll
      for (int o = 0; o < 8; o++) sg |= limb[3][o];
      if (__any_sync(0xffffffffu, (int32_t)sg < 0)) emit(std::true_type{});
      else emit(std::false_type{});
      return true;
    };
    stored(0);
    load((int64_t)blockIdx.x + gridDim.x);
    stored(1);
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, it++) {
      // the counts of the tile after the next on their way into L2
      const int64_t next = tile + 2 * (int64_t)gridDim.x;
      const int64_t off = (next * XP_ROWS + warp * (XP_ROWS / XP_WARPS)) * k * 8 + lane * 128;   // bytes: this warp's rows
      if (lane * 128 < (XP_ROWS / XP_WARPS) * k * 8 && off < R * k * 8)
        asm volatile("prefetch.global.L2 [%0];\n" ::"l"((const char *)F + off));
      int ps = 0;
#pragma unroll 1
      for (; ps < G::PASSES; ps++) {
        if (STASH) acc = stash[ps * 32 * XP_WARPS];
        if (!pass(ps, tile, acc)) break;
        if (STASH) stash[ps * 32 * XP_WARPS] = acc;
      }
      if (ps < G::PASSES) break;
      // every MMA of this tile is complete: its operand buffer takes the tile after the next
      load(next);
      stored(it + 2);
    }
  }
  if constexpr (MODE == XP_ARGMIN) {
    // the CTA's minimum per model over the 4 quarters x 8 row lanes, in the operand space
    ArgPart *red = (ArgPart *)smem;   // [32][64], 32 KB
    __syncthreads();
    if (active) {
#pragma unroll
      for (int ps = 0; ps < G::PASSES; ps++) {
        const XpAcc<MODE> x = STASH ? stash[ps * 32 * XP_WARPS] : acc;
#pragma unroll
        for (int e = 0; e < 2; e++)
          red[(quarter * 8 + (lane >> 2)) * XP_MAXM + 32 * ps + slice * 8 + 2 * (lane & 3) + e] = ArgPart{x.t[e], x.r[e]};
      }
    }
    __syncthreads();
    if (tid < M) {
      ArgPart b = red[tid];
      for (int w = 1; w < 32; w++) {
        const ArgPart x = red[w * XP_MAXM + tid];
        const int64_t kx = time_order(x.t), kb = time_order(b.t);
        if (kx < kb || (kx == kb && x.r < b.r)) b = x;
      }
      // a wait ran out: NaN (ordered below every time) and no row, for callers without a status
      if (s_abort) b = ArgPart{__longlong_as_double(-1ll), -1};
      part[(int64_t)blockIdx.x * M + tid] = b;
    }
  }
  if constexpr (MODE >= XP_SUMS_REL) {
    // the CTA's sums per model, in the operand space, then added to the totals
    double *sum = (double *)smem;   // [64][2]
    __syncthreads();
    if (tid < 2 * XP_MAXM) sum[tid] = 0;
    __syncthreads();
    if (active) {
#pragma unroll
      for (int ps = 0; ps < G::PASSES; ps++) {
        const XpAcc<MODE> x = STASH ? stash[ps * 32 * XP_WARPS] : acc;
#pragma unroll
        for (int e = 0; e < 2; e++) {
          const int m = 32 * ps + slice * 8 + 2 * (lane & 3) + e;
          if constexpr (MODE == XP_SUMS_REL) {
            atomicAdd(&sum[2 * m], (double)x.s[e] + (double)x.c[e]);
          } else {
            atomicAdd(&sum[2 * m], x.r[e]);
            atomicAdd(&sum[2 * m + 1], x.b[e]);
          }
        }
      }
    }
    __syncthreads();
    if (tid < M) {
      atomicAdd(&res.rr[tid], sum[2 * tid]);
      if (MODE == XP_SUMS_ABS) atomicAdd(&res.bb[tid], sum[2 * tid + 1]);
      else if (blockIdx.x == 0) res.bb[tid] = (double)R;   // b = 1 in every row
    }
  }
  xp_finish(&s_abort, status, warp == XP_WARPS, full, XP_RING, seq);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(G::TMEM_COLS));
}

bool exact_tc_ok(int k, int M) { return k >= 1 && k <= XP_MAXK && M >= 1 && M <= XP_MAXM; }

template <int MODE>
static cudaError_t launch_mode(const int64_t *F, int64_t R, int k, const double *W, int M, double *T, ArgPart *part,
                               int grid, int *status, const FitResidual &res, cudaStream_t st) {
  return xp_dispatch(k, M, [&](auto g) {
    using G = decltype(g);
    static_assert(G::SMEM >= 32 * XP_MAXM * sizeof(ArgPart) + 128, "the final reductions use the operand space");
    constexpr size_t smem = G::SMEM + xp_stash<G, MODE>();
    cudaError_t e = cudaFuncSetAttribute(k_predict_exact<G, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_predict_exact<G, MODE><<<grid, XP_THREADS, smem, st>>>(F, R, k, W, M, T, part, status, 256u, res);
    return cudaGetLastError();
  });
}

static int xp_grid(int64_t R, int sms) { return (int)std::max<int64_t>(1, std::min<int64_t>(sms, (R + XP_ROWS - 1) / XP_ROWS)); }

cudaError_t launch_predict_exact(const int64_t *F, int64_t R, int k, const double *W, int M, double *T, int *status,
                                 int sms, cudaStream_t st) {
  return launch_mode<XP_TIMES>(F, R, k, W, M, T, nullptr, xp_grid(R, sms), status, FitResidual{}, st);
}

// per-CTA minima to part[n_part][M]; every entry is written (n_part CTAs, some without rows)
cudaError_t launch_argmin_exact(const int64_t *F, int64_t R, int k, const double *W, int M, ArgPart *part, int n_part,
                                int *status, cudaStream_t st) {
  return launch_mode<XP_ARGMIN>(F, R, k, W, M, nullptr, part, n_part, status, FitResidual{}, st);
}

cudaError_t launch_fit_residual(const int64_t *F, int64_t R, int k, const double *W, int M, const FitResidual &res,
                                bool sums, int *status, int sms, cudaStream_t st) {
  const int grid = xp_grid(R, sms);
  if (!sums) return launch_mode<XP_RESIDUAL>(F, R, k, W, M, nullptr, nullptr, grid, status, res, st);
  if (res.relative) return launch_mode<XP_SUMS_REL>(F, R, k, W, M, nullptr, nullptr, grid, status, res, st);
  return launch_mode<XP_SUMS_ABS>(F, R, k, W, M, nullptr, nullptr, grid, status, res, st);
}

}  // namespace pmd

// Test hooks: the prediction, or the argmin, of one CTA whose issuing warp leaves after the
// first of its tiles.  F [R][k], T [R][M], part: M pairs; k <= 16, M <= 16.
template <int MODE>
static cudaError_t launch_held(const int64_t *F, int64_t R, int k, const double *W, int M, double *T, void *part,
                               int *status, void *stream) {
  using G = pmd::XpGeom<1, 16, 1>;
  if (R < 1 || k < 1 || k > 16 || M < 1 || M > 16) return cudaErrorInvalidValue;
  const auto kernel = pmd::k_predict_exact<G, MODE, true>;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
  if (e != cudaSuccess) return e;
  kernel<<<1, pmd::XP_THREADS, G::SMEM, (cudaStream_t)stream>>>(F, R, k, W, M, T, (pmd::ArgPart *)part, status, 256u,
                                                                pmd::FitResidual{});
  return cudaGetLastError();
}
extern "C" int pmx_predict_held(const int64_t *F, int64_t R, int k, const double *W, int M, double *T, int *status,
                                void *stream) {
  return launch_held<pmd::XP_TIMES>(F, R, k, W, M, T, nullptr, status, stream) == cudaSuccess ? PM_OK : PM_ERR_CUDA;
}
extern "C" int pmx_argmin_held(const int64_t *F, int64_t R, int k, const double *W, int M, void *part, int64_t *arg,
                               double *mn, int *status, void *stream) {
  if (launch_held<pmd::XP_ARGMIN>(F, R, k, W, M, nullptr, part, status, stream) != cudaSuccess) return PM_ERR_CUDA;
  return pmd::launch_argmin_reduce((const pmd::ArgPart *)part, 1, M, arg, mn, (cudaStream_t)stream) == cudaSuccess ? PM_OK
                                                                                                             : PM_ERR_CUDA;
}
