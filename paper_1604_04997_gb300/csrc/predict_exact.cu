// FP64-accurate prediction T = F W^T and the per-model argmin on the tensor cores, from
// exact digit products (exact_tc.cuh has the number scheme and the operand layouts).
//
// One CTA of 16 warps per SM, persistent over 128-row tiles.  Per tile: the counts' digits
// go to shared memory (the loads are issued before the previous tile's times are formed),
// one thread issues the MMAs of the groups of diagonals, and every thread gathers 16 exact
// sums limb by limb, turns them into times and hands them on.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "exact_tc.cuh"
#include "kernels.h"

namespace pmd {

// the order of times as integers (no NaN, no -0.0 among them)
__device__ __forceinline__ int64_t xp_order(double t) {
  const int64_t b = __double_as_longlong(t);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

// ARG false: write T (fp64 [R][M]).  ARG true: per-model minimum over the CTA's rows
// (smaller time, then smaller row) -> part[blockIdx.x][M].
template <bool ARG>
__global__ void __launch_bounds__(XP_THREADS, 1) k_predict_exact(const int64_t *__restrict__ F, int64_t R, int k,
                                                                 const double *__restrict__ W, int M,
                                                                 double *__restrict__ T, ArgPart *__restrict__ part,
                                                                 int *status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = smem_raw + ((128u - (xp_saddr(smem_raw) & 127u)) & 127u);
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ uint32_t tmem_base;
  __shared__ int s_E[XP_MAXM], s_nd[2];
  const XpGeom g = xp_geom(k, M);
  uint8_t *sA = smem, *sB = smem + 2 * g.a_buf();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int quarter = warp & 3, slice = warp >> 2;
  const int64_t ntiles = (R + XP_ROWS - 1) / XP_ROWS;
  const bool vec = (k & 1) == 0 && ((uintptr_t)F & 15) == 0;
  const bool vst = (M & 1) == 0 && ((uintptr_t)T & 15) == 0;
  const int row = xp_row(g.ks);   // this thread's row of a tile when it loads counts

  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(xp_saddr(&mbar[0])));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(xp_saddr(&mbar[1])));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
    s_nd[0] = s_nd[1] = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(xp_saddr(&tmem_base)),
                 "r"(g.tmem_cols()));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  int64_t v[8];
  auto load = [&](int64_t tile) {
    const int64_t r = tile * XP_ROWS + row;
#pragma unroll
    for (int c = 0; c < 8; c++) v[c] = 0;
    if (tile < ntiles && row < XP_ROWS && r < R) xp_load_row(F + r * k, k, g.ks, vec, v);
  };
  load(blockIdx.x);
  xp_load_weights(g, W, M, k, (double *)sA, sB, s_E);
  __syncthreads();   // the staged weights in sA have been read
  xp_store_digits(g, v, sA, &s_nd[0]);
  load((int64_t)blockIdx.x + gridDim.x);
  xp_store_digits(g, v, sA + g.a_buf(), &s_nd[1]);
  asm volatile("fence.proxy.async.shared::cta;\n" ::);
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
  const uint32_t tmem = tmem_base, sA32 = xp_saddr(sA), sB32 = xp_saddr(sB), half = 4u * (uint32_t)g.nb;
  const uint32_t tread = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(slice * 16);
  if (tid == 0 && blockIdx.x < ntiles) {
    for (int gr = 0; gr < 2; gr++) xp_issue(g, sA32, sB32, tmem + gr * half, gr, s_nd[0], xp_saddr(&mbar[gr]));
  }
  const bool active = slice * 16 < g.nb;   // this warp has models
  double bt[4];
  int64_t br[4];
  if (ARG) {
#pragma unroll
    for (int c = 0; c < 4; c++) { bt[c] = __longlong_as_double(0x7ff0000000000000ll); br[c] = INT64_MAX; }
  }
  uint32_t seq = 0;            // groups consumed so far: buffer seq & 1, phase parity (seq >> 1) & 1
  int cur = 0;
  bool aborted = false;
  for (int64_t tile = blockIdx.x; tile < ntiles && !aborted; tile += gridDim.x, cur ^= 1) {
    const int nd = s_nd[cur], ng = xp_groups(nd);
    const bool more = tile + gridDim.x < ntiles;
    const int nd_next = s_nd[cur ^ 1];
    uint32_t limb[3][16], cy[16];
#pragma unroll
    for (int o = 0; o < 16; o++) cy[o] = 0;
#pragma unroll
    for (int gr = 0; gr < 4; gr++) {
      const bool live = gr < ng;
      const uint32_t buf = seq & 1;
      if (live) {
        if (!cta_wait_bounded(xp_saddr(&mbar[buf]), (seq >> 1) & 1)) { aborted = true; break; }
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
      }
      if (active) {
        uint32_t top[16];
        xp_limb(g, tread + buf * half, gr, live, gr < 3 ? limb[gr < 3 ? gr : 0] : top, cy);
        if (gr == 3) {
#pragma unroll
          for (int o = 0; o < 16; o++) cy[o] = top[o];   // the fourth limb
        }
      }
      if (live) {
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
        __syncthreads();   // this group's columns are read: the group after the next may use them
        if (tid == 0) {
          const int ahead = gr + 2;
          if (ahead < ng)
            xp_issue(g, sA32 + cur * g.a_buf(), sB32, tmem + buf * half, ahead, nd, xp_saddr(&mbar[buf]));
          else if (more)
            xp_issue(g, sA32 + (cur ^ 1) * g.a_buf(), sB32, tmem + buf * half, ahead - ng, nd_next,
                     xp_saddr(&mbar[buf]));
        }
        seq++;
      }
    }
    if (aborted) break;
    // every MMA of this tile is complete: its operand buffer takes the tile after the next
    if (tid == 0) s_nd[cur] = 0;
    load(tile + 2 * (int64_t)gridDim.x);
    if (active) {
      const int64_t r0 = tile * XP_ROWS + quarter * 32 + (lane >> 2);
      const int c0 = slice * 16 + 2 * (lane & 3);
#pragma unroll
      for (int s = 0; s < 2; s++) {
#pragma unroll
        for (int h = 0; h < 2; h++) {
          const int64_t r = r0 + 16 * s + 8 * h;
#pragma unroll
          for (int j = 0; j < 2; j++) {
            const int m = c0 + 8 * j, o = 8 * s + 4 * j + 2 * h;
            double t[2];
#pragma unroll
            for (int e = 0; e < 2; e++) {
              xp_unbias(limb[0][o + e], limb[1][o + e], limb[2][o + e], cy[o + e]);
              t[e] = xp_value(limb[0][o + e], limb[1][o + e], limb[2][o + e], cy[o + e], s_E[m + e]);
            }
            if (ARG) {
#pragma unroll
              for (int e = 0; e < 2; e++)   // rows come in increasing order: only a smaller time improves
                if (r < R && xp_order(t[e]) < xp_order(bt[2 * j + e])) { bt[2 * j + e] = t[e]; br[2 * j + e] = r; }
            } else if (r < R) {
              double *out = T + r * M + m;
              if (vst) {
                if (m < M) __stcs((double2 *)out, make_double2(t[0], t[1]));
              } else {
                if (m < M) __stcs(out, t[0]);
                if (m + 1 < M) __stcs(out + 1, t[1]);
              }
            }
          }
        }
      }
    }
    __syncthreads();   // s_nd[cur] is cleared
    xp_store_digits(g, v, sA + cur * g.a_buf(), &s_nd[cur]);
    asm volatile("fence.proxy.async.shared::cta;\n" ::);
    __syncthreads();
  }
  if (aborted) {
    if (tid == 0 && status) atomicOr(status, ST_TIMEOUT);
    // let the MMAs in flight finish before TMEM is freed (bounded)
    cta_wait_bounded(xp_saddr(&mbar[(seq + 1) & 1]), ((seq + 1) >> 1) & 1);
  }
  if (ARG) {
    // the CTA's minimum per model over the 4 quarters x 8 row lanes, in the operand space
    ArgPart *red = (ArgPart *)smem;   // [32][64], 32 KB
    __syncthreads();
    if (active) {
#pragma unroll
      for (int c = 0; c < 4; c++)
        red[(quarter * 8 + (lane >> 2)) * XP_MAXM + slice * 16 + 2 * (lane & 3) + 8 * (c >> 1) + (c & 1)] =
            ArgPart{bt[c], br[c]};
    }
    __syncthreads();
    if (tid < M) {
      ArgPart b = red[tid];
      for (int w = 1; w < 32; w++) {
        const ArgPart x = red[w * XP_MAXM + tid];
        const int64_t kx = xp_order(x.t), kb = xp_order(b.t);
        if (kx < kb || (kx == kb && x.r < b.r)) b = x;
      }
      part[(int64_t)blockIdx.x * M + tid] = b;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(g.tmem_cols()));
}

bool exact_tc_ok(int k, int M) { return k >= 1 && k <= XP_MAXK && M >= 1 && M <= XP_MAXM; }

cudaError_t launch_predict_exact(const int64_t *F, int64_t R, int k, const double *W, int M, double *T, int *status,
                                 int sms, cudaStream_t st) {
  const size_t sm = xp_geom(k, M).smem();
  cudaError_t e = cudaFuncSetAttribute(k_predict_exact<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  const int grid = (int)std::min<int64_t>(sms, (R + XP_ROWS - 1) / XP_ROWS);
  k_predict_exact<false><<<grid, XP_THREADS, sm, st>>>(F, R, k, W, M, T, nullptr, status);
  return cudaGetLastError();
}

// per-CTA minima to part[n_part][M]; every entry is written (n_part CTAs, some without rows)
cudaError_t launch_argmin_exact(const int64_t *F, int64_t R, int k, const double *W, int M, ArgPart *part, int n_part,
                                int *status, cudaStream_t st) {
  const size_t sm = std::max<size_t>(xp_geom(k, M).smem(), 32 * XP_MAXM * sizeof(ArgPart) + 128);
  cudaError_t e = cudaFuncSetAttribute(k_predict_exact<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  k_predict_exact<true><<<n_part, XP_THREADS, sm, st>>>(F, R, k, W, M, nullptr, part, status);
  return cudaGetLastError();
}

}  // namespace pmd
