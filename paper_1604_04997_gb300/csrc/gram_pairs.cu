// Gram matrices of all models of the weight fit (Sec. 4.3) as one matrix product on the
// tensor cores.  With A_m = diag(rowfactor_m) U diag(2^-f_m),
//   G_m[a][b] = 2^-(f_ma + f_mb) sum_r (u_ra u_rb) rowfactor_rm^2,
// so the products u_ra u_rb (k (k + 1) / 2 pairs, the same for every model) meet the squared
// row factors of all models:  [pairs x rows] [rows x models].  A product is formed and split
// once instead of once per model (64 times the entries of U, 0.38e9 conversions for 200,000 x
// 32 x 64; the pairs are 0.11e9).
//
// Products and squares are rounded to FP32 and split into three bf16 terms each (24
// significant bits); the six term products down to 2^-24 accumulate in FP32 in tensor memory
// over at most GP_SUB rows (252 accumulation steps), then in FP64 into G.  The FP32 accumulation
// is what limits G: weights without refinement are off by 8e-7 (1,000 to 20,000 rows, cond(A)
// 20), 2.2e-6 (60,000) and 3.6e-6 (200,000 rows), where entries split into three terms per
// model and chunks of 4,096 rows gave 2e-6 (1,000) to 2e-5 (60,000); the rounding of the
// products alone is 2e-8.  Refinement with exact residuals recovers full accuracy as long as
// cond(G) 2^-18 is well below 1; else the fit falls back to the exact Gram (gram_tc.cu).
//
// One CTA per SM takes one contiguous range of rows, in stages of 16 rows (one K-step): 16
// warps write the stage's pairs (rows 0 .. 639 in five 128-row tiles), four its models (the N
// operand), K-major without swizzle, three terms each, 66 KB, into a ring of three, and a
// warp issues its 30 MMAs (M = 128, N = models).  Bound by the split arithmetic and the
// shared-memory reads of the MMAs (a 4 KB A tile per 48 cycles); the inputs of later stages
// are prefetched into L2 and, one or two stages ahead, into registers.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "exact_tc.cuh"
#include "kernels.h"
#include "pm.h"

namespace pmd {

namespace {

constexpr int GP_WARPS = 16, GP_WORK = 32 * GP_WARPS;   // warps that write pairs
constexpr int GP_BWARPS = 4;                            // warps that write models
constexpr int GP_ISSUER = GP_WARPS + GP_BWARPS, GP_THREADS = 32 * (GP_ISSUER + 1);
constexpr int GP_AHEAD = 8;           // stages whose inputs are on their way into L2
constexpr int GP_K = 16;              // rows per stage
constexpr int GP_RING = 3;
constexpr int GP_SUB = 42 * GP_K;     // rows accumulated in FP32
constexpr int GP_TILES = 5;           // 528 pairs of 32 columns
constexpr uint32_t GP_ATERM = GP_TILES * 128 * GP_K * 2, GP_BTERM = 64 * GP_K * 2;
constexpr uint32_t GP_STAGE = 3 * (GP_ATERM + GP_BTERM);
constexpr int GP_USTRIDE = GP_K + 4;  // floats per column of the staged U: 16-byte reads of 8 lanes hit distinct banks
constexpr uint32_t GP_SMEM = GP_RING * GP_STAGE + 2 * 32 * GP_USTRIDE * 4 + 64 * 32 * 2 + 128;

__device__ __forceinline__ uint32_t gp_pack(float x, float y) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  return *(const uint32_t *)&h;
}
// three bf16 terms of two floats, packed
__device__ __forceinline__ void gp_split(float x, float y, uint32_t &p1, uint32_t &p2, uint32_t &p3) {
  p1 = gp_pack(x, y);
  const float rx = __fsub_rn(x, __uint_as_float(p1 << 16)), ry = __fsub_rn(y, __uint_as_float(p1 & 0xFFFF0000u));
  p2 = gp_pack(rx, ry);
  p3 = gp_pack(__fsub_rn(rx, __uint_as_float(p2 << 16)), __fsub_rn(ry, __uint_as_float(p2 & 0xFFFF0000u)));
}
// eight floats to the three terms' 16-byte K-major rows
__device__ __forceinline__ void gp_store(const float (&x)[8], uint8_t *dst, uint32_t term) {
  uint32_t t[3][4];
#pragma unroll
  for (int i = 0; i < 4; i++) gp_split(x[2 * i], x[2 * i + 1], t[0][i], t[1][i], t[2][i]);
#pragma unroll
  for (int q = 0; q < 3; q++) *(uint4 *)(dst + q * term) = make_uint4(t[q][0], t[q][1], t[q][2], t[q][3]);
}

__device__ __forceinline__ int gp_exp(unsigned bits) {   // exponent e with x in [2^(e-1), 2^e), 0 for zero
  if (!bits) return 0;
  int e;
  frexpf(__uint_as_float(bits), &e);
  return e;
}

// pair p -> (a, b), a <= b, counting rows a of the upper triangle of a k x k matrix
__device__ __forceinline__ void gp_pair(int p, int k, int &a, int &b) {
  a = 0;
  while (a < k && p >= k - a) { p -= k - a; a++; }
  b = a + p;
}

}  // namespace

// Uh: [R][ldu] (zero columns beyond k); rfh, rfl: row factors as float-float [R][ld];
// rmax: their column maxima (float bits).  HELD: the issuing warp leaves without reporting its
// sums and the waits are short (pmx_gram_held).
template <bool HELD>
__global__ void __launch_bounds__(GP_THREADS, 1) k_gram_pairs(const float *__restrict__ Uh, int ldu, const float *__restrict__ rfh,
                                                              const float *__restrict__ rfl, int ld, int64_t R, int k,
                                                              int M, int64_t rows_per_cta, const unsigned *__restrict__ amax,
                                                              const unsigned *__restrict__ rmax,
                                                              double *__restrict__ G, int *status) {
  constexpr unsigned long long LIMIT = HELD ? XP_HELD_NS : MBAR_WAIT_NS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = smem_raw + ((128u - (xp_saddr(smem_raw) & 127u)) & 127u);
  float(*su)[32][GP_USTRIDE] = (float(*)[32][GP_USTRIDE])(smem + GP_RING * GP_STAGE);
  int16_t(*sf)[32] = (int16_t(*)[32])(smem + GP_RING * GP_STAGE + 2 * 32 * GP_USTRIDE * 4);
  __shared__ __align__(8) uint64_t ready[GP_RING], freed[GP_RING], summed, drained;
  __shared__ uint32_t tmem_base;
  __shared__ int s_sh[64];
  __shared__ volatile int s_abort;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int np = k * (k + 1) / 2, tiles = (np + 127) / 128, nb = (M + 15) & ~15;
  const int64_t r0 = (int64_t)blockIdx.x * rows_per_cta, r1 = min(R, r0 + rows_per_cta);

  // rows of pairs and models that do not exist stay zero
  for (uint32_t i = tid; i < GP_RING * GP_STAGE / 16; i += GP_THREADS) ((uint4 *)smem)[i] = make_uint4(0, 0, 0, 0);
  for (int i = tid; i < M * k; i += GP_THREADS) sf[i / k][i % k] = (int16_t)gp_exp(amax[(i / k) * 32 + i % k]);
  if (tid < 64) {
    // row factors are scaled to about 2^20 at most: squares up to 2^40, and 2^-102 (full
    // precision of the split) is reached at factors 2^-71 of the largest
    const int e = tid < M ? min(126, max(-100, gp_exp(rmax[tid]))) : 0;
    s_sh[tid] = e - 20;
  }
  if (tid == 0) {
    for (int b = 0; b < GP_RING; b++) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(xp_saddr(&ready[b])), "n"(GP_WARPS + GP_BWARPS));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(xp_saddr(&freed[b])));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(xp_saddr(&summed)));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(xp_saddr(&drained)), "n"(GP_WARPS));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
    s_abort = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(xp_saddr(&tmem_base)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  asm volatile("fence.proxy.async.shared::cta;\n" ::);
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
  const uint32_t tmem = xp_uniform(tmem_base), s0 = xp_uniform(xp_saddr(smem));
  bool ok = true;
  uint32_t n = 0, sub = 0;   // stages and FP32 sums so far

  if (warp == GP_ISSUER) {
    // kind::f16: D fp32, A and B bf16, both K-major
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t)(nb >> 3) << 17 | (128u >> 4) << 24;
    for (int64_t rb = r0; rb < r1 && ok; rb += GP_SUB, sub++) {
      if (sub && !(ok = xp_wait(xp_saddr(&drained), (sub - 1) & 1, &s_abort, LIMIT))) break;
      for (int64_t rs = rb; rs < min(r1, rb + GP_SUB); rs += GP_K, n++) {
        const uint32_t b = n % GP_RING;
        if (!(ok = xp_wait(xp_saddr(&ready[b]), (n / GP_RING) & 1, &s_abort, LIMIT))) break;
        const uint32_t sa = s0 + b * GP_STAGE, sb = sa + 3 * GP_ATERM;
#pragma unroll
        for (int p = 0; p < 6; p++) {   // term products 11, 12, 21, 13, 22, 31
          const uint32_t pa = p == 2 || p == 4 ? 1 : (p == 5 ? 2 : 0), pb = p == 1 || p == 4 ? 1 : (p == 3 ? 2 : 0);
#pragma unroll
          for (int t = 0; t < GP_TILES; t++)
            if (t < tiles)
              xp_mma(tmem + t * 64, xp_desc(sa + pa * GP_ATERM + t * 4096, 256), xp_desc(sb + pb * GP_BTERM, 256), idesc,
                     p != 0 || rs != rb);
        }
        xp_commit(xp_saddr(&freed[b]));
      }
      if (ok && !HELD) xp_commit(xp_saddr(&summed));
    }
    if (!ok) xp_drain(freed, GP_RING, n);
    __syncwarp();
  } else if (warp >= GP_WARPS) {
    // one row (8 rows of U of one model) of the N operand per thread: 64 models x 2 K-groups
    const int mop = tid - GP_WORK, mm = mop & 63, mkg = mop >> 6;
    const bool has = mm < M;
    const float msc = has ? __uint_as_float((uint32_t)(127 - s_sh[mm]) << 23) : 0.f;   // 2^-sh
    float nh[2][8], nl[2][8];   // two stages ahead
    auto fetch = [&](int64_t rs, float (&h)[8], float (&l)[8]) {
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const int64_t q = rs + mkg * 8 + i;
        const bool in = has && q < r1;
        h[i] = in ? rfh[q * ld + mm] : 0.f;
        l[i] = in ? rfl[q * ld + mm] : 0.f;
      }
    };
    auto stage = [&](int64_t rs, float (&h)[8], float (&l)[8]) {
      const uint32_t buf = n % GP_RING;
      float w[8];
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const float x = __fmul_rn(h[i], msc), y = __fmul_rn(l[i], msc);
        w[i] = __fmaf_rn(x, x, __fmul_rn(2.f, __fmul_rn(x, y)));
      }
      fetch(rs + 2 * GP_K, h, l);
      if (n >= GP_RING) ok = xp_wait(xp_saddr(&freed[buf]), (n / GP_RING - 1) & 1, &s_abort, LIMIT);
      if (!ok) return;
      if (has) gp_store(w, smem + buf * GP_STAGE + 3 * GP_ATERM + (mm >> 3) * 256 + mkg * 128 + (mm & 7) * 16, GP_BTERM);
      asm volatile("fence.proxy.async.shared::cta;\n" ::);
      __syncwarp();
      if (lane == 0) xp_arrive(xp_saddr(&ready[buf]));
      n++;
    };
    fetch(r0, nh[0], nl[0]);
    fetch(r0 + GP_K, nh[1], nl[1]);
    for (int64_t rs = r0; rs < r1 && ok; rs += 2 * GP_K) {
      // the row factors of a later pair of stages on their way: 32 rows, 128 bytes per prefetch
      const int64_t off = ((rs + GP_AHEAD * GP_K) * ld + (int64_t)mop * 32) * 4;
      if (mop < ld && off < R * ld * 4) {
        asm volatile("prefetch.global.L2 [%0];\n" ::"l"((const char *)rfh + off));
        asm volatile("prefetch.global.L2 [%0];\n" ::"l"((const char *)rfl + off));
      }
      stage(rs, nh[0], nl[0]);
      if (rs + GP_K < r1 && ok) stage(rs + GP_K, nh[1], nl[1]);
    }
  } else {
    // this thread's pair operations of a stage: 8 rows (K-group) of one pair; operation i
    // is pair 8 (i / 16) + i % 8, K-group (i / 8) % 2
    constexpr int OPS = (GP_TILES * 128 * 2 + GP_WORK - 1) / GP_WORK;
    uint32_t op_src[OPS], op_dst[OPS];
#pragma unroll
    for (int j = 0; j < OPS; j++) {
      const int i = tid + j * GP_WORK, p = (i >> 4) * 8 + (i & 7), kg = (i >> 3) & 1;
      int a = 0, b = 0;
      if (p < np) gp_pair(p, k, a, b);
      op_src[j] = p < np ? (uint32_t)(a * GP_USTRIDE + kg * 8) | (uint32_t)(b * GP_USTRIDE + kg * 8) << 16 : 0xFFFFFFFFu;
      op_dst[j] = (uint32_t)((p >> 3) * 256 + kg * 128 + (p & 7) * 16);
    }
    auto fetch = [&](int64_t rs) {   // this thread's entry of the stage at row rs
      const int64_t r = rs + (tid >> 5);
      return r < r1 && lane < ldu ? Uh[r * ldu + lane] : 0.f;
    };
    float nu = fetch(r0), nu2 = fetch(r0 + GP_K);
    bool dead = false;   // some warp's wait ran out: all working warps leave at the next stage's barrier
    for (int64_t rb = r0; rb < r1 && !dead; rb += GP_SUB, sub++) {
      const int64_t re = min(r1, rb + GP_SUB);
      for (int64_t rs = rb; rs < re; rs += GP_K, n++) {
        const uint32_t buf = n % GP_RING;
        su[n & 1][lane][tid >> 5] = nu;
        nu = nu2;
        nu2 = fetch(rs + 2 * GP_K);
        if (lane == 0 && rs + GP_AHEAD * GP_K + (tid >> 5) < R)   // one row of U per warp
          asm volatile("prefetch.global.L2 [%0];\n" ::"l"(Uh + (rs + GP_AHEAD * GP_K + (tid >> 5)) * ldu));
        if (n >= GP_RING) ok = xp_wait(xp_saddr(&freed[buf]), (n / GP_RING - 1) & 1, &s_abort, LIMIT) && ok;
        uint32_t any;   // the stage's U is complete once all have arrived
        asm volatile(
            "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.or.pred q, 1, %2, p;\nselp.u32 %0, 1, 0, q;\n}\n"
            : "=r"(any)
            : "r"((uint32_t)!ok), "n"(GP_WORK)
            : "memory");
        if ((dead = any != 0)) break;
        uint8_t *st = smem + buf * GP_STAGE;
        const float *u = &su[n & 1][0][0];
#pragma unroll
        for (int j = 0; j < OPS; j++) {
          if (op_src[j] == 0xFFFFFFFFu) continue;
          const float4 a0 = *(const float4 *)(u + (op_src[j] & 0xFFFF)), a1 = *(const float4 *)(u + (op_src[j] & 0xFFFF) + 4);
          const float4 b0 = *(const float4 *)(u + (op_src[j] >> 16)), b1 = *(const float4 *)(u + (op_src[j] >> 16) + 4);
          const float x[8] = {a0.x * b0.x, a0.y * b0.y, a0.z * b0.z, a0.w * b0.w,
                              a1.x * b1.x, a1.y * b1.y, a1.z * b1.z, a1.w * b1.w};
          gp_store(x, st + op_dst[j], GP_ATERM);
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::);
        __syncwarp();
        if (lane == 0) xp_arrive(xp_saddr(&ready[buf]));
      }
      if (dead) break;
      if (!xp_wait(xp_saddr(&summed), sub & 1, &s_abort, LIMIT)) {
        ok = false;
        continue;
      }
      // add the sums into G: warp w reads pairs 32 (w % 4) .. of each tile, models 16 (w / 4) ..
      const int quarter = warp & 3, m0 = (warp >> 2) * 16;
      if (m0 < nb) {
#pragma unroll 1
        for (int t = 0; t < tiles; t++) {
          uint32_t d[16];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
              : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]), "=r"(d[4]), "=r"(d[5]), "=r"(d[6]), "=r"(d[7]),
                "=r"(d[8]), "=r"(d[9]), "=r"(d[10]), "=r"(d[11]), "=r"(d[12]), "=r"(d[13]), "=r"(d[14]), "=r"(d[15])
              : "r"(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(t * 64 + m0)));
          asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::);
          const int p = t * 128 + quarter * 32 + lane;
          if (p < np) {
            int a, b;
            gp_pair(p, k, a, b);
#pragma unroll
            for (int j = 0; j < 16; j++) {
              const int m = m0 + j;
              const uint32_t mag = d[j] & 0x7FFFFFFFu;
              if (m < M && mag) {
                // the FP32 sum times 2^(2 sh - f_a - f_b) as FP64, by its exponent field
                const int sh = 2 * s_sh[m] - sf[m][a] - sf[m][b];
                double v;
                if (mag - 0x00800000u < 0x7F000000u) {
                  const uint32_t hi = (d[j] & 0x80000000u) | ((mag >> 3) + ((uint32_t)(896 + sh) << 20));
                  v = __hiloint2double((int)hi, (int)(mag << 29));
                } else {   // subnormal, infinite or NaN
                  v = ldexp((double)__uint_as_float(d[j]), sh);
                }
                atomicAdd(&G[((int64_t)m * 32 + a) * 32 + b], v);
              }
            }
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
      __syncwarp();
      if (lane == 0) xp_arrive(xp_saddr(&drained));
    }
  }
  xp_finish(&s_abort, status, warp == GP_ISSUER, freed, GP_RING, n);
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
}

template <bool HELD>
static cudaError_t launch(const float *Uh, int ldu, const float *rfh, const float *rfl, int ld, int64_t R, int k, int M,
                          int64_t rows, const unsigned *amax, const unsigned *rmax, double *G, int *status,
                          cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_gram_pairs<HELD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GP_SMEM);
  if (e != cudaSuccess) return e;
  k_gram_pairs<HELD><<<(unsigned)((R + rows - 1) / rows), GP_THREADS, GP_SMEM, st>>>(Uh, ldu, rfh, rfl, ld, R, k, M, rows, amax,
                                                                                  rmax, G, status);
  return cudaGetLastError();
}

cudaError_t launch_gram_pairs(const float *Uh, int ldu, const float *rfh, const float *rfl, int ld, int64_t R, int k, int M,
                              const unsigned *amax, const unsigned *rmax, double *G, int sms, int *status,
                              cudaStream_t st) {
  if (R <= 0 || M <= 0) return cudaSuccess;
  // one range of rows per SM, at least eight stages of them
  const int64_t rows = std::max<int64_t>(8 * GP_K, ((R + sms - 1) / sms + GP_K - 1) / GP_K * GP_K);
  return launch<false>(Uh, ldu, rfh, rfl, ld, R, k, M, rows, amax, rmax, G, status, st);
}

}  // namespace pmd

// Test hook: the Gram of one CTA whose issuing warp leaves without reporting its sums.  U, rfh,
// rfl: [R][32]; amax [M][32], rmax [M]; G [M][32][32]; R <= 1,024, k <= 32, M <= 32.
extern "C" int pmx_gram_held(const float *U, const float *rfh, const float *rfl, int64_t R, int k, int M,
                             const unsigned *amax, const unsigned *rmax, double *G, int *status, void *stream) {
  if (R < 1 || R > 1024 || k < 1 || k > 32 || M < 1 || M > 32) return PM_ERR_INVALID_ARG;
  return pmd::launch<true>(U, 32, rfh, rfl, 32, R, k, M, 1024, amax, rmax, G, status, (cudaStream_t)stream) == cudaSuccess
             ? PM_OK : PM_ERR_CUDA;
}
