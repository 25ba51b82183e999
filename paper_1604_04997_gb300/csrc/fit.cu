// Weight fit (Sec. 4.3): for every device model m, find w_m minimising
//   relative objective  sum_j (1 - F_j w_m / t_jm)^2     (the paper's)
//   absolute objective  sum_j (t_jm - F_j w_m)^2
// The least-squares matrix of model m is A_m = diag(1/t_m) F (relative) or F
// (absolute); its columns are scaled by powers of two so that max_r |A_rc| lies in
// [1/2, 1).  The normal equations A^T A x = A^T b (b = 1, or b = t_m) are formed
// in float-float arithmetic on the FP32 pipes (entries split exactly into hi + lo
// pairs, error-free products by FMA, compensated sums; about 2^-44 relative) per row
// chunk, chunks summed in FP64 (precision PM_PREC_FP64), or on the tensor cores from
// three bf16 terms with FP32 accumulation (PM_PREC_BF16X3, gram_pairs.cu), or exactly from
// bf16 digits of a 47-bit fixed-point image of A when refinement on the three-term Gram
// does not converge (gram_tc.cu);
// the k x k systems are factored by FP64 Cholesky.  Iterative refinement then
// recovers the accuracy: r = b - A x is formed from the exact fixed-point product
// F w (the prediction kernel itself, predict_exact.cu), t - F w in FP64 and float-float
// products with 1/t (about 2^-45), the correction solves G d = A^T r with the same factor, and
// x += d.  FP64 is kept to the Cholesky factors, the substitutions and the sums: this
// GPU's FP64 pipe is narrow.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "eval_common.cuh"
#include "float_float.cuh"
#include "kernels.h"
#include "pm.h"

namespace pmd {

constexpr int FIT_MAXK = 32;
constexpr int FIT_ROWS = 64;      // rows staged per batch
constexpr int FIT_THREADS = 256;

// ---- column maxima of |F| (as unsigned bit patterns, for atomicMax)
__global__ void k_colmax(const int64_t *__restrict__ F, int64_t R, int k, unsigned long long *cmax) {
  __shared__ unsigned long long s[FIT_MAXK];
  if (threadIdx.x < FIT_MAXK) s[threadIdx.x] = 0;
  __syncthreads();
  const int c = threadIdx.x % k;
  const int rstep = blockDim.x / k;
  unsigned long long m = 0;
  if (threadIdx.x < rstep * k) {
    for (int64_t r = (int64_t)blockIdx.x * rstep + threadIdx.x / k; r < R; r += (int64_t)gridDim.x * rstep) {
      const int64_t v = F[r * k + c];
      const unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
      m = a > m ? a : m;
    }
    atomicMax(&s[c], m);
  }
  __syncthreads();
  if (threadIdx.x < k) atomicMax(&cmax[threadIdx.x], s[threadIdx.x]);
}

// exponent e_c with max |F_c| in [2^(e-1), 2^e) (0 for an all-zero column)
__device__ __forceinline__ int col_exp(unsigned long long mx) { return mx ? 64 - __clzll((long long)mx) : 0; }

// ---- U = F diag(2^-e) as float-float pairs: Uh = rn(F), Ul = rn(F - Uh), scaled exactly;
// rows of ldu floats (k rounded up to 4), zero beyond column k
__global__ void k_scale(const int64_t *__restrict__ F, int64_t R, int k, int ldu, const unsigned long long *cmax,
                        float *__restrict__ Uh, float *__restrict__ Ul) {
  const int c = threadIdx.x & 31;
  const int e = c < k ? col_exp(cmax[c]) : 0;
  const int64_t step = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < R; r += step) {
    const int64_t v = c < k ? F[r * k + c] : 0;
    const float h = __ll2float_rn(v);
    if (c < ldu) {
      Uh[r * ldu + c] = ldexpf(h, -e);
      Ul[r * ldu + c] = ldexpf(__ll2float_rn(v - (int64_t)h), -e);
    }
  }
}

// 1/t for t > 0 as float-float (within ~2^-46): FP32 reciprocal, one Newton step with
// the residual formed by FMA; FP64 division outside [2^-100, 2^100].
__device__ __forceinline__ float2 ff_recip(double t) {
  const uint64_t b = (uint64_t)__double_as_longlong(t);
  const int e = (int)((b >> 52) & 0x7FF) - 1023;
  if (e < -100 || e > 100) {
    const double r = 1.0 / t;
    const float h = __double2float_rn(r);
    return make_float2(h, __double2float_rn(r - (double)h));
  }
  const float2 tt = ff_of_double(t);
  const float y = __frcp_rn(tt.x);
  float res = __fmaf_rn(-tt.x, y, 1.0f);       // 1 - th y, exact: th y is within 2^-23 of 1
  res = __fmaf_rn(-tt.y, y, res);              // - tl y
  const float lo = __fmul_rn(y, res);
  const float hi = __fadd_rn(y, lo);           // renormalise (Fast2Sum: |y| >= |lo|)
  return make_float2(hi, __fsub_rn(lo, __fsub_rn(hi, y)));
}

// ---- row factors as float-float, rows of ld floats: 1/t (relative) or 1 (absolute); beta
// (if wanted) = 1 or t.  The residual passes reuse the relative row factor as 1/t.  Entries
// beyond model M are zero.
// From them the maxima per (model, column) of |A_rc| = |U_rc| * rowfactor_rm, and per model
// of the row factors (float bits, atomicMax): a (max, x) matrix product over 32-row stages of
// U and of the row factors in shared memory, 4 columns x 4 models per thread, the two halves
// of the CTA on 16 rows each, so one 16-byte read feeds eight products.
constexpr int AM_ROWS = 32;
__global__ void __launch_bounds__(FIT_THREADS) k_rowfac(const float *__restrict__ U, int ldu, const double *__restrict__ T, int ld,
                                                        int64_t R, int k, int M, int objective, float *__restrict__ rfh,
                                                        float *__restrict__ rfl, float *__restrict__ bh,
                                                        float *__restrict__ bl, unsigned *__restrict__ amax,
                                                        unsigned *__restrict__ rmax, int *status) {
  __shared__ __align__(16) float su[AM_ROWS][32], sr[AM_ROWS][64];
  __shared__ unsigned best[64][33];
  const int tid = threadIdx.x, cg = tid & 7, mg = (tid >> 3) & 15, half = tid >> 7;
  for (int i = tid; i < 64 * 33; i += FIT_THREADS) (&best[0][0])[i] = 0;
  for (int i = tid; i < AM_ROWS * 64; i += FIT_THREADS) (&sr[0][0])[i] = 0.f;
  const int64_t big = __double_as_longlong(1e300);
  const int m4 = ld / 4, inv4 = (65536 + m4 - 1) / m4;   // i / m4 = i inv4 / 2^16 for i < 512
  const bool vec = (M & 1) == 0 && ((uintptr_t)T & 15) == 0;
  float mx[4][4], mr[4];
#pragma unroll
  for (int i = 0; i < 4; i++) {
    mr[i] = 0.f;
#pragma unroll
    for (int j = 0; j < 4; j++) mx[i][j] = 0.f;
  }
  // this thread's items of a stage: four models of a row each, their timings one stage ahead
  constexpr int ITEMS = AM_ROWS * 16 / FIT_THREADS;
  double tn[ITEMS][4];
  auto fetch = [&](int64_t rb) {
#pragma unroll
    for (int q = 0; q < ITEMS; q++) {
      const int i = tid + q * FIT_THREADS, r = (i * inv4) >> 16, m = (i - r * m4) * 4;
#pragma unroll
      for (int e = 0; e < 4; e++) tn[q][e] = 1.0;
      if (r < AM_ROWS && rb + r < R) {
        const double *src = T + (rb + r) * M + m;
        if (vec && m + 3 < M) {
          const double2 x = __ldcs((const double2 *)src), y = __ldcs((const double2 *)src + 1);
          tn[q][0] = x.x, tn[q][1] = x.y, tn[q][2] = y.x, tn[q][3] = y.y;
        } else {
#pragma unroll
          for (int e = 0; e < 4; e++)
            if (m + e < M) tn[q][e] = __ldcs(src + e);
        }
      }
    }
  };
  fetch((int64_t)blockIdx.x * AM_ROWS);
  for (int64_t rb = (int64_t)blockIdx.x * AM_ROWS; rb < R; rb += (int64_t)gridDim.x * AM_ROWS) {
    const int nr = (int)min((int64_t)AM_ROWS, R - rb);
    __syncthreads();
    for (int i = tid; i < AM_ROWS * 8; i += FIT_THREADS) {
      const int r = i >> 3, c = (i & 7) * 4;
      const float4 x = r < nr && c < ldu ? *(const float4 *)(U + (rb + r) * ldu + c) : make_float4(0.f, 0.f, 0.f, 0.f);
      *(float4 *)&su[r][c] = make_float4(fabsf(x.x), fabsf(x.y), fabsf(x.z), fabsf(x.w));
    }
#pragma unroll
    for (int q = 0; q < ITEMS; q++) {
      const int i = tid + q * FIT_THREADS, r = (i * inv4) >> 16, m = (i - r * m4) * 4;
      if (r >= AM_ROWS) continue;
      const double(&t)[4] = tn[q];
      float fh[4], fl[4], gh[4], gl[4];
#pragma unroll
      for (int e = 0; e < 4; e++) {
        float2 x = make_float2(0.f, 0.f), b = x;
        const int64_t tb = __double_as_longlong(t[e]);   // 0 < t <= 1e300 (NaN excluded) by its bits
        if (r >= nr || m + e >= M) {
        } else if (tb <= 0 || tb > big) {
          atomicOr(status, ST_BAD_INPUT);
        } else if (objective == PM_FIT_RELATIVE) {
          x = ff_recip(t[e]);
          b = make_float2(1.f, 0.f);
        } else {
          x = make_float2(1.f, 0.f);
          b = ff_of_double(t[e]);
        }
        fh[e] = x.x, fl[e] = x.y, gh[e] = b.x, gl[e] = b.y;
      }
      *(float4 *)&sr[r][m] = make_float4(fh[0], fh[1], fh[2], fh[3]);
      if (r < nr) {
        const int64_t o = (rb + r) * ld + m;
        *(float4 *)(rfh + o) = make_float4(fh[0], fh[1], fh[2], fh[3]);
        *(float4 *)(rfl + o) = make_float4(fl[0], fl[1], fl[2], fl[3]);
        if (bh) {
          *(float4 *)(bh + o) = make_float4(gh[0], gh[1], gh[2], gh[3]);
          *(float4 *)(bl + o) = make_float4(gl[0], gl[1], gl[2], gl[3]);
        }
      }
    }
    fetch(rb + (int64_t)gridDim.x * AM_ROWS);
    __syncthreads();
    if (mg * 4 < ld) {
#pragma unroll 4
      for (int r = half * (AM_ROWS / 2); r < (half + 1) * (AM_ROWS / 2); r++) {
        const float4 u4 = *(const float4 *)&su[r][4 * cg], f4 = *(const float4 *)&sr[r][4 * mg];
        const float u[4] = {u4.x, u4.y, u4.z, u4.w}, f[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
        for (int i = 0; i < 4; i++) {
          mr[i] = fmaxf(mr[i], f[i]);
#pragma unroll
          for (int j = 0; j < 4; j++) mx[i][j] = fmaxf(mx[i][j], __fmul_rn(u[j], f[i]));
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const int m = 4 * mg + i;
    if (cg == 0) atomicMax(&best[m][32], __float_as_uint(mr[i]));   // non-negative floats order as integers
#pragma unroll
    for (int j = 0; j < 4; j++) atomicMax(&best[m][4 * cg + j], __float_as_uint(mx[i][j]));
  }
  __syncthreads();
  for (int i = tid; i < M * 33; i += FIT_THREADS) {
    const int m = i / 33, c = i - m * 33;
    if (c == 32) atomicMax(&rmax[m], best[m][32]);
    else if (c < k) atomicMax(&amax[m * FIT_MAXK + c], best[m][c]);
  }
}

// power-of-two exponent f with max |A_c| * 2^-f in [1/2, 1) (0 for an all-zero column)
__device__ __forceinline__ int acol_exp(unsigned bits) {
  if (!bits) return 0;
  int e;
  frexpf(__uint_as_float(bits), &e);
  return e;
}

// ---- Gram matrices and right-hand sides.
// Grid (row chunks, models).  Each CTA accumulates, for its model, the upper triangle
// of sum_r v_r v_r^T and sum_r v_r * beta_r over its rows, where
// relative: v = u / t, beta = 1;   absolute: v = u, beta = t.
// The row [v | beta] (k + 1 <= 33 values, padded to 36) is staged in shared memory as
// float-float pairs; the 36 x 36 upper triangle is cut into the 45 4x4 blocks (bi <=
// bj) of a 9 x 9 block grid, and each of 5 row groups of 45 threads takes every
// block once: a thread reads two 4-column slices per row and forms 16 error-free
// products, accumulated with TwoSum compensation.  Chunk results are added to the
// FP64 totals with atomics.
constexpr int GB_COLS = 36, GB_BLOCKS = 9, GB_TASKS = 45, GB_GROUPS = 5;
__global__ void __launch_bounds__(FIT_THREADS) k_gram(const float *__restrict__ Uh, const float *__restrict__ Ul, int ldu,
                                                      const float *__restrict__ rfh, const float *__restrict__ rfl,
                                                      const float *__restrict__ bh, const float *__restrict__ bl,
                                                      int ld, int64_t R, int k, int M, int64_t rows_per_chunk,
                                                      const unsigned *__restrict__ amax, double *__restrict__ G,
                                                      double *__restrict__ rhs) {
  __shared__ __align__(16) float vh[FIT_ROWS][GB_COLS], vl[FIT_ROWS][GB_COLS];
  __shared__ int f[FIT_MAXK];
  const int m = blockIdx.y;
  if (threadIdx.x < FIT_MAXK) f[threadIdx.x] = threadIdx.x < k ? acol_exp(amax[m * FIT_MAXK + threadIdx.x]) : 0;
  const int64_t r0 = (int64_t)blockIdx.x * rows_per_chunk;
  const int64_t r1 = min(R, r0 + rows_per_chunk);
  // this thread's block (bi, bj) and row group
  const int task = threadIdx.x % GB_TASKS, grp = threadIdx.x / GB_TASKS;
  int bi = 0, rest = task;
  while (rest >= GB_BLOCKS - bi) { rest -= GB_BLOCKS - bi; bi++; }
  const int bj = bi + rest;
  const bool active = grp < GB_GROUPS && 4 * bi <= k && 4 * bj <= k;   // column k is beta
  constexpr int RPG = (FIT_ROWS + GB_GROUPS - 1) / GB_GROUPS;
  float s[16], c[16];
#pragma unroll
  for (int q = 0; q < 16; q++) s[q] = c[q] = 0.f;
  for (int64_t rb = r0; rb < r1; rb += FIT_ROWS) {
    __syncthreads();
    const int nr = (int)min((int64_t)FIT_ROWS, r1 - rb);
    const int64_t u0 = rb * ldu, m0 = rb * ld + m;
    for (int i = threadIdx.x; i < FIT_ROWS * GB_COLS; i += FIT_THREADS) {
      const int rr = i / GB_COLS, cc = i - rr * GB_COLS;
      float2 v = make_float2(0.f, 0.f);
      if (rr < nr) {
        const int o = rr * ldu + cc, q = rr * ld;
        if (cc < k) {
          v = ff_mul(Uh[u0 + o], Ul[u0 + o], rfh[m0 + q], rfl[m0 + q]);
          v.x = ldexpf(v.x, -f[cc]);
          v.y = ldexpf(v.y, -f[cc]);
        } else if (cc == k) {
          v = make_float2(bh[m0 + q], bl[m0 + q]);
        }
      }
      vh[rr][cc] = v.x;
      vl[rr][cc] = v.y;
    }
    __syncthreads();
    if (active) {
      const int rend = min(nr, (grp + 1) * RPG);
      for (int rr = grp * RPG; rr < rend; rr++) {
        const float4 ah = *(const float4 *)&vh[rr][4 * bi], al = *(const float4 *)&vl[rr][4 * bi];
        const float4 bh = *(const float4 *)&vh[rr][4 * bj], bl = *(const float4 *)&vl[rr][4 * bj];
        const float xa[4] = {ah.x, ah.y, ah.z, ah.w}, ya[4] = {al.x, al.y, al.z, al.w};
        const float xb[4] = {bh.x, bh.y, bh.z, bh.w}, yb[4] = {bl.x, bl.y, bl.z, bl.w};
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
          for (int j = 0; j < 4; j++) ff_acc(s[4 * i + j], c[4 * i + j], ff_mul(xa[i], ya[i], xb[j], yb[j]));
      }
    }
  }
  if (!active) return;
#pragma unroll
  for (int i = 0; i < 4; i++) {
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const int a = 4 * bi + i, b = 4 * bj + j;
      if (a > b || a >= k || b > k) continue;
      const double val = (double)s[4 * i + j] + (double)c[4 * i + j];
      if (b < k) atomicAdd(&G[((int64_t)m * FIT_MAXK + a) * FIT_MAXK + b], val);
      else atomicAdd(&rhs[(int64_t)m * FIT_MAXK + a], val);
    }
  }
}

// L L^T d = g of one model by a warp, lane a owning row a: forward and backward substitution
// column by column, each step one product with the diagonal's reciprocal in lane a and one
// multiply-add in every lane below (or above) it.  Dead directions give 0.
__device__ __forceinline__ double chol_substitute(const double (*L)[FIT_MAXK + 1], int k, unsigned dead, double g) {
  const int a = threadIdx.x & 31;
  const bool live = a < k && !((dead >> a) & 1);
  const double inv = live ? 1.0 / L[a][a] : 0.0;
  double s = live ? g : 0.0, y = 0.0;
  for (int c = 0; c < k; c++) {
    if (a == c) y = s * inv;
    const double yc = __shfl_sync(0xffffffffu, y, c);
    if (a > c) s -= L[a][c] * yc;
  }
  double t = y, d = 0.0;
  for (int c = k - 1; c >= 0; c--) {
    if (a == c) d = t * inv;
    const double dc = __shfl_sync(0xffffffffu, d, c);
    if (a < c) t -= L[c][a] * dc;
  }
  return live ? d : 0.0;
}

// the weights of scaled coordinates x (w_c = x_c 2^-e_c), and the sums of the pass that
// follows cleared
__device__ __forceinline__ void fit_publish(int m, int k, int M, double xa, const unsigned long long *cmax,
                                            const unsigned *amax, double *W, double *g, double *rr, double *bb) {
  const int a = threadIdx.x & 31;
  if (a < k)
    W[(int64_t)m * k + a] = cmax[a] ? ldexp(xa, -col_exp(cmax[a]) - acol_exp(amax[m * FIT_MAXK + a])) : 0.0;
  g[(int64_t)m * FIT_MAXK + a] = 0;
  if (a == 0) rr[m] = bb[m] = 0;
}

// 1/sqrt(d) to FP64 accuracy from the FP32 value by Newton's iteration (each step squares
// the relative error: 2^-22, 2^-43, below 2^-52), a fraction of the FP64 root and quotient on
// this GPU.  Pivots lie in FP32's normal range: above 1e-13 of the largest diagonal entry,
// which is at least 1/4 (scaled columns) and at most the row count.
__device__ __forceinline__ double rsqrt_newton(double d) {
  double y = (double)rsqrtf((float)d);
#pragma unroll
  for (int i = 0; i < 3; i++) {
    const double e = fma(-d * y, y, 1.0);
    y = fma(0.5 * y, e, y);
  }
  return y;
}

// ---- Cholesky of each model's Gram (one warp per model), FP64, and the first solution.
// Columns whose scale exponent marks them all-zero are replaced by identity rows
// (weight 0).  A pivot below tol * (largest diagonal) marks the model rank deficient
// and its direction is dropped likewise.  Lane a owns row a; after each column the lanes
// subtract its outer product from the columns to the right (independent multiply-adds, so
// the FP64 latency is paid per column, not per term; unrolled over all columns the code
// outgrows the instruction cache).
__global__ void __launch_bounds__(32) k_chol_solve(double *__restrict__ G, const double *__restrict__ rhs, int k, int M,
                                                   const unsigned long long *cmax, const unsigned *__restrict__ amax,
                                                   double *__restrict__ x, int *__restrict__ info,
                                                   double *__restrict__ diag_ratio, double *__restrict__ upd,
                                                   double *__restrict__ W, double *__restrict__ g,
                                                   double *__restrict__ rr, double *__restrict__ bb) {
  const int m = blockIdx.x;
  __shared__ double L[FIT_MAXK][FIT_MAXK + 1];
  const int a = threadIdx.x;
  double *Gm = G + (int64_t)m * FIT_MAXK * FIT_MAXK;
  for (int i = a; i < FIT_MAXK * FIT_MAXK; i += 32) {
    const int r = i / FIT_MAXK, c = i % FIT_MAXK;
    L[r][c] = r < k && c < k ? (r <= c ? Gm[r * FIT_MAXK + c] : Gm[c * FIT_MAXK + r]) : 0.0;   // the upper triangle, mirrored
  }
  const unsigned zero = __ballot_sync(0xffffffffu, a < k && cmax[a] == 0);
  unsigned dead = zero;
  __syncwarp();
  double dmax = a < k && !((dead >> a) & 1) ? L[a][a] : 0.0;
#pragma unroll
  for (int o = 16; o; o >>= 1) dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
  const double tol = dmax * 1e-13;
  int rank = 0;
  double pmin = 1e300, pmax = 0;
#pragma unroll 1
  for (int j = 0; j < k; j++) {
    const double d = L[j][j];
    __syncwarp();
    if (((dead >> j) & 1) || !(d > tol)) {
      dead |= 1u << j;
      if (a > j) L[a][j] = 0.0;
      if (a <= j) L[j][a] = a == j ? 1.0 : 0.0;
    } else {
      const double inv = rsqrt_newton(d), ljj = d * inv;
      rank++;
      pmin = fmin(pmin, ljj);
      pmax = fmax(pmax, ljj);
      const double l = a > j ? L[a][j] * inv : a == j ? ljj : 0.0;
      if (a >= j) L[a][j] = l;
      __syncwarp();
      for (int c0 = j + 1; c0 < k; c0 += 8) {   // eight columns at a time, their loads ahead of the stores
        double own[8], col[8];
#pragma unroll
        for (int i = 0; i < 8; i++) {
          const int c = min(c0 + i, FIT_MAXK - 1);
          own[i] = L[a][c];
          col[i] = L[c][j];
        }
#pragma unroll
        for (int i = 0; i < 8; i++)
          if (c0 + i < k && a >= c0 + i) L[a][c0 + i] = own[i] - l * col[i];
      }
    }
    __syncwarp();
  }
#pragma unroll 4
  for (int c = a + 1; c < FIT_MAXK; c++) L[a][c] = 0.0;
  __syncwarp();
  const double xa = chol_substitute(L, k, dead, a < k ? rhs[(int64_t)m * FIT_MAXK + a] : 0.0);
  x[(int64_t)m * FIT_MAXK + a] = xa;
  fit_publish(m, k, M, xa, cmax, amax, W, g, rr, bb);
  if (a == 0) {
    const int nz = __popc(zero);
    info[m * 4 + 0] = rank;
    info[m * 4 + 1] = nz;
    info[m * 4 + 2] = rank < k - nz ? 1 : 0;
    info[m * 4 + 3] = (int)dead;
    diag_ratio[m] = pmin > 0 ? (pmax / pmin) * (pmax / pmin) : 1e300;
    upd[m] = 0;
  }
  for (int i = a; i < FIT_MAXK * FIT_MAXK; i += 32) Gm[i] = L[i / FIT_MAXK][i % FIT_MAXK];   // L, for the refinement solves
}

// ---- g_m = U^T q_m  (float-float products and sums per warp, FP64 totals): bound by the
// twelve FP32 operations of each error-free product and compensated sum.  Grid (row chunks,
// groups of 16 models); a thread owns two columns and eight models (lanes 0-15 and 16-31 of a
// warp share the columns), so a row's 4 + 16 floats feed 16 products, and the eight warps
// take every eighth row.  Stages of 64 rows come through shared memory, two ahead (cp.async):
// read straight from L2, the loads' latency took half of the time (242 us for 200,000 x 32 x
// 64 with 16 warps per SM).
constexpr int ATQ_MODELS = 16, ATQ_ROWS = 64, ATQ_RING = 3;
struct AtqStage { float u[ATQ_ROWS][2][32], q[ATQ_ROWS][2][ATQ_MODELS]; };   // [hi, lo]
struct AtqSmem { AtqStage st[ATQ_RING]; float2 red[FIT_THREADS / 32][32][17]; };

__device__ __forceinline__ void cp_async16_zfill(void *dst, const void *src, bool in) {   // 16 bytes, zeros if !in
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(in ? 16 : 0));
}

__global__ void __launch_bounds__(FIT_THREADS, 2) k_atq(const float *__restrict__ Uh, const float *__restrict__ Ul, int ldu,
                                                        const float *__restrict__ Qh, const float *__restrict__ Ql, int ld,
                                                        int64_t R, int k, int M, int64_t rows_per_chunk,
                                                        const unsigned *__restrict__ amax, double *__restrict__ g) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  AtqSmem &S = *(AtqSmem *)smem_raw;
  auto &red = S.red;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c0 = 2 * (lane & 15), mg = 8 * (lane >> 4), mb = blockIdx.y * ATQ_MODELS;
  const int64_t r0 = (int64_t)blockIdx.x * rows_per_chunk;
  const int64_t r1 = min(R, r0 + rows_per_chunk);
  const int nst = (int)max((int64_t)0, (r1 - r0 + ATQ_ROWS - 1) / ATQ_ROWS);
  auto fetch = [&](int s) {   // stage s on its way; rows and models that do not exist are zero
    if (s < nst) {
      AtqStage &T = S.st[s % ATQ_RING];
      const int64_t rb = r0 + (int64_t)s * ATQ_ROWS;
#pragma unroll
      for (int i = 0; i < ATQ_ROWS * 16 / FIT_THREADS; i++) {
        const int x = tid + i * FIT_THREADS, row = x >> 4, h = (x >> 3) & 1, c = (x & 7) * 4;
        const bool in = rb + row < r1 && c < ldu;
        cp_async16_zfill(&T.u[row][h][c], (h ? Ul : Uh) + (in ? (rb + row) * ldu + c : 0), in);
      }
#pragma unroll
      for (int i = 0; i < ATQ_ROWS * 8 / FIT_THREADS; i++) {
        const int x = tid + i * FIT_THREADS, row = x >> 3, h = (x >> 2) & 1, m = (x & 3) * 4;
        const bool in = rb + row < r1 && mb + m < ld;
        cp_async16_zfill(&T.q[row][h][m], (h ? Ql : Qh) + (in ? (rb + row) * ld + mb + m : 0), in);
      }
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  fetch(0);
  fetch(1);
  // this thread's sums so far; a compensated sum's error grows with the square of its length,
  // so runs of 64 rows (8 stages) are added up in float-float
#pragma unroll
  for (int j = 0; j < 16; j++) red[warp][lane][j] = make_float2(0.f, 0.f);
  float s[16], c[16];
#pragma unroll
  for (int j = 0; j < 16; j++) s[j] = c[j] = 0.f;
  for (int st = 0; st < nst; st++) {
    asm volatile("cp.async.wait_group 1;\n" ::);
    __syncthreads();   // stage st is complete, and the buffer of stage st - 1 is free
    fetch(st + 2);
    const AtqStage &T = S.st[st % ATQ_RING];
#pragma unroll 2
    for (int row = warp; row < ATQ_ROWS; row += FIT_THREADS / 32) {
      const float2 uh = *(const float2 *)&T.u[row][0][c0], ul = *(const float2 *)&T.u[row][1][c0];
      const float4 h0 = *(const float4 *)&T.q[row][0][mg], h1 = *(const float4 *)&T.q[row][0][mg + 4];
      const float4 l0 = *(const float4 *)&T.q[row][1][mg], l1 = *(const float4 *)&T.q[row][1][mg + 4];
      const float qh[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
      const float ql[8] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w};
#pragma unroll
      for (int j = 0; j < 8; j++) {
        ff_acc(s[2 * j], c[2 * j], ff_mul(uh.x, ul.x, qh[j], ql[j]));
        ff_acc(s[2 * j + 1], c[2 * j + 1], ff_mul(uh.y, ul.y, qh[j], ql[j]));
      }
    }
    if ((st & 7) == 7 || st + 1 == nst) {
#pragma unroll
      for (int j = 0; j < 16; j++) {
        float2 t = red[warp][lane][j];
        ff_acc(t.x, t.y, make_float2(s[j], c[j]));
        red[warp][lane][j] = t;
        s[j] = c[j] = 0.f;
      }
    }
  }
  __syncthreads();
  // the eight warps' sums of 32 columns x 16 models, added up no worse than in FP64
  for (int o = tid; o < 32 * 16; o += FIT_THREADS) {
    const int l = o >> 4, j = o & 15;
    const int col = 2 * (l & 15) + (j & 1), m = mb + 8 * (l >> 4) + (j >> 1);
    if (m < M && col < k) {
      float ts = 0.f, tc = 0.f, td = 0.f;
#pragma unroll
      for (int w = 0; w < FIT_THREADS / 32; w++) ff_acc3(ts, tc, td, red[w][l][j]);
      atomicAdd(&g[(int64_t)m * FIT_MAXK + col],
                ldexp(((double)ts + (double)tc) + (double)td, -acol_exp(amax[m * FIT_MAXK + col])));
    }
  }
}

// ---- x += L^-T L^-1 g per model (one warp each); records |d| / |x|, and publishes the
// weights for the next residual pass.
__global__ void __launch_bounds__(32) k_refine_update(const double *__restrict__ Lall, double *__restrict__ g, int k, int M,
                                                      const int *__restrict__ info, const unsigned long long *cmax,
                                                      const unsigned *__restrict__ amax, double *__restrict__ x,
                                                      double *__restrict__ upd, double *__restrict__ W,
                                                      double *__restrict__ rr, double *__restrict__ bb) {
  const int m = blockIdx.x, a = threadIdx.x;
  __shared__ double L[FIT_MAXK][FIT_MAXK + 1];
  const double *Lm = Lall + (int64_t)m * FIT_MAXK * FIT_MAXK;
#pragma unroll 8
  for (int r = 0; r < FIT_MAXK; r++) L[r][a] = Lm[r * FIT_MAXK + a];
  __syncwarp();
  const double d = chol_substitute(L, k, (unsigned)info[m * 4 + 3], a < k ? g[(int64_t)m * FIT_MAXK + a] : 0.0);
  const double xa = x[(int64_t)m * FIT_MAXK + a] + d;
  x[(int64_t)m * FIT_MAXK + a] = xa;
  fit_publish(m, k, M, xa, cmax, amax, W, g, rr, bb);
  double dn = d * d, xn = xa * xa;
  for (int o = 16; o; o >>= 1) {
    dn += __shfl_xor_sync(0xffffffffu, dn, o);
    xn += __shfl_xor_sync(0xffffffffu, xn, o);
  }
  if (a == 0) upd[m] = xn > 0 ? sqrt(dn / xn) : 0.0;
}

// ------------------------------------------------------------------------------------ host side

// row lengths of the row factors and residuals, and of the scaled counts: whole 16-byte pieces
static int fit_ld(int M) { return (M + 3) & ~3; }
static int fit_ldu(int k) { return (k + 3) & ~3; }

size_t fit_scratch_bytes(int64_t R, int k, int M) {
  size_t b = 0;
  b += 256;                                        // cmax
  b += (size_t)M * (FIT_MAXK + 1) * 4;             // amax, rmax
  b += (size_t)R * fit_ldu(k) * 8;                 // Uh, Ul
  b += (size_t)R * fit_ld(M) * 8 * 2;              // row factors; beta, then Q (hi and lo)
  b += (size_t)M * FIT_MAXK * FIT_MAXK * 8;        // G / L
  b += (size_t)M * FIT_MAXK * 8 * 3;               // rhs, x, g
  b += (size_t)M * FIT_REPORT_BYTES;               // info, ratio, upd, rr, bb
  return b + 32 * 256;                             // every carve rounds up to 256 bytes
}

static char *carve(char *&p, size_t bytes) {
  char *r = p;
  p += (bytes + 255) & ~(size_t)255;
  return r;
}

cudaError_t launch_fit(const int64_t *F, int64_t R, int k, const double *T, int M, int objective, int gram,
                       int steps, void *scratch, double *W_out, void *h_report, int *status, cudaStream_t st) {
  const int ld = fit_ld(M), ldu = fit_ldu(k);
  char *p = (char *)scratch;
  // cleared together: cmax, amax, rmax, G, rhs
  char *zero = p;
  unsigned long long *cmax = (unsigned long long *)carve(p, 256);
  unsigned *amax = (unsigned *)carve(p, (size_t)M * FIT_MAXK * 4);
  unsigned *rmax = (unsigned *)carve(p, (size_t)M * 4);
  double *G = (double *)carve(p, (size_t)M * FIT_MAXK * FIT_MAXK * 8);
  double *rhs = (double *)carve(p, (size_t)M * FIT_MAXK * 8);
  const size_t zero_bytes = (size_t)(p - zero);
  float *U = (float *)carve(p, (size_t)R * ldu * 4);
  float *Ul = (float *)carve(p, (size_t)R * ldu * 4);
  float *rfh = (float *)carve(p, (size_t)R * ld * 4);
  float *rfl = (float *)carve(p, (size_t)R * ld * 4);
  float *bh = (float *)carve(p, (size_t)R * ld * 4);
  float *bl = (float *)carve(p, (size_t)R * ld * 4);
  float *Qh = bh, *Ql = bl;   // the residuals: beta has been read when the first are written
  double *x = (double *)carve(p, (size_t)M * FIT_MAXK * 8);
  double *g = (double *)carve(p, (size_t)M * FIT_MAXK * 8);
  void *report = carve(p, (size_t)M * FIT_REPORT_BYTES);
  const FitHost rep = fit_report(report, M);
  cudaError_t e;
  if ((e = cudaMemsetAsync(zero, 0, zero_bytes, st)) != cudaSuccess) return e;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const bool relative = objective == PM_FIT_RELATIVE;
  const bool beta = gram == 0 || !relative;   // else beta is 1 and the right-hand side takes the row factors
  k_colmax<<<sms * 4, 256, 0, st>>>(F, R, k, cmax);
  k_scale<<<sms * 8, 256, 0, st>>>(F, R, k, ldu, cmax, U, Ul);
  k_rowfac<<<(int)std::min<int64_t>(sms * 4, (R + AM_ROWS - 1) / AM_ROWS), FIT_THREADS, 0, st>>>(
      U, ldu, T, ld, R, k, M, objective, rfh, rfl, beta ? bh : nullptr, beta ? bl : nullptr, amax, rmax, status);
  const int groups = (M + ATQ_MODELS - 1) / ATQ_MODELS;
  // one wave of two CTAs per SM: the sums are issue-bound, and a partial second wave idles
  const int achunks = (int)std::max<int64_t>(1, std::min<int64_t>(2 * sms / groups, (R + ATQ_ROWS - 1) / ATQ_ROWS));
  const int64_t arpc = (R + achunks - 1) / achunks;
  if ((e = cudaFuncSetAttribute(k_atq, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(AtqSmem))) != cudaSuccess) return e;
  if (gram != 0) {
    // the Gram on the tensor cores; the right-hand side A^T b = U^T (rowfactor b) with the
    // float-float product kernel
    e = gram == 2 ? launch_gram_tc(U, Ul, ldu, rfh, rfl, ld, R, k, M, amax, G, sms, status, st)
                  : launch_gram_pairs(U, ldu, rfh, rfl, ld, R, k, M, amax, rmax, G, sms, status, st);
    if (e != cudaSuccess) return e;
    k_atq<<<dim3(achunks, groups), FIT_THREADS, sizeof(AtqSmem), st>>>(U, Ul, ldu, relative ? rfh : bh, relative ? rfl : bl, ld, R, k, M, arpc,
                                                         amax, rhs);
  } else {
    const int chunks = (int)std::max<int64_t>(1, std::min<int64_t>(4 * sms / std::max(1, M) + 1, (R + 255) / 256));
    k_gram<<<dim3(chunks, M), FIT_THREADS, 0, st>>>(U, Ul, ldu, rfh, rfl, bh, bl, ld, R, k, M, (R + chunks - 1) / chunks, amax, G, rhs);
  }
  k_chol_solve<<<M, 32, 0, st>>>(G, rhs, k, M, cmax, amax, x, rep.info, rep.ratio, rep.upd, W_out, g, rep.rr, rep.bb);
  FitResidual res;
  res.T = T;
  res.rfh = rfh;
  res.rfl = rfl;
  res.Qh = Qh;
  res.Ql = Ql;
  res.rr = rep.rr;
  res.bb = rep.bb;
  res.ld = ld;
  res.relative = relative;
  for (int it = 0; it < steps; it++) {
    if ((e = launch_fit_residual(F, R, k, W_out, M, res, false, status, sms, st)) != cudaSuccess) return e;
    k_atq<<<dim3(achunks, groups), FIT_THREADS, sizeof(AtqSmem), st>>>(U, Ul, ldu, Qh, Ql, ld, R, k, M, arpc, amax, g);
    k_refine_update<<<M, 32, 0, st>>>(G, g, k, M, rep.info, cmax, amax, x, rep.upd, W_out, rep.rr, rep.bb);
  }
  // the final residual, for the report
  if ((e = launch_fit_residual(F, R, k, W_out, M, res, true, status, sms, st)) != cudaSuccess) return e;
  if ((e = cudaMemcpyAsync(h_report, report, (size_t)M * FIT_REPORT_BYTES, cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace pmd

// Test hook: bytes of context scratch that a fit takes.
extern "C" size_t pmx_fit_scratch(int64_t R, int k, int M) { return pmd::fit_scratch_bytes(R, k, M); }

// Test hook: g [M][32] += U^T q of one row chunk (columns unscaled).  Uh, Ul [R][32]; Qh, Ql
// [R][16]; M <= 16; amax [M][32]: 1.0f each.
extern "C" int pmx_atq(const float *Uh, const float *Ul, const float *Qh, const float *Ql, int64_t R, int k, int M,
                       const unsigned *amax, double *g, void *stream) {
  if (R < 1 || k < 1 || k > 32 || M < 1 || M > 16) return PM_ERR_INVALID_ARG;
  if (cudaFuncSetAttribute(pmd::k_atq, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(pmd::AtqSmem)) != cudaSuccess)
    return PM_ERR_CUDA;
  pmd::k_atq<<<dim3(1, 1), pmd::FIT_THREADS, sizeof(pmd::AtqSmem), (cudaStream_t)stream>>>(Uh, Ul, 32, Qh, Ql, 16, R, k, M, R, amax, g);
  return cudaGetLastError() == cudaSuccess ? PM_OK : PM_ERR_CUDA;
}
