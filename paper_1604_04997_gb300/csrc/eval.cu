// K1: materialised count evaluation (pm_eval_counts), Sec. 2's re-evaluation of the
//     properties p_i(n) of compiled tables at many parameter points.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "eval_common.cuh"
#include "kernels.h"

namespace pmd {

// ------------------------------------------------------------------------------------ K1

constexpr int K1_THREADS = 128;

// One block: 128 points of one distinct table, one thread per point; the rows are staged in
// shared memory and written to every output position that names the table, as contiguous
// 16-byte pieces (the counts of a tuning space repeat: 2,656 matmul variants have 32 distinct
// tables).  Bound by the HBM writes where tables repeat (2,656 tables x 1,024 points, 696 MB:
// 201 us with every position evaluated, 109 now, 6.4 TB/s); else by the evaluation's latency,
// at the warps that the staged rows and slots (57 KB per block, and the largest table's words)
// leave room for.
template <int K>
__global__ void __launch_bounds__(K1_THREADS) k_eval_counts(const uint32_t *__restrict__ arena,
                                                           const int4 *__restrict__ items,
                                                           const int32_t *__restrict__ members, int table_words,
                                                           const int64_t *__restrict__ points, int64_t n_points,
                                                           int P, int64_t *__restrict__ out, int *status) {
  extern __shared__ __align__(16) uint8_t smem[];
  uint32_t *sT = (uint32_t *)smem;                                   // the table
  int64_t *stage = (int64_t *)(smem + table_words * 4);              // [threads][K+1]
  int64_t *slots = stage + K1_THREADS * (K + 1);                     // [24][threads]
  const int tid = threadIdx.x;
  const int4 item = items[blockIdx.y];
  const uint32_t *gT = arena + ((int64_t)item.w << 32 | (uint32_t)item.x);
  const int64_t first = members[item.y];   // read here, so that its latency is the header's
  const int words = (int)gT[pmt::H_WORDS];
  if (gT[pmt::H_MAGIC] != pmt::MAGIC || words > table_words || (int)gT[pmt::H_K] != K) {
    if (tid == 0) atomicOr(status, ST_BAD_TABLE);
    return;
  }
  for (int i = tid; i < words / 4; i += K1_THREADS) ((uint4 *)sT)[i] = ((const uint4 *)gT)[i];
  int64_t *row = stage + tid * (K + 1);
#pragma unroll
  for (int c = 0; c < K; c++) row[c] = 0;
  __syncthreads();
  const int64_t p0 = (int64_t)blockIdx.x * K1_THREADS;
  const int64_t p = p0 + tid;
  if (p < n_points) {
    int32_t n[4];
    if (!point_in_box(sT, points + p * P, P, n)) {
      atomicOr(status, ST_OUT_OF_BOX);
    } else {
      bool ok = eval_table(
          sT, n, slots + tid, K1_THREADS,
          [&](int col, int64_t v) { if (col < K) row[col] = v; },
          [&](int col, int64_t v) { if (col < K) row[col] = v; });
      if (!ok) {
        atomicOr(status, ST_BAD_TABLE);
#pragma unroll
        for (int c = 0; c < K; c++) row[c] = 0;
      }
    }
  }
  __syncthreads();
  // Streaming stores: the rows are not reread.  A table of one position is written in plain
  // order, 8 bytes a lane (no bank conflict and no member to look up: 64 distinct tables x
  // 20,000 points, 32 columns, 87 us; through the loop over positions below 113, and with 16
  // bytes a lane 90); a table of several reads a piece of 16 bytes once for all of them.
  const int nvalid = (int)min((int64_t)K1_THREADS, n_points - p0);
  constexpr int H = K / 2;
  if (item.z == 1) {
    int64_t *dst = out + (first * n_points + p0) * K;
    for (int i = tid; i < nvalid * K; i += K1_THREADS) {
      const int r = i / K, c = i - r * K;
      __stcs(dst + i, stage[r * (K + 1) + c]);
    }
  } else if (((uintptr_t)out & 15) == 0) {
    for (int i = tid; i < nvalid * H; i += K1_THREADS) {
      const int r = i / H, c2 = i - r * H;
      const longlong2 v = make_longlong2(stage[r * (K + 1) + 2 * c2], stage[r * (K + 1) + 2 * c2 + 1]);
      for (int m = 0; m < item.z; m++)
        __stcs((longlong2 *)(out + ((int64_t)members[item.y + m] * n_points + p0) * K) + i, v);
    }
  } else {
    for (int i = tid; i < nvalid * K; i += K1_THREADS) {
      const int r = i / K, c = i - r * K;
      for (int m = 0; m < item.z; m++)
        __stcs(out + ((int64_t)members[item.y + m] * n_points + p0) * K + i, stage[r * (K + 1) + c]);
    }
  }
}

cudaError_t launch_eval_counts(const uint32_t *arena, const int32_t *items, const int32_t *members, int n_items,
                               int max_words, const int64_t *points, int64_t n_points, int P, int K, int64_t *out,
                               int *status, cudaStream_t st) {
  if (n_points == 0 || n_items == 0) return cudaSuccess;
  const dim3 grid((unsigned)((n_points + K1_THREADS - 1) / K1_THREADS), (unsigned)n_items);
  const int words = (max_words + 3) & ~3;
  const size_t sm = (size_t)words * 4 + (size_t)K1_THREADS * (K + 1) * 8 + (size_t)pmt::MAX_SLOTS * K1_THREADS * 8;
  auto launch = [&](auto kernel) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    kernel<<<grid, K1_THREADS, sm, st>>>(arena, (const int4 *)items, members, words, points, n_points, P, out, status);
    return cudaGetLastError();
  };
  if (K == 32) return launch(k_eval_counts<32>);
  if (K == 12) return launch(k_eval_counts<12>);
  return cudaErrorInvalidValue;
}

}  // namespace pmd
