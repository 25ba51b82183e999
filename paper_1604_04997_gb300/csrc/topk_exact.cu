// Top-k rows per (group, model) over materialised features (configuration selection,
// Sec. 6.1) for more than a few models, on the exact tensor-core prediction (exact_tc.cuh):
// the times are those of k_predict_exact, bit for bit.
//
// One CTA of 16 working warps and an issuing warp per SM; the CTA takes units (up to
// topk_chunk positions of one group) in turn, in tiles of 128 positions.  Each model has one
// sorted list and a buffer of TX_BUF candidates in shared memory.  A time that is not above
// the list's last entry reserves a slot of its model's buffer; the warp that fills the buffer
// merges it into the list (topk_list.cuh) and empties it, and warps that find it full wait for
// that.  The warps meet only where a unit ends.  Kept in step by barriers around the buffers
// they could not hide each other's latencies (0.84 ms for 1e6 x 32 x 64, against 0.32 for the
// times alone), and merging each candidate as it came cost 400 instructions for one or two
// (1.19 ms).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "exact_tc.cuh"
#include "kernels.h"
#include "pm.h"
#include "topk_list.cuh"

namespace pmd {

constexpr int TX_BUF = 16;           // buffered candidates per model
constexpr int TX_TRIES = 1 << 22;    // polls of a buffer before giving up

// The tiles of a CTA, in order: units blockIdx.x, blockIdx.x + gridDim.x, .., each cut into
// 128 positions (a unit without positions is one empty tile).
struct TxCursor {
  int64_t p, p0, p1;   // this tile; its unit
  int32_t u, g, part, pad;
  __device__ void open(const TopkUnit *units, int n_units) {
    if (u < n_units) {
      const TopkUnit U = units[u];
      p = p0 = U.p0;
      p1 = U.p1;
      g = U.g;
      part = U.part;
    }
  }
  __device__ void start(const TopkUnit *units, int n_units) {
    p = p0 = p1 = 0;
    g = part = pad = 0;
    u = blockIdx.x;
    open(units, n_units);
  }
  __device__ bool more(int n_units) const { return u < n_units; }
  __device__ bool last() const { return p + XP_ROWS >= p1; }   // of its unit
  __device__ void next(const TopkUnit *units, int n_units) {
    if (!more(n_units)) return;
    if (last()) {
      u += gridDim.x;
      open(units, n_units);
    } else {
      p += XP_ROWS;
    }
  }
};

constexpr int TX_ROWRING = 8;
struct TxSmem {                      // beyond the operands of XpGeom
  int64_t lt[XP_MAXM][TOPK_MAX];     // sorted lists: times (as bits), rows
  int64_t lr[XP_MAXM][TOPK_MAX];
  int64_t thr[XP_MAXM];              // time_order of the list's last entry, and its row
  int64_t thr_row[XP_MAXM];
  int64_t ct[XP_MAXM][TX_BUF];       // candidates: times, positions within the unit
  int32_t cp[XP_MAXM][TX_BUF];
  int32_t cnt[XP_MAXM], wr[XP_MAXM]; // slots reserved and written
  uint8_t live[TX_ROWRING][XP_ROWS]; // positions of the tiles in flight (by tile modulo 8) that have a row
  TxCursor cursor[2][XP_WARPS + 1];  // per warp: its tile, and the tile it loads for
};

// For tests, with short waits: HELD: the issuing warp leaves after its first tile
// (pmx_topk_held); UNWRITTEN: every buffer has a slot that is never counted as written
// (pmx_topk_unwritten).
enum TxTest { TX_NORMAL, TX_HELD, TX_UNWRITTEN };
template <class G, TxTest TEST = TX_NORMAL>
__global__ void __launch_bounds__(XP_THREADS, 1) k_topk_exact(const int64_t *__restrict__ F, int64_t R, int k,
                                                              const double *__restrict__ W, int M,
                                                              const int64_t *__restrict__ rows,
                                                              const TopkUnit *__restrict__ units, int n_units, int topk,
                                                              double *__restrict__ part_t, int64_t *__restrict__ part_r,
                                                              int64_t *__restrict__ top_idx, double *__restrict__ top_t,
                                                              int *status, uint32_t m256) {
  constexpr unsigned long long LIMIT = TEST != TX_NORMAL ? XP_HELD_NS : MBAR_WAIT_NS;
  constexpr int TRIES = TEST != TX_NORMAL ? 1 << 10 : TX_TRIES;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = smem_raw + ((128u - (xp_saddr(smem_raw) & 127u)) & 127u);
  TxSmem &X = *(TxSmem *)(smem + G::SMEM - 128);
  __shared__ __align__(8) uint64_t full[XP_RING], empty[XP_RING], digits[2];
  __shared__ __align__(16) int s_nd[4][XP_WARPS];
  __shared__ uint32_t tmem_base;
  __shared__ int s_E[XP_MAXM];
  __shared__ volatile int s_abort;
  uint8_t *sA = smem, *sB = smem + G::OFF_B;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int quarter = warp & 3, slice = warp >> 2;
  const bool vec = (k & 1) == 0 && ((uintptr_t)F & 15) == 0;
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
  const int64_t INF = 0x7ff0000000000000ll;
  auto reset = [&](int m) {   // an empty list for model m (a warp)
    if (lane < TOPK_MAX) {
      X.lt[m][lane] = INF;
      X.lr[m][lane] = INT64_MAX;
    }
    if (lane == 0) {
      X.thr[m] = INF;
      X.thr_row[m] = INT64_MAX;
      X.cnt[m] = 0;
      X.wr[m] = TEST == TX_UNWRITTEN ? -1 : 0;
    }
  };
  if (warp < XP_WARPS)
    for (int m = warp; m < XP_MAXM; m += XP_WARPS) reset(m);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(xp_saddr(&tmem_base)),
                 "r"(G::TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  xp_load_weights<G>(W, M, k, (double *)sA, sB, s_E);
  asm volatile("fence.proxy.async.shared::cta;\n" ::);
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();   // the staged weights in sA have been read
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
  const uint32_t tmem = xp_uniform(tmem_base), s0 = xp_uniform(xp_saddr(smem));
  uint32_t seq = 0, it = 0;
  bool ok = true;
  // a warp's cursors, in shared memory: held in registers next to the limbs they make the
  // kernel spill, and shared memory leaves L1 too little room for that
  TxCursor &cur = X.cursor[0][warp], &ahead = X.cursor[1][warp];
  if (lane == 0) {
    cur.start(units, n_units);
    ahead.start(units, n_units);
  }
  __syncwarp();
  auto advance = [&](TxCursor &c) {
    __syncwarp();
    if (lane == 0) c.next(units, n_units);
    __syncwarp();
  };
  if (warp == XP_WARPS) {
    // this warp issues, ahead of the working warps as far as digits and columns allow
    for (; cur.more(n_units) && ok && !(TEST == TX_HELD && it); advance(cur), it++) {
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
    if (!ok) xp_drain(full, XP_RING, seq);
    __syncwarp();
  } else {
    const bool active = slice * 8 < G::NB;   // this warp has models
    const int c0 = slice * 8 + 2 * (lane & 3);
    const uint32_t tread = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(slice * 8);
    auto meet = [&]() { asm volatile("bar.sync 1, %0;\n" ::"n"(32 * XP_WARPS) : "memory"); };   // all working warps
    // find the rows of this warp's share of the n-th tile (at cursor ahead), and prefetch
    // them into L2, 128 bytes per instruction
    int64_t nrow = -1;
    auto locate = [&](uint32_t n) {
      nrow = -1;
      if (row < XP_ROWS) {
        const int64_t pos = ahead.p + row;
        int64_t r = -1;
        if (ahead.more(n_units) && pos < ahead.p1) {
          r = rows ? rows[pos] : pos;
          if (r < 0 || r >= R) {
            if (xp_kg<G>() == 0) atomicOr(status, ST_BAD_ROW);
            r = -1;
          }
        }
        if (xp_kg<G>() == 0) X.live[n % TX_ROWRING][row] = r >= 0;
        nrow = r;
        if (r >= 0 && (xp_kg<G>() & 1) == 0 && xp_kg<G>() * 64 < k * 8)
          asm volatile("prefetch.global.L2 [%0];\n" ::"l"((const char *)(F + r * k) + xp_kg<G>() * 64));
      }
      advance(ahead);
    };
    // load this thread's share of the n-th tile and store its digits
    auto feed = [&](uint32_t n) {
      int64_t v[8];
#pragma unroll
      for (int i = 0; i < 8; i++) v[i] = 0;
      if (nrow >= 0) xp_load_row<G>(F + nrow * k, k, vec, v);
      xp_store_digits<G>(v, sA + (n & 1) * G::A_BUF, s_nd[n & 3]);
      asm volatile("fence.proxy.async.shared::cta;\n" ::);
      __syncwarp();
      if (lane == 0) xp_arrive(xp_saddr(&digits[n & 1]));
    };
    // whether the time o (as ordered bits) of position pos may be among model m's topk
    auto below = [&](int64_t o, int64_t pos, int m) {
      const int64_t th = *(volatile int64_t *)&X.thr[m];
      if (o != th) return o < th;
      return (rows ? rows[pos] : pos) < *(volatile int64_t *)&X.thr_row[m];
    };
    // model m's n candidates into its list (a warp; all n are written)
    auto merge = [&](int m, int n) {
      double t = TK_INF, lt = TK_INF;
      int64_t r = INT64_MAX, lr = INT64_MAX;
      if (lane < n) {
        t = __longlong_as_double(*(volatile int64_t *)&X.ct[m][lane]);
        const int64_t pos = cur.p0 + *(volatile int32_t *)&X.cp[m][lane];
        r = rows ? rows[pos] : pos;
      }
      if (lane < TOPK_MAX) {
        lt = __longlong_as_double(*(volatile int64_t *)&X.lt[m][lane]);
        lr = *(volatile int64_t *)&X.lr[m][lane];
      }
      warp_list_merge(lt, lr, t, r, lane < n, topk, lane);
      if (lane < TOPK_MAX) {
        X.lt[m][lane] = __double_as_longlong(lt);
        X.lr[m][lane] = lr;
      }
      const int64_t th = time_order(__shfl_sync(0xffffffffu, lt, topk - 1)), thr = __shfl_sync(0xffffffffu, lr, topk - 1);
      __threadfence_block();
      __syncwarp();
      if (lane == 0) {
        *(volatile int64_t *)&X.thr_row[m] = thr;   // the row first: who reads the time and then the row (above)
        __threadfence_block();                      // never compares with a looser pair's row
        *(volatile int64_t *)&X.thr[m] = th;
        *(volatile int32_t *)&X.wr[m] = 0;
        __threadfence_block();
        atomicExch(&X.cnt[m], 0);   // the buffer is open again
      }
    };
    auto wait = [&]() { return xp_wait(xp_saddr(&full[seq % XP_RING]), (seq / XP_RING) & 1, &s_abort, LIMIT); };
    auto done = [&]() {   // this warp has read its share of a group
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
      __syncwarp();
      if (lane == 0) xp_arrive(xp_saddr(&empty[seq % XP_RING]));
      seq++;
    };
    // one (tile, pass): the exact sums, the times, the candidates.  After a wait that ran out
    // the warp only keeps the order of the meetings.
    auto pass = [&](int ps) {
      uint32_t limb[4][8], cy[8];
      ok = ok && wait();
      int ng = 4;
      if (ok) {
        ng = xp_groups(xp_tile_digits(s_nd[it & 3]));
        if (active) xp_limb<G, 0>(m256, tread + (seq % XP_RING) * G::RANGE, limb[0], cy);
        done();
        ok = wait();
      }
      if (ok) {
        if (active) xp_limb<G, 1>(m256, tread + (seq % XP_RING) * G::RANGE, limb[1], cy);
        done();
      }
      if (ng > 2) {
        if (ok) ok = wait();
        if (ok) {
          if (active) xp_limb<G, 2>(m256, tread + (seq % XP_RING) * G::RANGE, limb[2], cy);
          done();
        }
      } else {
#pragma unroll
        for (int o = 0; o < 8; o++) {
          limb[2][o] = cy[o] - XP_HI;
          cy[o] = (uint32_t)((int32_t)limb[2][o] >> 31) + XP_HI;
        }
      }
      if (ng > 3) {
        if (ok) ok = wait();
        if (ok) {
          if (active) xp_limb<G, 3>(m256, tread + (seq % XP_RING) * G::RANGE, limb[3], cy);
          done();
        }
      } else {
#pragma unroll
        for (int o = 0; o < 8; o++) limb[3][o] = cy[o] - XP_HI;
      }
      if (!ok || !active) return;
      const int m = 32 * ps + c0;
      int64_t t[8];           // row quarter 32 + lane / 4 + 8 i, model m + e: 2 i + e
      uint32_t pending = 0;   // bit 2 i + e: a candidate
      const int x0[2] = {1150 - s_E[m], 1150 - s_E[m + 1]};
      const bool wide = min(x0[0], x0[1]) < XP_XMIN || max(x0[0], x0[1]) > XP_XMAX;
      const int64_t th[2] = {*(volatile int64_t *)&X.thr[m], *(volatile int64_t *)&X.thr[m + 1]};
      const uint8_t *tile_live = X.live[it % TX_ROWRING] + quarter * 32 + (lane >> 2);
      const int32_t off = (int32_t)(cur.p - cur.p0) + quarter * 32 + (lane >> 2);   // of this thread's first row in the unit
      auto emit = [&](auto neg) {
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const bool live = tile_live[8 * i];
          double x[2];
          bool bad = wide;
#pragma unroll
          for (int e = 0; e < 2; e++)
            x[e] = xp_value<decltype(neg)::value>(limb[0][2 * i + e], limb[1][2 * i + e], limb[2][2 * i + e], limb[3][2 * i + e], x0[e], bad);
          if (bad) {
#pragma unroll
            for (int e = 0; e < 2; e++)
              x[e] = xp_value_rare(limb[0][2 * i + e], limb[1][2 * i + e], limb[2][2 * i + e], limb[3][2 * i + e], 1150 - x0[e]);
          }
#pragma unroll
          for (int e = 0; e < 2; e++) {
            t[2 * i + e] = __double_as_longlong(x[e]);
            if (live && m + e < M && time_order(x[e]) <= th[e]) pending |= 1u << (2 * i + e);
          }
        }
      };
      uint32_t sg = 0;
#pragma unroll
      for (int o = 0; o < 8; o++) sg |= limb[3][o];
      if (__any_sync(0xffffffffu, (int32_t)sg < 0)) emit(std::true_type{});
      else emit(std::false_type{});
      // offer the candidates; the warp that fills a buffer merges it
      for (int tries = 0; __any_sync(0xffffffffu, pending); tries++) {
        if (tries == TRIES) s_abort = 1;   // never: a full buffer's owner empties it
        if (__any_sync(0xffffffffu, s_abort)) {
          ok = false;
          break;
        }
        // one candidate of every lane that has any (unrolled over the eight, the code outgrows
        // the instruction cache)
        int mm = 0;
        bool filled = false;
        if (pending) {
          const int o = __ffs(pending) - 1;
          mm = m + (o & 1);
          int64_t x = t[0];
#pragma unroll
          for (int n = 1; n < 8; n++) x = o == n ? t[n] : x;
          const int32_t at = off + 8 * (o >> 1);
          bool gone = !below(time_order(__longlong_as_double(x)), cur.p0 + at, mm);   // tightened since, or a tie with a larger row
          if (!gone && *(volatile int32_t *)&X.cnt[mm] < TX_BUF) {
            const int slot = atomicAdd(&X.cnt[mm], 1);
            if (slot < TX_BUF) {
              *(volatile int64_t *)&X.ct[mm][slot] = x;
              *(volatile int32_t *)&X.cp[mm][slot] = at;
              __threadfence_block();
              atomicAdd(&X.wr[mm], 1);
              gone = true;
              filled = slot == TX_BUF - 1;
            }
          }
          if (gone) pending &= pending - 1;
        }
        unsigned who;
        while ((who = __ballot_sync(0xffffffffu, filled)) != 0) {
          const int from = __ffs(who) - 1;
          const int full_m = __shfl_sync(0xffffffffu, mm, from);
          if (lane == from) filled = false;
          int polls = 0;   // the other writers of the buffer are between reserving and writing
          while (*(volatile int32_t *)&X.wr[full_m] < TX_BUF && ++polls < TRIES) {}
          if (__any_sync(0xffffffffu, polls == TRIES)) {   // never; a buffer with unwritten slots is not merged
            s_abort = 1;
            break;
          }
          __threadfence_block();
          __syncwarp();
          merge(full_m, TX_BUF);
        }
      }
    };
    locate(0);
    feed(0);
    locate(1);
    feed(1);
    for (; cur.more(n_units); it++) {
      locate(it + 2);
#pragma unroll 1
      for (int ps = 0; ps < G::PASSES; ps++) pass(ps);
      const bool end = cur.last();
      if (end) {
        meet();   // every candidate of the unit is in a buffer or merged
        for (int m = warp; m < M; m += XP_WARPS) {
          merge(m, min(X.cnt[m], TX_BUF));
          __syncwarp();
          if (lane < topk) {
            const int64_t r = X.lr[m][lane];
            const double t = __longlong_as_double(X.lt[m][lane]);
            if (cur.part < 0) {
              const int64_t o = ((int64_t)cur.g * M + m) * topk + lane;
              top_idx[o] = r == INT64_MAX ? -1 : r;
              top_t[o] = t;
            } else {
              const int64_t o = ((int64_t)cur.part * M + m) * topk + lane;
              part_t[o] = t;
              part_r[o] = r;
            }
          }
          __syncwarp();
          reset(m);
        }
      }
      // every MMA of this tile is complete: its operand buffer takes the tile after the next
      if (ok) feed(it + 2);
      advance(cur);
      if (end) meet();   // the lists are reset
    }
  }
  xp_finish(&s_abort, status, warp == XP_WARPS, full, XP_RING, seq);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(G::TMEM_COLS));
}

cudaError_t launch_topk_exact(const int64_t *F, int64_t R, int k, const double *W, int M, const int64_t *rows,
                              const TopkUnit *units, int n_units, int topk, double *part_t, int64_t *part_r,
                              int64_t *top_idx, double *top_t, int *status, int sms, cudaStream_t st) {
  return xp_dispatch(k, M, [&](auto g) {
    using G = decltype(g);
    constexpr size_t smem = G::SMEM + sizeof(TxSmem);
    static_assert(smem <= 227 * 1024 - 1024, "one CTA per SM");
    cudaError_t e = cudaFuncSetAttribute(k_topk_exact<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_topk_exact<G><<<std::min(n_units, sms), XP_THREADS, smem, st>>>(F, R, k, W, M, rows, units, n_units, topk, part_t, part_r,
                                                                   top_idx, top_t, status, 256u);
    return cudaGetLastError();
  });
}

}  // namespace pmd

// Test hooks: the top-k of one CTA whose issuing warp leaves after the first of its tiles
// (held), or whose buffers never count as written.  F [R][k]; units [n_units] (each of one
// whole group: part -1); outputs [groups][M][topk]; k <= 16, M <= 16.
template <pmd::TxTest TEST>
static int topk_test(const int64_t *F, int64_t R, int k, const double *W, int M, const void *units, int n_units, int topk,
                     int64_t *idx, double *t, int *status, void *stream) {
  using G = pmd::XpGeom<1, 16, 1>;
  if (R < 1 || k < 1 || k > 16 || M < 1 || M > 16 || topk < 1 || topk > pmd::TOPK_MAX) return PM_ERR_INVALID_ARG;
  constexpr size_t smem = G::SMEM + sizeof(pmd::TxSmem);
  const auto kernel = pmd::k_topk_exact<G, TEST>;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return PM_ERR_CUDA;
  kernel<<<1, pmd::XP_THREADS, smem, (cudaStream_t)stream>>>(F, R, k, W, M, nullptr, (const pmd::TopkUnit *)units, n_units, topk,
                                                             nullptr, nullptr, idx, t, status, 256u);
  return cudaGetLastError() == cudaSuccess ? PM_OK : PM_ERR_CUDA;
}
extern "C" int pmx_topk_held(const int64_t *F, int64_t R, int k, const double *W, int M, const void *units, int n_units,
                             int topk, int64_t *idx, double *t, int *status, void *stream) {
  return topk_test<pmd::TX_HELD>(F, R, k, W, M, units, n_units, topk, idx, t, status, stream);
}
extern "C" int pmx_topk_unwritten(const int64_t *F, int64_t R, int k, const double *W, int M, const void *units,
                                  int n_units, int topk, int64_t *idx, double *t, int *status, void *stream) {
  return topk_test<pmd::TX_UNWRITTEN>(F, R, k, W, M, units, n_units, topk, idx, t, status, stream);
}
