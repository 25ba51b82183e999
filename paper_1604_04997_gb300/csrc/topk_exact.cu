// Top-k rows per (group, model) over materialised features (configuration selection,
// Sec. 6.1) for more than a few models, on the exact tensor-core prediction (exact_tc.cuh):
// the times are those of k_predict_exact, bit for bit.
//
// One CTA of 16 working warps and an issuing warp per SM; the CTA takes units (up to
// topk_chunk positions of one group) in turn, in tiles of 128 positions.  A time that is not
// above the model's current 16th is offered to the model's buffer of TX_BUF candidates in
// shared memory; when some buffer is half full (or cannot take a candidate), all warps meet
// and warp w merges the buffers of models w, w + 16, .. into their sorted lists (entry i in
// lane i, predict.cu's merge).  After the first tiles of a unit few candidates pass, so the
// warps rarely meet: the products bound the kernel, not the lists.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "exact_tc.cuh"
#include "kernels.h"
#include "topk_list.cuh"

namespace pmd {

constexpr int TX_BUF = 16;           // buffered candidates per model

struct TxSmem {                      // beyond the operands of XpGeom
  int64_t lt[XP_MAXM][TOPK_MAX];     // sorted lists: times (as bits), rows
  int64_t lr[XP_MAXM][TOPK_MAX];
  int64_t ct[XP_MAXM][TX_BUF];       // candidates: times, positions within the unit
  int32_t cp[XP_MAXM][TX_BUF];
  int64_t thr[XP_MAXM];              // time_order of the list's last entry
  int32_t cnt[XP_MAXM];
  int64_t rows[4][XP_ROWS];          // rows of the tiles in flight (by tile modulo 4), -1: none
};

// The tiles of a CTA, in order: units blockIdx.x, blockIdx.x + gridDim.x, .., each cut into
// 128 positions (a unit without positions is one empty tile).
struct TxCursor {
  const TopkUnit *units;
  int n_units, u;
  int64_t p, p1;
  int32_t g, part;
  __device__ void open() {
    if (u < n_units) {
      const TopkUnit U = units[u];
      p = U.p0;
      p1 = U.p1;
      g = U.g;
      part = U.part;
    }
  }
  __device__ TxCursor(const TopkUnit *units, int n_units) : units(units), n_units(n_units), u(blockIdx.x), p(0), p1(0), g(0), part(0) {
    open();
  }
  __device__ bool more() const { return u < n_units; }
  __device__ bool last() const { return p + XP_ROWS >= p1; }   // of its unit
  __device__ void next() {
    if (last()) {
      u += gridDim.x;
      open();
    } else {
      p += XP_ROWS;
    }
  }
};

template <class G>
__global__ void __launch_bounds__(XP_THREADS, 1) k_topk_exact(const int64_t *__restrict__ F, int64_t R, int k,
                                                              const double *__restrict__ W, int M,
                                                              const int64_t *__restrict__ rows,
                                                              const TopkUnit *__restrict__ units, int n_units, int topk,
                                                              double *__restrict__ part_t, int64_t *__restrict__ part_r,
                                                              int64_t *__restrict__ top_idx, double *__restrict__ top_t,
                                                              int *status, uint32_t m256) {
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
      X.cnt[m] = 0;
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
  TxCursor cur(units, n_units);
  if (warp == XP_WARPS) {
    // this warp issues, ahead of the working warps as far as digits and columns allow
    for (; cur.more() && ok; cur.next(), it++) {
      if (!(ok = xp_wait(xp_saddr(&digits[it & 1]), (it >> 1) & 1, &s_abort))) break;
      const int nd = (int)xp_uniform((uint32_t)xp_tile_digits(s_nd[it & 3])), ng = xp_groups(nd);
      for (int n = 0; n < G::PASSES * ng && ok; n++, seq++) {
        const uint32_t b = seq % XP_RING;
        const int ps = n >= ng;
        if (seq >= XP_RING && !(ok = xp_wait(xp_saddr(&empty[b]), (seq / XP_RING - 1) & 1, &s_abort))) break;
        xp_issue<G>(s0, s0 + (it & 1) * G::A_BUF, s0 + G::OFF_B + ps * G::B_PASS, tmem + b * G::RANGE, n - ps * ng, nd,
                    xp_saddr(&full[b]));
      }
    }
    if (!ok) {
      if (lane == 0) atomicOr(status, ST_TIMEOUT);
      // let the MMAs in flight finish before TMEM is freed (bounded)
      const unsigned long long t0 = globaltimer_ns();
      for (uint32_t n = seq >= XP_RING ? seq - XP_RING : 0; n < seq; n++)
        while (!xp_try(xp_saddr(&full[n % XP_RING]), (n / XP_RING) & 1) && globaltimer_ns() - t0 < MBAR_WAIT_NS) {}
    }
    __syncwarp();
  } else {
    const bool active = slice * 8 < G::NB;   // this warp has models
    const int c0 = slice * 8 + 2 * (lane & 3);
    const uint32_t tread = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(slice * 8);
    // the working warps meet; true if any of their threads says so
    auto meet = [&](bool say) -> bool {
      uint32_t any;
      asm volatile(
          "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.or.pred q, 1, %2, p;\nselp.u32 %0, 1, 0, q;\n}\n"
          : "=r"(any)
          : "r"((uint32_t)say), "n"(32 * XP_WARPS)
          : "memory");
      return any != 0;
    };
    // the feature row of this thread's share of the tile at cursor c, or -1
    auto locate = [&](const TxCursor &c) -> int64_t {
      const int64_t pos = c.p + row;
      if (row >= XP_ROWS || !c.more() || pos >= c.p1) return -1;
      const int64_t r = rows ? rows[pos] : pos;
      if (r >= 0 && r < R) return r;
      if (xp_kg<G>() == 0) atomicOr(status, ST_BAD_ROW);
      return -1;
    };
    // load this thread's share of the n-th tile, from row r, and store its digits
    auto feed = [&](int64_t r, uint32_t n) {
      int64_t v[8];
#pragma unroll
      for (int i = 0; i < 8; i++) v[i] = 0;
      if (row < XP_ROWS) {
        if (xp_kg<G>() == 0) X.rows[n & 3][row] = r;
        if (r >= 0) xp_load_row<G>(F + r * k, k, vec, v);
      }
      xp_store_digits<G>(v, sA + (n & 1) * G::A_BUF, s_nd[n & 3]);
      asm volatile("fence.proxy.async.shared::cta;\n" ::);
      __syncwarp();
      if (lane == 0) xp_arrive(xp_saddr(&digits[n & 1]));
    };
    // the candidates of this warp's models into their lists
    int64_t base = 0;   // first position of the current unit
    auto merge = [&]() {
      for (int m = warp; m < M; m += XP_WARPS) {
        const int n = min(X.cnt[m], TX_BUF);
        if (n == 0) continue;   // warp-uniform
        double t = TK_INF, lt = TK_INF;
        int64_t r = INT64_MAX, lr = INT64_MAX;
        if (lane < n) {
          t = __longlong_as_double(X.ct[m][lane]);
          const int64_t pos = base + X.cp[m][lane];
          r = rows ? rows[pos] : pos;
        }
        if (lane < TOPK_MAX) {
          lt = __longlong_as_double(X.lt[m][lane]);
          lr = X.lr[m][lane];
        }
        warp_list_merge(lt, lr, t, r, lane < n, topk, lane);
        if (lane < TOPK_MAX) {
          X.lt[m][lane] = __double_as_longlong(lt);
          X.lr[m][lane] = lr;
        }
        const int64_t th = time_order(__shfl_sync(0xffffffffu, lt, topk - 1));
        if (lane == 0) {
          X.thr[m] = th;
          X.cnt[m] = 0;
        }
        __syncwarp();
      }
    };
    auto wait = [&]() { return xp_wait(xp_saddr(&full[seq % XP_RING]), (seq / XP_RING) & 1, &s_abort); };
    auto done = [&]() {   // this warp has read its share of a group
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
      __syncwarp();
      if (lane == 0) xp_arrive(xp_saddr(&empty[seq % XP_RING]));
      seq++;
    };
    // one (tile, pass): the exact sums, the times, the candidates.  On a wait that ran out the
    // warp goes on without sums to the meeting point, where all leave together (false).
    auto pass = [&](int ps) -> bool {
      uint32_t limb[4][8], cy[8];
      ok = wait();
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
      const int m = 32 * ps + c0;
      const int rl = quarter * 32 + (lane >> 2);   // this thread's rows of the tile: rl + 8 i, i < 4
      int64_t t[8];
      uint32_t pending = 0;   // bit 2 i + e: the time of row rl + 8 i, model m + e is still to be offered
      if (ok && active) {
        const int x0[2] = {1150 - s_E[m], 1150 - s_E[m + 1]};
        const bool wide = min(x0[0], x0[1]) < XP_XMIN || max(x0[0], x0[1]) > XP_XMAX;
        uint32_t sg = 0;
#pragma unroll
        for (int o = 0; o < 8; o++) sg |= limb[3][o];
        const bool neg = __any_sync(0xffffffffu, (int32_t)sg < 0);
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const bool live = X.rows[it & 3][rl + 8 * i] >= 0;
#pragma unroll
          for (int e = 0; e < 2; e++) {
            const int o = 2 * i + e;
            bool bad = wide;
            double x = neg ? xp_value<true>(limb[0][o], limb[1][o], limb[2][o], limb[3][o], x0[e], bad)
                           : xp_value<false>(limb[0][o], limb[1][o], limb[2][o], limb[3][o], x0[e], bad);
            if (bad) x = xp_value_rare(limb[0][o], limb[1][o], limb[2][o], limb[3][o], 1150 - x0[e]);
            t[o] = __double_as_longlong(x);
            if (live && m + e < M && time_order(x) <= X.thr[m + e]) pending |= 1u << o;
          }
        }
      }
      // offer; when a buffer is half full, or full, merge and offer the rest
      while (true) {
        bool call = false;
#pragma unroll
        for (int o = 0; o < 8; o++) {
          if (pending & (1u << o)) {
            const int mm = m + (o & 1);
            if (time_order(__longlong_as_double(t[o])) > X.thr[mm]) {   // tightened since
              pending &= ~(1u << o);
            } else {
              const int slot = atomicAdd(&X.cnt[mm], 1);
              if (slot < TX_BUF) {
                X.ct[mm][slot] = t[o];
                X.cp[mm][slot] = (int32_t)(cur.p - base) + rl + 8 * (o >> 1);
                pending &= ~(1u << o);
              }
              call |= slot >= TX_BUF / 2;
            }
          }
        }
        if (meet(!ok)) return false;          // (also: every offer is written)
        if (!meet(call || pending)) break;
        merge();
        meet(false);                          // lists, thresholds and counts are up to date
        if (!meet(pending != 0)) break;
      }
      return true;
    };
    TxCursor ahead(units, n_units);
    feed(locate(ahead), 0);
    if (ahead.more()) ahead.next();
    feed(locate(ahead), 1);
    if (ahead.more()) ahead.next();
    base = cur.p;
    for (; cur.more(); it++) {
      // the rows of the tile after the next on their way into L2, 128 bytes per prefetch
      const int64_t next = locate(ahead);
      if (next >= 0 && (xp_kg<G>() & 1) == 0 && xp_kg<G>() * 64 < k * 8)
        asm volatile("prefetch.global.L2 [%0];\n" ::"l"((const char *)(F + next * k) + xp_kg<G>() * 64));
      int ps = 0;
#pragma unroll 1
      for (; ps < G::PASSES; ps++)
        if (!pass(ps)) break;
      if (ps < G::PASSES) break;
      const bool end = cur.last();
      if (end) {
        // the unit's lists
        merge();
        for (int m = warp; m < M; m += XP_WARPS) {
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
      feed(next, it + 2);
      if (ahead.more()) ahead.next();
      cur.next();
      if (end) {
        base = cur.p;
        meet(false);   // the lists are reset
      }
    }
    if (!ok) s_abort = 1;
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();
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
