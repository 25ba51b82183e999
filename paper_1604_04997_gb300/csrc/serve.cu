// Serving kernels: one batch of autotuner queries (Sec. 6.1 configuration selection).
//
// A query asks for the topk fastest of n candidate (kernel variant, parameter point)
// pairs under one device model.  Each candidate's properties p_i(n) are evaluated from
// its compiled table (Sec. 2: counts re-evaluated for changed n) and contracted with the
// model's weights to FP64 accuracy (exact fixed-point products and 128-bit sums, as in
// the batched ranking kernel).  Two launches per batch:
//   k_serve_eval  one thread per candidate -> a monotone 64-bit ranking key
//   k_serve_topk  one CTA per query -> topk (key, candidate) pairs, ordered by
//                 (time, candidate index), converted to times.
#include "eval_common.cuh"
#include "topk_list.cuh"

namespace pmd {

constexpr int SV_THREADS = 128;      // candidates per k_serve_eval CTA
constexpr int SV_TOPK_WARPS = 16;

// Per-model fixed-point weights W_i = round(w_i 2^E) (sum |W_i| <= 2^62) as 28-bit limb
// triples, by the block's first warp (E by weight_exponent_warp: one thread's chain of 32
// FP64 additions cost every block of a batch more than the rest of its prologue).
__device__ __forceinline__ void load_model_limbs(const double *w, Limbs3 *s_w) {
  if (threadIdx.x < 32) s_w[threadIdx.x] = to_limbs3(llrint(ldexp(w[threadIdx.x], weight_exponent_warp(w))));
}

__global__ void __launch_bounds__(SV_THREADS) k_serve_eval(ServeArgs a) {
  __shared__ int64_t slots[pmt::MAX_SLOTS * SV_THREADS];
  __shared__ Limbs3 s_w[32];
  const int2 b = a.blocks[blockIdx.x];
  const SQuery q = a.queries[b.x];
  load_model_limbs(a.models + (int64_t)q.model * 32, s_w);
  __syncthreads();
  const int i = b.y * SV_THREADS + threadIdx.x;
  if (i >= q.n) return;
  const int64_t c = q.begin + i;
  const uint32_t *T = a.arena + a.cand_off[c];
  int64_t key = INT64_MAX;   // out-of-box candidates never rank
  int32_t n[4];
  if (!point_in_box(T, a.points + c * 4, (int)T[pmt::H_NPARAMS], n)) {
    atomicOr(a.q_status + b.x, ST_OUT_OF_BOX);
  } else {
    LimbAcc la;
    la.zero();
    const bool ok = eval_table(
        T, n, slots + threadIdx.x, SV_THREADS,
        [&](int col, int64_t val) { if (col < 32) la.add((uint64_t)val, s_w[col]); },
        [&](int col, int64_t val) { la.add((uint64_t)val, s_w[col]); });
    if (!ok) atomicOr(a.q_status + b.x, ST_BAD_TABLE);
    else key = acc_key(la.sum());
  }
  a.keys[c] = key;
}

// One CTA per query.  Each warp keeps one sorted list of its smallest (key, index) pairs, an
// entry per lane, and merges 32 keys at a time into it.  Bound by the issue of those merges
// (some 400 instructions each), so the warps share the least of their lists' last entries:
// after the first batches nearly every key falls to one comparison and a vote.  Largest and
// smallest query of a burst, by the kernel's time: 126 and 12.6 us with a list of 16 per
// thread (every lane inserting on its own, then topk rounds over the block), 80 and 6.1 with
// 32 warps and no shared bound, 58 and 5.3 now; one query of 16 candidates from submission to
// result 51 -> 37 us.
//
// Keys ride through the list as the doubles whose time_order they are; they stay below that
// of +inf (|S| < 2^126, so a key's top byte is at most 0x7e).
__global__ void __launch_bounds__(SV_TOPK_WARPS * 32) k_serve_topk(ServeArgs a) {
  __shared__ double s_k[SV_TOPK_WARPS][SV_MAX_TOPK];
  __shared__ int64_t s_i[SV_TOPK_WARPS][SV_MAX_TOPK];
  __shared__ long long s_thr;   // no key above it is among the topk: the least of the warps' last entries
  static_assert(SV_MAX_TOPK == 16 && SV_TOPK_WARPS % 2 == 0, "two warps' lists are merged at a time");
  const SQuery q = a.queries[blockIdx.x];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t *keys = a.keys + q.begin;
  if (threadIdx.x == 0) s_thr = INT64_MAX;
  __syncthreads();
  double lt = TK_INF;
  int64_t lr = INT64_MAX;
  for (int64_t b = 32 * warp; b < q.n; b += 4 * 32 * SV_TOPK_WARPS) {   // warp-uniform
    int64_t k[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const int64_t i = b + u * 32 * SV_TOPK_WARPS + lane;
      k[u] = i < q.n ? keys[i] : INT64_MAX;
    }
#pragma unroll 1
    for (int u = 0; u < 4; u++) {   // one copy of the merge's code
      const bool ok = k[0] != INT64_MAX && k[0] <= *(volatile long long *)&s_thr;
      if (__any_sync(0xffffffffu, ok)) {
        const double t = __longlong_as_double(k[0] ^ ((k[0] >> 63) & 0x7fffffffffffffffll));
        warp_list_merge(lt, lr, t, b + u * 32 * SV_TOPK_WARPS + lane, ok, q.topk, lane);
        if (lane == q.topk - 1 && lr != INT64_MAX && time_order(lt) < *(volatile long long *)&s_thr)
          atomicMin(&s_thr, (long long)time_order(lt));
      }
      k[0] = k[1], k[1] = k[2], k[2] = k[3], k[3] = INT64_MAX;
    }
  }
  if (lane < SV_MAX_TOPK) {
    s_k[warp][lane] = lt;
    s_i[warp][lane] = lr;
  }
  __syncthreads();
  if (warp) return;
  const int E = weight_exponent_warp(a.models + (int64_t)q.model * 32);
#pragma unroll 1
  for (int w = 0; w < SV_TOPK_WARPS; w += 2) {
    const int64_t r = w ? s_i[w + (lane >> 4)][lane & 15] : s_i[1][lane & 15];
    const double t = w ? s_k[w + (lane >> 4)][lane & 15] : s_k[1][lane & 15];
    warp_list_merge(lt, lr, t, r, r != INT64_MAX && (w || lane < 16), q.topk, lane);   // the warp's own list is held
  }
  if (lane < q.topk) {
    const bool real = lr != INT64_MAX;
    a.out_idx[(int64_t)blockIdx.x * SV_MAX_TOPK + lane] = real ? (int32_t)lr : -1;
    a.out_t[(int64_t)blockIdx.x * SV_MAX_TOPK + lane] =
        real ? key_value(time_order(lt), E) : __longlong_as_double(0x7ff0000000000000ll);
  }
}

cudaError_t launch_serve(const ServeArgs &a, int n_blocks, cudaStream_t st) {
  if (n_blocks > 0) k_serve_eval<<<n_blocks, SV_THREADS, 0, st>>>(a);
  if (a.n_queries > 0) k_serve_topk<<<a.n_queries, SV_TOPK_WARPS * 32, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace pmd
