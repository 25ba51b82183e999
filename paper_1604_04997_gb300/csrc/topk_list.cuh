// Ordered times, and a warp's sorted list of its smallest (time, row) pairs, shared by the
// ranking kernels over materialised features (predict.cu, topk_exact.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace pmd {

// The order of the times as 64-bit integers: a double's bit pattern, with the magnitude
// bits of negative values flipped, orders like the double itself for everything these
// kernels produce (no NaN, no -0.0).  Comparing integers keeps the comparisons off this
// GPU's narrow FP64 pipe.
__device__ __forceinline__ int64_t time_order(double t) {
  const int64_t b = __double_as_longlong(t);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

__device__ __forceinline__ bool arg_less(double a, int64_t ra, double b, int64_t rb) {
  const int64_t ka = time_order(a), kb = time_order(b);
  return ka < kb || (ka == kb && ra < rb);
}

constexpr double TK_INF = __builtin_huge_val();

// One compare-exchange stage across lanes lane and lane ^ j: this lane keeps the
// smaller (take_min) or the larger (t, r) pair of the two.
__device__ __forceinline__ void lane_cmp_swap(double &t, int64_t &r, int j, bool take_min) {
  const double ot = __shfl_xor_sync(0xffffffffu, t, j);
  const int64_t orr = __shfl_xor_sync(0xffffffffu, r, j);
  if (arg_less(ot, orr, t, r) == take_min) { t = ot; r = orr; }
}

// Merge this lane's candidate (t, r), if ok, into the warp's sorted list (lt, lr):
// entry i in lane i for i < topk, (+inf, INT64_MAX) in the other lanes.  Warp-uniform
// call; every shuffle and ballot is executed by all 32 lanes (none sits behind a
// short-circuit or a lane-dependent branch).  Candidates not below the list's last
// entry are dropped; one or two survivors are inserted one at a time (warp argmin,
// then a shift), more are sorted by a bitonic network and merged in one pass (the
// elementwise minimum of the list and the reversed candidates holds the 32 smallest
// as a bitonic sequence, which a 5-stage bitonic merge sorts).
__device__ __forceinline__ void warp_list_merge(double &lt, int64_t &lr, double t, int64_t r, bool ok, int topk,
                                                int lane) {
  constexpr unsigned FULL = 0xffffffffu;
  double kt = __shfl_sync(FULL, lt, topk - 1);     // the list's last entry: the threshold
  int64_t kr = __shfl_sync(FULL, lr, topk - 1);
  bool pass = ok && arg_less(t, r, kt, kr);
  unsigned mask = __ballot_sync(FULL, pass);
  if (__popc(mask) > 2) {
    double ct = pass ? t : TK_INF;
    int64_t cr = pass ? r : INT64_MAX;
#pragma unroll
    for (int kk = 2; kk <= 32; kk <<= 1)
#pragma unroll
      for (int j = kk >> 1; j > 0; j >>= 1) lane_cmp_swap(ct, cr, j, ((lane & j) == 0) == ((lane & kk) == 0));
    const double rt = __shfl_sync(FULL, ct, 31 - lane);
    const int64_t rr = __shfl_sync(FULL, cr, 31 - lane);
    if (arg_less(rt, rr, lt, lr)) { lt = rt; lr = rr; }
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) lane_cmp_swap(lt, lr, j, (lane & j) == 0);
    mask = 0;
  }
  for (int round = 0; mask && round < 32; round++) {   // one insertion per round; the winning lane drops out
    double bt = pass ? t : TK_INF;
    int64_t br = pass ? r : INT64_MAX;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const double ot = __shfl_xor_sync(FULL, bt, o);
      const int64_t orr = __shfl_xor_sync(FULL, br, o);
      if (arg_less(ot, orr, bt, br)) { bt = ot; br = orr; }
    }
    const int win = __ffs(__ballot_sync(FULL, pass && __double_as_longlong(t) == __double_as_longlong(bt) && r == br)) - 1;
    const int pos = __popc(__ballot_sync(FULL, lane < topk && arg_less(lt, lr, bt, br)));   // <= topk - 1
    const double ut = __shfl_up_sync(FULL, lt, 1);
    const int64_t ur = __shfl_up_sync(FULL, lr, 1);
    if (lane > pos) { lt = ut; lr = ur; }
    else if (lane == pos) { lt = bt; lr = br; }
    if (lane == win) pass = false;
    kt = __shfl_sync(FULL, lt, topk - 1);
    kr = __shfl_sync(FULL, lr, topk - 1);
    pass = pass && arg_less(t, r, kt, kr);
    mask = __ballot_sync(FULL, pass);
  }
  if (lane >= topk) { lt = TK_INF; lr = INT64_MAX; }
}

}  // namespace pmd
