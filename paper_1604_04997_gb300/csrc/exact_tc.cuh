// FP64-accurate prediction on the tensor cores, exactly in integer arithmetic: the
// device pieces shared by the kernels of predict_exact.cu.
//
//   S_rm = sum_i F_ri W_mi,   F int64 counts, W_mi = round(w_mi 2^E_m) (|W| <= 2^62)
//
// Every count and every weight is written as eight balanced base-256 digits,
// v = sum_q d_q 256^q with d_q in [-128, 127] (the top digit in [-128, 128], which
// covers all of int64).  A digit is exact in f16, a digit product is at most 2^14, and
//   P_d = sum_{q + q' = d} sum_i F_digit_q(r, i) W_digit_q'(m, i)
// sums at most 8 x 32 of them: below 2^22 in magnitude (the weights' top digit is at most
// 65), so tcgen05.mma (kind::f16, FP32 accumulation) forms every P_d without rounding, and
// S = sum_d 256^d P_d is exact in 128 bits, as the 32-bit multiply-add kernel (predict.cu)
// forms it: the same sums, the same times bit for bit.
//
// Four diagonals d = 4 g .. 4 g + 3 make one group (one 32-bit limb of S) and lie side by
// side in tensor memory, 4 x nb columns (nb: the models of one pass, 16 or 32).  With the
// weight digits stored one after another, and zero blocks before and after them, the digits
// 4 g - q .. 4 g - q + 3 that digit q of the counts meets are one window of the B operand:
// one MMA (M = 128 rows, N = 4 nb, K = 16) per (group, digit q, 16 features), at most 44
// per 128-row tile and pass, all of a group with the same shape and accumulator.  Four
// column ranges are used in turn, so the MMAs of a pass run while the sums of the one before
// are read back; a tile's operands are double-buffered likewise.  More than 32 models take
// two passes: 8 sums per thread, so that four limbs of each stay in registers.
//
// Digits that no count of the tile reaches are skipped (counts below 2^46 need 6 of 8).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "eval_common.cuh"
#include "kernels.h"
#include "mbar_wait.cuh"

namespace pmd {

constexpr int XP_ROWS = 128;      // MMA M: rows per tile
constexpr int XP_WARPS = 16;      // working warps: warp w reads TMEM lanes 32 (w % 4) .., models 8 (w / 4) .. of a pass
constexpr int XP_THREADS = 32 * XP_WARPS + 32;   // and one warp of which a thread issues the MMAs
constexpr int XP_RING = 4;        // column ranges in TMEM
constexpr int XP_DIG = 8;
constexpr int XP_MAXK = 32;
constexpr int XP_MAXM = 64;
constexpr int XP_BLOCKS = 14;     // weight-digit blocks: three zero, eight digits, three zero
// Every accumulator starts at XP_BIAS's float 1.5 2^23 = 4096 x 3072, the third of a group
// at 2^15 more (one more MMA per group): |P| <= 3,936,256 keeps the sum inside [2^23, 2^24),
// so the bits read back are P + XP_BIAS (+ 2^15), an integer.
constexpr uint32_t XP_BIAS = 0x4B400000u;
constexpr uint32_t XP_BIAS_A = 0x3C006C00u, XP_BIAS_B = 0x6A00u, XP_BIAS_B2 = 0x78006A00u;   // f16: 4096, 1; 3072, 0; 3072, 32768
// Gathering a limb (xp_limb) leaves the high word at its value plus XP_HI.
constexpr uint32_t XP_HI = 0x8B41u;

// sizes that depend on the problem: KS K-steps of 16 features, NB models per pass (padded),
// PASSES passes; offsets in bytes from the operands' start
template <int KS_, int NB_, int PASSES_>
struct XpGeom {
  static constexpr int KS = KS_, NB = NB_, PASSES = PASSES_;
  static constexpr uint32_t SBO = 256 * KS;                      // between 8-row groups
  static constexpr uint32_t A_DIG = XP_ROWS * 32 * KS;           // one digit of a row tile
  static constexpr uint32_t A_BUF = XP_DIG * A_DIG;
  static constexpr uint32_t B_BLK = NB * 32 * KS;                // one digit of a pass's weights
  static constexpr uint32_t B_PASS = XP_BLOCKS * B_BLK;
  static constexpr uint32_t OFF_B = 2 * A_BUF;
  // operands of the bias MMA, K = 16: 128 rows and 4 NB models, element 0 of each row set
  static constexpr uint32_t OFF_BIAS_A = OFF_B + PASSES * B_PASS;
  static constexpr uint32_t OFF_BIAS_B = OFF_BIAS_A + XP_ROWS * 32;
  static constexpr size_t SMEM = OFF_BIAS_B + NB * 128 + 128;
  static constexpr uint32_t RANGE = 4 * NB;                      // TMEM columns of one group
  static constexpr uint32_t TMEM_COLS = XP_RING * RANGE;         // 256 or 512
};

// the geometry of a problem: f(XpGeom) with k <= 16 or 32 and M <= 16, 32 or 64
template <class Fn>
inline cudaError_t xp_dispatch(int k, int M, Fn &&f) {
  if (k <= 16) return M <= 16 ? f(XpGeom<1, 16, 1>{}) : M <= 32 ? f(XpGeom<1, 32, 1>{}) : f(XpGeom<1, 32, 2>{});
  return M <= 16 ? f(XpGeom<2, 16, 1>{}) : M <= 32 ? f(XpGeom<2, 32, 1>{}) : f(XpGeom<2, 32, 2>{});
}

__device__ __forceinline__ uint32_t xp_saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor, no swizzle: 8-row x 16-byte core matrices, K-groups
// 128 B apart, 8-row groups sbo apart
__device__ __forceinline__ uint64_t xp_desc(uint32_t saddr, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | (uint64_t)(128u >> 4) << 16 | (uint64_t)((sbo >> 4) & 0x3FFFu) << 32 |
         (uint64_t)1 << 46;
}

// One MMA, issued by one elected lane of a converged warp.  The whole warp runs the issuing
// loops with warp-uniform operands: inside a branch of one thread the operands are not known
// to be uniform, and every MMA then waits about 150 cycles for its registers to be collected.
__device__ __forceinline__ void xp_mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p, e;\nsetp.ne.u32 p, %4, 0;\nelect.sync _|e, 0xffffffff;\n"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

// the same lane's commit of its MMAs so far: one arrival at mbar when they are complete
__device__ __forceinline__ void xp_commit(uint32_t mbar) {
  asm volatile(
      "{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\n"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(mbar)
      : "memory");
}

// a value that is the same in all lanes, known as such to the compiler
__device__ __forceinline__ uint32_t xp_uniform(uint32_t x) { return __shfl_sync(0xffffffffu, x, 0); }

// 16 TMEM lanes x 8 columns: thread t holds lanes t/4 and t/4 + 8, columns 2 (t%4) and + 1
// as words {0, 1} (lane t/4) and {2, 3} (lane t/4 + 8)
__device__ __forceinline__ void xp_ld16x8(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

// ---------------------------------------------------------------- digits

// Balanced base-256 digits of a 64-bit value as bytes: byte q of (lo, hi) is d_q + 128 for
// q < 7 (adding 128 to every digit makes them plain bytes); the top digit comes back apart.
struct XpBytes { uint32_t lo, hi; int top; };
__device__ __forceinline__ XpBytes xp_bytes(int64_t v) {
  const uint32_t l = (uint32_t)v, h = (uint32_t)((uint64_t)v >> 32);
  XpBytes b;
  uint32_t c;
  asm("add.cc.u32 %0, %2, 0x80808080;\n\taddc.u32 %1, %3, 0x00808080;\n\t" : "=r"(b.lo), "=r"(c) : "r"(l), "r"(h & 0xFFFFFFu));
  b.hi = c;                                     // bytes 4..6, and the carry into digit 7 above them
  b.top = ((int32_t)h >> 24) + (int)(c >> 24);  // [-128, 128]
  return b;
}

// digits q and q' of two values, given as bytes (b, b'), to packed f16: (1024 + b) - 1152
__device__ __forceinline__ uint32_t xp_half2(uint32_t bytes01, uint32_t sel) {
  const uint32_t x = __byte_perm(bytes01, 0x64646464u, sel);
  const __half2 h = __hsub2(*(const __half2 *)&x, __half2half2(__ushort_as_half(0x6480)));   // 1152
  return *(const uint32_t *)&h;
}

// the eight digits of a pair of values as packed f16 (first value in the low half)
__device__ __forceinline__ void xp_digits(int64_t v0, int64_t v1, uint32_t (&d)[XP_DIG]) {
  const XpBytes a = xp_bytes(v0), b = xp_bytes(v1);
  const uint32_t l01 = __byte_perm(a.lo, b.lo, 0x5140), l23 = __byte_perm(a.lo, b.lo, 0x7362);
  const uint32_t h01 = __byte_perm(a.hi, b.hi, 0x5140), h2 = __byte_perm(a.hi, b.hi, 0x7362);
  d[0] = xp_half2(l01, 0x4140);
  d[1] = xp_half2(l01, 0x4342);
  d[2] = xp_half2(l23, 0x4140);
  d[3] = xp_half2(l23, 0x4342);
  d[4] = xp_half2(h01, 0x4140);
  d[5] = xp_half2(h01, 0x4342);
  d[6] = xp_half2(h2, 0x4140);
  // top digits: 1024 + 512 + d as f16 bits, less 1536
  const uint32_t t = 0x66006600u + (uint32_t)a.top + ((uint32_t)b.top << 16);
  const __half2 h = __hsub2(*(const __half2 *)&t, __half2half2(__ushort_as_half(0x6600)));
  d[7] = *(const uint32_t *)&h;
}

// digits that values of this magnitude need: |v| <= 2^(8 n - 2) is covered by n
__device__ __forceinline__ int xp_ndigits(uint64_t mag) {   // mag: OR of v ^ (v >> 63)
  const int bits = 64 - __clzll((long long)mag);
  return min(XP_DIG, (bits + 9) >> 3);
}

// feature of K slot 8 kg + 2 c + e (c: 16-byte chunk of the slot's K-group): lanes of
// neighbouring K-groups read neighbouring 16-byte chunks of a row
__device__ __forceinline__ int xp_feature(int kg, int c, int e, int ks) { return 2 * (2 * ks * c + kg) + e; }

// ---------------------------------------------------------------- operands

// Weights (fp64 [M][k], staged through `scratch`, M k doubles in shared memory) to the
// digit blocks sB and the exponents sE, and the operands of the bias MMA.  Every thread of
// the CTA calls it.
template <class G>
__device__ __forceinline__ void xp_load_weights(const double *__restrict__ W, int M, int k,
                                                double *scratch, uint8_t *sB, int *sE) {
  for (int i = threadIdx.x; i < M * k; i += blockDim.x) scratch[i] = W[i];
  for (uint32_t i = threadIdx.x; i < G::PASSES * G::B_PASS / 16; i += blockDim.x)
    ((uint4 *)sB)[i] = make_uint4(0, 0, 0, 0);
  uint8_t *bias = sB + G::PASSES * G::B_PASS;   // rows of 2 x 16 bytes, 8-row groups of 2 x 128
  for (int i = threadIdx.x; i < 2 * (XP_ROWS + 4 * G::NB); i += blockDim.x) {
    const int kg = (i >> 3) & 1, r = (i >> 4) * 8 + (i & 7);
    const int n = r - XP_ROWS;   // column of the group: diagonal n / nb
    ((uint4 *)bias)[i] = make_uint4(kg ? 0u : n < 0 ? XP_BIAS_A : n / G::NB == 2 ? XP_BIAS_B2 : XP_BIAS_B, 0, 0, 0);
  }
  __syncthreads();
  if ((int)threadIdx.x < XP_MAXM) sE[threadIdx.x] = (int)threadIdx.x < M ? weight_exponent(scratch + threadIdx.x * k, k) : 0;
  __syncthreads();
  const int kslots = 16 * G::KS;
  for (int i = threadIdx.x; i < M * kslots / 2; i += blockDim.x) {
    const int m = i / (kslots / 2), p = i - m * (kslots / 2);   // slots 2 p and 2 p + 1
    const int kg = p >> 2, c = p & 3;
    const int f = xp_feature(kg, c, 0, G::KS);
    const int64_t w0 = f < k ? fixed_weight(scratch[m * k + f], sE[m]) : 0;
    const int64_t w1 = f + 1 < k ? fixed_weight(scratch[m * k + f + 1], sE[m]) : 0;
    uint32_t d[XP_DIG];
    xp_digits(w0, w1, d);
    uint8_t *dst = sB + (m >> 5) * G::B_PASS + ((m & 31) >> 3) * G::SBO + kg * 128 + (m & 7) * 16 + c * 4;
#pragma unroll
    for (int q = 0; q < XP_DIG; q++) *(uint32_t *)(dst + (3 + q) * G::B_BLK) = d[q];
  }
}

// A working thread's share of a row tile: row `xp_row` of the tile, K-group `xp_kg`, eight
// counts.  With one K-step only the first eight warps have a share.
template <class G>
__device__ __forceinline__ int xp_row() {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  return G::KS == 2 ? warp * 8 + (lane & 7) : warp * 16 + (lane >> 4) * 8 + (lane & 7);
}
template <class G>
__device__ __forceinline__ int xp_kg() { return ((threadIdx.x & 31) >> 3) & (2 * G::KS - 1); }

// vec: k even and F 16-byte aligned
template <class G>
__device__ __forceinline__ void xp_load_row(const int64_t *__restrict__ f, int k, bool vec, int64_t (&v)[8]) {
  const int kg = xp_kg<G>();
#pragma unroll
  for (int c = 0; c < 4; c++) {
    const int j = xp_feature(kg, c, 0, G::KS);
    v[2 * c] = v[2 * c + 1] = 0;
    if (vec) {
      if (j < k) {
        const longlong2 x = __ldg((const longlong2 *)(f + j));
        v[2 * c] = x.x;
        v[2 * c + 1] = x.y;
      }
    } else {
      if (j < k) v[2 * c] = __ldg(f + j);
      if (j + 1 < k) v[2 * c + 1] = __ldg(f + j + 1);
    }
  }
}

// digits of this thread's eight counts into operand buffer sA; s_nd[warp] receives the
// number of digits the warp's counts need
template <class G>
__device__ __forceinline__ void xp_store_digits(const int64_t (&v)[8], uint8_t *sA, int *s_nd) {
  if (G::KS == 1 && threadIdx.x >= 16 * XP_WARPS) return;   // warp-uniform; those warps' entries stay 1
  uint64_t mag = 0;
#pragma unroll
  for (int c = 0; c < 8; c++) mag |= (uint64_t)(v[c] ^ (v[c] >> 63));
  const int nd = __reduce_max_sync(0xffffffffu, xp_ndigits(mag));
  if ((threadIdx.x & 31) == 0) s_nd[threadIdx.x >> 5] = nd;
  const int row = xp_row<G>();
  uint8_t *dst = sA + (row >> 3) * G::SBO + xp_kg<G>() * 128 + (row & 7) * 16;
  uint32_t d[4][XP_DIG];
#pragma unroll
  for (int c = 0; c < 4; c++) xp_digits(v[2 * c], v[2 * c + 1], d[c]);
#pragma unroll
  for (int q = 0; q < XP_DIG; q++) *(uint4 *)(dst + q * G::A_DIG) = make_uint4(d[0][q], d[1][q], d[2][q], d[3][q]);
}

// the digits a tile needs: the largest of its warps' entries (any thread)
__device__ __forceinline__ int xp_tile_digits(const int *s_nd) {
  int n = 1;
#pragma unroll
  for (int w = 0; w < XP_WARPS; w += 4) {
    const int4 x = *(const int4 *)(s_nd + w);
    n = max(max(max(n, x.x), max(x.y, x.z)), x.w);
  }
  return n;
}

// groups of diagonals that have any digit product, for nd digits (a prefix of the four)
__device__ __forceinline__ int xp_groups(int nd) { return nd >= 6 ? 4 : nd >= 2 ? 3 : 2; }

// Issue group gr's MMAs into TMEM columns tmem .. (a whole warp; s0: the operands' shared
// address, sA: the tile's digits, sB: the pass's weight digits).  Their completion and the
// issuing lane's own arrival complete one phase of mbar (two arrivals): whoever waits for it
// sees the sums and everything the issuing warp has seen.
template <class G>
__device__ __forceinline__ void xp_issue(uint32_t s0, uint32_t sA, uint32_t sB, uint32_t tmem, int gr, int nd, uint32_t mbar) {
  // kind::f16: D fp32, A and B f16, both K-major; the fourth diagonal of group 3 is empty
  const uint32_t n = (uint32_t)((gr == 3 ? 3 : 4) * G::NB);
  const uint32_t idesc = (1u << 4) | (n >> 3) << 17 | (uint32_t)(XP_ROWS >> 4) << 24;
  const int q0 = max(0, 4 * gr - 7), q1 = min(nd - 1, 4 * gr + 3);
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
  xp_mma(tmem, xp_desc(s0 + G::OFF_BIAS_A, 256), xp_desc(s0 + G::OFF_BIAS_B, 256), idesc, 0);
  for (int q = q0; q <= q1; q++) {
    const uint32_t a = sA + q * G::A_DIG, b = sB + (uint32_t)(3 + 4 * gr - q) * G::B_BLK;
#pragma unroll
    for (int kc = 0; kc < G::KS; kc++) xp_mma(tmem, xp_desc(a + kc * 256, G::SBO), xp_desc(b + kc * 256, G::SBO), idesc, 1);
  }
  xp_commit(mbar);
  if ((threadIdx.x & 31) == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(mbar) : "memory");
  __syncwarp();
}

// One poll of mbar's phase that lets the hardware suspend the warp for a few microseconds,
// so that waiting warps leave the issue slots to the others.
__device__ __forceinline__ bool xp_try(uint32_t mbar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 4000;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(mbar), "r"(parity)
      : "memory");
  return done != 0;
}

constexpr unsigned long long XP_HELD_NS = 2000000ull;   // the waits of the HELD kernels (tests)

// Wait for one phase of mbar: false if it took longer than limit_ns, or if another thread has
// given up; *s_abort is set in both cases.
__device__ __forceinline__ bool xp_wait_one(uint32_t mbar, uint32_t parity, volatile int *s_abort,
                                            unsigned long long limit_ns) {
  bool ok = xp_try(mbar, parity);
  if (!ok) {
    const unsigned long long t0 = globaltimer_ns();
    while (!ok && !*s_abort) {
      ok = xp_try(mbar, parity);
      if (!ok && globaltimer_ns() - t0 > limit_ns) *s_abort = 1;
    }
  }
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
  return ok;
}

// the same for a whole warp, with the same result in all lanes
__device__ __forceinline__ bool xp_wait(uint32_t mbar, uint32_t parity, volatile int *s_abort,
                                        unsigned long long limit_ns = MBAR_WAIT_NS) {
  return __all_sync(0xffffffffu, xp_wait_one(mbar, parity, s_abort, limit_ns));
}

// The n-th commit that a warp made in turn to the `ring` barriers mbar[0 .. ring), and all
// before it, complete (bounded): the MMAs in flight, before their TMEM is freed.
__device__ __forceinline__ void xp_drain(const uint64_t *mbar, uint32_t ring, uint32_t n) {
  const unsigned long long t0 = globaltimer_ns();
  for (uint32_t i = n >= ring ? n - ring : 0; i < n; i++)
    while (!xp_try(xp_saddr(&mbar[i % ring]), (i / ring) & 1) && globaltimer_ns() - t0 < MBAR_WAIT_NS) {}
}

// What a kernel does before it frees its TMEM, after a wait of any warp ran out: the status bit,
// and the issuing warp's (issuer) n commits complete.  Every thread of the CTA calls it, past
// all of its waits.  The issuing warp cannot report alone: it runs ahead of the others, and has
// left when they wait for the last sums.
__device__ __forceinline__ void xp_finish(volatile int *s_abort, int *status, bool issuer, const uint64_t *mbar,
                                          uint32_t ring, uint32_t n) {
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();
  if (!*s_abort) return;   // the same for all threads
  if (threadIdx.x == 0 && status) atomicOr(status, ST_TIMEOUT);
  if (issuer) xp_drain(mbar, ring, n);
  __syncthreads();
}

__device__ __forceinline__ void xp_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(mbar) : "memory");
}

// One limb of this thread's 8 sums from group GR's diagonals:
//   limb + 2^32 (cy' - XP_HI) = (cy - XP_HI) + P_0 + 256 P_1 + 256^2 P_2 + 256^3 P_3
// (cy: the high word of the group before, none for group 0).  Sum 2 i + e: row 8 i of the
// thread's four, model e of its two.
// The pairs u = P_0 + 256 P_1 + carry and v = P_2 + 256 P_3 fit in 32 signed bits; as
// unsigned words u + 2^31 and v + 0x8B408000 (the biases of b_2 + 256 b_3) they add up to
// the limb's 64 bits plus 2^31 + 2^16 0x8B408000 = 2^32 XP_HI, which leaves the low word as
// it is.  m256 is 256 as a kernel argument: a literal would become a shift and add on the
// integer ALU, this kernel's busiest pipe.  (A 32 x 32 + 64-bit multiply-add is four
// instructions on this GPU.)
template <class G, int GR>
__device__ __forceinline__ void xp_limb(uint32_t m256, uint32_t tmem, uint32_t (&limb)[8],
                                        uint32_t (&cy)[8]) {
  constexpr uint32_t K = 0x80000000u - XP_BIAS * 257u - (GR == 0 ? 0u : XP_HI);
  uint32_t p[4][2][4];
#pragma unroll
  for (int s = 0; s < 2; s++)
#pragma unroll
    for (int j = 0; j < (GR == 3 ? 3 : 4); j++) xp_ld16x8(tmem + ((uint32_t)(16 * s) << 16) + (uint32_t)(j * G::NB), p[j][s]);
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::);
#pragma unroll
  for (int i = 0; i < 8; i++) {
    const int s = i >> 2, e = i & 3;
    const uint32_t u = p[1][s][e] * m256 + (p[0][s][e] + (GR == 0 ? K : cy[i] + K));
    const uint32_t v = GR == 3 ? p[2][s][e] : p[3][s][e] * m256 + p[2][s][e];
    const uint64_t t = (uint64_t)u + ((uint64_t)v << 16);
    limb[i] = (uint32_t)t;
    cy[i] = (uint32_t)(t >> 32);
  }
}

static __device__ __noinline__ double xp_value_rare(uint32_t a, uint32_t b, uint32_t c, uint32_t d, int E) {
  Acc128 A;
  A.lo = (uint64_t)a | ((uint64_t)b << 32);
  A.hi = (uint64_t)c | ((uint64_t)d << 32);
  return key_value(acc_key(A), E);
}

// The time of an exact sum S (limbs x0 .. x3, two's complement; NEG: S may be negative):
// key_value(acc_key(S), E) of eval_common.cuh (57 leading bits, rounded once to FP64's 53)
// in one pass over the limbs.  x: 1150 - E, the biased exponent of a leading one in bit 31
// of x3, in [XP_XMIN, XP_XMAX], which keeps every time in FP64's normal range.  bad is set,
// and the result is not to be used, for S = 0.
constexpr int XP_XMIN = 130, XP_XMAX = 2044;
template <bool NEG>
__device__ __forceinline__ double xp_value(uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3, int x, bool &bad) {
  uint32_t sg = 0;
  if (NEG) {
    sg = (uint32_t)((int32_t)x3 >> 31);
    x0 ^= sg, x1 ^= sg, x2 ^= sg, x3 ^= sg;
    asm("sub.cc.u32 %0, %0, %4;\n\tsubc.cc.u32 %1, %1, %4;\n\tsubc.cc.u32 %2, %2, %4;\n\tsubc.u32 %3, %3, %4;\n\t"
        : "+r"(x0), "+r"(x1), "+r"(x2), "+r"(x3)
        : "r"(sg));
  }
  // shift whole limbs out at the top until the leading one is in x3
  if ((x3 | x2) == 0) { x3 = x1; x2 = x0; x1 = x0 = 0; x -= 64; }
  if (x3 == 0) { x3 = x2; x2 = x1; x1 = x0; x -= 32; }
  bad = bad || x3 == 0;
  uint32_t lz;
  asm("bfind.shiftamt.u32 %0, %1;" : "=r"(lz) : "r"(x3));
  uint32_t nh, nl;   // the 64 bits from the leading one down
  nh = __funnelshift_l(x2, x3, lz);
  nl = __funnelshift_l(x1, x2, lz);
  // drop the leading one and all below bit 7, round to nearest even at bit 11; a carry out
  // of the fraction moves into the exponent
  const uint32_t bit = (nl >> 11) & 1u;
  uint64_t y = ((uint64_t)(nh & 0x7FFFFFFFu) << 32 | (nl & ~127u)) + (0x3FFu + bit);
  const uint32_t lo = (uint32_t)(y >> 11);
  const uint32_t hi = (uint32_t)(y >> 43) + ((uint32_t)(x - (int)lz) << 20);
  return __hiloint2double((int)(NEG ? hi | (sg & 0x80000000u) : hi), (int)lo);
}

}  // namespace pmd
