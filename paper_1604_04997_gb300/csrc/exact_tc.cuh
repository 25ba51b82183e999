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
// side in tensor memory, 4 x nb columns (nb: models rounded up to 16).  With the weight
// digits stored one after another, and zero blocks before and after them, the digits
// 4 g - q .. 4 g - q + 3 that digit q of the counts meets are one window of the B operand:
// one MMA (M = 128 rows, N = 4 nb, K = 16) per (group, digit q, 16 features), at most 44
// per 128-row tile, all of a group with the same shape and accumulator.  Two groups
// alternate between two column ranges, so the MMAs of the next groups run while a
// group's sums are read back; a tile's operands are double-buffered likewise.
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
constexpr int XP_THREADS = 512;   // 16 warps: warp w reads TMEM lanes 32 (w % 4) .., models 16 (w / 4) ..
constexpr int XP_DIG = 8;
constexpr int XP_MAXK = 32;
constexpr int XP_MAXM = 64;
constexpr int XP_BLOCKS = 14;     // weight-digit blocks: three zero, eight digits, three zero
constexpr float XP_MAGIC = 12582912.0f;        // 1.5 2^23: (P + XP_MAGIC) has P + 0x4B400000 as its bits
constexpr uint32_t XP_BIAS = 0x4B400000u;
// the bias of the four limbs: XP_BIAS (1 + 256 + ... + 256^15) modulo 2^128
constexpr uint64_t XP_BIAS_W = (uint64_t)XP_BIAS * 0x01010101u;
constexpr uint32_t XP_B0 = (uint32_t)XP_BIAS_W;
constexpr uint64_t XP_S1 = (XP_BIAS_W >> 32) + XP_BIAS_W;
constexpr uint32_t XP_B1 = (uint32_t)XP_S1;
constexpr uint64_t XP_S2 = (XP_S1 >> 32) + XP_BIAS_W;
constexpr uint32_t XP_B2 = (uint32_t)XP_S2;
constexpr uint32_t XP_B3 = (uint32_t)((XP_S2 >> 32) + XP_BIAS_W);

// sizes that depend on the problem: K-steps of 16 features and padded models
struct XpGeom {
  int ks, nb;
  __host__ __device__ uint32_t a_dig() const { return (uint32_t)(XP_ROWS * 32 * ks); }   // one digit of a row tile
  __host__ __device__ uint32_t a_buf() const { return XP_DIG * a_dig(); }
  __host__ __device__ uint32_t b_blk() const { return (uint32_t)(nb * 32 * ks); }        // one digit of the weights
  __host__ __device__ uint32_t sbo() const { return (uint32_t)(256 * ks); }              // between 8-row groups
  __host__ __device__ size_t smem() const { return 2 * a_buf() + XP_BLOCKS * b_blk() + 128; }
  __host__ __device__ uint32_t tmem_cols() const { return nb <= 16 ? 128u : nb <= 32 ? 256u : 512u; }
};

__host__ __device__ inline XpGeom xp_geom(int k, int M) { return XpGeom{k <= 16 ? 1 : 2, (M + 15) & ~15}; }

__device__ __forceinline__ uint32_t xp_saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor, no swizzle: 8-row x 16-byte core matrices, K-groups
// 128 B apart, 8-row groups sbo apart
__device__ __forceinline__ uint64_t xp_desc(uint32_t saddr, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | (uint64_t)(128u >> 4) << 16 | (uint64_t)((sbo >> 4) & 0x3FFFu) << 32 |
         (uint64_t)1 << 46;
}

__device__ __forceinline__ void xp_mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

// 16 TMEM lanes x 16 columns: thread t holds lanes t/4 and t/4 + 8, columns 8 j + 2 (t%4)
// and + 1 (j = 0, 1) as v[4 j + {0, 1}] (lane t/4) and v[4 j + {2, 3}] (lane t/4 + 8)
__device__ __forceinline__ void xp_ld16x16(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 8; i++) v[i] = __uint_as_float(r[i]);
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

// W = round(w 2^E) to nearest even, as llrint(ldexp(w, E)), with integer operations (this
// GPU's FP64 pipe is narrow); infinities and NaN take the FP64 path.
__device__ __forceinline__ int64_t xp_fixed_weight(double w, int E) {
  const uint64_t b = (uint64_t)__double_as_longlong(w);
  const int e = (int)((b >> 52) & 0x7FF);
  if (e == 0x7FF) return llrint(ldexp(w, E));
  const uint64_t mant = (b & 0xFFFFFFFFFFFFFull) | (e ? 1ull << 52 : 0ull);
  const int s = (e ? e : 1) - 1075 + E;
  uint64_t q;
  if (s >= 0) {
    q = mant << min(s, 63);
  } else if (s > -55) {
    const uint64_t half = 1ull << (-s - 1), rem = mant & (2 * half - 1);
    q = mant >> -s;
    if (rem > half || (rem == half && (q & 1))) q++;
  } else {
    q = 0;
  }
  return (b >> 63) ? -(int64_t)q : (int64_t)q;
}

// feature of K slot 8 kg + 2 c + e (c: 16-byte chunk of the slot's K-group): lanes of
// neighbouring K-groups read neighbouring 16-byte chunks of a row
__device__ __forceinline__ int xp_feature(int kg, int c, int e, int ks) { return 2 * (2 * ks * c + kg) + e; }

// ---------------------------------------------------------------- operands

// Weights (fp64 [M][k], staged through `scratch`, M k doubles in shared memory) to the
// digit blocks sB and the exponents sE.  Every thread of the CTA calls it.
__device__ __forceinline__ void xp_load_weights(const XpGeom &g, const double *__restrict__ W, int M, int k,
                                                double *scratch, uint8_t *sB, int *sE) {
  for (int i = threadIdx.x; i < M * k; i += XP_THREADS) scratch[i] = W[i];
  for (uint32_t i = threadIdx.x; i < XP_BLOCKS * g.b_blk() / 16; i += XP_THREADS)
    ((uint4 *)sB)[i] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  if ((int)threadIdx.x < XP_MAXM) sE[threadIdx.x] = (int)threadIdx.x < M ? weight_exponent(scratch + threadIdx.x * k, k) : 0;
  __syncthreads();
  const int kslots = 16 * g.ks;
  for (int i = threadIdx.x; i < M * kslots / 2; i += XP_THREADS) {
    const int m = i / (kslots / 2), p = i - m * (kslots / 2);   // slots 2 p and 2 p + 1
    const int kg = p >> 2, c = p & 3;
    const int f = xp_feature(kg, c, 0, g.ks);
    const int64_t w0 = f < k ? xp_fixed_weight(scratch[m * k + f], sE[m]) : 0;
    const int64_t w1 = f + 1 < k ? xp_fixed_weight(scratch[m * k + f + 1], sE[m]) : 0;
    uint32_t d[XP_DIG];
    xp_digits(w0, w1, d);
    uint8_t *dst = sB + (m >> 3) * g.sbo() + kg * 128 + (m & 7) * 16 + c * 4;
#pragma unroll
    for (int q = 0; q < XP_DIG; q++) *(uint32_t *)(dst + (3 + q) * g.b_blk()) = d[q];
  }
}

// This thread's share of a row tile: row `xp_row` of the tile, K-group `xp_kg`, eight
// counts.  With one K-step only the first eight warps have a share.
__device__ __forceinline__ int xp_row(int ks) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  return ks == 2 ? warp * 8 + (lane & 7) : warp * 16 + (lane >> 4) * 8 + (lane & 7);
}
__device__ __forceinline__ int xp_kg(int ks) { return ((threadIdx.x & 31) >> 3) & (2 * ks - 1); }

// vec: k even and F 16-byte aligned
__device__ __forceinline__ void xp_load_row(const int64_t *__restrict__ f, int k, int ks, bool vec, int64_t (&v)[8]) {
  const int kg = xp_kg(ks);
#pragma unroll
  for (int c = 0; c < 4; c++) {
    const int j = xp_feature(kg, c, 0, ks);
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

// digits of this thread's eight counts into operand buffer sA; *s_nd collects the number
// of digits the tile needs
__device__ __forceinline__ void xp_store_digits(const XpGeom &g, const int64_t (&v)[8], uint8_t *sA, int *s_nd) {
  if (g.ks == 1 && threadIdx.x >= XP_THREADS / 2) return;   // warp-uniform
  uint64_t mag = 0;
#pragma unroll
  for (int c = 0; c < 8; c++) mag |= (uint64_t)(v[c] ^ (v[c] >> 63));
  const int nd = __reduce_max_sync(0xffffffffu, xp_ndigits(mag));
  if ((threadIdx.x & 31) == 0) atomicMax(s_nd, nd);
  const int row = xp_row(g.ks);
  uint8_t *dst = sA + (row >> 3) * g.sbo() + xp_kg(g.ks) * 128 + (row & 7) * 16;
  uint32_t d[4][XP_DIG];
#pragma unroll
  for (int c = 0; c < 4; c++) xp_digits(v[2 * c], v[2 * c + 1], d[c]);
#pragma unroll
  for (int q = 0; q < XP_DIG; q++) *(uint4 *)(dst + q * g.a_dig()) = make_uint4(d[0][q], d[1][q], d[2][q], d[3][q]);
}

// groups of diagonals that have any digit product, for nd digits (a prefix of the four)
__device__ __forceinline__ int xp_groups(int nd) { return nd >= 6 ? 4 : nd >= 2 ? 3 : 2; }

// issue group gr's MMAs (one thread) into TMEM columns tmem .. and commit them to mbar
__device__ __forceinline__ void xp_issue(const XpGeom &g, uint32_t sA, uint32_t sB, uint32_t tmem, int gr, int nd,
                                         uint32_t mbar) {
  // kind::f16: D fp32, A and B f16, both K-major; the fourth diagonal of group 3 is empty
  const uint32_t n = (uint32_t)((gr == 3 ? 3 : 4) * g.nb);
  const uint32_t idesc = (1u << 4) | (n >> 3) << 17 | (uint32_t)(XP_ROWS >> 4) << 24;
  const int q0 = max(0, 4 * gr - 7), q1 = min(nd - 1, 4 * gr + 3);
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
  uint32_t acc = 0;
  for (int q = q0; q <= q1; q++) {
    const uint32_t a = sA + q * g.a_dig(), b = sB + (uint32_t)(3 + 4 * gr - q) * g.b_blk();
    for (int kc = 0; kc < g.ks; kc++) {
      xp_mma(tmem, xp_desc(a + kc * 256, g.sbo()), xp_desc(b + kc * 256, g.sbo()), idesc, acc);
      acc = 1;
    }
  }
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(mbar));
}

// One limb of this thread's 16 sums from group gr's diagonals (live: the group was issued;
// else its sums are zero): limb = low word of carry + sum_j 256^j (P_j + bias), cy = high word.
__device__ __forceinline__ void xp_limb(const XpGeom &g, uint32_t tmem, int gr, bool live, uint32_t (&limb)[16],
                                        uint32_t (&cy)[16]) {
#pragma unroll
  for (int s = 0; s < 2; s++) {
    float p[4][8];
    if (live) {
#pragma unroll
      for (int j = 0; j < 4; j++)
        if (gr < 3 || j < 3) xp_ld16x16(tmem + ((uint32_t)(16 * s) << 16) + (uint32_t)(j * g.nb), p[j]);
      asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::);
    }
#pragma unroll
    for (int o = 0; o < 8; o++) {
      uint32_t b[4];
#pragma unroll
      for (int j = 0; j < 4; j++)
        b[j] = live && (gr < 3 || j < 3) ? __float_as_uint(__fadd_rn(p[j][o], XP_MAGIC)) : XP_BIAS;
      uint64_t t = (uint64_t)(b[0] + cy[8 * s + o]);   // below 2^31 + 2^24
      asm("mad.wide.u32 %0, %1, 256, %0;" : "+l"(t) : "r"(b[1]));
      asm("mad.wide.u32 %0, %1, 65536, %0;" : "+l"(t) : "r"(b[2]));
      asm("mad.wide.u32 %0, %1, 16777216, %0;" : "+l"(t) : "r"(b[3]));
      limb[8 * s + o] = (uint32_t)t;
      cy[8 * s + o] = (uint32_t)(t >> 32);
    }
  }
}

// Remove the bias from four limbs: the exact sum S, two's complement.
__device__ __forceinline__ void xp_unbias(uint32_t &a, uint32_t &b, uint32_t &c, uint32_t &d) {
  asm("sub.cc.u32 %0, %0, %4;\n\tsubc.cc.u32 %1, %1, %5;\n\tsubc.cc.u32 %2, %2, %6;\n\tsubc.u32 %3, %3, %7;\n\t"
      : "+r"(a), "+r"(b), "+r"(c), "+r"(d)
      : "n"(XP_B0), "n"(XP_B1), "n"(XP_B2), "n"(XP_B3));
}

__device__ __noinline__ double xp_value_rare(uint32_t a, uint32_t b, uint32_t c, uint32_t d, int E) {
  Acc128 A;
  A.lo = (uint64_t)a | ((uint64_t)b << 32);
  A.hi = (uint64_t)c | ((uint64_t)d << 32);
  return key_value(acc_key(A), E);
}

// The time of an exact sum: key_value(acc_key(S), E) of eval_common.cuh (57 leading bits,
// rounded once to FP64's 53) in one pass over the limbs.
__device__ __forceinline__ double xp_value(uint32_t a, uint32_t b, uint32_t c, uint32_t d, int E) {
  const uint32_t sg = (uint32_t)((int32_t)d >> 31);
  uint32_t x0 = a ^ sg, x1 = b ^ sg, x2 = c ^ sg, x3 = d ^ sg;
  asm("sub.cc.u32 %0, %0, %4;\n\tsubc.cc.u32 %1, %1, %4;\n\tsubc.cc.u32 %2, %2, %4;\n\tsubc.u32 %3, %3, %4;\n\t"
      : "+r"(x0), "+r"(x1), "+r"(x2), "+r"(x3)
      : "r"(sg));
  // the three limbs from the leading one down
  const bool p3 = x3 != 0, p2 = x2 != 0, p1 = x1 != 0;
  const uint32_t h = p3 ? x3 : p2 ? x2 : p1 ? x1 : x0;
  const uint32_t m = p3 ? x2 : p2 ? x1 : p1 ? x0 : 0;
  const uint32_t l = p3 ? x1 : p2 ? x0 : 0;
  const int lz = __clz((int)h);
  const uint32_t nh = __funnelshift_l(m, h, lz), nl = __funnelshift_l(l, m, lz);   // bit 31 of nh: the leading one
  const int x = (p3 ? 127 : p2 ? 95 : p1 ? 63 : 31) - lz - E + 1022;               // biased exponent - 1
  if (h == 0 || x < 0 || x > 2043) return xp_value_rare(a, b, c, d, E);
  uint64_t y = (((uint64_t)nh << 32) | nl) >> 7;   // 57 bits
  y += 7 + ((y >> 4) & 1);                         // to nearest, ties to even, at bit 4
  const uint64_t bits = (y >> 4) + ((uint64_t)(uint32_t)x << 52);
  return __longlong_as_double((long long)(bits | ((uint64_t)sg << 63)));
}

}  // namespace pmd
