// Launch interfaces between the host API layer and the CUDA kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace pmd {

// bits of the device status word
enum StatusBits { ST_OUT_OF_BOX = 1, ST_BAD_TABLE = 2, ST_TIMEOUT = 4, ST_BAD_INPUT = 8, ST_BAD_ROW = 16 };

// K1 (eval.cu)
// items: [n_items][4] (arena word offset low, first member, members, offset high); members: the table
// positions an item's rows are written to; max_words: the largest table
cudaError_t launch_eval_counts(const uint32_t *arena, const int32_t *items, const int32_t *members, int n_items,
                               int max_words, const int64_t *points, int64_t n_points, int P, int K, int64_t *out,
                               int *status, cudaStream_t st);

// Fused ranking (rank.cu).  A ranking group's image (32-bit words, 16-byte aligned
// sections; built by plan.cpp):
//   header [HDR_WORDS]: basis entries B, dependency levels, conditions, image words,
//     the end of each level (entries are ordered by level), section offsets;
//   basis definitions, 8 words each: [a0 a1 a2 a3 | b c magic kind] for an atom
//     floor((a . n + b) / c) (kind = 2 | shift << 8 | numerator-may-be-negative << 16),
//     [i j . . | . . . kind] for a parameter (kind 0, i = its index), the constant
//     (kind 1) or a product of entries i and j (kind 3);
//   conditions (at most 64): [n_terms, const_lo, const_hi, (entry, coef_lo, coef_hi) *
//     n_terms], bit q of a point's two mask words when const + sum coef * value >= 0:
//     the tables' piece conditions and the signs of undecided post-op differences A - B;
//     then the word offset of each condition in the image;
//   programs (one per distinct table), as records of four words:
//     condition node [1 | n << 8 | piece records << 16, condition ids 0-4 (6 bits each),
//       ids 5-9, LUT offset]: the LUT byte of the n condition bits names a piece record;
//     sub node [2 | n << 8, condition ids, children, 0]: child record = children + 4 * bits;
//     leaf [n64 << 8 | n32 << 16 | nwide << 24, term records, denominator block or 0,
//       constant present]: term records are the constant's 128-bit weight (if present),
//       then [w0 w1 w2 entry] per term with a 96-bit weight (n64 terms whose basis value
//       may leave [0, 2^32), then n32 terms), then [w0 w1 w2 w3][entry 0 0 0] per term
//       with a 128-bit weight; the denominator block is [shift, 0, 0, 0, d^-1 mod 2^128];
//   the program table, in walk order (by shape: every leaf of a program is padded to one
//     count of 64-bit- and of 32-bit-class terms): [root record offset | program id << 16],
//     program ids in the order of their first variants;
//   per program id its span [first entry | count << 16] in the list of variant indices (16
//     bits each), which holds at most the first 16 variants of each program;
//   runs of one shape [shape = n64 | n32 << 8 (0xFFFF: 128-bit weights), first position,
//     count, first program]; H_STAGED: the words up to here, which the kernel stages;
//   the whole walk, variant by variant (positions): per position the program's root record
//     offset and the variant's index in the group (16 bits each).
struct RankLayout {
  static constexpr int POINTS = 32;   // points per work unit: one per lane
  enum { H_B = 0, H_NLEV = 1, H_NCOND = 2, H_WORDS = 3, H_LEVEL_END = 4, H_OFF_BASIS = 12, H_OFF_COND = 13,
         H_OFF_VARMAP = 14, H_OFF_VIDMAP = 15, H_OFF_RUNS = 16, H_NRUNS = 17, H_NPROGS = 18, H_OFF_PROGS = 19, H_OFF_SPAN = 20,
         H_OFF_PVID = 21, H_STAGED = 22, H_OFF_CINDEX = 23, HDR_WORDS = 24 };
  static constexpr int SPAN_MAX = 16; // variants listed per program: the longest ranking
};
struct RankArgs {
  const uint32_t *img;         // every group's image (weights filled per call)
  const int4 *groups;          // [n_groups][2]: (image word offset, image words, first variant
                               //   (template-relative), variants), (template, group index in template, staged words, 0)
  const int4 *tmpl;            // [T][3]: (parameters, groups, 0, 0), box lo, box hi
  const int4 *chunks;          // [n_chunks] (template, first point, point count <= 32, first partial slot or -1)
  const int2 *units;           // [n_units] (chunk, group or -1 for a template without variants), schedule order
  int n_units;
  int *unit_counter;           // units handed out beyond the first of each CTA; 0 before each launch
  int *chunk_count;            // [n_chunks] groups finished; 0 before each launch
  int64_t *part_k;             // [slots][16][32] partial lists of chunks with several groups
  const int64_t *points;       // [total][4]
  const int *exponent;         // E of the fixed-point weights round(w 2^E)
  int topk;
  int32_t *top_idx;            // [total][topk]
  double *top_t;               // [total][topk]
  int *status;
  int img_words, basis_cap;    // shared-memory layout: the largest staged image and basis of the plan
};
cudaError_t launch_rank(const RankArgs &args, int nw, int grid, cudaStream_t st);
int rank_max_blocks_per_sm(int nw, int img_words, int basis_cap);
// fill the 128-bit term weights of the ranking programs from w (fp64 [32]), zero the
// launch's n_counters counters and write the weights' exponent E
cudaError_t launch_k2_weights(uint32_t *prog, const uint4 *targets, const uint4 *contrib, int n_targets,
                              const double *w, int *counters, int n_counters, int *exponent, cudaStream_t st);

// predict.cu
struct ArgPart { double t; int64_t r; };   // a partial per-model minimum: time and row
// per-model minimum over n_part partials part[p][M] (smaller time, then smaller row);
// n_part == 0 gives -1 and +inf
cudaError_t launch_argmin_reduce(const ArgPart *part, int n_part, int M, int64_t *arg, double *mn, cudaStream_t st);
cudaError_t launch_predict(const int64_t *F, int64_t R, int k, const double *W, int M, int precision, double *T,
                           int *status, cudaStream_t st);
// argmin: per-model partial results go to scratch (n_part [M] (double, int64) pairs), then reduced.
size_t argmin_scratch_bytes(int M, int n_part);
int argmin_parts();
cudaError_t launch_predict_argmin(const int64_t *F, int64_t R, int k, const double *W, int M, int precision,
                                  void *scratch, int64_t *arg, double *mn, int *status, cudaStream_t st);

// predict_exact.cu: the same exact sums from digit products on the tensor cores, for
// k <= 32 (exact_tc_ok); status (may be null) receives ST_TIMEOUT
bool exact_tc_ok(int k, int M);
cudaError_t launch_predict_exact(const int64_t *F, int64_t R, int k, const double *W, int M, double *T, int *status,
                                 int sms, cudaStream_t st);
cudaError_t launch_argmin_exact(const int64_t *F, int64_t R, int k, const double *W, int M, ArgPart *part, int n_part,
                                int *status, cudaStream_t st);
// a residual pass of the fit: predictions p = F w, then the residuals of the measured times
// T [R][M] as float-float (Qh, Ql), or (sums) the sums rr of their squares and bb of b^2
struct FitResidual {
  const double *T = nullptr;
  const float *rfh = nullptr, *rfl = nullptr;   // 1 / t (relative)
  float *Qh = nullptr, *Ql = nullptr;
  double *rr = nullptr, *bb = nullptr;          // [M]
  int ld = 0;                                   // row length of rf and Q: M rounded up to 4
  int relative = 0;
};
cudaError_t launch_fit_residual(const int64_t *F, int64_t R, int k, const double *W, int M, const FitResidual &res,
                                bool sums, int *status, int sms, cudaStream_t st);

// top-k rows per (group, model): work units of at most topk_chunk(...) positions of one
// group; a group of one unit is written directly (part < 0), the partial lists of the
// others ([part][M][topk]) are merged per group (TopkMerge)
constexpr int TOPK_MAX = 16;
constexpr int64_t TOPK_CHUNK = 1024;
// the kernel that M models over `total` positions in G groups take (row per lane, tensor
// cores, integer tile), and its largest unit
enum class TopkPath { ROWS, TENSOR, INTEGER };
TopkPath topk_path(int k, int M, int topk, int64_t total, int64_t G);
int64_t topk_chunk(int k, int M, int topk, int64_t total, int64_t G);
struct TopkUnit { int64_t p0, p1; int32_t g, part; };
struct TopkMerge { int32_t g, part0, n_parts, pad; };
// topk_exact.cu: more than a few models, k <= 32, on the tensor cores
cudaError_t launch_topk_exact(const int64_t *F, int64_t R, int k, const double *W, int M, const int64_t *rows,
                              const TopkUnit *units, int n_units, int topk, double *part_t, int64_t *part_r,
                              int64_t *top_idx, double *top_t, int *status, int sms, cudaStream_t st);
cudaError_t launch_predict_topk(const int64_t *F, int64_t R, int k, const double *W, int M, const int64_t *rows,
                                const TopkUnit *units, int n_units, const TopkMerge *merges, int n_merges, int topk,
                                double *part_t, int64_t *part_r, int64_t *top_idx, double *top_t, TopkPath path,
                                int *status, cudaStream_t st);

// predict_tc.cu (tensor cores, three-term bf16 split)
int tc_parts(int sms);
size_t tc_argmin_scratch_bytes(int M, int sms);
cudaError_t launch_predict_tc(const int64_t *F, int64_t R, int k, const double *W, int M, double *T, int64_t *arg,
                              double *mn, void *scratch, int sms, int *status, cudaStream_t st);

// serve.cu: one batch of queries, all arrays inside one device region
constexpr int SV_MAX_TOPK = 16;
struct SQuery {               // 24 bytes
  int64_t begin;              // first candidate of the query in the batch
  int32_t n;                  // candidates
  int32_t model;              // row of models
  int32_t topk;               // 1..16
  int32_t pad;
};
struct ServeArgs {
  const uint32_t *arena;      // compiled tables
  const SQuery *queries;
  int n_queries;
  const int2 *blocks;         // per k_serve_eval CTA: (query, chunk of 128 candidates)
  const uint32_t *cand_off;   // [N] arena word offset of each candidate's table
  const int64_t *points;      // [N][4]
  const double *models;       // [n_models][32]
  int64_t *keys;              // [N] scratch
  int32_t *q_status;          // [n_queries] status bits
  int32_t *out_idx;           // [n_queries][16]
  double *out_t;              // [n_queries][16]
};
cudaError_t launch_serve(const ServeArgs &a, int n_blocks, cudaStream_t st);

// fit.cu
struct FitHost {            // what the fit reports per model, copied to the host as one block
  int *info;                // [M][4] rank, zero columns, rank deficient, dropped-direction mask
  double *ratio, *upd, *rr, *bb;
};
constexpr size_t FIT_REPORT_BYTES = 16 + 4 * 8;   // per model
inline FitHost fit_report(void *p, int M) {
  double *d = (double *)((char *)p + (size_t)M * 16);
  return FitHost{(int *)p, d, d + M, d + 2 * M, d + 3 * M};
}
size_t fit_scratch_bytes(int64_t R, int k, int M);
// gram: 0 float-float (k_gram), 1 three bf16 terms (k_gram_pairs), 2 exact digits (k_gram_tc)
cudaError_t launch_fit(const int64_t *F, int64_t R, int k, const double *T, int M, int objective, int gram,
                       int steps, void *scratch, double *W_out, void *h_report, int *status, cudaStream_t st);
// Gram matrices of the fit on the tensor cores (add into G, upper triangle, [M][32][32])
cudaError_t launch_gram_pairs(const float *Uh, int ldu, const float *rfh, const float *rfl, int ld, int64_t R, int k, int M,
                              const unsigned *amax, const unsigned *rmax, double *G, int sms, int *status,
                              cudaStream_t st);
cudaError_t launch_gram_tc(const float *Uh, const float *Ul, int ldu, const float *rfh, const float *rfl, int ld, int64_t R,
                           int k, int M, const unsigned *amax, double *G, int sms, int *status, cudaStream_t st);

}  // namespace pmd
