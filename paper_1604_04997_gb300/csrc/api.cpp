// Host side of the C ABI: context, resident tables, argument checks, launches.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include "kernels.h"
#include "pm.h"
#include "pm_internal.h"
#include "pm_table.h"
#include "trace.h"

int pm_compile_table(const char *ir, size_t len, int layout, const int64_t *plo, const int64_t *phi,
                     std::vector<uint32_t> &words, int info[8], std::string &msg);

// Last error of the calling thread, in a fixed buffer (reporting an error allocates nothing).
static thread_local char g_err[512];

pm_status pm_set_error_c(pm_status code, const char *m) {
  size_t n = 0;
  while (m[n] && n < sizeof(g_err) - 1) { g_err[n] = m[n]; n++; }
  g_err[n] = 0;
  return code;
}

pm_status pm_set_error(pm_status code, const std::string &m) { return pm_set_error_c(code, m.c_str()); }

extern "C" const char *pm_last_error(void) { return g_err; }

#define CU(x)                                                                                          \
  do {                                                                                                 \
    cudaError_t e__ = (x);                                                                             \
    if (e__ != cudaSuccess) return pm_set_error(PM_ERR_CUDA, std::string(#x) + ": " + cudaGetErrorString(e__)); \
  } while (0)

// ------------------------------------------------------------------------------------- context

pm_status ctx_device_guard(pm_ctx *c) {
  if (!c) return pm_set_error(PM_ERR_INVALID_ARG, "null context");
  if (c->device < 0) return pm_set_error(PM_ERR_INVALID_ARG, "host-only context has no device");
  CU(cudaSetDevice(c->device));
  return PM_OK;
}

extern "C" pm_status pm_create(pm_ctx **out, int device, size_t mem_budget_bytes) {
  if (!out) return pm_set_error(PM_ERR_INVALID_ARG, "out is null");
  *out = nullptr;
  std::unique_ptr<pm_ctx> c(new pm_ctx());
  c->device = device;
  c->budget = mem_budget_bytes ? mem_budget_bytes : (size_t(16) << 30);
  if (device >= 0) {
    int n = 0;
    CU(cudaGetDeviceCount(&n));
    if (device >= n) return pm_set_error(PM_ERR_INVALID_ARG, "no such device");
    CU(cudaSetDevice(device));
    CU(cudaMalloc(&c->d_status, sizeof(int)));
    CU(cudaMemset(c->d_status, 0, sizeof(int)));
    CU(cudaMallocHost(&c->h_status, sizeof(int)));
    CU(cudaDeviceGetAttribute(&c->n_sms, cudaDevAttrMultiProcessorCount, device));
  }
  *out = c.release();
  return PM_OK;
}

extern "C" void pm_destroy(pm_ctx *c) {
  if (!c) return;
  serve_destroy(c);
  if (c->device >= 0) {
    cudaSetDevice(c->device);
    cudaDeviceSynchronize();
    for (auto &kv : c->dcache) cudaFree(kv.second);
    for (auto &kv : c->plans) {
      if (kv.second->graph_exec) cudaGraphExecDestroy(kv.second->graph_exec);
      for (void *p : kv.second->dev) cudaFree(p);
      delete kv.second;
    }
    cudaFree(c->arena);
    cudaFree(c->d_status);
    cudaFree(c->scratch);
    cudaFreeHost(c->h_status);
    if (c->fit_host) cudaFreeHost(c->fit_host);
  }
  delete c;
}

extern "C" pm_status pm_sync_status(pm_ctx *c, void *stream) {
  pm_status g = ctx_device_guard(c);
  if (g) return g;
  cudaStream_t st = (cudaStream_t)stream;
  CU(cudaMemcpyAsync(c->h_status, c->d_status, sizeof(int), cudaMemcpyDeviceToHost, st));
  CU(cudaMemsetAsync(c->d_status, 0, sizeof(int), st));
  CU(cudaStreamSynchronize(st));
  int s = *c->h_status;
  if (s & pmd::ST_OUT_OF_BOX) return pm_set_error(PM_ERR_OUT_OF_BOX, "a parameter point lies outside its table's box");
  if (s & pmd::ST_BAD_TABLE) return pm_set_error(PM_ERR_INVALID_ARG, "malformed table reached the device");
  if (s & pmd::ST_TIMEOUT) return pm_set_error(PM_ERR_TIMEOUT, "a device wait ran out");
  if (s & pmd::ST_BAD_INPUT) return pm_set_error(PM_ERR_INVALID_ARG, "a timing is not positive and finite");
  if (s & pmd::ST_BAD_ROW) return pm_set_error(PM_ERR_INVALID_ARG, "a listed row lies outside [0, R)");
  return PM_OK;
}

// Device copy of a small host array, cached by content (schedules, offsets).
pm_status ctx_dcopy(pm_ctx *c, const void *h, size_t bytes, void **d) {
  std::string key((const char *)h, bytes);
  auto it = c->dcache.find(key);
  if (it != c->dcache.end()) { *d = it->second; return PM_OK; }
  if (c->dcache.size() > 4096) {
    CU(cudaDeviceSynchronize());
    for (auto &kv : c->dcache) cudaFree(kv.second);
    c->dcache.clear();
    c->eval_plans.clear();   // their device arrays are in dcache
  }
  void *p = nullptr;
  CU(cudaMalloc(&p, std::max<size_t>(bytes, 16)));
  CU(cudaMemcpy(p, h, bytes, cudaMemcpyHostToDevice));
  c->dcache[key] = p;
  *d = p;
  return PM_OK;
}

pm_status ctx_scratch(pm_ctx *c, size_t bytes, void **d) {
  if (bytes > c->scratch_cap) {
    CU(cudaDeviceSynchronize());
    cudaFree(c->scratch);
    c->scratch = nullptr;
    c->scratch_cap = 0;
    CU(cudaMalloc(&c->scratch, bytes));
    c->scratch_cap = bytes;
  }
  *d = c->scratch;
  return PM_OK;
}

static pm_status upload_table(pm_ctx *c, int id) {
  const auto &w = c->tables[id];
  if (c->canon[id] != id) {   // the same words are there already
    c->dev_off[id] = c->dev_off[c->canon[id]];
    return PM_OK;
  }
  size_t need = c->arena_used + w.size();
  if (need > c->arena_cap) {
    size_t cap = std::max<size_t>(need * 2, size_t(1) << 20);
    uint32_t *na = nullptr;
    CU(cudaMalloc(&na, cap * 4));
    if (c->arena_used) CU(cudaMemcpy(na, c->arena, c->arena_used * 4, cudaMemcpyDeviceToDevice));
    CU(cudaDeviceSynchronize());
    cudaFree(c->arena);
    c->arena = na;
    c->arena_cap = cap;
  }
  CU(cudaMemcpy(c->arena + c->arena_used, w.data(), w.size() * 4, cudaMemcpyHostToDevice));
  c->dev_off[id] = (int64_t)c->arena_used;
  c->arena_used += w.size();
  return PM_OK;
}

// ------------------------------------------------------------------------------------- counting

// Add a table's image: its id, and the first table with the same image (tables of equal
// images are evaluated once, and share their device words).
static pm_status add_table(pm_ctx *c, std::vector<uint32_t> words, int *out_id) {
  const int id = (int)c->tables.size();
  uint64_t h = 1469598103934665603ull;   // FNV-1a over the words
  for (uint32_t w : words) h = (h ^ w) * 1099511628211ull;
  auto &same = c->by_hash[h];
  int canon = id;
  for (int t : same)
    if (c->tables[t] == words) { canon = t; break; }
  c->tables.push_back(std::move(words));
  c->dev_off.push_back(-1);
  c->canon.push_back(canon);
  if (canon == id) same.push_back(id);
  if (c->device >= 0) {
    pm_status s = ctx_device_guard(c);
    if (!s) s = upload_table(c, id);
    if (s) {   // taken back out, so that no id refers to a table without device words
      if (canon == id) c->by_hash[h].pop_back();
      c->tables.pop_back();
      c->dev_off.pop_back();
      c->canon.pop_back();
      return s;
    }
  }
  *out_id = id;
  return PM_OK;
}

extern "C" pm_status pm_compile_counts(pm_ctx *c, const char *ir, size_t len, int32_t layout, const int64_t *lo,
                                       const int64_t *hi, int32_t *out_id, pm_table_info *info) {
  PM_TRACE("pm_compile_counts");
  if (!c || !ir || !lo || !hi || !out_id) return pm_set_error(PM_ERR_INVALID_ARG, "null argument");
  if (layout != PM_LAYOUT_12 && layout != PM_LAYOUT_32) return pm_set_error(PM_ERR_INVALID_ARG, "layout must be 12 or 32");
  std::vector<uint32_t> words;
  int inf[8];
  std::string msg;
  int rc = pm_compile_table(ir, len, layout, lo, hi, words, inf, msg);
  if (rc) return pm_set_error(rc, msg);
  std::lock_guard<std::mutex> lk(c->mu);
  if (pm_status u = add_table(c, std::move(words), out_id)) return u;
  if (info) {
    info->n_params = inf[0]; info->n_atoms = inf[1]; info->n_conds = inf[2]; info->n_pieces = inf[3];
    info->n_monomials = inf[4]; info->n_columns = inf[5]; info->n_words = inf[6]; info->degree = inf[7];
  }
  return PM_OK;
}

bool pm_table_valid(const uint32_t *w, size_t n, std::string &why);   // table_check.cpp

extern "C" pm_status pm_table_load(pm_ctx *c, const uint32_t *words, size_t n_words, int32_t *out_id) {
  PM_TRACE("pm_table_load");
  if (!c || !words || !out_id) return pm_set_error(PM_ERR_INVALID_ARG, "null argument");
  std::string why;
  if (!pm_table_valid(words, n_words, why)) return pm_set_error(PM_ERR_INVALID_ARG, "table image rejected: " + why);
  std::lock_guard<std::mutex> lk(c->mu);
  return add_table(c, std::vector<uint32_t>(words, words + n_words), out_id);
}

extern "C" pm_status pm_table_image(pm_ctx *c, int32_t id, uint32_t *buf, size_t cap, size_t *out_words) {
  if (!c || id < 0 || id >= (int)c->tables.size()) return pm_set_error(PM_ERR_NOT_FOUND, "no such table");
  const auto &w = c->tables[id];
  if (out_words) *out_words = w.size();
  if (buf) {
    if (cap < w.size()) return pm_set_error(PM_ERR_INVALID_ARG, "buffer too small");
    std::memcpy(buf, w.data(), w.size() * 4);
  }
  return PM_OK;
}

static pm_status eval_plan(pm_ctx *c, const int32_t *ids, int n, const EvalPlan **out) {
  // by the first tables of equal images: a list of other ids with the same images is the same,
  // so there are no more plans than device arrays in dcache, which is bounded
  std::string key((size_t)n * sizeof(int), 0);
  for (int i = 0; i < n; i++) {
    if (ids[i] < 0 || ids[i] >= (int)c->tables.size()) return pm_set_error(PM_ERR_NOT_FOUND, "unknown table id");
    memcpy(&key[i * sizeof(int)], &c->canon[ids[i]], sizeof(int));
  }
  auto it = c->eval_plans.find(key);
  if (it != c->eval_plans.end()) { *out = &it->second; return PM_OK; }
  EvalPlan p;
  std::unordered_map<int, int> slot;             // canonical table -> its members
  std::vector<std::vector<int32_t>> members;
  std::vector<int> tab;
  for (int i = 0; i < n; i++) {
    const int id = c->canon[ids[i]];
    const auto &w = c->tables[id];
    if (i == 0) { p.P = (int)w[pmt::H_NPARAMS]; p.K = (int)w[pmt::H_K]; }
    if (p.P != (int)w[pmt::H_NPARAMS]) return pm_set_error(PM_ERR_INVALID_ARG, "tables differ in parameter count");
    if (p.K != (int)w[pmt::H_K]) return pm_set_error(PM_ERR_INVALID_ARG, "tables differ in layout");
    if (c->dev_off[id] < 0) return pm_set_error(PM_ERR_INVALID_ARG, "table not on the device");
    const auto at = slot.emplace(id, (int)tab.size());
    if (at.second) {
      tab.push_back(id);
      members.emplace_back();
      p.max_words = std::max(p.max_words, (int)w.size());
    }
    members[at.first->second].push_back(i);
  }
  std::vector<int32_t> list, first;              // the members, table by table
  int most = 0;
  for (auto &m : members) {
    first.push_back((int32_t)list.size());
    list.insert(list.end(), m.begin(), m.end());
    most = std::max(most, (int)m.size());
  }
  list.resize((list.size() + 3) & ~(size_t)3);   // the items are read as 16-byte records
  size_t at[EVAL_ITEM];
  for (int per = 1; per <= EVAL_ITEM; per++) {
    p.n_items[per - 1] = per > 1 && per > most ? p.n_items[per - 2] : 0;   // the same items again
    at[per - 1] = p.n_items[per - 1] ? at[per - 2] : list.size();
    if (p.n_items[per - 1]) continue;
    for (size_t t = 0; t < tab.size(); t++) {
      const int cnt = (int)members[t].size();
      const int64_t off = c->dev_off[tab[t]];
      for (int m = 0; m < cnt; m += per) {
        list.insert(list.end(), {(int32_t)(uint32_t)off, first[t] + m, std::min(per, cnt - m), (int32_t)(off >> 32)});
        p.n_items[per - 1]++;
      }
    }
  }
  void *d = nullptr;
  pm_status s = ctx_dcopy(c, list.data(), list.size() * sizeof(int32_t), &d);
  if (s) return s;
  p.members = (const int32_t *)d;
  for (int i = 0; i < EVAL_ITEM; i++) p.items[i] = p.members + at[i];
  *out = &(c->eval_plans[key] = p);
  return PM_OK;
}

// Test hook: the work lists that pm_eval_counts keeps.
extern "C" int pmx_eval_plans(const pm_ctx *c) { return c ? (int)c->eval_plans.size() : -1; }

extern "C" pm_status pm_eval_counts(pm_ctx *c, const int32_t *ids, int32_t n_tables, const int64_t *d_points,
                                    int64_t n_points, int64_t *d_counts, void *stream) {
  PM_TRACE("pm_eval_counts");
  pm_status g = ctx_device_guard(c);
  if (g) return g;
  if (n_tables < 0 || n_points < 0 || (n_tables && !ids)) return pm_set_error(PM_ERR_INVALID_ARG, "bad sizes");
  if (n_tables == 0 || n_points == 0) return PM_OK;
  if (!d_points || !d_counts) return pm_set_error(PM_ERR_INVALID_ARG, "null device buffer");
  // the launch puts points on grid x (128 per block) and work items on grid y (at most 65,535)
  if (n_points > (int64_t(1) << 37)) return pm_set_error(PM_ERR_INVALID_ARG, "too many points");
  // A block evaluates 128 points of one table and writes the rows of up to eight positions
  // that name it: about 2,800 blocks of eight take 109 us where 21,248 of one took 201 (2,656
  // tables x 1,024 points).  Fewer positions a block where that would leave fewer than 16
  // blocks per SM (three are resident): small calls keep one block per position.
  const int64_t chunks = (n_points + 127) / 128;
  const int per = (int)std::min<int64_t>(EVAL_ITEM, std::max<int64_t>(1, chunks * n_tables / ((int64_t)c->n_sms * 16)));
  const EvalPlan *p = nullptr;
  pm_status s = eval_plan(c, ids, n_tables, &p);
  if (s) return s;
  constexpr int64_t MAX_GRID_Y = 65535;
  const int n_items = p->n_items[per - 1];
  for (int64_t t0 = 0; t0 < n_items; t0 += MAX_GRID_Y)
    CU(pmd::launch_eval_counts(c->arena, p->items[per - 1] + 4 * t0, p->members, (int)std::min<int64_t>(MAX_GRID_Y, n_items - t0),
                               p->max_words, d_points, n_points, p->P, p->K, d_counts, c->d_status, (cudaStream_t)stream));
  return PM_OK;
}

// ------------------------------------------------------------------------------------- prediction

extern "C" pm_status pm_predict(pm_ctx *c, const int64_t *F, int64_t R, int32_t k, const double *W, int32_t M,
                                int32_t precision, double *T, void *stream) {
  PM_TRACE("pm_predict");
  pm_status g = ctx_device_guard(c);
  if (g) return g;
  if (R < 0 || k <= 0 || M <= 0) return pm_set_error(PM_ERR_INVALID_ARG, "bad sizes");
  if (R == 0) return PM_OK;
  if (!F || !W || !T) return pm_set_error(PM_ERR_INVALID_ARG, "null device buffer");
  if (precision == PM_PREC_BF16X3) return pm_predict_bf16x3(c, F, R, k, W, M, T, nullptr, nullptr, stream);
  if (precision != PM_PREC_FP64 && precision != PM_PREC_NATIVE_FP64)
    return pm_set_error(PM_ERR_INVALID_ARG, "unknown precision");
  if (precision == PM_PREC_FP64 && (k > 40 || M > 64)) return pm_set_error(PM_ERR_INVALID_ARG, "k <= 40 and M <= 64");
  CU(pmd::launch_predict(F, R, k, W, M, precision, T, c->d_status, (cudaStream_t)stream));
  return PM_OK;
}

extern "C" pm_status pm_predict_argmin(pm_ctx *c, const int64_t *F, int64_t R, int32_t k, const double *W,
                                       int32_t M, int32_t precision, int64_t *arg, double *mn, void *stream) {
  PM_TRACE("pm_predict_argmin");
  pm_status g = ctx_device_guard(c);
  if (g) return g;
  if (R < 0 || k <= 0 || k > 40 || M <= 0 || M > 64) return pm_set_error(PM_ERR_INVALID_ARG, "bad sizes");
  if ((!F && R > 0) || !W || !arg || !mn) return pm_set_error(PM_ERR_INVALID_ARG, "null device buffer");
  if (precision == PM_PREC_BF16X3) return pm_predict_bf16x3(c, F, R, k, W, M, nullptr, arg, mn, stream);
  if (precision != PM_PREC_FP64) return pm_set_error(PM_ERR_INVALID_ARG, "argmin supports PM_PREC_FP64 and PM_PREC_BF16X3");
  void *scr = nullptr;
  pm_status s = ctx_scratch(c, pmd::argmin_scratch_bytes(M, pmd::argmin_parts()), &scr);
  if (s) return s;
  CU(pmd::launch_predict_argmin(F, R, k, W, M, precision, scr, arg, mn, c->d_status, (cudaStream_t)stream));
  return PM_OK;
}

extern "C" pm_status pm_predict_topk(pm_ctx *c, const int64_t *F, int64_t R, int32_t k, const double *W, int32_t M,
                                     int32_t precision, const int64_t *h_seg_off, int32_t G, const int64_t *d_rows,
                                     int32_t topk, int64_t *d_top_idx, double *d_top_t, void *stream) {
  PM_TRACE("pm_predict_topk");
  pm_status g = ctx_device_guard(c);
  if (g) return g;
  if (R < 0 || k <= 0 || k > 40 || M <= 0 || M > 64 || G < 0 || topk < 1 || topk > pmd::TOPK_MAX)
    return pm_set_error(PM_ERR_INVALID_ARG, "bad sizes (need 0 < k <= 40, 0 < M <= 64, G >= 0, 1 <= topk <= 16)");
  if (precision != PM_PREC_FP64) return pm_set_error(PM_ERR_INVALID_ARG, "pm_predict_topk supports PM_PREC_FP64");
  if (G == 0) return PM_OK;
  if (!h_seg_off || !W || !d_top_idx || !d_top_t || (!F && R > 0)) return pm_set_error(PM_ERR_INVALID_ARG, "null buffer");
  if (h_seg_off[0] < 0) return pm_set_error(PM_ERR_INVALID_ARG, "group offsets must start at 0 or above");
  for (int32_t i = 0; i < G; i++)
    if (h_seg_off[i + 1] < h_seg_off[i]) return pm_set_error(PM_ERR_INVALID_ARG, "group offsets must be non-decreasing");
  if (!d_rows && h_seg_off[G] > R) return pm_set_error(PM_ERR_INVALID_ARG, "without a row list the groups must lie in [0, R)");
  // work units: groups cut into even chunks; a one-chunk group
  // (an empty one too) is written directly, the others through partial lists
  std::vector<pmd::TopkUnit> units;
  std::vector<pmd::TopkMerge> merges;
  int64_t parts = 0;
  const int64_t total = h_seg_off[G] - h_seg_off[0], most = pmd::topk_chunk(k, M, topk, total, G);
  for (int32_t i = 0; i < G; i++) {
    const int64_t p0 = h_seg_off[i], p1 = h_seg_off[i + 1];
    const int64_t nch = std::max<int64_t>(1, (p1 - p0 + most - 1) / most);
    const int64_t each = ((p1 - p0 + nch - 1) / nch + 31) & ~(int64_t)31;   // a multiple of 32, at most `most`
    if (nch == 1) {
      units.push_back(pmd::TopkUnit{p0, p1, i, -1});
      continue;
    }
    if (parts + nch > INT32_MAX) return pm_set_error(PM_ERR_INVALID_ARG, "too many rows");
    merges.push_back(pmd::TopkMerge{i, (int32_t)parts, (int32_t)nch, 0});
    for (int64_t q = 0; q < nch; q++)
      units.push_back(pmd::TopkUnit{std::min(p1, p0 + q * each), std::min(p1, p0 + (q + 1) * each), i,
                                    (int32_t)(parts + q)});
    parts += nch;
  }
  if (units.size() > (size_t)INT32_MAX) return pm_set_error(PM_ERR_INVALID_ARG, "too many groups");
  const size_t ub = units.size() * sizeof(pmd::TopkUnit), mb = merges.size() * sizeof(pmd::TopkMerge);
  std::vector<uint8_t> meta(ub + mb);
  std::memcpy(meta.data(), units.data(), ub);
  if (mb) std::memcpy(meta.data() + ub, merges.data(), mb);
  void *d_meta = nullptr, *scr = nullptr;
  pm_status s = ctx_dcopy(c, meta.data(), meta.size(), &d_meta);
  if (s) return s;
  const size_t pb = (size_t)parts * M * topk * sizeof(double);
  if (parts) {
    s = ctx_scratch(c, 2 * pb, &scr);
    if (s) return s;
  }
  CU(pmd::launch_predict_topk(F, R, k, W, M, d_rows, (const pmd::TopkUnit *)d_meta, (int)units.size(),
                              (const pmd::TopkMerge *)((uint8_t *)d_meta + ub), (int)merges.size(), topk,
                              (double *)scr, (int64_t *)((uint8_t *)scr + pb), d_top_idx, d_top_t,
                              pmd::topk_path(k, M, topk, total, G), c->d_status, (cudaStream_t)stream));
  return PM_OK;
}

// Tensor-core path (three-term bf16 split, FP32 accumulation): T, or per-model argmin.
pm_status pm_predict_bf16x3(pm_ctx *c, const int64_t *F, int64_t R, int k, const double *W, int M, double *T,
                            int64_t *arg, double *mn, void *stream) {
  if (k != 32 || M > 64) return pm_set_error(PM_ERR_INVALID_ARG, "PM_PREC_BF16X3 needs k == 32 and M <= 64");
  if ((uintptr_t)F % 16 != 0) return pm_set_error(PM_ERR_INVALID_ARG, "PM_PREC_BF16X3 needs F 16-byte aligned");
  void *scr = nullptr;
  if (arg) {
    pm_status s = ctx_scratch(c, pmd::tc_argmin_scratch_bytes(M, c->n_sms), &scr);
    if (s) return s;
  }
  CU(pmd::launch_predict_tc(F, R, k, W, M, T, arg, mn, scr, c->n_sms, c->d_status, (cudaStream_t)stream));
  return PM_OK;
}

// ------------------------------------------------------------------------------------- batched eval+predict+top-k

extern "C" pm_status pm_eval_predict_topk(pm_ctx *c, const int32_t *tables, const int32_t *var_off,
                                          int32_t n_templates, const int64_t *d_points, const int64_t *pt_off,
                                          const double *d_w, int32_t topk, int32_t *d_top_idx, double *d_top_t,
                                          void *stream) {
  PM_TRACE("pm_eval_predict_topk");
  pm_status g = ctx_device_guard(c);
  if (g) return g;
  if (n_templates <= 0 || !tables || !var_off || !pt_off || !d_points || !d_w || !d_top_idx || !d_top_t)
    return pm_set_error(PM_ERR_INVALID_ARG, "null argument");
  if (topk < 1 || topk > PM_MAX_TOPK) return pm_set_error(PM_ERR_INVALID_ARG, "topk must be 1..16");
  Plan *plan = nullptr;
  pm_status s = ctx_plan_k2(c, tables, var_off, n_templates, pt_off, &plan);
  if (s) return s;
  return ctx_run_k2(c, plan, tables, var_off, pt_off, d_points, d_w, topk, d_top_idx, d_top_t, (cudaStream_t)stream);
}

// ------------------------------------------------------------------------------------- fit (Sec. 4.3)

extern "C" pm_status pm_fit_weights(pm_ctx *c, const int64_t *F, int64_t R, int32_t k, const double *T, int32_t M,
                                    int32_t objective, int32_t precision, int32_t refine_steps, double *W_out,
                                    pm_fit_report *rep, void *stream) {
  PM_TRACE("pm_fit_weights");
  pm_status g = ctx_device_guard(c);
  if (g) return g;
  if (R <= 0 || k <= 0 || k > 32 || M <= 0 || M > 64 || refine_steps < 0 || refine_steps > 50)
    return pm_set_error(PM_ERR_INVALID_ARG, "need R > 0, 0 < k <= 32, 0 < M <= 64, 0 <= refine_steps <= 50");
  if (!F || !T || !W_out || !rep) return pm_set_error(PM_ERR_INVALID_ARG, "null argument");
  if (objective != PM_FIT_RELATIVE && objective != PM_FIT_ABSOLUTE) return pm_set_error(PM_ERR_INVALID_ARG, "objective");
  if (precision != PM_PREC_FP64 && precision != PM_PREC_BF16X3) return pm_set_error(PM_ERR_INVALID_ARG, "precision");
  void *scr = nullptr;
  pm_status s = ctx_scratch(c, pmd::fit_scratch_bytes(R, k, M), &scr);
  if (s) return s;
  if (!c->fit_host) CU(cudaMallocHost(&c->fit_host, 64 * pmd::FIT_REPORT_BYTES));
  const pmd::FitHost h = pmd::fit_report(c->fit_host, M);
  cudaStream_t st = (cudaStream_t)stream;
  // PM_PREC_BF16X3: the Gram from three bf16 terms first, within 2^-21 (1,000 rows) to 2^-18
  // (200,000) of its diagonal; refinement with exact residuals makes the weights accurate when
  // cond(G) 2^-18 is well below one.  If some model's last correction is still large, or
  // without refinement its smallest pivot is known to less than a hundredth, or its factor reports a rank
  // drop that the exact Gram may not have, the fit is repeated with the exact digit Gram.
  int gram = precision == PM_PREC_BF16X3 ? 1 : 0;
  for (;;) {
    CU(pmd::launch_fit(F, R, k, T, M, objective, gram, refine_steps, scr, W_out, c->fit_host, c->d_status, st));
    s = pm_sync_status(c, stream);
    if (s) return s;
    if (gram != 1) break;
    bool converged = true;
    for (int m = 0; m < M; m++)
      converged &= h.info[m * 4 + 2] == 0 && (refine_steps ? h.upd[m] < 1e-10 : h.ratio[m] < 0x1p12);
    if (converged) break;
    gram = 2;
  }
  bool deficient = false;
  for (int m = 0; m < M; m++) {
    pm_fit_report &r = rep[m];
    r.rank = h.info[m * 4 + 0];
    r.n_dropped = h.info[m * 4 + 1];
    r.iters = refine_steps;
    r.cond_est = h.ratio[m];
    r.rel_resid = h.bb[m] > 0 ? std::sqrt(h.rr[m] / h.bb[m]) : 0.0;
    r.last_update = h.upd[m];
    r.status = h.info[m * 4 + 2] ? 1 : (refine_steps > 0 && !(r.last_update < 1e-6) ? 2 : 0);
    deficient |= h.info[m * 4 + 2] != 0;
  }
  return deficient ? PM_WARN_RANK_DEFICIENT : PM_OK;
}
