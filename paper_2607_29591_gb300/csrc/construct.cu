// Construction of the compressed cache (Alg. 1), layer by layer, on the
// caller's stream.  Every step is a kernel of construct_kernels.cuh; the host
// only validates, sizes the scratch buffers and sequences the launches.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "construct_kernels.cuh"
#include "lloyd_assign.cuh"
#include "internal.h"

namespace reskv {

reskv_status alloc_handle(const reskv_config& cfg, cudaStream_t stream, reskv_cache** out);
void release_handle(reskv_cache* c);
reskv_status finalize_ragged_layout(reskv_cache* c);

namespace {

using namespace build;

reskv_status fail(reskv_status st, const std::string& msg) {
  set_error(msg);
  return st;
}

// The construction's scratch arrays, in one device allocation: every cudaMalloc
// and cudaFree costs 10 us of host time beside its kernels, up to 700 for 1 GB (a
// build of 8 units of 32K keys spent 1.4 of its 5.3 ms on 37 pairs of them).  get() places
// an array, commit() allocates and sets every pointer.
class Scratch {
 public:
  ~Scratch() {
    if (block_) cudaFree(block_);
  }
  template <typename T>
  void get(T** p, size_t count) {
    *p = nullptr;
    arrays_.push_back({reinterpret_cast<void**>(p), size_});
    size_ += (std::max<size_t>(count, 1) * sizeof(T) + 255) & ~size_t(255);
  }
  bool commit() {
    if (device_alloc(&block_, size_) != cudaSuccess) {
      cudaGetLastError();
      block_ = nullptr;
      return false;
    }
    for (const Array& a : arrays_) *a.p = static_cast<uint8_t*>(block_) + a.offset;
    return true;
  }

 private:
  struct Array {
    void** p;
    size_t offset;
  };
  std::vector<Array> arrays_;
  size_t size_ = 0;
  void* block_ = nullptr;
};

#define RESKV_LAUNCH_CHECK(what)                                                      \
  do {                                                                               \
    cudaError_t e_ = cudaGetLastError();                                             \
    if (e_ != cudaSuccess)                                                           \
      return fail(RESKV_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e_)); \
  } while (0)

template <typename K>
cudaError_t set_smem(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
}

int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

// One cluster of CTAs of kTopThreads threads per item: as many CTAs as the SMs
// hold (a power of two, at most 8).
template <typename Kernel, typename Args>
cudaError_t launch_clusters(Kernel kernel, int items, int num_sms, size_t smem, cudaStream_t stream, const Args& args) {
  int cs = 8;
  while (cs > 1 && int64_t(items) * cs > num_sms) cs /= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(items) * unsigned(cs), 1, 1);
  cfg.blockDim = dim3(kTopThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = unsigned(cs);
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args);
}

// Device time per construction stage: an event is recorded on the stream at
// every stage boundary of a layer; at the end of the layer the intervals are
// added to their stages (events are reused from layer to layer).
class StageTimer {
 public:
  explicit StageTimer(cudaStream_t s) : stream_(s) {}
  ~StageTimer() {
    for (cudaEvent_t e : pool_) cudaEventDestroy(e);
  }
  // the interval that starts now belongs to `stage` (-1: not timed)
  bool mark(int stage) {
    if (n_ == pool_.size()) {
      cudaEvent_t e;
      if (cudaEventCreate(&e) != cudaSuccess) return false;
      pool_.push_back(e);
    }
    stage_.resize(n_ + 1);
    stage_[n_] = stage;
    return cudaEventRecord(pool_[n_++], stream_) == cudaSuccess;
  }
  // close the layer: wait for its last event, accumulate, start over
  bool flush(float* ms) {
    if (n_ == 0) return true;
    if (cudaEventSynchronize(pool_[n_ - 1]) != cudaSuccess) return false;
    for (size_t i = 0; i + 1 < n_; ++i) {
      float t = 0.f;
      if (cudaEventElapsedTime(&t, pool_[i], pool_[i + 1]) != cudaSuccess) return false;
      if (stage_[i] >= 0) ms[stage_[i]] += t;
    }
    n_ = 0;
    return true;
  }

 private:
  cudaStream_t stream_;
  std::vector<cudaEvent_t> pool_;
  std::vector<int> stage_;
  size_t n_ = 0;
};

enum { kStScore = 0, kStRank, kStValTargets, kStLloyd, kStValLoss, kStPack };

}  // namespace

reskv_status build_all_layers(reskv_cache** out, const reskv_config& cfg,
                              const int32_t* override_host, const void* const* Kl,
                              const void* const* Vl, const void* const* Ql, cudaStream_t stream) {
  // ---------------- validation ----------------
  const int64_t s = cfg.seq_len;
  const int b = cfg.budget;
  if (cfg.recent_window < 0) return fail(RESKV_ERR_INVALID_ARG, "recent_window must be >= 0");
  const int P = int(std::min<int64_t>(cfg.recent_window, s));
  const int UL = cfg.batch * cfg.n_kv_heads;
  const int G = cfg.group;
  const int64_t U_all = int64_t(cfg.n_layers) * UL;
  if (cfg.budget_mode != RESKV_BUDGET_UNIFORM && cfg.budget_mode != RESKV_BUDGET_ADAKV)
    return fail(RESKV_ERR_INVALID_ARG, "unknown budget_mode");
  // AdaKV allocation across the KV heads of each (layer, batch element); with
  // b >= s nothing is evicted and the layout keeps one budget
  const bool adakv = cfg.budget_mode == RESKV_BUDGET_ADAKV && int64_t(b) < s;
  if (cfg.budget_mode == RESKV_BUDGET_ADAKV) {
    if (cfg.unit_budgets)
      return fail(RESKV_ERR_INVALID_ARG, "budget_mode ADAKV allocates the budgets: unit_budgets must be NULL");
    if (!(cfg.adakv_safeguard >= 0.f && cfg.adakv_safeguard <= 1.f))
      return fail(RESKV_ERR_INVALID_ARG, "adakv_safeguard must be in [0, 1]");
  }
  const bool per_unit = cfg.unit_budgets != nullptr || adakv;
  const int n_free_head = b - P;                       // selectable slots per head (AdaKV)
  const int ada_f = adakv ? std::min(n_free_head, std::max(0, int(std::floor(
                                double(cfg.adakv_safeguard) * double(n_free_head))))) : 0;
  if (adakv && double(cfg.n_kv_heads) * double(s) >= double(int64_t(1) << 31))
    return fail(RESKV_ERR_UNSUPPORTED, "AdaKV: n_kv_heads * seq_len must be < 2^31");
  if (adakv && n_free_head > kTopMax)
    return fail(RESKV_ERR_UNSUPPORTED, "AdaKV: budget - recent_window must be <= 8192");
  // the largest budget a unit can get (sizes the scratch), and whether any unit evicts
  int64_t b_hi = b;
  bool any_evict = int64_t(b) < s;
  if (cfg.unit_budgets) {
    b_hi = 0;
    any_evict = false;
    for (int64_t u = 0; u < U_all; ++u) {
      const int64_t bu = cfg.unit_budgets[u];
      if (std::min(bu, s) < P)
        return fail(RESKV_ERR_INVALID_ARG, "unit_budgets must be >= min(recent_window, seq_len)");
      b_hi = std::max(b_hi, bu);
      any_evict |= bu < s;
    }
  } else if (int64_t(std::min<int64_t>(b, s)) < P) {
    return fail(RESKV_ERR_INVALID_ARG, "budget must be >= min(recent_window, seq_len)");
  }
  if (adakv)   // |P| + f + every shared slot, within s and the ranking limit
    b_hi = std::min<int64_t>(std::min<int64_t>(s, int64_t(P) + kTopMax),
                             int64_t(P) + ada_f + int64_t(cfg.n_kv_heads) * (n_free_head - ada_f));
  const int n_top = int(std::min<int64_t>(b_hi, s)) - P;   // ranking width per unit
  if (n_top > kTopMax)
    return fail(RESKV_ERR_UNSUPPORTED, "budget - recent_window must be <= 8192");
  const bool all_main = !any_evict;
  const bool proxy = override_host == nullptr && !all_main;
  if (cfg.score_mode != RESKV_SCORE_OBS_POOL && cfg.score_mode != RESKV_SCORE_KEYNORM)
    return fail(RESKV_ERR_INVALID_ARG, "unknown score_mode");
  if (cfg.pool_kernel < 1 || cfg.pool_kernel % 2 == 0)
    return fail(RESKV_ERR_INVALID_ARG, "pool_kernel must be a positive odd number");
  const bool need_q = cfg.score_mode == RESKV_SCORE_OBS_POOL || proxy;
  if (need_q) {
    if (!Ql) return fail(RESKV_ERR_INVALID_ARG, "observation queries are required");
    for (int l = 0; l < cfg.n_layers; ++l)
      if (!Ql[l]) return fail(RESKV_ERR_INVALID_ARG, "NULL observation-query layer");
    if (cfg.score_mode == RESKV_SCORE_OBS_POOL && (cfg.n_fit < 1 || cfg.n_fit > cfg.n_obs))
      return fail(RESKV_ERR_INVALID_ARG, "need 1 <= n_fit <= n_obs");
    if (proxy) {
      const int used_fit = cfg.score_mode == RESKV_SCORE_OBS_POOL ? cfg.n_fit : 0;
      if (cfg.n_val < 1 || used_fit + cfg.n_val > cfg.n_obs)
        return fail(RESKV_ERR_INVALID_ARG, "need n_val >= 1 and n_fit + n_val <= n_obs");
    }
  }
  for (int l = 0; l < cfg.n_layers; ++l)
    if (!Kl[l] || !Vl[l]) return fail(RESKV_ERR_INVALID_ARG, "NULL K or V layer");
  if (cfg.lloyd_iters < 1 || cfg.lloyd_iters > 64)
    return fail(RESKV_ERR_INVALID_ARG, "lloyd_iters must be in [1, 64]");
  if (cfg.n_grid < 0 || cfg.n_grid > RESKV_MAX_GRID)
    return fail(RESKV_ERR_INVALID_ARG, "n_grid must be in [0, 8]");
  if (!(cfg.delta >= 0.f && cfg.delta < 1.f) || !std::isfinite(cfg.beta))
    return fail(RESKV_ERR_INVALID_ARG, "delta must be in [0, 1) and beta finite");

  // candidate budgets r = floor(ratio * b) > 0, distinct, ascending (App. B).
  // One budget: the columns are those r.  Per-unit budgets: the columns are
  // the distinct positive ratios, ascending; unit u's r in a column is
  // floor(ratio * b_u), dropped (0) when zero, equal to the previous column's,
  // or leaving less than |P| main slots (unit_cands).
  std::vector<int32_t> cands;          // one budget: r of every column
  std::vector<float> col_ratio;        // per-unit budgets: ratio of every column
  std::vector<int32_t> col_rmax;       // per column: the largest r any unit can have
  for (int i = 0; i < cfg.n_grid; ++i)
    if (!(cfg.grid_ratios[i] >= 0.f && cfg.grid_ratios[i] <= 1.f))
      return fail(RESKV_ERR_INVALID_ARG, "grid ratios must be in [0, 1]");
  if (proxy && !per_unit) {
    for (int i = 0; i < cfg.n_grid; ++i) {
      const int r = int(std::floor(double(cfg.grid_ratios[i]) * double(b)));
      if (r > 0 && b - r >= P && std::find(cands.begin(), cands.end(), r) == cands.end())
        cands.push_back(r);
    }
    std::sort(cands.begin(), cands.end());
    col_rmax = cands;
  } else if (proxy) {
    for (int i = 0; i < cfg.n_grid; ++i)
      if (cfg.grid_ratios[i] > 0.f &&
          std::find(col_ratio.begin(), col_ratio.end(), cfg.grid_ratios[i]) == col_ratio.end())
        col_ratio.push_back(cfg.grid_ratios[i]);
    std::sort(col_ratio.begin(), col_ratio.end());
    for (float ratio : col_ratio)
      col_rmax.push_back(int(std::floor(double(ratio) * double(b_hi))));
  }
  // r of every candidate column for the units of one layer ([ncol, UL], column 0 = 0)
  auto unit_candidates = [&](const int32_t* bl, std::vector<int32_t>& out) {
    const int nc = 1 + int(col_rmax.size());
    out.assign(size_t(nc) * UL, 0);
    for (int i = 0; i < UL; ++i) {
      const int64_t bu = bl ? bl[i] : b;
      int prev = 0;
      for (int c = 1; c < nc; ++c) {
        int r = cands.empty() ? int(std::floor(double(col_ratio[c - 1]) * double(bu))) : cands[c - 1];
        if (r <= 0 || r == prev || bu - r < P || bu >= s) r = 0;
        else prev = r;
        out[size_t(c) * UL + i] = r;
      }
    }
  };
  std::vector<int32_t> ovr;
  int rmax = 0;
  if (override_host) {
    ovr.assign(override_host, override_host + U_all);
    for (int64_t u = 0; u < U_all; ++u) {
      const int r = ovr[u];
      const int64_t bu = cfg.unit_budgets ? cfg.unit_budgets[u] : b;
      if (r < 0 || r >= bu) return fail(RESKV_ERR_INVALID_ARG, "residual_override out of [0, budget)");
      if (r > 0 && !adakv && (bu >= s || bu - r < P))
        return fail(RESKV_ERR_INVALID_ARG,
                    "residual_override needs budget < seq_len and budget - r >= recent_window");
      rmax = std::max(rmax, r);
    }
  }
  for (int32_t r : col_rmax) rmax = std::max(rmax, r);
  if (rmax > kMaxR) return fail(RESKV_ERR_UNSUPPORTED, "residual entries per unit must be <= 8192");
  const int rstride = (rmax + 15) & ~15;             // stride of the per-centre arrays
  // What the kernels read at once: whole key tiles and 16-byte chunks for
  // observation scores, the assignment (tiles of 128 keys by TMA; fewer keys are
  // copied) and the proxy, whose losses take the values the same way; else rows in
  // 8-byte pieces.  Queries come in 4-byte words.
  const uintptr_t k_align = cfg.score_mode == RESKV_SCORE_OBS_POOL || proxy ||
                            (rmax > 0 && int64_t(UL) * s >= kTile) ? 16 : 8;
  const uintptr_t v_align = proxy ? 16 : 8;
  auto aligned = [](const void* p, uintptr_t to) { return reinterpret_cast<uintptr_t>(p) % to == 0; };
  for (int l = 0; l < cfg.n_layers; ++l)
    if (!aligned(Kl[l], k_align) || !aligned(Vl[l], v_align) || (need_q && !aligned(Ql[l], 4)))
      return fail(RESKV_ERR_INVALID_ARG,
                  "layer " + std::to_string(l) + ": K must be " + std::to_string(k_align) + "-byte aligned, V " +
                      std::to_string(v_align) + "-byte, Qobs 4-byte");

  // ---------------- handle and scratch ----------------
  reskv_cache* c = nullptr;
  reskv_status st;
  std::vector<int32_t> budgets_host;   // per-unit budgets (every layer)
  if (adakv) {
    // provisional layout with b per unit: the allocation keeps every
    // (layer, batch element)'s total, so only offsets inside it move
    budgets_host.assign(size_t(U_all), b);
    reskv_config lay = cfg;
    lay.unit_budgets = budgets_host.data();
    st = alloc_handle(lay, stream, &c);
  } else {
    if (cfg.unit_budgets) budgets_host.assign(cfg.unit_budgets, cfg.unit_budgets + U_all);
    st = alloc_handle(cfg, stream, &c);
  }
  if (st != RESKV_OK) return st;
  c->candidates = per_unit ? std::vector<int32_t>() : cands;
  c->n_candidates = int32_t(col_rmax.size());
  c->ranked_width = std::max(n_top, 0);
  if (proxy) c->unit_cands.assign(size_t(U_all) * col_rmax.size(), 0);
  const int ncol = 1 + int(col_rmax.size());         // run 0 = pure-main cache
  const int ntiles = int(cdiv(s, kTile));
  const int n_fit_rows = cfg.score_mode == RESKV_SCORE_OBS_POOL ? G * cfg.n_fit : 0;
  const int n_val_rows = proxy ? G * cfg.n_val : 0;
  // Chunks of the validation targets: at most 16 tiles per CTA, and as many CTAs
  // as fill whole waves of one CTA per SM.
  const int row_blocks = int(cdiv(std::max(n_val_rows, 1), kValRows));
  int64_t nchunks = 1;
  for (int64_t wave = 1;; ++wave) {
    nchunks = std::max<int64_t>(1, wave * c->num_sms / (int64_t(UL) * row_blocks));
    if (cdiv(ntiles, nchunks) <= 16) break;
  }
  const int chunk_tiles = int(cdiv(ntiles, nchunks));
  nchunks = cdiv(ntiles, chunk_tiles);
  const int nparts = int(nchunks) * val_shape(std::max(n_val_rows, 1) - (row_blocks - 1) * kValRows).splits;
  // entry storage: one slice per run with r > 0
  std::vector<int32_t> run_off(std::max(ncol, 2), 0);
  int64_t ent_stride = 0;
  if (proxy) {
    for (int i = 0; i < int(col_rmax.size()); ++i) {
      run_off[1 + i] = int32_t(ent_stride);
      ent_stride += col_rmax[i];
    }
  } else {
    ent_stride = rmax;
  }

  Scratch S;
  double* scores = nullptr;
  float* A = nullptr;
  uint4* qfrag = nullptr;
  float2* tstats = nullptr;
  float2* rstats = nullptr;
  int32_t *top = nullptr, *rank_pos = nullptr, *assign = nullptr;
  int32_t *ccount = nullptr, *ecount = nullptr;
  int32_t *r_runs = nullptr, *r_final = nullptr, *chosen = nullptr, *run_off_d = nullptr;
  int32_t* budgets_d = nullptr;        // [U_all] per-unit budgets (per_unit only)
  int32_t* ada_counts = nullptr;       // [UL, 2]
  float *cnorm = nullptr, *vpart = nullptr, *oS = nullptr;
  __nv_bfloat16* cplanes = nullptr;
  __nv_bfloat16* kpad = nullptr;       // the layer's keys where they are fewer than a tile
  double* centers64 = nullptr;
  long long *msum = nullptr, *tsum = nullptr;
  uint32_t* mflag = nullptr;
  float* knorm = nullptr;
  int4* amb = nullptr;
  int2* cand = nullptr;
  int* amb_count = nullptr;
  float* centers32 = nullptr;
  int32_t *assign2 = nullptr, *lbase = nullptr, *lsize = nullptr, *list = nullptr, *mcount = nullptr;
  __nv_bfloat16 *kbar = nullptr, *vbar = nullptr;
  double *rowerr = nullptr, *losses = nullptr;
  const size_t US = size_t(UL) * size_t(s);
  const int nruns = proxy ? ncol : 2;
  // Candidates whose Lloyd runs share their launches: a layer of few tokens does
  // not fill the GPU with one (8 units of 32K keys: 1.45 ms one by one, 0.78
  // together), one of more than 2^20 tokens does, and would pay for its small
  // candidates being swept like the largest.
  const int n_cands = proxy ? ncol - 1 : 1;
  const int n_batch = int(std::max<int64_t>(
      1, std::min({int64_t(n_cands), (int64_t(1) << 20) / int64_t(US), int64_t(65535) / UL})));   // (a grid dimension)
  const size_t UR = size_t(UL) * n_batch;          // run units of a launch
  S.get(&scores, US);
  S.get(&top, size_t(UL) * std::max(n_top, 1));
  S.get(&rank_pos, US);
  S.get(&r_runs, size_t(nruns) * UL);
  S.get(&r_final, UL);
  S.get(&chosen, UL);
  S.get(&run_off_d, run_off.size());
  if (per_unit) S.get(&budgets_d, size_t(U_all));
  if (adakv) S.get(&ada_counts, size_t(UL) * 2);
  if (n_fit_rows > 0) {
    S.get(&A, US);
    S.get(&qfrag, size_t(UL) * cdiv(n_fit_rows, 16) * 256);
    S.get(&tstats, size_t(UL) * n_fit_rows * ntiles);
    S.get(&rstats, size_t(UL) * n_fit_rows);
  }
  if (rmax > 0) {
    const size_t n_c = UR * rstride;                 // centres
    S.get(&assign, UR * s);
    S.get(&assign2, UR * s);
    S.get(&list, 2 * UR * s);
    S.get(&mcount, n_c * 2 * 2);
    S.get(&lbase, n_c * 2);
    S.get(&lsize, UR);
    S.get(&ccount, n_c);
    S.get(&centers64, n_c * kHeadDim);
    S.get(&centers32, n_c * kHeadDim);
    S.get(&cplanes, n_c * 2 * kHeadDim);
    S.get(&cnorm, n_c);
    S.get(&kbar, size_t(UL) * ent_stride * kHeadDim);
    S.get(&vbar, size_t(UL) * ent_stride * kHeadDim);
    S.get(&ecount, size_t(UL) * ent_stride);
    S.get(&msum, n_c * 2 * kHeadDim * 2);
    S.get(&mflag, n_c);
    S.get(&knorm, US);
    S.get(&amb, UR * ntiles * kTile);
    S.get(&amb_count, kResMaxCtas);
    if (rmax > kAsgRmax) S.get(&cand, UR * s);
    if (US < size_t(kTile)) S.get(&kpad, kTile * kHeadDim);
  }
  if (proxy) {
    S.get(&vpart, size_t(UL) * n_val_rows * nparts * kValRec);
    S.get(&oS, size_t(UL) * n_val_rows * kHeadDim);
    S.get(&rowerr, size_t(UL) * ncol * n_val_rows);
    S.get(&losses, size_t(UL) * ncol);
  }
  bool ok = S.commit();
  // the member sums start at zero; each pass's k_lloyd_finish clears what it
  // read.  Assignments start at -1 (no centre), so that a tile a failed
  // assignment never reached holds no index
  if (ok && rmax > 0)
    ok = cudaMemsetAsync(assign, 0xff, UR * s * sizeof(int32_t), stream) == cudaSuccess &&
         cudaMemsetAsync(assign2, 0xff, UR * s * sizeof(int32_t), stream) == cudaSuccess &&
         (!kpad || cudaMemsetAsync(kpad, 0, kTile * kHeadDim * 2, stream) == cudaSuccess);
  if (ok && rmax > 0) {
    const size_t n = UR * rstride * 2 * kHeadDim;
    tsum = msum + n;
    ok = cudaMemsetAsync(msum, 0, 2 * n * sizeof(long long), stream) == cudaSuccess &&
         cudaMemsetAsync(mflag, 0, UR * rstride * sizeof(uint32_t), stream) == cudaSuccess;
  }
  if (ok && cfg.keep_debug) {
    const size_t U = size_t(c->n_units);
    cudaError_t e = device_alloc(reinterpret_cast<void**>(&c->dbg_scores), U * size_t(s) * 8);
    if (e == cudaSuccess)
      e = device_alloc(reinterpret_cast<void**>(&c->dbg_ranked), U * std::max(n_top, 1) * 4);
    if (e == cudaSuccess) e = device_alloc(reinterpret_cast<void**>(&c->dbg_losses), U * ncol * 8);
    if (e == cudaSuccess) e = cudaMemsetAsync(c->dbg_losses, 0, U * ncol * 8, stream);
    ok = e == cudaSuccess;
    c->dbg_n_top = n_top;
  }
  if (!ok) {
    cudaGetLastError();
    release_handle(c);
    return fail(RESKV_ERR_OOM, "construction scratch allocation failed");
  }

  auto cleanup_fail = [&](reskv_status e) {
    release_handle(c);
    return e;
  };

  // per-run r arrays [nruns, UL] (proxy: per layer from the units' budgets;
  // override: filled per layer)
  std::vector<int32_t> hr;
  if (proxy) unit_candidates(nullptr, hr);
  if (cudaMemcpyAsync(run_off_d, run_off.data(), run_off.size() * 4, cudaMemcpyHostToDevice,
                      stream) != cudaSuccess ||
      (cfg.unit_budgets && cudaMemcpyAsync(budgets_d, budgets_host.data(), size_t(U_all) * 4,
                                           cudaMemcpyHostToDevice, stream) != cudaSuccess) ||
      cudaStreamSynchronize(stream) != cudaSuccess)
    return cleanup_fail(fail(RESKV_ERR_CUDA, "copying run tables"));

  // kernel attributes
  const size_t sm_obs1 = size_t(kTile) * kAsgRowBytes;               // the key tile
  const size_t sm_obs2 = sm_obs1 + size_t(8) * kTile * 4;  // + the partial sums
  // the ranked keys and positions, up to the next power of two of kTopThreads
  size_t n_sort = kTopThreads;
  while (n_sort < size_t(std::max(n_top, 1))) n_sort *= 2;
  const size_t sm_top = n_sort * 12;
  const size_t sm_scatter = size_t(std::max(rmax, 1)) * 4 * sizeof(int);
  // two ranking CTAs per SM where there are more units than SMs (else one has an SM
  // to itself, and 32 registers only spill: 32 units of 128K 93 -> 97 us)
  auto* topk_k = UL > c->num_sms && n_top <= 2 * kTopThreads ? k_topk<2> : k_topk<8>;
  if (set_smem(k_obs_pass1, sm_obs1) != cudaSuccess || set_smem(k_obs_pass2, sm_obs2) != cudaSuccess ||
      set_smem(k_topk<2>, sm_top) != cudaSuccess || set_smem(k_topk<8>, sm_top) != cudaSuccess || set_smem(k_lloyd_scatter<false, 1>, sm_scatter) != cudaSuccess ||
      set_smem(k_lloyd_scatter<true, 1>, sm_scatter) != cudaSuccess ||
      set_smem(k_lloyd_scatter<false, 4>, sm_scatter) != cudaSuccess ||
      set_smem(k_lloyd_scatter<true, 4>, sm_scatter) != cudaSuccess ||
      set_smem(k_lloyd_assign<1>, kAsgSmemMax) != cudaSuccess ||
      set_smem(k_lloyd_assign<2>, kAsgSmemMax) != cudaSuccess ||
      set_smem(k_lloyd_assign<3>, kAsgSmemMax) != cudaSuccess ||
      set_smem(k_lloyd_assign<4>, kAsgSmemMax) != cudaSuccess ||
      set_smem(k_lloyd_accum<false, true>, kAccSmem) != cudaSuccess ||
      set_smem(k_lloyd_accum<true, true>, kAccSmem) != cudaSuccess ||
      set_smem(k_lloyd_accum<false, false>, kAccSmem) != cudaSuccess ||
      set_smem(k_lloyd_accum<true, false>, kAccSmem) != cudaSuccess ||
      set_smem(k_val_loss, kValSmemLoss) != cudaSuccess ||
      set_smem(k_val_full, kValSmemFull) != cudaSuccess)
    return cleanup_fail(fail(RESKV_ERR_CUDA, "setting kernel shared-memory limits"));

  const double one_minus_delta = 1.0 - double(cfg.delta);
  StageTimer timer(stream);
  bool timing_ok = true;

  int test_fault = take_test_wait_fault() ? 1 : 0;   // test hook (reskv_test_inject)
  for (int l = 0; l < cfg.n_layers; ++l) {
    const __nv_bfloat16* K = static_cast<const __nv_bfloat16*>(Kl[l]);
    const __nv_bfloat16* V = static_cast<const __nv_bfloat16*>(Vl[l]);
    const __nv_bfloat16* Q = Ql ? static_cast<const __nv_bfloat16*>(Ql[l]) : nullptr;

    // ---- token scores ----
    timing_ok &= timer.mark(kStScore);
    if (cfg.score_mode == RESKV_SCORE_OBS_POOL) {
      ObsArgs oa{K, Q, s, G, cfg.n_obs, n_fit_rows, cfg.n_fit, ntiles, qfrag, tstats, rstats, A};
      k_obs_frag<<<dim3(unsigned(cdiv(n_fit_rows, 16)), UL), 256, 0, stream>>>(oa);
      k_obs_pass1<<<dim3(ntiles, UL), 32 * obs_warps1(n_fit_rows), sm_obs1, stream>>>(oa);
      k_obs_rowstats<<<unsigned(cdiv(int64_t(UL) * n_fit_rows, 32)), 256, 0, stream>>>(oa, UL);
      k_obs_pass2<<<dim3(ntiles, UL), 32 * obs_warps2(n_fit_rows), sm_obs2, stream>>>(oa);
      k_pool<<<unsigned(cdiv(int64_t(UL) * cdiv(s, int64_t(4)), 256)), 256, 0, stream>>>(A, scores, s, UL, cfg.pool_kernel,
                                                                                     1.0 / double(cfg.pool_kernel));
    } else {
      k_key_norms<true><<<unsigned(cdiv(int64_t(US), 256)), 256, 0, stream>>>(K, scores, knorm, int64_t(US));
    }
    RESKV_LAUNCH_CHECK("scoring");
    timing_ok &= timer.mark(kStRank);
    int32_t* bl_d = per_unit ? budgets_d + size_t(l) * UL : nullptr;   // this layer's budgets
    const int32_t* bl_h = per_unit ? budgets_host.data() + size_t(l) * UL : nullptr;
    if (adakv) {
      // AdaKV: mark every head's safeguard (its top f), split the shared slots
      TopArgs tf{scores, s, P, ada_f, top, rank_pos, c->status, nullptr};
      const cudaError_t e1 = launch_clusters(topk_k, UL, c->num_sms, sm_top, stream, tf);
      AdaArgs aa{scores, rank_pos, s, P, cfg.n_kv_heads, ada_f, P + ada_f,
                 int64_t(cfg.n_kv_heads) * (n_free_head - ada_f), bl_d, ada_counts};
      const cudaError_t e2 = launch_clusters(k_adakv, cfg.batch, c->num_sms, 0, stream, aa);
      if (e1 != cudaSuccess || e2 != cudaSuccess)
        return cleanup_fail(fail(RESKV_ERR_CUDA, "launching the AdaKV budgets"));
      RESKV_LAUNCH_CHECK("AdaKV budgets");
      if (cudaMemcpyAsync(budgets_host.data() + size_t(l) * UL, bl_d, size_t(UL) * 4,
                          cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
          cudaStreamSynchronize(stream) != cudaSuccess)
        return cleanup_fail(fail(RESKV_ERR_CUDA, "reading the AdaKV budgets"));
      // the layer's units keep their region; place them inside it
      const int64_t u0 = int64_t(l) * UL;
      for (int i = 0; i < UL; ++i) {
        const int64_t bu = bl_h[i];
        if (bu < P + ada_f || bu > b_hi)
          return cleanup_fail(fail(bu > b_hi ? RESKV_ERR_UNSUPPORTED : RESKV_ERR_CUDA,
                                   "AdaKV budget " + std::to_string(bu) + " of unit " +
                                       std::to_string(u0 + i) +
                                       " is outside what construction covers"));
        if (!ovr.empty() && ovr[size_t(u0 + i)] > 0 &&
            (bu >= s || bu - ovr[size_t(u0 + i)] < P))
          return cleanup_fail(fail(RESKV_ERR_INVALID_ARG,
                                   "residual_override of unit " + std::to_string(u0 + i) +
                                       " leaves less than recent_window main slots of its AdaKV budget"));
        c->h_offsets[size_t(u0 + i) + 1] = c->h_offsets[size_t(u0 + i)] + int32_t(bu) + c->append_capacity;
      }
      if (cudaMemcpyAsync(c->offsets + u0, c->h_offsets.data() + u0, size_t(UL + 1) * 4,
                          cudaMemcpyHostToDevice, stream) != cudaSuccess)
        return cleanup_fail(fail(RESKV_ERR_CUDA, "copying unit offsets"));
    }
    if (per_unit && n_top > 0 &&
        cudaMemsetAsync(top, 0xff, size_t(UL) * n_top * 4, stream) != cudaSuccess)
      return cleanup_fail(fail(RESKV_ERR_CUDA, "clearing the ranking"));
    TopArgs ta{scores, s, P, n_top, top, rank_pos, c->status, bl_d};
    if (launch_clusters(topk_k, UL, c->num_sms, sm_top, stream, ta) != cudaSuccess)
      return cleanup_fail(fail(RESKV_ERR_CUDA, "launching the ranking"));
    RESKV_LAUNCH_CHECK("ranking");
    // candidate r per unit of this layer
    if (proxy) {
      if (per_unit || l == 0) unit_candidates(bl_h, hr);
      for (int c2 = 1; c2 < ncol; ++c2)
        for (int i = 0; i < UL; ++i)
          c->unit_cands[(size_t(l) * UL + i) * (ncol - 1) + (c2 - 1)] = hr[size_t(c2) * UL + i];
      if ((per_unit || l == 0) &&
          cudaMemcpyAsync(r_runs, hr.data(), hr.size() * 4, cudaMemcpyHostToDevice, stream) != cudaSuccess)
        return cleanup_fail(fail(RESKV_ERR_CUDA, "copying candidate budgets"));
    }

    LloydArgs la{};
    la.K = K;
    la.V = V;
    la.s = s;
    la.UL = UL;
    la.recent = P;
    la.n_top = n_top;
    la.budget = b;
    la.ntiles = ntiles;
    la.rmax = rstride;
    la.top = top;
    la.rank_pos = rank_pos;
    la.budgets = bl_d;
    la.cnorm = cnorm;
    la.centers64 = centers64;
    la.centers32 = centers32;
    la.cplanes = cplanes;
    la.knorm = knorm;
    la.cand = cand;
    la.amb = amb;
    la.amb_count = amb_count;
    la.mcount = mcount;
    la.cursor = mcount + 2 * UR * rstride;
    la.ccount = ccount;
    la.lbase = lbase;
    la.lsize = lsize;
    la.list = list;
    la.msum = msum;
    la.tsum = tsum;
    la.mflag = mflag;
    la.kbar = kbar;
    la.vbar = vbar;
    la.ecount = ecount;
    la.ent_stride = ent_stride;
    la.status = c->status;
    // the assignment loads tiles of 128 keys by TMA: a layer with fewer rows is
    // read from a padded copy
    CUtensorMap tmK;
    if (rmax > 0) {
      if (cfg.score_mode == RESKV_SCORE_OBS_POOL)         // (the query-free scores come with the norms)
        k_key_norms<false><<<unsigned(cdiv(int64_t(US), 256)), 256, 0, stream>>>(K, nullptr, knorm, int64_t(US));
      if (kpad && cudaMemcpyAsync(kpad, K, US * kHeadDim * 2, cudaMemcpyDeviceToDevice, stream) != cudaSuccess)
        return cleanup_fail(fail(RESKV_ERR_CUDA, "copying the keys"));
      if (!encode_key_tiles(&tmK, kpad ? kpad : K, std::max<uint64_t>(US, kTile)))
        return cleanup_fail(fail(RESKV_ERR_CUDA, "creating the TMA tensor map of the keys"));
    }
    // the Lloyd runs of n_run candidates at once: r_unit [n_run, UL], entries at
    // run_off_d[run0 ..]
    auto lloyd_run = [&](const int32_t* r_unit, int run0, int n_run, int r_hi) -> reskv_status {
      const int U = UL * n_run;
      la.r_unit = r_unit;
      la.n_units = U;
      la.run_off = run_off_d + run0;
      timing_ok &= timer.mark(kStLloyd);
      const bool k16 = (reinterpret_cast<uintptr_t>(K) & 15u) == 0, v16 = (reinterpret_cast<uintptr_t>(V) & 15u) == 0;
      const unsigned gr = unsigned(cdiv((r_hi + 15) & ~15, kFinWarps));
      const unsigned asg_grid = unsigned(std::min<int64_t>(std::min(c->num_sms, kResMaxCtas), int64_t(U) * ntiles));
      // segments of at most 256 centres, of equal width
      const int nseg = int(cdiv(r_hi, kAsgRmax));
      const int segw = (int(cdiv(r_hi, nseg)) + 15) & ~15;
      // tokens per thread of the list kernel: four where two CTAs per SM remain
      const int tok = cdiv(s, int64_t(4 * kScatterThreads)) * U >= 2 * c->num_sms ? 4 : 1;
      const dim3 gs(unsigned(cdiv(s, int64_t(tok * kScatterThreads))), unsigned(U));
      const dim3 ga(unsigned(cdiv(s, int64_t(kAccRows))), unsigned(U));
      auto clear = [&](int32_t* counts, size_t n) {
        return cudaMemsetAsync(counts, 0, n * sizeof(int32_t), stream) == cudaSuccess;
      };
      k_lloyd_init<<<dim3(gr, U), kFinWarps * 32, 0, stream>>>(la);
      for (int it = 0; it < cfg.lloyd_iters; ++it) {
        const bool last = it == cfg.lloyd_iters - 1;
        la.assign = (it & 1) ? assign2 : assign;
        la.assign_prev = it == 0 ? nullptr : (it & 1) ? assign : assign2;
        if (!clear(la.mcount, UR * rstride * 2 * 2))      // and the cursors
          return fail(RESKV_ERR_CUDA, "clearing the move counts");
        la.test_fault = test_fault;       // an injected fault is taken by the first launch only
        test_fault = 0;
        for (int sg = 0; sg < nseg; ++sg) {
          auto* assign_k = segw <= 64 ? k_lloyd_assign<1> : segw <= 128 ? k_lloyd_assign<2>
                           : segw <= 192 ? k_lloyd_assign<3> : k_lloyd_assign<4>;
          assign_k<<<asg_grid, kAsgThreads, lloyd_asg_smem(segw), stream>>>(
              la, sg * segw, segw, lloyd_asg_key_bufs(segw), tmK);
          la.test_fault = 0;
        }
        k_lloyd_resolve<<<unsigned(3 * c->num_sms), kResWarps * 32, 0, stream>>>(la, int(asg_grid));
        (tok == 4 ? k_lloyd_scatter<false, 4> : k_lloyd_scatter<false, 1>)
            <<<gs, kScatterThreads, size_t(r_hi) * 4 * sizeof(int), stream>>>(la);
        (k16 ? k_lloyd_accum<false, true> : k_lloyd_accum<false, false>)<<<ga, kThreads, kAccSmem, stream>>>(la);
        if (last) {                       // the values of every member
          if (it > 0) {
            if (!clear(la.cursor, UR * rstride * 2))
              return fail(RESKV_ERR_CUDA, "clearing the list cursors");
            (tok == 4 ? k_lloyd_scatter<true, 4> : k_lloyd_scatter<true, 1>)
                <<<gs, kScatterThreads, size_t(r_hi) * 2 * sizeof(int), stream>>>(la);
          }
          (v16 ? k_lloyd_accum<true, true> : k_lloyd_accum<true, false>)<<<ga, kThreads, kAccSmem, stream>>>(la);
        }
        k_lloyd_finish<<<dim3(unsigned(cdiv(r_hi, kFinWarps)), U), kFinWarps * 32, 0, stream>>>(la, last);
      }
      RESKV_LAUNCH_CHECK("residual entries");
      return RESKV_OK;
    };

    if (proxy) {
      // ---- validation targets, candidates, choice of r ----
      timing_ok &= timer.mark(kStValTargets);
      ValArgs va{K, V, Q, s, G, cfg.n_obs, cfg.n_val, n_val_rows, chunk_tiles, int(nchunks), nparts, vpart, oS};
      k_val_full<<<dim3(unsigned(nchunks), unsigned(row_blocks), UL), kThreads, kValSmemFull, stream>>>(va);
      k_val_combine<<<dim3(n_val_rows, UL), kHeadDim, 0, stream>>>(va);
      RESKV_LAUNCH_CHECK("validation targets");
      for (int run = 1; run < ncol; run += n_batch) {
        const int n_run = std::min(n_batch, ncol - run);
        int r_hi = 0;                    // (0: no unit of the layer has these candidates)
        for (int i = 0; i < UL * n_run; ++i) r_hi = std::max(r_hi, hr[size_t(run) * UL + i]);
        if (r_hi > 0 && (st = lloyd_run(r_runs + size_t(run) * UL, run, n_run, r_hi)) != RESKV_OK)
          return cleanup_fail(st);
      }
      timing_ok &= timer.mark(kStValLoss);
      LossArgs lo{K, V, Q, s, UL, G, cfg.n_obs, cfg.n_val, n_val_rows, P, n_top, b, top, r_runs,
                  kbar, vbar, ecount, ent_stride, run_off_d, cfg.beta, cfg.gate_mode,
                  cfg.tau, cfg.alpha, cfg.g_min, cfg.g_fixed, oS, rowerr, cfg.softmax_mode, bl_d};
      k_val_loss<<<dim3(unsigned(row_blocks), UL, ncol), kThreads, kValSmemLoss, stream>>>(lo);
      k_loss_reduce<<<unsigned(cdiv(int64_t(UL) * ncol, 8)), 256, 0, stream>>>(rowerr, losses, n_val_rows, UL,
                                                                             ncol, r_runs);
      RESKV_LAUNCH_CHECK("validation loss");
      k_choose<<<unsigned(cdiv(UL, 128)), 128, 0, stream>>>(losses, ncol, r_runs, UL,
                                                           one_minus_delta, r_final, chosen);
      RESKV_LAUNCH_CHECK("choosing r");
    } else {
      // fixed r per unit (or the budget covers every token: r = 0)
      timing_ok &= timer.mark(-1);
      std::vector<int32_t> rl(UL, 0), ch(UL, 0);
      bool any = false;
      if (!ovr.empty())
        for (int i = 0; i < UL; ++i) {
          rl[i] = ovr[size_t(l) * UL + i];
          ch[i] = rl[i] > 0 ? 1 : 0;
          any |= rl[i] > 0;
        }
      if (cudaMemcpyAsync(r_final, rl.data(), UL * 4, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
          cudaMemcpyAsync(chosen, ch.data(), UL * 4, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
          cudaStreamSynchronize(stream) != cudaSuccess)
        return cleanup_fail(fail(RESKV_ERR_CUDA, "copying residual counts"));
      if (any) {
        st = lloyd_run(r_final, 0, 1, *std::max_element(rl.begin(), rl.end()));
        if (st != RESKV_OK) return cleanup_fail(st);
      }
    }

    // ---- pack the chosen cache ----
    timing_ok &= timer.mark(kStPack);
    PackArgs pa{K, V, s, P, b, c->stride, rank_pos, r_final, chosen, run_off_d, kbar, vbar, ecount,
                ent_stride, cfg.beta, int64_t(l) * UL, c->kslots, c->vslots, c->logc,
                c->slot_pos, c->counts, c->n_main, c->n_res, bl_d,
                per_unit ? c->offsets : nullptr};
    if (launch_clusters(k_pack, UL, c->num_sms, 0, stream, pa) != cudaSuccess)
      return cleanup_fail(fail(RESKV_ERR_CUDA, "packing launch"));
    RESKV_LAUNCH_CHECK("packing");
    timing_ok &= timer.mark(-1);
    timing_ok &= timer.flush(c->build_ms);

    if (cfg.keep_debug) {
      cudaError_t e = cudaMemcpyAsync(c->dbg_scores + size_t(l) * US, scores, US * 8,
                                      cudaMemcpyDeviceToDevice, stream);
      if (e == cudaSuccess && n_top > 0)
        e = cudaMemcpyAsync(c->dbg_ranked + size_t(l) * UL * n_top, top, size_t(UL) * n_top * 4,
                            cudaMemcpyDeviceToDevice, stream);
      if (e == cudaSuccess && proxy)
        e = cudaMemcpyAsync(c->dbg_losses + size_t(l) * UL * ncol, losses, size_t(UL) * ncol * 8,
                            cudaMemcpyDeviceToDevice, stream);
      if (e != cudaSuccess) return cleanup_fail(fail(RESKV_ERR_CUDA, "keeping intermediates"));
    }
  }
  if (!timing_ok)                        // timing is reported, not needed: clear it
    for (float& t : c->build_ms) t = 0.f;
  if (adakv && (st = finalize_ragged_layout(c)) != RESKV_OK) return cleanup_fail(st);
  // scratch is freed (cudaFree synchronises) when S leaves scope
  cudaError_t e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) return cleanup_fail(fail(RESKV_ERR_CUDA, std::string("construction: ") +
                                                                   cudaGetErrorString(e)));
  *out = c;
  return RESKV_OK;
}

}  // namespace reskv
