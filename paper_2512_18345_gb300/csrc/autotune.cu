// Schedule autotuner for batched plans (the batching / CUDA-graph row of the
// hot path; Section IV-A multi-polynomial caching, Section IV-C graphs).
//
// The paper sizes its batches by the L2 capacity; on GB300 the stage kernels
// are bound by the integer pipes rather than by L2 traffic, so larger groups
// that amortise each launch's ramp can win even when their working set spills
// from L2, and concurrent lanes overlap one group's DRAM-bound inner product
// with another group's transforms.  fhe_autotune measures the candidates on
// the device -- real graph plans of synthetic key switches at the caller's
// level and batch size -- and keeps the fastest.  Timing does not depend on
// the residues or the key, so the inputs are filler residues below 2^20 (valid
// for every prime of a context) and, when no relinearisation key is set, a
// temporary filler key is installed for the run and removed afterwards.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <map>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/fhe.h"
#include "ctx.h"
#include "internal.h"

namespace {
__global__ void k_fill(uint32_t *p, size_t n, uint32_t seed) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    uint32_t x = (uint32_t)i * 2654435761u ^ seed;
    x ^= x >> 15;
    x *= 0x2C1B3C6Du;
    x ^= x >> 12;
    p[i] = x & 0xFFFFFu;
  }
}
}  // namespace

extern "C" int fhe_autotune(fhe_ctx *c, int level, int n_items, int flags, fhe_tune_result *out,
                            fhe_stream stream) {
  if (!c || !out) return fhe_fail(FHE_EINVAL, "fhe_autotune: null argument");
  if (level < 1 || level > c->L) return fhe_fail(FHE_ELEVEL, "fhe_autotune: level %d", level);
  if (n_items < 1 || n_items > 64) return fhe_fail(FHE_EINVAL, "fhe_autotune: n_items %d (1..64)", n_items);
  if (flags & ~(FHE_TUNE_BCONV | FHE_TUNE_NTT | FHE_TUNE_SHAPE))
    return fhe_fail(FHE_EINVAL, "fhe_autotune: flags %d", flags);
  cudaSetDevice(c->device);
  cudaStream_t s = (cudaStream_t)stream;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone)
    return fhe_fail(FHE_EINVAL, "fhe_autotune: stream is capturing");
  const size_t N = c->N, poly = (size_t)level * N;
  uint32_t *ins = nullptr, *outs = nullptr, *tmp_key = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  const size_t key_words = (size_t)c->dnum * 2 * (c->L + c->K) * N;
  auto release = [&]() {
    cudaFree(ins);
    cudaFree(outs);
    if (tmp_key) {
      cudaFree(tmp_key);
      c->relin_key = nullptr;
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
  };
  if (cudaMalloc(&ins, 4 * poly * n_items) != cudaSuccess || cudaMalloc(&outs, 8 * poly * n_items) != cudaSuccess ||
      cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    release();
    return fhe_fail(FHE_ENOMEM, "fhe_autotune: buffers");
  }
  k_fill<<<1024, 256, 0, s>>>(ins, poly * n_items, 0x9E3779B9u);
  if (!c->relin_key) {
    if (cudaMalloc(&tmp_key, 4 * key_words) != cudaSuccess) {
      release();
      return fhe_fail(FHE_ENOMEM, "fhe_autotune: filler key");
    }
    k_fill<<<1024, 256, 0, s>>>(tmp_key, key_words, 0x85EBCA6Bu);
    c->relin_key = tmp_key;
  }
  std::vector<fhe_ks_item> items(n_items);
  for (int i = 0; i < n_items; i++) {
    fhe_ks_item &it = items[i];
    memset(&it, 0, sizeof it);
    it.op = FHE_OP_KS;
    it.level = level;
    it.rot = FHE_RELIN_KEY;
    it.in = ins + poly * i;
    it.out = outs + 2 * poly * i;
  }

  int l2 = 0;
  cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, c->device);
  const size_t saved_budget = c->batch_budget;
  const int saved_group = c->batch_max_group, saved_lanes = c->batch_lanes, saved_mode = c->bconv_mode;
  std::vector<int> modes{c->bconv_mode};
  if (flags & FHE_TUNE_BCONV) {
    modes = {FHE_BCONV_SCALAR};
    if (fhe_ctx_set_bconv(c, FHE_BCONV_TC) == FHE_OK) modes.push_back(FHE_BCONV_TC);
    c->bconv_mode = saved_mode;
  }
  // budget 0 is the default grouping (fhe_ctx_set_batch), which no explicit budget gives beyond
  // 8 items; first, so that it is the one kept where another budget forms the same groups
  const size_t budgets[] = {0, (size_t)l2 * 3 / 4, (size_t)l2, (size_t)l2 * 2, (size_t)l2 * 4};
  std::map<std::tuple<int, int, std::vector<int>>, double> seen;  // (mode, lanes, group sizes) -> us per KS
  fhe_tune_result best;
  memset(&best, 0, sizeof best);
  best.us_per_ks = 1e30;
  int rc = FHE_OK, tried = 0;
  const int saved_ip = c->tabs.ip_ctas_per_sm, saved_comp = c->comp_pipe;
  const int saved_ntt = (c->tabs.ntt_otf ? FHE_NTT_OTF : 0) | (c->tabs.ntt_single ? FHE_NTT_SINGLE_PASS : 0) |
                        (c->tabs.ntt_stream ? FHE_NTT_STREAM : 0) | (c->tabs.ntt_persist ? FHE_NTT_PERSIST : 0);
  fhe_kernel_shape saved_shape;
  fhe_ctx_get_kernel_shape(c, &saved_shape);
  fhe_tune_result by_ip[2];  // fastest schedule with one / two inner-product CTAs per SM
  memset(by_ip, 0, sizeof by_ip);
  by_ip[0].us_per_ks = by_ip[1].us_per_ks = 1e30;
  // time a graph plan of the items: two warm-up launches, then the fastest of three runs of
  // five (the minimum is robust to a run that met interference, so that candidates a few
  // percent apart are ranked by their own speed)
  auto measure = [&](fhe_plan *p, double &us) -> int {
    const int reps = 5, trials = 3;
    int r = FHE_OK;
    for (int w = 0; w < 2 && r == FHE_OK; w++) r = fhe_batch_launch(p, stream);
    float best = 0.f;
    for (int tr = 0; tr < trials && r == FHE_OK; tr++) {
      cudaEventRecord(e0, s);
      for (int k = 0; k < reps && r == FHE_OK; k++) r = fhe_batch_launch(p, stream);
      cudaEventRecord(e1, s);
      float ms = 0.f;
      if (r == FHE_OK && (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess))
        r = fhe_fail(FHE_ECUDA, "fhe_autotune: timing");
      if (tr == 0 || ms < best) best = ms;
    }
    us = 1e3 * best / (reps * n_items);
    return r;
  };
  for (int mode : modes)
    for (int comp = 0; comp <= 1; comp++)
    for (int ipc = 1; ipc <= 2; ipc++)
    for (int lanes = 1; lanes <= 4 && rc == FHE_OK; lanes++)
      for (size_t budget : budgets) {
        c->comp_pipe = comp;
        c->tabs.ip_ctas_per_sm = ipc;
        c->bconv_mode = mode;
        c->batch_budget = budget;
        c->batch_lanes = lanes;
        c->batch_max_group = 0;
        fhe_plan *p = nullptr;
        rc = fhe_batch_plan(c, items.data(), n_items, FHE_PLAN_GRAPH, &p);
        if (rc != FHE_OK) break;
        std::vector<int> gs(64);
        const int ng = fhe_plan_groups(p, gs.data(), 64);
        gs.resize(std::min(ng, 64));
        const int eff_lanes = std::min(lanes, ng);
        const bool is_default = mode == saved_mode && comp == 1 && ipc == 2 && lanes == 2 && budget == 0;
        const auto key = std::make_tuple(mode * 8 + comp * 4 + ipc, eff_lanes, gs);
        auto found = seen.find(key);
        if (found != seen.end()) {  // the same schedule as one already measured
          if (is_default) best.default_us_per_ks = found->second;
          fhe_plan_destroy(p);
          continue;
        }
        double us = 0;
        rc = measure(p, us);
        fhe_plan_destroy(p);
        if (rc != FHE_OK) break;
        tried++;
        seen[key] = us;
        if (is_default) best.default_us_per_ks = us;
        fhe_tune_result &b = by_ip[ipc - 1];
        if (us < b.us_per_ks) {
          b.us_per_ks = us;
          b.lanes = lanes;
          b.l2_budget_bytes = budget;
          b.max_group = 0;
          b.bconv_mode = mode;
          b.n_groups = ng;
          b.ip_ctas_per_sm = ipc;
          b.comp_pipe = comp;
        }
      }
  // one resident inner-product CTA per SM only when it beats the best two-CTA schedule by
  // more than the timing noise (2 %): alone, the two-CTA kernel streams faster
  {
    const double dflt = best.default_us_per_ks;
    best = by_ip[0].us_per_ks < 0.98 * by_ip[1].us_per_ks ? by_ip[0] : by_ip[1];
    best.default_us_per_ks = dflt;
  }
  best.ntt_mode = saved_ntt;
  best.shape = saved_shape;
  // the NTT variants under the chosen schedule: another mode only when it is faster by more
  // than the timing noise (1 %)
  if (rc == FHE_OK && tried > 0 && (flags & FHE_TUNE_NTT)) {
    c->batch_budget = best.l2_budget_bytes;
    c->batch_lanes = best.lanes;
    c->batch_max_group = best.max_group;
    c->bconv_mode = best.bconv_mode;
    c->tabs.ip_ctas_per_sm = best.ip_ctas_per_sm;
    c->comp_pipe = best.comp_pipe;
    const double base = best.us_per_ks;
    for (int m : {0, FHE_NTT_OTF, FHE_NTT_SINGLE_PASS, FHE_NTT_SINGLE_PASS | FHE_NTT_OTF, FHE_NTT_STREAM,
                  FHE_NTT_STREAM | FHE_NTT_OTF, FHE_NTT_STREAM | FHE_NTT_SINGLE_PASS, FHE_NTT_PERSIST}) {
      if (m == saved_ntt || fhe_ctx_set_ntt(c, m) != FHE_OK) continue;
      fhe_plan *p = nullptr;
      rc = fhe_batch_plan(c, items.data(), n_items, FHE_PLAN_GRAPH, &p);
      if (rc != FHE_OK) break;
      int ng = fhe_plan_groups(p, nullptr, 0);
      double us = 0;
      rc = measure(p, us);
      fhe_plan_destroy(p);
      if (rc != FHE_OK) break;
      tried++;
      if (us < 0.99 * base && us < best.us_per_ks) {
        best.us_per_ks = us;
        best.ntt_mode = m;
        best.n_groups = ng;
      }
    }
    fhe_ctx_set_ntt(c, saved_ntt);
  }
  // kernel shapes under the chosen schedule and NTT mode, one parameter at a time: another
  // value only when it is faster by more than the timing noise (1 %)
  if (rc == FHE_OK && tried > 0 && (flags & FHE_TUNE_SHAPE)) {
    c->batch_budget = best.l2_budget_bytes;
    c->batch_lanes = best.lanes;
    c->batch_max_group = best.max_group;
    c->bconv_mode = best.bconv_mode;
    c->tabs.ip_ctas_per_sm = best.ip_ctas_per_sm;
    c->comp_pipe = best.comp_pipe;
    fhe_ctx_set_ntt(c, best.ntt_mode);
    fhe_kernel_shape cur = saved_shape;
    double cur_us = best.us_per_ks;
    auto try_shape = [&](const fhe_kernel_shape &cand) {
      if (rc != FHE_OK || memcmp(&cand, &cur, sizeof cand) == 0) return;
      if (fhe_ctx_set_kernel_shape(c, &cand) != FHE_OK) return;  // not available here: skip
      fhe_plan *p = nullptr;
      rc = fhe_batch_plan(c, items.data(), n_items, FHE_PLAN_GRAPH, &p);
      if (rc != FHE_OK) return;
      const int ng = fhe_plan_groups(p, nullptr, 0);
      double us = 0;
      rc = measure(p, us);
      fhe_plan_destroy(p);
      if (rc != FHE_OK) return;
      tried++;
      if (us < 0.99 * cur_us) {
        cur_us = us;
        cur = cand;
        best.n_groups = ng;
      }
    };
    for (int f = 0; f <= 1; f++) {
      fhe_kernel_shape k = cur;
      k.fuse_ip_moddown = f;
      try_shape(k);
    }
    if (best.bconv_mode == FHE_BCONV_TC) {
      for (int pl = 0; pl <= 1; pl++) {
        fhe_kernel_shape k = cur;
        k.bconv_tc_pipeline = pl;
        try_shape(k);
      }
      for (int n : {2, 3, 4}) {
        fhe_kernel_shape k = cur;
        k.bconv_tc_ctas = n;
        try_shape(k);
      }
    }
    if (best.ntt_mode & FHE_NTT_STREAM) {
      for (int st : {2, 3}) {
        fhe_kernel_shape k = cur;
        k.ntt_stream_stages = st;
        try_shape(k);
      }
      for (int n : {2, 3}) {
        fhe_kernel_shape k = cur;
        k.ntt_stream_ctas = n;
        try_shape(k);
      }
    }
    best.shape = cur;
    best.us_per_ks = cur_us;
    fhe_ctx_set_kernel_shape(c, &saved_shape);
    fhe_ctx_set_ntt(c, saved_ntt);
  }
  if (rc == FHE_OK) rc = fhe_ctx_sync(c);  // an expired bounded device wait voids the timings
  if (rc == FHE_OK && tried > 0) {
    best.candidates = tried;
    c->batch_budget = best.l2_budget_bytes;
    c->batch_lanes = best.lanes;
    c->batch_max_group = best.max_group;
    c->bconv_mode = best.bconv_mode;
    c->tabs.ip_ctas_per_sm = best.ip_ctas_per_sm;
    c->comp_pipe = best.comp_pipe;
    fhe_ctx_set_ntt(c, best.ntt_mode);
    fhe_ctx_set_kernel_shape(c, &best.shape);
    *out = best;
  } else {
    c->tabs.ip_ctas_per_sm = saved_ip;
    c->comp_pipe = saved_comp;
    fhe_ctx_set_ntt(c, saved_ntt);
    c->batch_budget = saved_budget;
    c->batch_lanes = saved_lanes;
    c->batch_max_group = saved_group;
    c->bconv_mode = saved_mode;
    fhe_ctx_set_kernel_shape(c, &saved_shape);
  }
  release();
  return rc;
}

// ---- tuning cache: one text line per (set of candidates, ring, level, special primes, digit size,
// batch, flags, GPU) -> chosen schedule; the last matching line wins, unreadable lines are skipped.
// sched=2: the candidates include the default grouping; entries without it were chosen among
// explicit budgets alone and are measured again.

static std::string tune_key(const fhe_ctx *c, int level, int n_items, int flags) {
  cudaDeviceProp prop;
  memset(&prop, 0, sizeof prop);
  cudaGetDeviceProperties(&prop, c->device);
  std::string gpu(prop.name);
  for (char &ch : gpu)
    if (ch == ' ' || ch == '|') ch = '_';
  char buf[384];
  snprintf(buf, sizeof buf, "sched=2 N=%zu level=%d K=%d alpha=%d dnum=%d items=%d flags=%d gpu=%s sms=%d", (size_t)c->N,
           level, c->K, c->alpha, c->dnum, n_items, flags, gpu.c_str(), prop.multiProcessorCount);
  return buf;
}

static bool tune_parse(const char *rest, const fhe_kernel_shape &dflt, fhe_tune_result *r) {
  fhe_tune_result t;
  memset(&t, 0, sizeof t);
  unsigned long long budget = 0;
  fhe_kernel_shape &k = t.shape;
  // entries with the kernel shape, and older ones without it (the context's shape then)
  if (sscanf(rest,
             " lanes=%d budget=%llu group=%d bconv=%d ip=%d comp=%d ntt=%d fuse=%d tcctas=%d tcpipe=%d nst=%d nsc=%d "
             "us=%lf",
             &t.lanes, &budget, &t.max_group, &t.bconv_mode, &t.ip_ctas_per_sm, &t.comp_pipe, &t.ntt_mode,
             &k.fuse_ip_moddown, &k.bconv_tc_ctas, &k.bconv_tc_pipeline, &k.ntt_stream_stages, &k.ntt_stream_ctas,
             &t.us_per_ks) != 13) {
    k = dflt;
    if (sscanf(rest, " lanes=%d budget=%llu group=%d bconv=%d ip=%d comp=%d ntt=%d us=%lf", &t.lanes, &budget,
               &t.max_group, &t.bconv_mode, &t.ip_ctas_per_sm, &t.comp_pipe, &t.ntt_mode, &t.us_per_ks) != 8)
      return false;
  }
  k.ip_staged_gather = dflt.ip_staged_gather;  // not tuned (key switches read their digits directly)
  k.ip_staged_ctas = dflt.ip_staged_ctas;
  k.ip_staged_depth = dflt.ip_staged_depth;
  if (k.fuse_ip_moddown < 0 || k.fuse_ip_moddown > 1 || k.bconv_tc_ctas < 1 || k.bconv_tc_ctas > 4 ||
      k.ntt_stream_stages < 2 || k.ntt_stream_stages > 3 || k.ntt_stream_ctas < 1 || k.ntt_stream_ctas > 3 ||
      k.bconv_tc_pipeline < 0 || k.bconv_tc_pipeline > 1)
    return false;
  if (t.comp_pipe != 0 && t.comp_pipe != 1) return false;
  if (t.ntt_mode & ~(FHE_NTT_OTF | FHE_NTT_SINGLE_PASS | FHE_NTT_STREAM | FHE_NTT_PERSIST)) return false;
  if (t.lanes < 1 || t.lanes > 4 || t.ip_ctas_per_sm < 1 || t.ip_ctas_per_sm > 2 ||
      (t.bconv_mode != FHE_BCONV_SCALAR && t.bconv_mode != FHE_BCONV_TC) || t.max_group < 0)
    return false;
  t.l2_budget_bytes = (size_t)budget;
  *r = t;
  return true;
}

extern "C" int fhe_autotune_cached(fhe_ctx *c, const char *path, int level, int n_items, int flags,
                                   fhe_tune_result *out, fhe_stream stream) {
  if (!c || !out || !path || !*path) return fhe_fail(FHE_EINVAL, "fhe_autotune_cached: null argument");
  if (level < 1 || level > c->L) return fhe_fail(FHE_ELEVEL, "fhe_autotune_cached: level %d", level);
  const std::string key = tune_key(c, level, n_items, flags);
  fhe_tune_result hit;
  bool found = false;
  if (FILE *f = fopen(path, "r")) {
    char line[1024];
    while (fgets(line, sizeof line, f)) {
      const char *bar = strchr(line, '|');
      if (!bar || (size_t)(bar - line) != key.size() + 1 || strncmp(line, key.c_str(), key.size()) != 0) continue;
      fhe_tune_result r;
      fhe_kernel_shape dflt;
      fhe_ctx_get_kernel_shape(c, &dflt);
      if (tune_parse(bar + 1, dflt, &r)) {
        hit = r;
        found = true;
      }
    }
    fclose(f);
  }
  if (found) {
    if (hit.bconv_mode == FHE_BCONV_TC && fhe_ctx_set_bconv(c, FHE_BCONV_TC) != FHE_OK)
      hit.bconv_mode = c->bconv_mode;  // not available on this context: keep its kernel
    c->batch_budget = hit.l2_budget_bytes;
    c->batch_lanes = hit.lanes;
    c->batch_max_group = hit.max_group;
    c->bconv_mode = hit.bconv_mode;
    c->tabs.ip_ctas_per_sm = hit.ip_ctas_per_sm;
    c->comp_pipe = hit.comp_pipe;
    if (fhe_ctx_set_ntt(c, hit.ntt_mode) != FHE_OK) hit.ntt_mode = 0, fhe_ctx_set_ntt(c, 0);
    if (fhe_ctx_set_kernel_shape(c, &hit.shape) != FHE_OK) fhe_ctx_get_kernel_shape(c, &hit.shape);
    hit.candidates = 0;  // served from the cache
    *out = hit;
    return FHE_OK;
  }
  int rc = fhe_autotune(c, level, n_items, flags, out, stream);
  if (rc != FHE_OK) return rc;
  char line[1024];
  const int len = snprintf(line, sizeof line,
                           "%s | lanes=%d budget=%llu group=%d bconv=%d ip=%d comp=%d ntt=%d fuse=%d tcctas=%d "
                           "tcpipe=%d nst=%d nsc=%d us=%.3f\n",
                           key.c_str(), out->lanes, (unsigned long long)out->l2_budget_bytes, out->max_group,
                           out->bconv_mode, out->ip_ctas_per_sm, out->comp_pipe, out->ntt_mode,
                           out->shape.fuse_ip_moddown, out->shape.bconv_tc_ctas, out->shape.bconv_tc_pipeline,
                           out->shape.ntt_stream_stages, out->shape.ntt_stream_ctas, out->us_per_ks);
  FILE *f = fopen(path, "a");
  if (!f) return fhe_fail(FHE_EINVAL, "fhe_autotune_cached: cannot append to %s", path);
  const bool ok = fwrite(line, 1, (size_t)len, f) == (size_t)len;  // one write per entry
  fclose(f);
  return ok ? FHE_OK : fhe_fail(FHE_EINVAL, "fhe_autotune_cached: write to %s failed", path);
}
