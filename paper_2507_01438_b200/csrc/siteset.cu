// A set of linear sites that see the same mixed batch (paper Section 3.4: every LoRA-augmented
// linear layer of the model is evaluated over the same batch of requests; Section 4.3: the mapping
// from adapter ids to samples is worked out once).  The set builds one routing plan per batch and
// hands its sites to the device in runs: one launch computes the shrink of every site of a run, the next
// one their base products with the expand, so that launches, ramp-ups and partly empty last waves are paid
// per run and not per site.
#include <cuda_runtime.h>

#include <cstring>
#include <new>
#include <vector>

#include "guard.h"
#include "pool.h"
#include "prefill.h"

using namespace edgelora;

struct edgelora_siteset {
  std::vector<edgelora_pool *> pools;
  std::vector<const void *> W;
  std::vector<int32_t> input_of;
  int32_t n_inputs = 0, max_tokens = 0;
  std::vector<int32_t> in_width;          // h_in of every input
  std::vector<int32_t> first_writer;      // per input, of the call at hand: the first site that writes into its memory
  edgelora_plan *plan = nullptr;
  DecodeWorkspace ws;                     // of the launches of decode-sized batches
  // host-buffer path (allocated on first use)
  std::vector<uint16_t *> dx;             // [n_inputs] device mirrors of the inputs
  int32_t *dids = nullptr;
  std::vector<uint16_t *> dy;             // [n_sites] device results of the sites that are read back
  std::vector<std::pair<int32_t, uint16_t *>> dy_scratch;  // (h_out, buffer) for the others
  cudaStream_t copy_stream = nullptr;     // read-back of results beside the sites that follow
  std::vector<cudaEvent_t> done_ev;       // [n_sites] recorded behind a site whose result is read back
  std::vector<cudaEvent_t> up_ev;         // [n_inputs] an input uploaded on the second stream has arrived
};

namespace {

bool capturing(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return st != cudaStreamCaptureStatusNone;
}

// Sites of a run that holds a result to be read back: the copy starts behind the run, so a long run delays it, and a short
// one pays for its own launches.  28 sites of four decoder layers, host call, us for runs of 1 / 4 / 7 / 14 / 32 sites:
// T = 2112, last layer read back 6512 / 6509 / 6857 / 6858 / 7161, the down projections 4092 / 4109 / 4214 / 4397 / 5015, k
// and v 3839 / 3836 / 3779 / 3932 / 4209; T = 320, last layer 1412 / 1322 / 1444 / 1438 / 1449, the down projections 1081 /
// 1083 / 1028 / 1055 / 1173, k and v 1264 / 1100 / 1013 / 1034 / 1061; all results: no difference.
constexpr int kReadBackRun = 7;

bool overlap(const void *a, size_t na, const void *b, size_t nb) {
  const uintptr_t pa = reinterpret_cast<uintptr_t>(a), pb = reinterpret_cast<uintptr_t>(b);
  return pa < pb + nb && pb < pa + na;
}

// after: optional, one event per site (or null): recorded on the stream behind that site's launch.
// before: optional, one event per site (or null): the stream waits for it in front of that site's launch.
int run_sites(edgelora_siteset *s, const void *const *x_dev, const int32_t *ids_dev, int32_t T,
              void *const *y_dev, cudaStream_t stream, const std::vector<cudaEvent_t> *after = nullptr,
              const std::vector<cudaEvent_t> *before = nullptr) {
  int rc = EDGELORA_OK;
  const int n = static_cast<int>(s->pools.size());
  const bool in_capture = capturing(stream);
  // A result that lies in an input's memory is seen by the sites behind it: a site that reads such an input starts
  // when the site in front of it is done (which is when all before that are), whatever overlap the pools allow.
  const size_t row = static_cast<size_t>(T) * 2;
  bool chained = false;
  for (int k = 0; k < s->n_inputs; ++k) {
    int i = 0;
    while (i < n && !(s->in_width[k] && overlap(x_dev[k], row * s->in_width[k], y_dev[i], row * s->pools[i]->cfg.h_out))) ++i;
    s->first_writer[k] = i;
    chained = chained || i < n;
  }
  // The sites go to the device in runs that share one shrink launch and one base-product launch, when every pool
  // runs in its default configuration and no result is an input.
  const bool decode = T <= kDecodeMaxT;
  bool runs = !chained;
  for (auto *p : s->pools) {
    runs = runs && p->opt_regime == 0 && p->opt_pdl >= 1 && !p->a_q8;
    if (decode)
      runs = runs && !p->opt_profile && T <= p->opt_gather_min_t && p->opt_decode_splits == 0 && p->opt_shrink_items == 0 &&
             p->opt_shrink_depth == 0;
  }
  if (!runs || !decode) {  // (the decode kernels derive the plan themselves)
    rc = edgelora_plan_build(s->plan, ids_dev, T, stream);
    if (rc != EDGELORA_OK) return rc;
  }
  if (!runs) {
    for (int i = 0; i < n; ++i) {
      if (before && (*before)[i] && cudaStreamWaitEvent(stream, (*before)[i], 0) != cudaSuccess) return EDGELORA_ERR_CUDA;
      // (otherwise the sites are independent given their inputs and results, so a site's shrink may start under the
      // previous site's base product)
      const Order order = s->first_writer[s->input_of[i]] < i ? Order::kAfter : i > 0 ? Order::kIndependent : Order::kPool;
      rc = lora_linear_impl(s->pools[i], s->plan, nullptr, s->W[i], x_dev[s->input_of[i]], T, y_dev[i], stream, order);
      if (rc != EDGELORA_OK) return rc;
      if (after && (*after)[i] && cudaEventRecord((*after)[i], stream) != cudaSuccess) return EDGELORA_ERR_CUDA;
    }
    return EDGELORA_OK;
  }
  for (int i = 0; i < n; ++i) {
    if ((reinterpret_cast<uintptr_t>(x_dev[s->input_of[i]]) | reinterpret_cast<uintptr_t>(s->W[i]) |
         reinterpret_cast<uintptr_t>(y_dev[i])) & 15)
      return EDGELORA_ERR_INVALID_ARG;
    rc = wait_for_loads(s->pools[i], stream, in_capture);
    if (rc != EDGELORA_OK) return rc;
  }
  for (int i0 = 0; i0 < n;) {
    // A run ends where the launch's tables are full, where a pool would come twice (its z workspace holds one
    // site's z), where two sites write the same memory (the later one is to be seen; results that the host call
    // does not read back share a buffer nobody looks at), where the pools' wait limits differ (a launch has one), in
    // front of a site whose input is still on its way, and behind kReadBackRun sites when results are read back beside
    // the sites that follow.  Profiled pools go one by one.
    SiteCall calls[kPairSites];
    SiteCall inputs[kPairInputs];  // the first site on each input
    int m = 0, n_inputs = 0;
    bool read_back = false;
    for (int i = i0; i < n && m < kPairSites; ++i) {
      edgelora_pool *p = s->pools[i];
      const SiteCall call{p, s->W[i], static_cast<const uint16_t *>(x_dev[s->input_of[i]]), y_dev[i]};
      if (m > 0 && ((before && (*before)[i]) || p->opt_profile || calls[0].p->opt_profile ||
                    p->wait_cycles != calls[0].p->wait_cycles || (read_back && m >= kReadBackRun)))
        break;
      bool again = false;
      for (int k = 0; k < m; ++k)
        again = again || calls[k].p == p ||
                (!(after && !(*after)[i] && !(*after)[i0 + k]) &&
                 overlap(y_dev[i], row * p->cfg.h_out, calls[k].y, row * calls[k].p->cfg.h_out));
      if (again) break;
      int xi = 0;
      while (xi < n_inputs && !inputs[xi].same_input(call)) ++xi;
      if (xi == kPairInputs) break;
      if (xi == n_inputs) inputs[n_inputs++] = call;
      if (m == 0 && before && (*before)[i] && cudaStreamWaitEvent(stream, (*before)[i], 0) != cudaSuccess)
        return EDGELORA_ERR_CUDA;
      calls[m++] = call;
      read_back = read_back || (after && (*after)[i]);
    }
    // The kernel in front of a run is the plan kernel, launched behind everything before it, or the base product of the run
    // before.  A decode-sized batch has no plan kernel: its first run starts behind everything before the set, whatever
    // overlap its pools allow (the sites read inputs of their own, which no pool's option speaks for).
    rc = decode ? decode_sites(calls, m, s->plan, ids_dev, T, s->ws, stream, i0 > 0)
                : prefill_sites(calls, m, s->plan, nullptr, T, stream, true);
    if (rc != EDGELORA_OK) return rc;
    for (int i = i0; i < i0 + m; ++i)
      if (after && (*after)[i] && cudaEventRecord((*after)[i], stream) != cudaSuccess) return EDGELORA_ERR_CUDA;
    i0 += m;
  }
  if (!in_capture) {  // slot loads issued later wait for this step
    for (auto *p : s->pools) {
      if (cudaEventRecord(p->use_ev, stream) != cudaSuccess) return EDGELORA_ERR_CUDA;
      p->use_recorded = true;
    }
  }
  return EDGELORA_OK;
}

}  // namespace

extern "C" {

int edgelora_siteset_create(int32_t n_sites, edgelora_pool_t *const *pools, const void *const *W_dev,
                            const int32_t *input_of_site, int32_t n_inputs, int32_t max_tokens,
                            edgelora_siteset_t **set_out) {
  if (n_sites < 1 || !pools || !W_dev || !input_of_site || n_inputs < 1 || !set_out) return EDGELORA_ERR_INVALID_ARG;
  if (max_tokens == 0) max_tokens = 8192;
  if (max_tokens < 0 || max_tokens > kMaxTokensLimit) return EDGELORA_ERR_TOO_MANY_TOKENS;
  edgelora_siteset *s = new (std::nothrow) edgelora_siteset();
  if (!s) return EDGELORA_ERR_INVALID_ARG;
  s->n_inputs = n_inputs;
  s->max_tokens = max_tokens;
  s->in_width.assign(n_inputs, 0);
  s->first_writer.assign(n_inputs, n_sites);
  for (int i = 0; i < n_sites; ++i) {
    edgelora_pool *p = pools[i];
    const int in = input_of_site[i];
    bool ok = p && W_dev[i] && in >= 0 && in < n_inputs && p->cfg.n_slots == pools[0]->cfg.n_slots &&
              p->cfg.max_tokens >= max_tokens;
    if (ok) {
      if (s->in_width[in] == 0) s->in_width[in] = p->cfg.h_in;
      ok = s->in_width[in] == p->cfg.h_in;  // every site on an input has that input's width
    }
    if (!ok) {
      delete s;
      return EDGELORA_ERR_INVALID_ARG;
    }
    s->pools.push_back(p);
    s->W.push_back(W_dev[i]);
    s->input_of.push_back(in);
  }
  int rc = edgelora_plan_create(max_tokens, pools[0]->cfg.n_slots, &s->plan);
  if (rc != EDGELORA_OK) {
    delete s;
    return rc;
  }
  s->ws.ctas = decode_workspace_ctas(pools, n_sites, max_tokens);
  const size_t planes = decode_workspace_planes(s->ws.ctas, max_tokens);
  const cudaError_t e = el_malloc(&s->ws.partial, (planes + static_cast<size_t>(s->ws.ctas) * 4) * 4);
  if (e != cudaSuccess) {
    set_last_cuda_error(e, "workspace of a site set");
    cudaGetLastError();
    edgelora_plan_destroy(s->plan);
    delete s;
    return EDGELORA_ERR_CUDA;
  }
  s->ws.arrivals = reinterpret_cast<int32_t *>(s->ws.partial + planes);
  s->dx.assign(n_inputs, nullptr);
  s->dy.assign(n_sites, nullptr);
  *set_out = s;
  return EDGELORA_OK;
}

int edgelora_siteset_destroy(edgelora_siteset_t *s) {
  if (!s) return EDGELORA_ERR_INVALID_ARG;
  cudaDeviceSynchronize();
  if (s->plan) edgelora_plan_destroy(s->plan);
  for (auto *q : s->dx) if (q) el_free(q);
  for (auto *q : s->dy) if (q) el_free(q);
  for (auto &e : s->dy_scratch) if (e.second) el_free(e.second);
  if (s->dids) el_free(s->dids);
  if (s->ws.partial) el_free(s->ws.partial);
  for (auto e : s->done_ev) if (e) cudaEventDestroy(e);
  for (auto e : s->up_ev) if (e) cudaEventDestroy(e);
  if (s->copy_stream) cudaStreamDestroy(s->copy_stream);
  cudaGetLastError();
  delete s;
  return EDGELORA_OK;
}

int edgelora_siteset_plan(edgelora_siteset_t *s, edgelora_plan_t **plan_out) {
  if (!s || !plan_out) return EDGELORA_ERR_INVALID_ARG;
  *plan_out = s->plan;
  return EDGELORA_OK;
}

int edgelora_siteset_run(edgelora_siteset_t *s, const void *const *x_dev, const int32_t *adapter_id_dev,
                         int32_t T, void *const *y_dev, void *stream) {
  if (!s || T < 0) return EDGELORA_ERR_INVALID_ARG;
  if (T == 0) return EDGELORA_OK;
  if (T > s->max_tokens) return EDGELORA_ERR_TOO_MANY_TOKENS;
  if (!x_dev || !adapter_id_dev || !y_dev) return EDGELORA_ERR_INVALID_ARG;
  for (int i = 0; i < s->n_inputs; ++i)
    if (!x_dev[i] && s->in_width[i]) return EDGELORA_ERR_INVALID_ARG;
  for (size_t i = 0; i < s->pools.size(); ++i)
    if (!y_dev[i]) return EDGELORA_ERR_INVALID_ARG;
  return run_sites(s, x_dev, adapter_id_dev, T, y_dev, static_cast<cudaStream_t>(stream));
}

int edgelora_siteset_run_host(edgelora_siteset_t *s, const uint16_t *const *x_host,
                              const int32_t *adapter_id_host, int32_t T, uint16_t *const *y_host,
                              void *stream) {
  if (!s || T < 0) return EDGELORA_ERR_INVALID_ARG;
  if (T == 0) return EDGELORA_OK;
  if (T > s->max_tokens) return EDGELORA_ERR_TOO_MANY_TOKENS;
  if (!x_host || !adapter_id_host || !y_host) return EDGELORA_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t mt = s->max_tokens;
  const int n = static_cast<int>(s->pools.size());
#define SET_TRY(expr)                                                                  \
  do {                                                                                 \
    cudaError_t _e = (expr);                                                           \
    if (_e != cudaSuccess) {                                                           \
      set_last_cuda_error(_e, #expr);                                                  \
      return EDGELORA_ERR_CUDA;                                                        \
    }                                                                                  \
  } while (0)
  // device mirrors, on first use: the inputs, the ids, one result buffer per site that is read
  // back and one shared buffer per output width for the sites that are not
  for (int i = 0; i < s->n_inputs; ++i) {
    if (!s->in_width[i]) continue;
    if (!x_host[i]) return EDGELORA_ERR_INVALID_ARG;
    if (!s->dx[i]) SET_TRY(el_malloc(&s->dx[i], mt * s->in_width[i] * 2));
  }
  if (!s->dids) SET_TRY(el_malloc(&s->dids, mt * 4));
  std::vector<void *> y_dev(n, nullptr);
  for (int i = 0; i < n; ++i) {
    const int32_t h_out = s->pools[i]->cfg.h_out;
    if (y_host[i]) {
      if (!s->dy[i]) SET_TRY(el_malloc(&s->dy[i], mt * h_out * 2));
      y_dev[i] = s->dy[i];
    } else {
      uint16_t *buf = nullptr;
      for (auto &e : s->dy_scratch)
        if (e.first == h_out) buf = e.second;
      if (!buf) {
        SET_TRY(el_malloc(&buf, mt * h_out * 2));
        s->dy_scratch.emplace_back(h_out, buf);
      }
      y_dev[i] = buf;
    }
  }
  // An input that the first sites do not need is uploaded on the second stream, beside them; the launches of its
  // first consumer wait for it.
  if (!s->copy_stream) SET_TRY(cudaStreamCreateWithFlags(&s->copy_stream, cudaStreamNonBlocking));
  if (s->up_ev.empty()) s->up_ev.assign(s->n_inputs, nullptr);
  std::vector<cudaEvent_t> before(n, nullptr);
  SET_TRY(cudaMemcpyAsync(s->dids, adapter_id_host, static_cast<size_t>(T) * 4, cudaMemcpyHostToDevice, st));
  for (int i = 0; i < s->n_inputs; ++i) {
    if (!s->in_width[i]) continue;
    int first = n;
    for (int k = 0; k < n; ++k)
      if (s->input_of[k] == i) {
        first = k;
        break;
      }
    const size_t bytes = static_cast<size_t>(T) * s->in_width[i] * 2;
    if (first == 0 || first == n) {
      SET_TRY(cudaMemcpyAsync(s->dx[i], x_host[i], bytes, cudaMemcpyHostToDevice, st));
    } else {
      if (!s->up_ev[i]) SET_TRY(cudaEventCreateWithFlags(&s->up_ev[i], cudaEventDisableTiming));
      SET_TRY(cudaMemcpyAsync(s->dx[i], x_host[i], bytes, cudaMemcpyHostToDevice, s->copy_stream));
      SET_TRY(cudaEventRecord(s->up_ev[i], s->copy_stream));
      before[first] = s->up_ev[i];
    }
  }
  std::vector<const void *> xd(s->dx.begin(), s->dx.end());
  // A result goes back to the host on a second stream as soon as its site is done, beside the sites
  // that follow (an event behind a launch keeps the next launch from starting under it, which is
  // paid only for the sites that are read back).
  if (s->done_ev.empty()) s->done_ev.assign(n, nullptr);
  for (int i = 0; i < n; ++i)
    if (y_host[i] && !s->done_ev[i]) SET_TRY(cudaEventCreateWithFlags(&s->done_ev[i], cudaEventDisableTiming));
  std::vector<cudaEvent_t> after(n, nullptr);
  for (int i = 0; i < n; ++i)
    if (y_host[i]) after[i] = s->done_ev[i];
  int rc = run_sites(s, xd.data(), s->dids, T, y_dev.data(), st, &after, &before);
  if (rc != EDGELORA_OK) return rc;
  for (int i = 0; i < n; ++i)
    if (y_host[i]) {
      SET_TRY(cudaStreamWaitEvent(s->copy_stream, s->done_ev[i], 0));
      SET_TRY(cudaMemcpyAsync(y_host[i], s->dy[i], static_cast<size_t>(T) * s->pools[i]->cfg.h_out * 2,
                              cudaMemcpyDeviceToHost, s->copy_stream));
    }
  SET_TRY(cudaStreamSynchronize(st));
  SET_TRY(cudaStreamSynchronize(s->copy_stream));
#undef SET_TRY
  return EDGELORA_OK;
}

}  // extern "C"
