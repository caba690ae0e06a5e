// Host side of the C ABI: the adapter pool (slot blocks + slot table in HBM, pinned staging,
// side-stream loads), the routing-plan objects and the launcher of the batched layer.
// Paper Section 3.3 / 4.2 (pre-allocated pool of fixed blocks, reuse after eviction) and
// Section 3.4 / 4.3 (batch LoRA inference).
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <utility>
#include <vector>

#include "decode_sites.h"
#include "decode_tile.h"
#include "guard.h"
#include "pool.h"
#include "prefill.h"
#include "shrink_tiles.h"
#include "tile_order.h"
#include "units.h"

using namespace edgelora;

namespace edgelora {
thread_local char g_last_error[256] = "";
void set_last_cuda_error(cudaError_t e, const char *what) {
  snprintf(g_last_error, sizeof g_last_error, "%s: %s", what, cudaGetErrorString(e));
  if (getenv("EDGELORA_LOG")) fprintf(stderr, "[edgelora] CUDA error: %s\n", g_last_error);
}
}  // namespace edgelora

namespace {

constexpr int kTmapCache = 32;
constexpr int kProfEvents = 8192;
constexpr size_t kSmemBudget = 220 * 1024;
constexpr int kMaxDecodeSplits = 8;  // K splits of a row tile form one (portable-size) cluster

#define CUDA_TRY(expr)                                   \
  do {                                                   \
    cudaError_t _e = (expr);                             \
    if (_e != cudaSuccess) {                             \
      set_last_cuda_error(_e, #expr);                    \
      return EDGELORA_ERR_CUDA;                          \
    }                                                    \
  } while (0)

inline int pad_rank(int r) { return r <= 16 ? 16 : (r <= 32 ? 32 : 64); }

// ---- cuTensorMapEncodeTiled through the runtime's driver entry point (no link to libcuda) ----
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// bf16 row-major [d2][d1][d0] (d2 == 0 => 2D), box = {box_cols, box_rows, 1}; out-of-range
// elements read as zero.  box_cols 64, 32, 16: operand tiles of the tensor core, rows of 128, 64 or 32 bytes with the
// swizzle of that width; otherwise (the decode shrink's row segments) no swizzle.
int encode_tmap(CUtensorMap *out, const void *base, uint64_t d0, uint64_t d1, uint64_t d2,
                uint32_t box_rows, uint32_t box_cols, uint64_t s1 = 0, uint64_t s2 = 0) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return EDGELORA_ERR_CUDA;
  const cuuint32_t rank = d2 ? 3 : 2;
  cuuint64_t dims[3] = {d0, d1, d2 ? d2 : 1};
  cuuint64_t strides[2] = {s1 ? s1 : d0 * 2, s2 ? s2 : d0 * d1 * 2};
  cuuint32_t box[3] = {box_cols, box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void *>(base), dims,
                  strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  box_cols == 64   ? CU_TENSOR_MAP_SWIZZLE_128B
                  : box_cols == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                  : box_cols == 16 ? CU_TENSOR_MAP_SWIZZLE_32B
                                   : CU_TENSOR_MAP_SWIZZLE_NONE,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    snprintf(g_last_error, sizeof g_last_error, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    return EDGELORA_ERR_CUDA;
  }
  return EDGELORA_OK;
}

}  // namespace

namespace {

// The descriptor is copied out: a later miss of the same call may reuse the cache entry it came
// from (the cache is a ring), and the launch takes its descriptors by value anyway.
int get_tmap(edgelora_pool *p, CUtensorMap *out, const void *base, uint64_t d0, uint64_t d1,
             uint64_t d2, uint32_t box_rows, uint32_t box_cols = kBlockK, uint64_t s1 = 0, uint64_t s2 = 0) {
  TmapKey key{base, d0, d1, d2, box_rows, box_cols, s1, s2};
  for (auto &e : p->tmaps)
    if (e.key == key) {
      *out = e.map;
      return EDGELORA_OK;
    }
  TmapEntry e;
  e.key = key;
  int rc = encode_tmap(&e.map, base, d0, d1, d2, box_rows, box_cols, s1, s2);
  if (rc != EDGELORA_OK) return rc;
  *out = e.map;
  if (p->tmaps.size() < static_cast<size_t>(kTmapCache)) {
    p->tmaps.push_back(e);
  } else {
    p->tmaps[p->tmap_next] = e;
    p->tmap_next = (p->tmap_next + 1) % kTmapCache;
  }
  return EDGELORA_OK;
}

bool stream_capturing(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return st != cudaStreamCaptureStatusNone;
}

struct ProfScope {
  edgelora_pool *p;
  cudaStream_t s;
  ProfRec *rec = nullptr;
  ProfScope(edgelora_pool *pool, int kernel, cudaStream_t stream) : p(pool), s(stream) {
    if (p->opt_profile && p->prof_used < p->prof.size() && !stream_capturing(s)) {
      rec = &p->prof[p->prof_used++];
      rec->kernel = kernel;
      cudaEventRecord(rec->start, s);
    }
  }
  ~ProfScope() {
    if (rec) cudaEventRecord(rec->stop, s);
  }
};

int check_cfg(const edgelora_pool_config *c) {
  if (!c) return EDGELORA_ERR_INVALID_ARG;
  if (c->h_in < 8 || c->h_out < 8 || (c->h_in % 8) || (c->h_out % 8)) return EDGELORA_ERR_INVALID_ARG;
  if (c->n_slots < 1 || c->n_slots > 65534) return EDGELORA_ERR_INVALID_ARG;
  if ((c->flags & EDGELORA_FLAG_A_Q8) && (c->h_in % 256)) return EDGELORA_ERR_INVALID_ARG;
  if (c->max_rank < 1) return EDGELORA_ERR_INVALID_ARG;
  if (c->max_rank > 64) return EDGELORA_ERR_RANK_TOO_LARGE;
  if (c->max_tokens < 0 || c->max_tokens > kMaxTokensLimit) return EDGELORA_ERR_TOO_MANY_TOKENS;
  return EDGELORA_OK;
}

size_t arena_bytes_for(const edgelora_pool_config *c) {
  const size_t R = pad_rank(c->max_rank);
  // A: bfloat16 rows, or Q8_0 rows of 34 bytes per 32 values; B: bfloat16
  const size_t a_row = (c->flags & EDGELORA_FLAG_A_Q8) ? static_cast<size_t>(c->h_in) / 32 * 34
                                                       : static_cast<size_t>(c->h_in) * 2;
  const size_t per_slot = R * a_row + 2 * R * static_cast<size_t>(c->h_out);
  return per_slot * c->n_slots;
}

int plan_alloc(edgelora_plan *pl) {
  const size_t mt = pl->max_tokens;
  const int max_tiles = pl->max_tokens / kSegMin + 8;
  // ids_valid, perm, group_adapter, seg_adapter, tok_seg, perm_short: mt each;
  // group_start, seg_start, gs_short, scratch: mt + 1 each; tiles; counts; status
  // lg_adapter: mt; mt_count: n_mt + 1; mt_list: n_mt * 256
  const size_t n_mt = (mt + kListTile - 1) / kListTile;
  const size_t ints = 7 * mt + 4 * (mt + 1) + 4 * static_cast<size_t>(max_tiles) + (n_mt + 1) +
                      n_mt * kListTile + 8 + 4;
  CUDA_TRY(el_malloc(&pl->block, ints * 4));
  CUDA_TRY(cudaMemset(pl->block, 0, ints * 4));
  int32_t *q = static_cast<int32_t *>(pl->block);
  PlanView &v = pl->pv;
  v.ids_valid = q; q += mt;
  v.perm = q; q += mt;
  v.group_adapter = q; q += mt;
  v.seg_adapter = q; q += mt;
  v.tok_seg = q; q += mt;
  v.perm_short = q; q += mt;
  v.group_start = q; q += mt + 1;
  v.seg_start = q; q += mt + 1;
  v.gs_short = q; q += mt + 1;
  v.scratch = q; q += mt + 1;
  v.sgmv_tiles = q; q += 4 * static_cast<size_t>(max_tiles);
  v.lg_adapter = q; q += mt;
  v.mt_count = q; q += n_mt + 1;
  v.mt_list = q; q += n_mt * kListTile;
  v.counts = q; q += 8;
  v.status = reinterpret_cast<uint32_t *>(q);
  v.max_sgmv_tiles = max_tiles;
  return EDGELORA_OK;
}

}  // namespace

extern "C" {

const char *edgelora_strerror(int code) {
  switch (code) {
    case EDGELORA_OK: return "ok";
    case EDGELORA_ERR_INVALID_ARG: return "invalid argument";
    case EDGELORA_ERR_BAD_SLOT: return "slot index out of range";
    case EDGELORA_ERR_RANK_TOO_LARGE: return "adapter rank exceeds the pool's max_rank (or 64)";
    case EDGELORA_ERR_ARENA_TOO_SMALL: return "caller arena smaller than edgelora_pool_bytes_required";
    case EDGELORA_ERR_CUDA: return g_last_error[0] ? g_last_error : "CUDA error";
    case EDGELORA_ERR_BAD_ADAPTER_ID: return "an adapter id outside [-1, n_slots) was seen (token computed base-only)";
    case EDGELORA_ERR_SLOT_EMPTY: return "an adapter id named an empty slot (token computed base-only)";
    case EDGELORA_ERR_TIMEOUT: return "a bounded in-kernel wait gave up";
    case EDGELORA_ERR_BOUNDS:
      return "checked build: a kernel met an index outside its array, or a guard zone around a device buffer was overwritten";
    case EDGELORA_ERR_TOO_MANY_TOKENS: return "T exceeds max_tokens (or max_tokens exceeds 32768)";
    case EDGELORA_ERR_CACHE_FULL: return "every block of the adapter cache is held by a running request";
    default: return "unknown error";
  }
}

int edgelora_pool_bytes_required(const edgelora_pool_config *cfg, size_t *bytes_out) {
  int rc = check_cfg(cfg);
  if (rc != EDGELORA_OK) return rc;
  if (!bytes_out) return EDGELORA_ERR_INVALID_ARG;
  *bytes_out = arena_bytes_for(cfg);
  return EDGELORA_OK;
}

int edgelora_plan_create(int32_t max_tokens, int32_t n_slots, edgelora_plan_t **plan_out) {
  if (!plan_out || n_slots < 1 || n_slots > 65534) return EDGELORA_ERR_INVALID_ARG;
  if (max_tokens == 0) max_tokens = 8192;
  if (max_tokens < 0 || max_tokens > kMaxTokensLimit) return EDGELORA_ERR_TOO_MANY_TOKENS;
  edgelora_plan *pl = new (std::nothrow) edgelora_plan();
  if (!pl) return EDGELORA_ERR_INVALID_ARG;
  pl->max_tokens = max_tokens;
  pl->n_slots = n_slots;
  int rc = plan_alloc(pl);
  if (rc != EDGELORA_OK) {
    if (pl->block) el_free(pl->block);
    delete pl;
    return rc;
  }
  init_plan_kernel();
  *plan_out = pl;
  return EDGELORA_OK;
}

int edgelora_plan_destroy(edgelora_plan_t *plan) {
  if (!plan) return EDGELORA_ERR_INVALID_ARG;
  cudaDeviceSynchronize();
  if (plan->block) el_free(plan->block);
  delete plan;
  return EDGELORA_OK;
}

int edgelora_plan_build(edgelora_plan_t *plan, const int32_t *ids_dev, int32_t T, void *stream) {
  if (!plan || T < 0 || (T > 0 && !ids_dev)) return EDGELORA_ERR_INVALID_ARG;
  if (T > plan->max_tokens) return EDGELORA_ERR_TOO_MANY_TOKENS;
  plan->last_T = T;
  if (T == 0) return EDGELORA_OK;
  plan->unread = true;
  launch_plan(ids_dev, T, plan->n_slots, plan->pv, false, static_cast<cudaStream_t>(stream));
  CUDA_TRY(cudaGetLastError());
  return EDGELORA_OK;
}

int edgelora_plan_export(edgelora_plan_t *plan, void *stream, int32_t *ids_valid, int32_t *perm,
                         int32_t *group_start, int32_t *group_adapter, int32_t *seg_start,
                         int32_t *seg_adapter, int32_t counts_out[2]) {
  if (!plan) return EDGELORA_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  CUDA_TRY(cudaStreamSynchronize(s));
  const int T = plan->last_T;
  int32_t counts[8] = {0};
  if (T > 0) CUDA_TRY(cudaMemcpy(counts, plan->pv.counts, sizeof counts, cudaMemcpyDeviceToHost));
  const int G = counts[0], NS = counts[1];
  auto get = [&](int32_t *dst, const int32_t *src, int n) -> cudaError_t {
    if (!dst || n <= 0) return cudaSuccess;
    return cudaMemcpy(dst, src, static_cast<size_t>(n) * 4, cudaMemcpyDeviceToHost);
  };
  CUDA_TRY(get(ids_valid, plan->pv.ids_valid, T));
  CUDA_TRY(get(perm, plan->pv.perm, T));
  CUDA_TRY(get(group_adapter, plan->pv.group_adapter, G));
  CUDA_TRY(get(seg_adapter, plan->pv.seg_adapter, NS));
  if (T > 0) {
    CUDA_TRY(get(group_start, plan->pv.group_start, G + 1));
    CUDA_TRY(get(seg_start, plan->pv.seg_start, NS + 1));
  } else {
    if (group_start) group_start[0] = 0;
    if (seg_start) seg_start[0] = 0;
  }
  if (counts_out) {
    counts_out[0] = G;
    counts_out[1] = NS;
  }
  return EDGELORA_OK;
}

int edgelora_pool_create(const edgelora_pool_config *cfg, edgelora_pool_t **pool_out) {
  int rc = check_cfg(cfg);
  if (rc != EDGELORA_OK) return rc;
  if (!pool_out) return EDGELORA_ERR_INVALID_ARG;
  const size_t need = arena_bytes_for(cfg);
  if (cfg->arena_dev) {
    if (cfg->arena_bytes < need) return EDGELORA_ERR_ARENA_TOO_SMALL;
    if (reinterpret_cast<uintptr_t>(cfg->arena_dev) % 256) return EDGELORA_ERR_INVALID_ARG;
  }
  int dev = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  cudaDeviceProp prop;
  CUDA_TRY(cudaGetDeviceProperties(&prop, dev));
  if (prop.major != 10) {
    snprintf(g_last_error, sizeof g_last_error, "device is sm_%d%d; this library is built for sm_100a only",
             prop.major, prop.minor);
    return EDGELORA_ERR_CUDA;
  }
  if (!get_encode_fn()) {
    snprintf(g_last_error, sizeof g_last_error, "cuTensorMapEncodeTiled not available from the driver");
    return EDGELORA_ERR_CUDA;
  }

  edgelora_pool *p = new (std::nothrow) edgelora_pool();
  if (!p) return EDGELORA_ERR_INVALID_ARG;
  p->cfg = *cfg;
  if (p->cfg.max_tokens == 0) p->cfg.max_tokens = 8192;
  p->R_pad = pad_rank(cfg->max_rank);
  p->device = dev;
  p->sms = prop.multiProcessorCount;
  p->a_q8 = (cfg->flags & EDGELORA_FLAG_A_Q8) != 0;
  // elements (2 bytes each) of a slot's A and B blocks; Q8_0 rows are 17 such elements per 32 values
  p->a_block = p->a_q8 ? static_cast<size_t>(p->R_pad) * (cfg->h_in / 32) * 17 : static_cast<size_t>(p->R_pad) * cfg->h_in;
  p->b_block = static_cast<size_t>(cfg->h_out) * p->R_pad;
  p->slots_host.assign(cfg->n_slots, SlotRow{0, 0.f, 0, 0});
  p->tmaps.reserve(kTmapCache);

#define POOL_TRY(expr)                         \
  do {                                         \
    cudaError_t _e = (expr);                   \
    if (_e != cudaSuccess) {                   \
      set_last_cuda_error(_e, #expr);          \
      edgelora_pool_destroy(p);                \
      return EDGELORA_ERR_CUDA;                \
    }                                          \
  } while (0)

  if (cfg->arena_dev) {
    p->arena = static_cast<uint8_t *>(cfg->arena_dev);
  } else {
    POOL_TRY(el_malloc(&p->arena, need));
    p->owns_arena = true;
  }
  p->A_pool = reinterpret_cast<uint16_t *>(p->arena);
  p->B_pool = p->A_pool + p->a_block * cfg->n_slots;
  POOL_TRY(el_malloc(&p->slots_dev, sizeof(SlotRow) * cfg->n_slots));
  POOL_TRY(cudaMemset(p->slots_dev, 0, sizeof(SlotRow) * cfg->n_slots));
  POOL_TRY(el_malloc(&p->status_dev, 16));
  POOL_TRY(cudaMemset(p->status_dev, 0, 16));
  // room for a block in its own layout or, for Q8_0 loads, A and B as 8-bit blocks (+ alignment)
  const size_t b_q8_bytes = static_cast<size_t>(cfg->h_out) * ((p->R_pad + 31) / 32) * 34;
  const size_t stage_bytes = p->a_block * 2 + 16 + std::max(p->b_block * 2, b_q8_bytes) + sizeof(SlotRow);
  for (auto &sb : p->staging) {
    POOL_TRY(cudaMallocHost(&sb.host, stage_bytes));
    POOL_TRY(cudaEventCreateWithFlags(&sb.done, cudaEventDisableTiming));
  }
  POOL_TRY(cudaStreamCreateWithFlags(&p->side, cudaStreamNonBlocking));
  POOL_TRY(cudaEventCreateWithFlags(&p->use_ev, cudaEventDisableTiming));
  // partial planes [0, kMaxZSplits) plus the final plane of the decode shrink
  POOL_TRY(el_malloc(&p->zws, sizeof(float) * (kMaxZSplits + 1) * static_cast<size_t>(p->cfg.max_tokens) * p->R_pad));
  POOL_TRY(el_malloc(&p->group_counters, sizeof(int32_t) * (kDecodeMaxT * 8 + 32)));
  POOL_TRY(cudaMemset(p->group_counters, 0, sizeof(int32_t) * (kDecodeMaxT * 8 + 32)));
  // an arrival counter per tile of the tensor-core shrink: segment tiles, then gather tiles (in parts)
  const int max_gather = (std::min(p->cfg.max_tokens, p->cfg.n_slots) * p->R_pad + kTileM - 1) / kTileM;
  p->n_tile_counters = p->cfg.max_tokens / kSegMin + 8 +
                       static_cast<int32_t>(gather_tiles_max(p->cfg.max_tokens, max_gather, p->sms));
  POOL_TRY(el_malloc(&p->tile_counters, sizeof(int32_t) * p->n_tile_counters));
  POOL_TRY(cudaMemset(p->tile_counters, 0, sizeof(int32_t) * p->n_tile_counters));
  POOL_TRY(gemm_set_smem_limit(kSmemBudget));
  POOL_TRY(shrink_set_smem_limit());
  POOL_TRY(shrink_tiles_set_smem_limit());
  POOL_TRY(pair_set_smem_limit());
  POOL_TRY(decode_sites_set_smem_limit());
  POOL_TRY(decode_tile_set_smem_limit());
  rc = edgelora_plan_create(p->cfg.max_tokens, cfg->n_slots, &p->plan);
  if (rc != EDGELORA_OK) {
    edgelora_pool_destroy(p);
    return rc;
  }
#undef POOL_TRY
  *pool_out = p;
  return EDGELORA_OK;
}

int edgelora_pool_destroy(edgelora_pool_t *p) {
  if (!p) return EDGELORA_ERR_INVALID_ARG;
  cudaDeviceSynchronize();
  if (p->plan) edgelora_plan_destroy(p->plan);
  if (p->owns_arena && p->arena) el_free(p->arena);
  if (p->slots_dev) el_free(p->slots_dev);
  if (p->status_dev) el_free(p->status_dev);
  for (auto &sb : p->staging) {
    if (sb.host) cudaFreeHost(sb.host);
    if (sb.done) cudaEventDestroy(sb.done);
  }
  if (p->side) cudaStreamDestroy(p->side);
  if (p->use_ev) cudaEventDestroy(p->use_ev);
  if (p->zws) el_free(p->zws);
  if (p->group_counters) el_free(p->group_counters);
  if (p->tile_counters) el_free(p->tile_counters);
  for (auto &r : p->prof) {
    cudaEventDestroy(r.start);
    cudaEventDestroy(r.stop);
  }
  if (p->hx) cudaFreeHost(p->hx);
  if (p->hy) cudaFreeHost(p->hy);
  if (p->hids) cudaFreeHost(p->hids);
  if (p->dx) el_free(p->dx);
  if (p->dy) el_free(p->dy);
  if (p->dids) el_free(p->dids);
  for (int b = 0; b < 2; ++b) {
    if (p->pdx[b]) el_free(p->pdx[b]);
    if (p->pdy[b]) el_free(p->pdy[b]);
    if (p->pdids[b]) el_free(p->pdids[b]);
    if (p->ev_in[b]) cudaEventDestroy(p->ev_in[b]);
    if (p->ev_done[b]) cudaEventDestroy(p->ev_done[b]);
    if (p->ev_out[b]) cudaEventDestroy(p->ev_out[b]);
  }
  if (p->h2d_stream) cudaStreamDestroy(p->h2d_stream);
  if (p->d2h_stream) cudaStreamDestroy(p->d2h_stream);
  cudaGetLastError();
  delete p;
  return EDGELORA_OK;
}

// where the slot-table row sits in a staging buffer: behind the largest payload
static size_t slot_row_offset(const edgelora_pool *p) {
  const size_t b_q8_bytes = static_cast<size_t>(p->cfg.h_out) * ((p->R_pad + 31) / 32) * 34;
  return p->a_block * 2 + 16 + std::max(p->b_block * 2, b_q8_bytes);
}

// Orders the side stream behind the last call that may still read this pool, once per call.
static int wait_for_use(edgelora_pool *p) {
  if (p->use_recorded) CUDA_TRY(cudaStreamWaitEvent(p->side, p->use_ev, 0));
  p->use_recorded = false;
  return EDGELORA_OK;
}
// A load is on the side stream: its staging buffer is free again, and the calls behind it may run, when its event is done.
static int load_issued(edgelora_pool *p, StagingBuf &sb) {
  CUDA_TRY(cudaEventRecord(sb.done, p->side));
  sb.in_flight = true;
  p->last_load = sb.done;
  p->load_seq += 1;
  return EDGELORA_OK;
}

static int stage_and_copy(edgelora_pool *p, int32_t slot, int32_t rank, float scale,
                          const uint16_t *A_host, const uint16_t *B_host) {
  if (p->a_q8 && rank > 0) return EDGELORA_ERR_INVALID_ARG;  // this pool takes Q8_0 adapters only
  StagingBuf &sb = p->staging[p->next_staging];
  p->next_staging = (p->next_staging + 1) % kStagingBuffers;
  if (sb.in_flight) {
    CUDA_TRY(cudaEventSynchronize(sb.done));
    sb.in_flight = false;
  }
  const int h_in = p->cfg.h_in, h_out = p->cfg.h_out, R = p->R_pad;
  uint16_t *sa = reinterpret_cast<uint16_t *>(sb.host);
  uint16_t *sbp = sa + p->a_block;
  SlotRow *srow = reinterpret_cast<SlotRow *>(sb.host + slot_row_offset(p));
  SlotRow &mirror = p->slots_host[slot];
  mirror.rank = rank;
  mirror.scale = scale;
  mirror.generation += 1;
  *srow = mirror;
  if (const int rc = wait_for_use(p)) return rc;
  if (rank > 0) {
    // A: rows [rank, R) are zero; B: columns [rank, R) are zero
    memcpy(sa, A_host, static_cast<size_t>(rank) * h_in * 2);
    memset(sa + static_cast<size_t>(rank) * h_in, 0, static_cast<size_t>(R - rank) * h_in * 2);
    if (rank == R) {
      memcpy(sbp, B_host, static_cast<size_t>(h_out) * R * 2);
    } else {
      for (int j = 0; j < h_out; ++j) {
        memcpy(sbp + static_cast<size_t>(j) * R, B_host + static_cast<size_t>(j) * rank, rank * 2);
        memset(sbp + static_cast<size_t>(j) * R + rank, 0, (R - rank) * 2);
      }
    }
    CUDA_TRY(cudaMemcpyAsync(p->A_pool + p->a_block * slot, sa, p->a_block * 2, cudaMemcpyHostToDevice, p->side));
    CUDA_TRY(cudaMemcpyAsync(p->B_pool + p->b_block * slot, sbp, p->b_block * 2, cudaMemcpyHostToDevice, p->side));
  }
  CUDA_TRY(cudaMemcpyAsync(p->slots_dev + slot, srow, sizeof(SlotRow), cudaMemcpyHostToDevice, p->side));
  return load_issued(p, sb);
}

int edgelora_pool_load_slot(edgelora_pool_t *p, int32_t slot, int32_t rank, float scale,
                            const uint16_t *A_host, const uint16_t *B_host) {
  if (!p || !A_host || !B_host) return EDGELORA_ERR_INVALID_ARG;
  if (slot < 0 || slot >= p->cfg.n_slots) return EDGELORA_ERR_BAD_SLOT;
  if (rank < 1) return EDGELORA_ERR_INVALID_ARG;
  if (rank > p->cfg.max_rank) return EDGELORA_ERR_RANK_TOO_LARGE;
  return stage_and_copy(p, slot, rank, scale, A_host, B_host);
}

int edgelora_pool_load_slot_pinned(edgelora_pool_t *p, int32_t slot, int32_t rank, float scale,
                                   const uint16_t *A_pinned, const uint16_t *B_pinned) {
  if (!p || !A_pinned || !B_pinned) return EDGELORA_ERR_INVALID_ARG;
  if (slot < 0 || slot >= p->cfg.n_slots) return EDGELORA_ERR_BAD_SLOT;
  if (rank != p->R_pad || p->a_q8) return EDGELORA_ERR_INVALID_ARG;  // already in the block's layout: nothing to pad
  cudaPointerAttributes at{};
  if (cudaPointerGetAttributes(&at, A_pinned) != cudaSuccess || at.type != cudaMemoryTypeHost ||
      cudaPointerGetAttributes(&at, B_pinned) != cudaSuccess || at.type != cudaMemoryTypeHost) {
    cudaGetLastError();
    return EDGELORA_ERR_INVALID_ARG;  // not page-locked: use edgelora_pool_load_slot
  }
  // the slot row still goes through a staging buffer (16 bytes the library owns)
  StagingBuf &sb = p->staging[p->next_staging];
  p->next_staging = (p->next_staging + 1) % kStagingBuffers;
  if (sb.in_flight) {
    CUDA_TRY(cudaEventSynchronize(sb.done));
    sb.in_flight = false;
  }
  SlotRow *srow = reinterpret_cast<SlotRow *>(sb.host + slot_row_offset(p));
  SlotRow &mirror = p->slots_host[slot];
  mirror.rank = rank;
  mirror.scale = scale;
  mirror.generation += 1;
  *srow = mirror;
  if (const int rc = wait_for_use(p)) return rc;
  CUDA_TRY(cudaMemcpyAsync(p->A_pool + p->a_block * slot, A_pinned, p->a_block * 2, cudaMemcpyHostToDevice, p->side));
  CUDA_TRY(cudaMemcpyAsync(p->B_pool + p->b_block * slot, B_pinned, p->b_block * 2, cudaMemcpyHostToDevice, p->side));
  CUDA_TRY(cudaMemcpyAsync(p->slots_dev + slot, srow, sizeof(SlotRow), cudaMemcpyHostToDevice, p->side));
  return load_issued(p, sb);
}

int edgelora_pool_load_slot_q8(edgelora_pool_t *p, int32_t slot, int32_t rank, float scale, const void *A_q8,
                               const void *B_q8) {
  if (!p || !A_q8 || !B_q8) return EDGELORA_ERR_INVALID_ARG;
  if (slot < 0 || slot >= p->cfg.n_slots) return EDGELORA_ERR_BAD_SLOT;
  if (rank < 1 || (p->cfg.h_in % 32)) return EDGELORA_ERR_INVALID_ARG;
  if (rank > p->cfg.max_rank) return EDGELORA_ERR_RANK_TOO_LARGE;
  const int h_in = p->cfg.h_in, h_out = p->cfg.h_out, R = p->R_pad;
  const size_t a_bytes = static_cast<size_t>(rank) * (h_in / 32) * 34;
  const size_t b_bytes = static_cast<size_t>(h_out) * ((rank + 31) / 32) * 34;
  const size_t b_off = (a_bytes + 15) & ~static_cast<size_t>(15);
  StagingBuf &sb = p->staging[p->next_staging];
  p->next_staging = (p->next_staging + 1) % kStagingBuffers;
  if (sb.in_flight) {
    CUDA_TRY(cudaEventSynchronize(sb.done));
    sb.in_flight = false;
  }
  // the 8-bit form is smaller than the block the staging buffer was sized for
  memcpy(sb.host, A_q8, a_bytes);
  memcpy(sb.host + b_off, B_q8, b_bytes);
  SlotRow &mirror = p->slots_host[slot];
  mirror.rank = rank;
  mirror.scale = scale;
  mirror.generation += 1;
  if (const int rc = wait_for_use(p)) return rc;
  CUDA_TRY(launch_q8_load(sb.host, a_bytes, sb.host + b_off, b_bytes, p->A_pool + p->a_block * slot,
                          p->B_pool + p->b_block * slot, mirror, p->slots_dev + slot, R, h_in, h_out, p->a_q8, p->side));
  return load_issued(p, sb);
}

int edgelora_pool_evict_slot(edgelora_pool_t *p, int32_t slot) {
  if (!p) return EDGELORA_ERR_INVALID_ARG;
  if (slot < 0 || slot >= p->cfg.n_slots) return EDGELORA_ERR_BAD_SLOT;
  return stage_and_copy(p, slot, 0, 0.f, nullptr, nullptr);
}

int edgelora_pool_wait_loads(edgelora_pool_t *p) {
  if (!p) return EDGELORA_ERR_INVALID_ARG;
  CUDA_TRY(cudaStreamSynchronize(p->side));
  for (auto &sb : p->staging) sb.in_flight = false;
  return EDGELORA_OK;
}

int edgelora_pool_plan(edgelora_pool_t *p, edgelora_plan_t **plan_out) {
  if (!p || !plan_out) return EDGELORA_ERR_INVALID_ARG;
  *plan_out = p->plan;
  return EDGELORA_OK;
}

int edgelora_pool_set_option(edgelora_pool_t *p, int32_t option, int32_t value) {
  if (!p) return EDGELORA_ERR_INVALID_ARG;
  switch (option) {
    case EDGELORA_OPT_REGIME:
      if (value < 0 || value > 2) return EDGELORA_ERR_INVALID_ARG;
      p->opt_regime = value;
      return EDGELORA_OK;
    case EDGELORA_OPT_PROFILE:
      p->opt_profile = value ? 1 : 0;
      if (p->opt_profile && p->prof.empty()) {
        p->prof.resize(kProfEvents);
        for (auto &r : p->prof) {
          CUDA_TRY(cudaEventCreate(&r.start));
          CUDA_TRY(cudaEventCreate(&r.stop));
        }
      }
      return EDGELORA_OK;
    case EDGELORA_OPT_PDL:
      if (value < 0 || value > 2) return EDGELORA_ERR_INVALID_ARG;
      p->opt_pdl = value;
      return EDGELORA_OK;
    case EDGELORA_OPT_DECODE_SPLITS:
      if (value < 0 || value > kMaxDecodeSplits) return EDGELORA_ERR_INVALID_ARG;
      p->opt_decode_splits = value;
      return EDGELORA_OK;
    case EDGELORA_OPT_WAIT_CYCLES:
      if (value < 0) return EDGELORA_ERR_INVALID_ARG;
      p->wait_cycles = value == 0 ? ptx::kWaitLimitCycles : static_cast<long long>(value) * 1024;
      return EDGELORA_OK;
    case EDGELORA_OPT_SHRINK_ITEMS:
      if (value < 0) return EDGELORA_ERR_INVALID_ARG;
      p->opt_shrink_items = value;
      return EDGELORA_OK;
    case EDGELORA_OPT_SHRINK_DEPTH:
      if (value != 0 && value != 2 && value != 4) return EDGELORA_ERR_INVALID_ARG;
      p->opt_shrink_depth = value;
      return EDGELORA_OK;
    case EDGELORA_OPT_FUSED_DECODE:
      if (value != 0 && value != 1) return EDGELORA_ERR_INVALID_ARG;
      p->opt_fused_decode = value;
      return EDGELORA_OK;
    case EDGELORA_OPT_GATHER_SPLITS:
      if (value < 0 || value > 8) return EDGELORA_ERR_INVALID_ARG;
      p->opt_gather_splits = value;
      return EDGELORA_OK;
    case EDGELORA_OPT_GATHER_MIN_T:
      if (value < 0 || value > kDecodeMaxT) return EDGELORA_ERR_INVALID_ARG;
      p->opt_gather_min_t = value;
      return EDGELORA_OK;
    default:
      return EDGELORA_ERR_INVALID_ARG;
  }
}

int edgelora_pool_last_launch(edgelora_pool_t *p, int64_t info_out[8]) {
  if (!p || !info_out) return EDGELORA_ERR_INVALID_ARG;
  memcpy(info_out, p->last_info, sizeof p->last_info);
  info_out[6] = p->total_launches;
  return EDGELORA_OK;
}

int edgelora_pool_kernel_times(edgelora_pool_t *p, double ms_out[5], int64_t launches_out[5],
                               int32_t reset) {
  if (!p) return EDGELORA_ERR_INVALID_ARG;
  for (size_t i = 0; i < p->prof_used; ++i) {
    ProfRec &r = p->prof[i];
    CUDA_TRY(cudaEventSynchronize(r.stop));
    float ms = 0.f;
    CUDA_TRY(cudaEventElapsedTime(&ms, r.start, r.stop));
    p->prof_ms[r.kernel] += ms;
    p->prof_n[r.kernel] += 1;
  }
  p->prof_used = 0;
  for (int k = 0; k < 5; ++k) {
    if (ms_out) ms_out[k] = p->prof_ms[k];
    if (launches_out) launches_out[k] = p->prof_n[k];
    if (reset) {
      p->prof_ms[k] = 0;
      p->prof_n[k] = 0;
    }
  }
  return EDGELORA_OK;
}

int edgelora_pool_sync_status(edgelora_pool_t *p, uint32_t *bits_out) {
  if (!p) return EDGELORA_ERR_INVALID_ARG;
  CUDA_TRY(cudaDeviceSynchronize());
  uint32_t a = 0, b = 0;
  CUDA_TRY(cudaMemcpy(&a, p->status_dev, 4, cudaMemcpyDeviceToHost));
  CUDA_TRY(cudaMemcpy(&b, p->plan->pv.status, 4, cudaMemcpyDeviceToHost));
  CUDA_TRY(cudaMemset(p->status_dev, 0, 4));
  CUDA_TRY(cudaMemset(p->plan->pv.status, 0, 8));
  const uint32_t bits = a | b;
  if (bits_out) *bits_out = bits;
  // a wait that ran out can leave arrival counters between their values: nothing is in flight now
  if (bits & EDGELORA_STATUS_TIMEOUT) {
    CUDA_TRY(cudaMemset(p->group_counters, 0, sizeof(int32_t) * (kDecodeMaxT * 8 + 32)));
    CUDA_TRY(cudaMemset(p->tile_counters, 0, sizeof(int32_t) * p->n_tile_counters));
  }
  if (bits & EDGELORA_STATUS_BOUNDS) {  // checked build: which test failed first
    uint32_t site = 0;
    CUDA_TRY(cudaMemcpy(&site, p->status_dev + 1, 4, cudaMemcpyDeviceToHost));
    CUDA_TRY(cudaMemset(p->status_dev + 1, 0, 4));
    snprintf(g_last_error, sizeof g_last_error, "a kernel's index test failed (test %u)", site);
    return EDGELORA_ERR_BOUNDS;
  }
  if (bits & EDGELORA_STATUS_TIMEOUT) return EDGELORA_ERR_TIMEOUT;
  if (edgelora_check_guards() != EDGELORA_OK) return EDGELORA_ERR_BOUNDS;  // always intact in the normal build
  if (bits & EDGELORA_STATUS_BAD_ADAPTER_ID) return EDGELORA_ERR_BAD_ADAPTER_ID;
  if (bits & EDGELORA_STATUS_SLOT_EMPTY) return EDGELORA_ERR_SLOT_EMPTY;
  return EDGELORA_OK;
}

int edgelora_plan_sync_status(edgelora_plan_t *plan, void *stream, uint32_t *bits_out) {
  if (!plan) return EDGELORA_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  CUDA_TRY(cudaStreamSynchronize(s));
  uint32_t bits = 0;
  CUDA_TRY(cudaMemcpy(&bits, plan->pv.status, 4, cudaMemcpyDeviceToHost));
  CUDA_TRY(cudaMemset(plan->pv.status, 0, 4));
  if (bits_out) *bits_out = bits;
  if (bits & EDGELORA_STATUS_BOUNDS) return EDGELORA_ERR_BOUNDS;
  if (bits & EDGELORA_STATUS_TIMEOUT) return EDGELORA_ERR_TIMEOUT;
  if (bits & EDGELORA_STATUS_BAD_ADAPTER_ID) return EDGELORA_ERR_BAD_ADAPTER_ID;
  if (bits & EDGELORA_STATUS_SLOT_EMPTY) return EDGELORA_ERR_SLOT_EMPTY;
  return EDGELORA_OK;
}

int edgelora_pool_selftest_wait(edgelora_pool_t *p, void *stream) {
  if (!p) return EDGELORA_ERR_INVALID_ARG;
  // only with a lowered limit: at the default the kernel would spin for seconds
  if (p->wait_cycles > (1LL << 24)) return EDGELORA_ERR_INVALID_ARG;
  CUDA_TRY(launch_wait_selftest(p->status_dev, p->wait_cycles, static_cast<cudaStream_t>(stream)));
  return EDGELORA_OK;
}

// The layer.  Decode regime (T <= 256): routing + shrink in one kernel, then the base product with
// the expand and the split-K reduction fused in.  Prefill regime: plan, gather shrink for short
// runs, segment shrink for long runs, base product with the expand fused in.
}  // extern "C"

namespace edgelora {

// Orders a call behind every load issued so far, once per stream and load (a wait node between two
// calls of one stream would also keep them from overlapping).  A captured call records no such wait:
// see the header for what a graph's owner has to do instead.
int wait_for_loads(edgelora_pool *p, cudaStream_t stream, bool capturing) {
  if (p->load_seq == 0 || capturing) return EDGELORA_OK;
  auto it = std::find_if(p->load_waited.begin(), p->load_waited.end(),
                         [&](const std::pair<cudaStream_t, uint64_t> &e) { return e.first == stream; });
  if (it == p->load_waited.end()) {
    if (p->load_waited.size() >= 64) p->load_waited.clear();  // streams come and go: start over
    p->load_waited.emplace_back(stream, 0);
    it = p->load_waited.end() - 1;
  }
  if (it->second != p->load_seq) {
    CUDA_TRY(cudaStreamWaitEvent(stream, p->last_load, 0));
    it->second = p->load_seq;
  }
  return EDGELORA_OK;
}

// ---- the tensor-core shrink (shrink_tiles.cu): what a site, its input and the plan contribute to a launch
static int fill_shrink_site(edgelora_pool *q, ShrinkSite *s, int splits, int x_index) {
  s->slots = q->slots_dev;
  s->zws = q->zws;
  s->tile_counters = q->tile_counters;
  s->status = q->status_dev;
  s->x_index = x_index;
  s->kb_total = (q->cfg.h_in + kBlockK - 1) / kBlockK;
  s->R_pad = q->R_pad;
  s->max_tokens = q->cfg.max_tokens;
  s->splits = splits;
  // the A blocks as one 2D matrix [n_slots * R_pad][h_in]: slot a is rows [a R_pad, (a + 1) R_pad)
  return get_tmap(q, &s->a, q->A_pool, q->cfg.h_in, static_cast<uint64_t>(q->R_pad) * q->cfg.n_slots, 0, q->R_pad);
}
static int fill_shrink_inputs(edgelora_pool *q, const uint16_t *x, int32_t T, CUtensorMap *mx, CUtensorMap *mg) {
  const int rc = get_tmap(q, mx, x, q->cfg.h_in, T, 0, kTileM);
  return rc ? rc : get_tmap(q, mg, x, q->cfg.h_in, T, 0, 1);
}
template <int kSites>
static void fill_shrink_plan(const edgelora_plan *plan, int32_t T, long long wait_cycles, int n_sites, int z_bf16,
                             ShrinkBatch<kSites> *b) {
  b->n_sites = n_sites;
  b->T = T;
  b->n_slots = plan->n_slots;
  b->z_bf16 = z_bf16;
  b->sgmv_tiles = plan->pv.sgmv_tiles;
  b->counts = plan->pv.counts;
  b->perm_short = plan->pv.perm_short;
  b->gs_short = plan->pv.gs_short;
  b->group_adapter = plan->pv.group_adapter;
  b->ids_valid = plan->pv.ids_valid;
  b->wait_cycles = wait_cycles;
}

// K splits of a site's shrink tiles.  A single site is split until every SM has an item, but not further than the
// sum of the planes at the end of a tile (1.6 us per plane of 128 x 64) gains over the K blocks (0.25 us each): the
// sum of both is least near sqrt(10 kb / R).  In a run of sites the items of all sites share the grid, and items
// of about 32 K blocks keep a wide input from making long ones.
static int shrink_splits(const edgelora_pool *q, int32_t T, int n_sites) {
  if (T <= kDecodeMaxT) return 1;
  const int kbt = (q->cfg.h_in + kBlockK - 1) / kBlockK;
  int z = n_sites > 1 ? std::min(8, std::max(1, kbt / 32)) : std::min(8, q->sms / std::max(1, T / kTileM));
  if (n_sites == 1) z = std::min(z, static_cast<int>(std::sqrt(10.0 * kbt / q->R_pad) + 0.5));
  z = std::max(1, std::min(z, kbt / 4));
  const int kb_per = (kbt + z - 1) / z;
  return (kbt + kb_per - 1) / kb_per;
}

// W rows of a pair tile.  A K block of a tile takes about 2 BN + 140 cycles (2 BN is the tensor pipe's share),
// below BN = 160 about 480 (the hand-over of a K block sets the pace), so the width whose last wave is fullest for
// the width's efficiency is taken; the sites' tiles form one list over all pairs.  Measured per call:
// 14336 -> 4096, T = 4096: 367 us at 256, 381 at 192; 4096 -> 4096, T = 300: 32 us at 160, 37 at 128 and 256;
// 3080 -> 5000, T = 1111: 68 us at 192, 72 at 256, 80 at 128.
static int pair_width(const SiteCall *sites, int n, int n_mtiles, int units) {
  int best = 0;
  double best_cost = 0;
  for (int BN = 256; BN >= 64; BN -= 32) {
    double work = 0;
    int64_t tiles = 0;
    int kb_max = 0;
    for (int i = 0; i < n; ++i) {
      const int kb = (sites[i].p->cfg.h_in + kBlockK - 1) / kBlockK + 4;
      const int64_t t = static_cast<int64_t>(n_mtiles) * ((sites[i].p->cfg.h_out + BN - 1) / BN);
      tiles += t;
      work += static_cast<double>(t) * kb;
      kb_max = std::max(kb_max, kb);
    }
    const double waves = static_cast<double>((tiles + units - 1) / units);
    // one site: whole waves; several: the list's total, and half a tile for its ragged end
    const double k = n == 1 ? waves * kb_max : std::max(work / units + 0.5 * kb_max, static_cast<double>(kb_max));
    const double cost = k * (BN >= 160 ? 2 * BN + 140 : 480) + 12.0 * BN;  // + the last tile's epilogue
    if (best == 0 || cost < best_cost) {
      best = BN;
      best_cost = cost;
    }
  }
  return best;
}

template <int kSites>
static int prefill_batch(const SiteCall *sites, int n, edgelora_plan *plan, int32_t T, cudaStream_t stream,
                         bool pdl_shrink, bool pdl_base) {
  edgelora_pool *p0 = sites[0].p;
  const int n_mtiles = (T + kListTile - 1) / kListTile;
  const int BN = pair_width(sites, n, n_mtiles, std::max(1, p0->sms / 2));
  ShrinkBatch<kSites> sb{};
  PairBatch<kSites> pb{};
  fill_shrink_plan(plan, T, p0->wait_cycles, n, 1, &sb);
  pb.n_sites = n;
  pb.T = T;
  pb.n_slots = plan->n_slots;
  pb.BN = BN;
  pb.stages = pair_stages(BN);
  pb.n_mtiles = n_mtiles;
  pb.ids_valid = plan->pv.ids_valid;
  pb.mt_count = plan->pv.mt_count;
  pb.mt_list = plan->pv.mt_list;
  pb.wait_cycles = p0->wait_cycles;
  const SiteCall *inputs[kPairInputs] = {};  // the first site on each input
  int n_inputs = 0, tiles = 0;
  for (int i = 0; i < n; ++i) {
    edgelora_pool *q = sites[i].p;
    int xi = 0;
    while (xi < n_inputs && !inputs[xi]->same_input(sites[i])) ++xi;
    if (xi == n_inputs) {
      inputs[n_inputs++] = &sites[i];
      const int rc = fill_shrink_inputs(q, sites[i].x, T, &sb.x[xi], &sb.xg[xi]);
      if (rc) return rc;
      pb.x[xi] = sb.x[xi];
    }
    PairSite &s = pb.site[i];
    int rc = fill_shrink_site(q, &sb.site[i], shrink_splits(q, T, n), xi);
    if (!rc) rc = get_tmap(q, &s.w, sites[i].W, q->cfg.h_in, q->cfg.h_out, 0, BN / 2);
    if (!rc) rc = get_tmap(q, &s.b, q->B_pool, q->R_pad, q->cfg.h_out, q->cfg.n_slots, BN / 2, q->R_pad);
    if (rc) return rc;
    tiles += n_mtiles * ((q->cfg.h_out + BN - 1) / BN);
    s.y = static_cast<uint16_t *>(sites[i].y);
    s.slots = q->slots_dev;
    s.zb = reinterpret_cast<const uint4 *>(q->zws + static_cast<size_t>(kMaxZSplits) * q->cfg.max_tokens * q->R_pad);
    s.status = q->status_dev;
    s.tile_end = tiles;
    s.x_index = xi;
    s.h_out = q->cfg.h_out;
    s.kb_total = (q->cfg.h_in + kBlockK - 1) / kBlockK;
    s.R_pad = q->R_pad;
  }
  {
    ProfScope ps(p0, 2, stream);
    CUDA_TRY(launch_shrink_tiles(sb, p0->sms, pdl_shrink, stream));
  }
  {
    ProfScope ps(p0, 3, stream);
    CUDA_TRY(launch_pair_gemm(pb, p0->sms, pdl_base, stream));
  }
  for (int i = 0; i < n; ++i) {
    int64_t *info = sites[i].p->last_info;
    info[1] = 2;
    info[2] = pair_grid(tiles, p0->sms);
    info[3] = 1;
    info[4] = pb.stages;
    info[5] = BN;
  }
  return EDGELORA_OK;
}

// Large batches: plan (when ids are given), shrink, base product with the expand, for one site or for a run of
// sites that share the plan: at most kPairSites sites on at most kPairInputs inputs, no pool twice.
int prefill_sites(const SiteCall *sites, int n, edgelora_plan *plan, const int32_t *ids_dev, int32_t T,
                  cudaStream_t stream, bool pdl_first) {
  edgelora_pool *p0 = sites[0].p;
  const bool pdl = p0->opt_pdl >= 1 && !p0->opt_profile;
  int launches = 2;
  if (ids_dev) {
    ProfScope ps(p0, 0, stream);
    plan->last_T = T;
    plan->unread = true;
    launch_plan(ids_dev, T, plan->n_slots, plan->pv, pdl_first, stream);
    CUDA_TRY(cudaGetLastError());
    ++launches;
  }
  const bool pdl_shrink = ids_dev ? pdl : (pdl_first && pdl);
  const int rc = n == 1 ? prefill_batch<1>(sites, n, plan, T, stream, pdl_shrink, pdl)
                        : prefill_batch<kPairSites>(sites, n, plan, T, stream, pdl_shrink, pdl);
  if (rc) return rc;
  for (int i = 0; i < n; ++i) sites[i].p->last_info[0] = i == 0 ? launches : 0;
  p0->total_launches += launches;
  return EDGELORA_OK;
}

// ---- decode-sized batches of a run of sites (decode_sites.cu)
static_assert(kPairSites <= kDecSites && kPairInputs <= kDecInputs, "the runs of a set are cut for either launch");
static int32_t decode_columns(int32_t T) { return std::max(16, (T + 15) / 16 * 16); }

int32_t decode_workspace_ctas(edgelora_pool *const *pools, int32_t n, int32_t max_tokens) {
  const int32_t T = std::min(max_tokens, kDecodeMaxT), stages = expand_stages_max(T, pools[0]->cfg.n_slots, kExpTok);
  int64_t units = 0;
  for (int32_t i = 0; i < n; ++i) {
    const edgelora_pool_config &c = pools[i]->cfg;
    units += static_cast<int64_t>((c.h_out + kTileM - 1) / kTileM) *
             ((c.h_in + kBlockK - 1) / kBlockK + expand_units(stages, pools[i]->R_pad));
  }
  return run_count(static_cast<int32_t>(std::min<int64_t>(units, INT32_MAX)), pools[0]->sms);
}
size_t decode_workspace_planes(int32_t ctas, int32_t max_tokens) {
  return static_cast<size_t>(ctas) * 2 * kTileM * decode_columns(std::min(max_tokens, kDecodeMaxT));
}

static int fill_decode_site(const SiteCall &c, int x_index, DecSite *d) {
  edgelora_pool *q = c.p;
  const int h_in = q->cfg.h_in, h_out = q->cfg.h_out, R = q->R_pad;
  const int rc = get_tmap(q, &d->w, c.W, h_in, h_out, 0, kTileM);
  if (rc) return rc;
  d->slots = q->slots_dev;
  d->z = q->zws + static_cast<size_t>(kMaxZSplits) * q->cfg.max_tokens * R;
  d->status = q->status_dev;
  d->x_index = x_index;
  d->R_pad = R;
  d->y = static_cast<uint16_t *>(c.y);
  d->h_out = h_out;
  d->kb = (h_in + kBlockK - 1) / kBlockK;
  return get_tmap(q, &d->b, q->B_pool, R, h_out, q->cfg.n_slots, kTileM, R);
}

int decode_sites(const SiteCall *sites, int n, edgelora_plan *plan, const int32_t *ids_dev, int32_t T,
                 const DecodeWorkspace &ws, cudaStream_t stream, bool pdl_first) {
  edgelora_pool *p0 = sites[0].p;
  const int32_t N = decode_columns(T);
  int32_t R_max = 0;
  for (int i = 0; i < n; ++i) R_max = std::max(R_max, sites[i].p->R_pad);
  const DecShape shape = decode_sites_shape(N, R_max);
  DecShrinkBatch sb{};
  DecBatch db{};
  sb.n_sites = db.n_sites = n;
  sb.T = T;
  sb.n_slots = db.n_slots = plan->n_slots;
  sb.ids = ids_dev;
  sb.pv = plan->pv;
  sb.zero = db.arrivals = ws.arrivals;
  sb.n_zero = 4 * ws.ctas;
  db.T = T;
  db.N = N;
  db.ids = ids_dev;
  db.stages = shape.stages;
  db.exp_stages = shape.exp_stages;
  db.exp_bytes = shape.exp_bytes;
  db.n_acc = shape.n_acc;
  db.tmem_cols = shape.tmem_cols;
  db.partial = ws.partial;
  db.wait_cycles = p0->wait_cycles;
  const SiteCall *inputs[kDecInputs] = {};  // the first site on each input
  int n_inputs = 0;
  for (int i = 0; i < n; ++i) {
    edgelora_pool *q = sites[i].p;
    const int h_in = q->cfg.h_in, R = q->R_pad;
    int xi = 0, rc = EDGELORA_OK;
    while (xi < n_inputs && !inputs[xi]->same_input(sites[i])) ++xi;
    if (xi == n_inputs) {
      inputs[n_inputs++] = &sites[i];
      rc = get_tmap(q, &sb.x[xi], sites[i].x, h_in, T, 0, 1, kShrinkStepElems);
      if (!rc) rc = get_tmap(q, &db.x[xi], sites[i].x, h_in, T, 0, N);
      if (rc) return rc;
    }
    DecShrinkSite &s = sb.site[i];
    rc = get_tmap(q, &s.a, q->A_pool, h_in, R, q->cfg.n_slots, 8, kShrinkStepElems);
    if (!rc) rc = fill_decode_site(sites[i], xi, &db.site[i]);
    if (rc) return rc;
    s.slots = q->slots_dev;
    s.zws = q->zws;
    s.counters = q->group_counters;
    s.status = q->status_dev;
    s.x_index = xi;
    s.n_ksteps = (h_in + kShrinkStepElems - 1) / kShrinkStepElems;
    // K chunks of eight steps or more, 32 KB of A per item (four and sixteen: no difference)
    s.ks = std::max(1, std::min(kMaxZSplits, s.n_ksteps / 8));
    s.R_pad = R;
    s.max_tokens = q->cfg.max_tokens;
  }
  plan->last_T = T;
  plan->unread = true;
  if (getenv("EDGELORA_LOG")) fprintf(stderr, "edgelora: decode T %d N %d sites %d grid %d\n", T, N, n, ws.ctas);
  // (two CTAs of the shrink per SM, 98 KB of ring each: 1 % less for 28 sites than one)
  CUDA_TRY(launch_decode_sites_shrink(sb, 2 * p0->sms, pdl_first, stream));
  CUDA_TRY(launch_decode_sites(db, shape, ws.ctas, true, stream));
  for (int i = 0; i < n; ++i) {
    int64_t *info = sites[i].p->last_info;
    info[0] = i == 0 ? 2 : 0;
    info[1] = 1;
    info[2] = ws.ctas;
    info[3] = 1;
    info[4] = shape.stages;
    info[5] = N;
  }
  p0->total_launches += 2;
  return EDGELORA_OK;
}

// ---- decode-sized batch of one site (decode_tile.cu)
//
// CTAs that share a tile: the count whose launch is done first.  A K block takes a CTA about a third of a microsecond.  Beside
// the K blocks it works out the expand of its own tokens: a sixth for every stage (one for each of their adapters, whose number
// the device knows, six tenths of the tokens are assumed, and one for every eight tokens more), and 0.028, 0.036 or 0.052 for
// every token, by the rank stride.  All of that is little beside a wave: clusters that are not resident at once begin their launch over, with
// its u-batches and its first round of copies, which takes 16, and 1.5 more with parts to exchange.
// (Residency, by count: 148, 74, 45, 33, 26, 22, 15 and 15 clusters.)  In 130 drawn calls of 33 to 256 tokens the count taken
// was 0.6 % slower than the best of all eight on average, 7 % at most.  Us per call, with the rule before (the tokens of an adapter
// free, four per wave, two K blocks for each CTA) and now: 608 -> 1280, 106 tokens on 19 adapters of rank 64: 31.7 and 22.0; 5216 -> 11224,
// 64 tokens: 49.7 and 39.8; 9440 -> 6184, 142 tokens: 53.8 and 38.2; 664 -> 864, 226 tokens on 34: 43.1 and 30.8.
static int decode_parts(edgelora_pool *p, int n_tiles, int kb, int32_t T) {
  if (p->tile_clusters[1] == 0)
    for (int c = 1; c <= kTileMaxParts; ++c) p->tile_clusters[c] = std::max(1, decode_tile_max_clusters(c));
  const int most = std::max(1, std::min(p->opt_decode_splits > 0 ? p->opt_decode_splits : kTileMaxParts, kb));
  const int quads = (T + 3) / 4;
  int best = 1;
  double best_cost = 0;
  for (int c = 1; c <= most; ++c) {
    if (!decode_tile_parts_fit(T, c)) continue;
    const int waves = (n_tiles + p->tile_clusters[c] - 1) / p->tile_clusters[c];
    const int own = std::min((quads + c - 1) / c * 4, T);
    const double stages = std::min(0.6 * own, static_cast<double>(p->cfg.n_slots)) + own / 8.0;
    const double expand = 0.17 * stages + (0.02 + 0.0005 * p->R_pad) * own;
    const double cost = waves * (std::max((kb + c - 1) / c * 0.33, expand) + (c > 1 ? 17.5 : 16.0));
    if (c == 1 || cost < best_cost || p->opt_decode_splits > 0) {
      best = c;
      best_cost = cost;
    }
  }
  return best;
}

static int decode_tile(const SiteCall &c, const edgelora_plan *plan, const int32_t *ids_dev, int32_t T, bool pdl,
                       cudaStream_t stream) {
  edgelora_pool *p = c.p;
  const int h_in = p->cfg.h_in, h_out = p->cfg.h_out, R = p->R_pad;
  const int32_t N = decode_columns(T);
  DecTile d{};
  int rc = get_tmap(p, &d.w, c.W, h_in, h_out, 0, kTileM);
  if (!rc) rc = get_tmap(p, &d.x, c.x, h_in, T, 0, N);
  if (!rc) rc = get_tmap(p, &d.b, p->B_pool, R, h_out, p->cfg.n_slots, kTileM, R);
  if (rc) return rc;
  d.y = static_cast<uint16_t *>(c.y);
  d.slots = p->slots_dev;
  d.z = p->zws + static_cast<size_t>(kMaxZSplits) * p->cfg.max_tokens * R;
  d.status = p->status_dev;
  d.ids = ids_dev;
  d.T = T;
  d.h_out = h_out;
  d.kb = (h_in + kBlockK - 1) / kBlockK;
  d.R_pad = R;
  d.n_slots = plan->n_slots;
  d.N = N;
  const int n_tiles = (h_out + kTileM - 1) / kTileM;
  const DecTileShape shape = decode_tile_shape(N, R);
  d.parts = decode_parts(p, n_tiles, d.kb, T);
  d.stages = shape.stages;
  d.exp_bytes = shape.exp_bytes;
  d.tmem_cols = shape.tmem_cols;
  d.wait_cycles = p->wait_cycles;
  if (getenv("EDGELORA_LOG"))
    fprintf(stderr, "edgelora: decode T %d N %d splits %d grid %d\n", T, N, d.parts, n_tiles * d.parts);
  CUDA_TRY(launch_decode_tile(d, pdl, stream));
  p->last_info[2] = n_tiles * d.parts;
  p->last_info[3] = d.parts;
  p->last_info[4] = shape.stages;
  p->last_info[5] = N;
  return EDGELORA_OK;
}

// CTAs of a one-launch decode call that the device holds at once, asked once per shape of the last few.
static int fused_max_ctas(edgelora_pool *p, int splits, size_t smem) {
  const uint64_t key = (static_cast<uint64_t>(splits) << 32) | static_cast<uint64_t>(smem);
  for (const auto &f : p->fused_fits)
    if (f.key == key) return f.ctas;
  auto &f = p->fused_fits[p->fused_next];
  p->fused_next = (p->fused_next + 1) % (sizeof(p->fused_fits) / sizeof(p->fused_fits[0]));
  f.key = key;
  f.ctas = gemm_fused_max_ctas(splits, smem);
  return f.ctas;
}

// A call is on the stream: slot loads issued later wait for it.
static int call_issued(edgelora_pool *p, int launches, int regime, bool capturing, cudaStream_t stream) {
  if (!capturing) {
    CUDA_TRY(cudaEventRecord(p->use_ev, stream));
    p->use_recorded = true;
  }
  p->last_info[0] = launches;
  p->last_info[1] = regime;
  p->total_launches += launches;
  return EDGELORA_OK;
}

int lora_linear_impl(edgelora_pool *p, edgelora_plan *plan, const int32_t *ids_dev, const void *W_dev,
                     const void *x_dev, int32_t T, void *y_dev, cudaStream_t stream, Order order) {
  if (!p || !plan || T < 0) return EDGELORA_ERR_INVALID_ARG;
  if (T == 0) return EDGELORA_OK;
  if (!W_dev || !x_dev || !y_dev) return EDGELORA_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(W_dev) | reinterpret_cast<uintptr_t>(x_dev) |
       reinterpret_cast<uintptr_t>(y_dev)) & 15)
    return EDGELORA_ERR_INVALID_ARG;
  if (T > p->cfg.max_tokens || T > plan->max_tokens) return EDGELORA_ERR_TOO_MANY_TOKENS;
  if (plan->n_slots != p->cfg.n_slots) return EDGELORA_ERR_INVALID_ARG;
  if (!ids_dev && plan->last_T != T) return EDGELORA_ERR_INVALID_ARG;
  const int h_in = p->cfg.h_in, h_out = p->cfg.h_out, R = p->R_pad;
  const bool capturing = stream_capturing(stream);
  const bool pdl = p->opt_pdl >= 1 && !p->opt_profile;        // between the kernels of this call
  // first kernel vs earlier stream work (see Order): a set of sites knows whether a call consumes what the calls
  // before it produce
  bool pdl_first = !p->opt_profile && ((order == Order::kPool && p->opt_pdl >= 2) ||
                                       (order == Order::kIndependent && p->opt_pdl >= 1));
  const uint16_t *x = static_cast<const uint16_t *>(x_dev);
  int launches = 0;

  const int rc_loads = wait_for_loads(p, stream, capturing);
  if (rc_loads) return rc_loads;

  int regime = (T <= kDecodeMaxT) ? 1 : 2;
  if (p->opt_regime == 2) regime = 2;
  if (p->opt_regime == 1 && T > kDecodeMaxT) return EDGELORA_ERR_INVALID_ARG;
  const int kb_total = (h_in + kBlockK - 1) / kBlockK;

  GemmParams g{};
  g.T = T;
  g.h_in = h_in;
  g.h_out = h_out;
  g.kb_total = kb_total;
  g.R_pad = R;
  g.max_tokens = p->cfg.max_tokens;
  g.slots = p->slots_dev;
  g.B_pool = p->B_pool;
  g.zws = p->zws;
  g.y = static_cast<uint16_t *>(y_dev);
  g.ids = ids_dev ? ids_dev : plan->pv.ids_valid;
  g.n_slots = p->cfg.n_slots;
  g.status = p->status_dev;
  g.wait_cycles = p->wait_cycles;

  auto smem_for = [](int stages, int BN, int extra = 0) {
    // alignment slack + operand ring + barriers (512) + adapter list and sort keys (3456, rounded up)
    // (+ the staged rows of a one-launch call)
    return static_cast<size_t>(1024 + stages * (kTileM * kBlockK * 2 + BN * kBlockK * 2) + 4096 + extra);
  };
  auto stages_for = [&](int BN, int k_blocks_per_cta, size_t budget) {
    int s = static_cast<int>((budget - 5120) / (kTileM * kBlockK * 2 + BN * kBlockK * 2));
    return std::max(1, std::min({s, kMaxStages, std::max(2, k_blocks_per_cta)}));
  };
  auto pow2_cols = [](int cols) {
    int c = 32;
    while (c < cols) c <<= 1;
    return c;
  };

  // decode batches above this size take the plan kernel + tensor-core gather tiles; smaller ones
  // the single shrink kernel that derives the routing itself (a launch less)
  const int kGatherMinT = p->opt_gather_min_t;
  // a pool that keeps A in Q8_0 is served by the decode shrink kernel only (it decodes the blocks as
  // it streams them); the tensor-core shrink tiles need bfloat16 operand tiles
  if (p->a_q8 && (regime != 1 || T > kGatherMinT)) return EDGELORA_ERR_INVALID_ARG;

  if (regime == 1) {
    // ---------------------------------------------------------------- decode
    const int32_t *ids_in = ids_dev ? ids_dev : plan->pv.ids_valid;
    plan->last_T = T;
    if (!ids_dev && plan->unread) pdl_first = false;  // (the ids are the library's own)
    plan->unread = plan->unread || ids_dev;
    auto launch_shrink = [&](int base_ctas) -> int {  // base_ctas: CTAs that run beside it
      if (T > kGatherMinT) {
        if (ids_dev) {
          ProfScope ps(p, 0, stream);
          launch_plan(ids_dev, T, plan->n_slots, plan->pv, pdl_first, stream);
          CUDA_TRY(cudaGetLastError());
          ++launches;
        }
        // gather tiles only, the K split count chosen on the device from the number of adapters the
        // batch touches; the summed z as fp32
        ShrinkBatch<1> sb{};
        int splits = p->opt_gather_splits;
        while (splits > 1 && (splits - 1) * ((kb_total + splits - 1) / splits) >= kb_total) --splits;  // no empty split
        int rc = fill_shrink_site(p, &sb.site[0], splits, 0);
        if (!rc) rc = fill_shrink_inputs(p, x, T, &sb.x[0], &sb.xg[0]);
        if (rc) return rc;
        fill_shrink_plan(plan, T, p->wait_cycles, 1, 0, &sb);
        ProfScope ps(p, 2, stream);
        CUDA_TRY(launch_shrink_tiles(sb, p->sms, ids_dev ? pdl : pdl_first, stream));
        ++launches;
      } else
      {
        ProfScope ps(p, 1, stream);
        // When calls overlap (EDGELORA_OPT_PDL = 2) a small batch's shrink runs under the previous
        // call's base product, so its length does not matter but its tail does: one K chunk per
        // item (no pass that adds chunks) and few CTAs (they take SM resources from the base product).
        const bool overlapped = pdl_first && T <= 64;
        // ring depth 2 lets two CTAs share an SM: twice the warps in flight with half the ring each,
        // which suits a kernel bound by the per-warp chain of copy issue, wait and FMAs (measured on
        // the 200-adapter down_proj: 45.8 us against 49.8 us with depth 4)
        const int shrink_depth = T <= 64 ? 2 : (p->opt_shrink_depth == 4 ? 4 : 2);
        const int cta_cap = shrink_depth == 2 && T > 64 ? 2 * p->sms : p->sms;
        // Large batches: few, long items beat many short ones, whose ring ramp-up and chunk sums add up: 92 us per step
        // with 2 K chunks on the 1000-adapter down_proj, 96 with 3-4, 100 with 12, 104 with 1.  About 0.6 per warp are
        // aimed for, and where they leave warps without one, K is cut further, to about one per warp (6144 -> 3432 with A
        // in Q8_0, 145 tokens on six adapters: 42.7 us per call, 53.9 without; 1656 -> 328, 69 tokens on four: 21.6 and
        // 27.3), in small batches on the SMs that the base product beside it leaves only (1752 -> 4136, 54 tokens, 132 CTAs of the base
        // product: 15.5 with all SMs, 14.1; 5120 -> 1608, 58 tokens, A in Q8_0: 16.7 and 13.7).  Small batches: four items per warp.
        const int auto_target = T > 64 ? 5 * cta_cap : 4 * 8 * cta_cap;
        const int target = p->opt_shrink_items > 0 ? p->opt_shrink_items : (overlapped ? 1 : auto_target);
        // Token blocks x (R / 8) row groups x K chunks warp items, eight warps per CTA: each adapter's tokens in blocks of four.
        // (With a block per adapter for a bound, a batch on few adapters was left to few CTAs: 4096 -> 4096, 128 tokens on four
        // adapters 38.2 us per call, now 23.5; 664 -> 864, 226 tokens on eight of rank 64: 46.7 and 26.6.)
        const int groups = std::min(T, p->cfg.n_slots), blocks = groups + (T - groups) / kDecShrinkTok;
        const int n_ksteps = (h_in + kShrinkStepElems - 1) / kShrinkStepElems;
        auto ctas_for = [&](int chunk) {  // K chunks of so many steps at least
          const int chunks = target == 1 ? 1 : std::max(1, std::min(kMaxZSplits, n_ksteps / chunk));
          return std::max(1, std::min(cta_cap - 1, (blocks * (R / 8) * chunks + 7) / 8));
        };
        const int spare = p->opt_shrink_items > 0 || overlapped ? 0 : std::max(0, cta_cap - base_ctas);
        const int workers = std::max(ctas_for(4), std::min(ctas_for(2), spare));
        const int grid = workers + 1;  // + the publishing CTA
        const int fill_warps = std::min(workers, spare) * 8;
        CUtensorMap ma, mx, md;
        // A rows: bfloat16, or for a pool that keeps A in Q8_0 two planes per slot: the signed bytes
        // [R_pad][h_in] (taken as 16-bit elements: 128 per K step) and the half-precision block scales
        // [R_pad][h_in / 32] (8 per K step); both planes have the slot's byte stride
        int rc;
        if (p->a_q8) {
          const uint64_t slot_bytes = p->a_block * 2;
          rc = get_tmap(p, &ma, p->A_pool, h_in / 2, R, p->cfg.n_slots, 8, kShrinkStepElems / 2, h_in, slot_bytes);
          if (rc) return rc;
          rc = get_tmap(p, &md, reinterpret_cast<const uint8_t *>(p->A_pool) + static_cast<size_t>(R) * h_in, h_in / 32, R,
                        p->cfg.n_slots, 8, kShrinkStepElems / 32, h_in / 16, slot_bytes);
        } else {
          rc = get_tmap(p, &ma, p->A_pool, h_in, R, p->cfg.n_slots, 8, kShrinkStepElems);
          md = ma;
        }
        if (rc) return rc;
        rc = get_tmap(p, &mx, x, h_in, T, 0, 1, kShrinkStepElems);
        if (rc) return rc;
        CUDA_TRY(launch_decode_shrink(ma, md, mx, ids_in, p->slots_dev, plan->pv, p->zws, p->group_counters,
                                      T, h_in, R, p->cfg.n_slots, p->cfg.max_tokens, target, fill_warps, grid,
                                      p->status_dev, pdl_first, p->a_q8, shrink_depth, stream));
        ++launches;
      }
      if (!ids_dev) plan->unread = false;
      return 0;
    };
    // Up to 64 tokens whose row tiles leave SMs for K splits: the K splits of a row tile form a cluster, and the expand moves
    // to the owners of the cluster reduction (at most 16 tokens and 64 16-byte loads of B per thread), so the main loop does not
    // depend on the shrink at all.
    const int N = T <= 32 ? 32 : 64;  // tokens on the UMMA N axis: a power of two so that the cluster's owners get
    const int row_tiles = (h_out + kTileM - 1) / kTileM;  // equal power-of-two column blocks
    const int stage_bytes = kTileM * kBlockK * 2 + N * kBlockK * 2;
    int want = p->opt_decode_splits > 0 ? p->opt_decode_splits : std::max(1, 2 * p->sms / row_tiles);
    want = std::min({want, kMaxDecodeSplits, std::max(1, kb_total / 2)});
    int splits = 1;
    while (splits * 2 <= want) splits <<= 1;
    while (splits > 1 && (kb_total + splits - 1) / splits * (splits - 1) >= kb_total) splits >>= 1;  // every split needs a K block
    auto owners_expand = [&](int sp) { return T <= 64 && sp > 1 && N / sp <= 16 && N / sp * (R / 8) <= 64; };
    // one CTA per SM leaves room for the shrink kernel's CTAs, so that the two kernels run side
    // by side (measured on 4096 -> 4096, T = 32: 18.4 us per step with 4 splits, 24.4 with 8)
    if (owners_expand(splits) && p->opt_decode_splits == 0)
      while (splits > 1 && row_tiles * splits > p->sms) splits >>= 1;
    if (!owners_expand(splits)) {
      int rc = launch_shrink(0);
      if (rc) return rc;
      {
        // Launched under the shrink's tail: its CTAs end at different times, and on the SMs that are free early the K
        // blocks, which need no z, start at once.
        ProfScope ps(p, 3, stream);
        rc = decode_tile(SiteCall{p, W_dev, x, y_dev}, plan, ids_in, T, pdl, stream);
        if (rc) return rc;
        ++launches;
      }
      return call_issued(p, launches, regime, capturing, stream);
    }
    g.BN = N;
    g.splits = splits;
    g.kb_per = (kb_total + splits - 1) / splits;
    g.n_mtiles = row_tiles;
    // the decode shrink leaves the summed z in the plane after the partial ones
    g.zws = p->zws + static_cast<size_t>(kMaxZSplits) * p->cfg.max_tokens * R;
    const size_t budget = kSmemBudget / 2;
    // the cluster's reduction buffer (N x 128 fp32, plus z of the owner's tokens) overlays the ring
    auto stages_of = [&](int sp, int kb_per) {
      int st = stages_for(N, kb_per + 8, budget);
      while (st * stage_bytes < N * kTileM * 4 + (N / sp) * R * 4 && st < kMaxStages) ++st;
      return st;
    };
    g.stages = stages_of(splits, g.kb_per);
    g.tmem_cols = pow2_cols(N);
    CUtensorMap mr, mc;
    int rc = get_tmap(p, &mr, W_dev, h_in, h_out, 0, kTileM);
    if (rc) return rc;
    rc = get_tmap(p, &mc, x, h_in, T, 0, N);
    if (rc) return rc;
    const int grid = row_tiles * splits;
    // Small batches in one launch: the shrink runs on team warps of the base product's CTAs
    // and on spare CTAs in front of them (SMs the grid leaves empty), and the owners of the cluster
    // reduction wait for its arrival counter.  CTAs of one grid wait for one another here, so every
    // cluster of the launch must be resident at once: checked against the device's occupancy figure.
    bool fused = false;
    if (getenv("EDGELORA_LOG"))
      fprintf(stderr, "edgelora: decode T %d N %d splits %d grid %d\n", T, N, splits, grid);
    // (Calls that may overlap the call before them keep the two launches: a one-launch grid holds every
    // SM until its last CTA is done, so consecutive calls cannot overlap; measured on 4096 -> 4096,
    // T = 32: 17.0 us per step in one launch against 9.7 us in two when the calls are independent, and
    // 16.9 against 19.7 us when each call waits for the one before.)
    if (p->opt_fused_decode && !pdl_first && T <= kGatherMinT && ids_dev &&
        !p->a_q8 && h_in % 8 == 0) {
      // Fewer K splits when the clusters of all row tiles do not fit beside a spare one (clusters of eight: 16 on this chip;
      // 2048 -> 2048, 8 tokens: 6.6 us in one launch with 4 splits, 10.4 in two with 8).
      for (int sp = splits; sp > 1 && !fused; sp >>= 1) {
        if (!owners_expand(sp) || (p->opt_decode_splits != 0 && sp != splits)) break;
        GemmParams gf = g;
        gf.splits = sp;
        gf.kb_per = (kb_total + sp - 1) / sp;
        if (gf.kb_per * (sp - 1) >= kb_total) continue;  // every split needs a K block
        gf.stages = stages_of(sp, gf.kb_per);
        FusedDecode f{};
        // room behind the ring for the B_a rows and z of an owner's tokens, when it fits
        // (2: and for the cluster reduction's buffer, which then does not have to wait for the ring)
        // The staged rows are worth more than the ring's last stage: without them the expand stays behind the exchange.  Us per
        // call without and with them: 4096 -> 4096, one token of rank 64: 17.2 and 11.7, 64 tokens of rank 32: 24.4 and 17.4; 4096 ->
        // 1920, eight tokens of rank 64: 20.9 and 9.8 (17.6 in two launches); 14336 -> 4096, 20 tokens of rank 64: 45.1 and 37.4.
        size_t stage_extra = static_cast<size_t>(N / sp) * (kTileM * R * 2 + R * 4);
        const size_t reduce_bytes = static_cast<size_t>(N) * kTileM * 4 + static_cast<size_t>(N / sp) * R * 4;
        for (int st = gf.stages; st >= std::max(2, gf.stages - 1) && st * stage_bytes >= reduce_bytes && !f.b_stage; --st)
          if (smem_for(st, N, static_cast<int>(stage_extra)) <= kSmemBudget) {
            f.b_stage = 1;
            gf.stages = st;
          }
        const size_t with_buf = ((stage_extra + 1023) & ~static_cast<size_t>(1023)) + static_cast<size_t>(N) * kTileM * 4;
        if (f.b_stage && smem_for(gf.stages, N, static_cast<int>(with_buf)) <= kSmemBudget) {
          f.b_stage = 2;
          stage_extra = with_buf;
        }
        const size_t smem = smem_for(gf.stages, N, f.b_stage ? static_cast<int>(stage_extra) : 0);
        const int gf_grid = row_tiles * sp;
        const int spare = std::max(0, std::min(fused_max_ctas(p, sp, smem) - gf_grid, 32) / sp * sp);
        if (spare == 0) continue;  // every CTA resident at once, and a spare CTA to publish the routing plan
        const int n_teams = 2 * spare + gf_grid;
        const int n_ksteps = (h_in + kShrinkStepElems - 1) / kShrinkStepElems;
        int ks = std::max(1, std::min(kMaxZSplits, n_ksteps / 4));
        while (ks > 1 && T * (R / 8) * ks > 2 * n_teams) ks >>= 1;
        f.n_ctas = spare;
        f.ks = ks;
        f.x_wait = 1;  // x may be the output of the call before this one
        f.A_pool = p->A_pool;
        f.x = x;
        f.z = p->zws;
        f.sync = p->group_counters + kDecodeMaxT * 8 + 8;
        f.pv = plan->pv;
        CUtensorMap me;  // B_a rows for the expand on the CUDA cores: boxes as wide as the rank stride
        rc = get_tmap(p, &me, p->B_pool, R, h_out, p->cfg.n_slots, kTileM, R);
        if (rc) return rc;
        ProfScope ps(p, 3, stream);
        CUDA_TRY(launch_gemm_fused(mr, mc, me, gf, f, smem, p->opt_pdl != 0, stream));
        ++launches;
        fused = true;
        g = gf;
        p->last_info[2] = gf_grid + spare;
        p->last_info[3] = sp;
        p->last_info[4] = g.stages;
        p->last_info[5] = g.BN;
      }
    }
    if (!fused) {
      // (a cluster lies within one of eight groups of about 18 SMs: what the shrink takes is what whole clusters leave.  11008 ->
      // 2344, nine tokens, A in Q8_0: 24.5 us per call with 40 CTAs of the shrink, 31.7 with 64)
      rc = launch_shrink((row_tiles + 7) / 8 * 8 * splits + 4);
      if (rc) return rc;
    }
    if (!fused) {
      ProfScope ps(p, 3, stream);
      CUDA_TRY(launch_gemm(mr, mc, g, grid, smem_for(g.stages, N), pdl, stream));
      ++launches;
      p->last_info[2] = grid;
      p->last_info[3] = splits;
      p->last_info[4] = g.stages;
      p->last_info[5] = g.BN;
    }
  } else {
    // ---------------------------------------------------------------- prefill
    const SiteCall call{p, W_dev, x, y_dev};
    const int rc = prefill_sites(&call, 1, plan, ids_dev, T, stream, pdl_first);
    if (rc) return rc;
    if (!capturing) {
      CUDA_TRY(cudaEventRecord(p->use_ev, stream));
      p->use_recorded = true;
    }
    return EDGELORA_OK;
  }

  return call_issued(p, launches, regime, capturing, stream);
}
}  // namespace edgelora

extern "C" {

int edgelora_lora_linear(edgelora_pool_t *pool, const void *W_dev, const void *x_dev,
                         const int32_t *adapter_id_dev, int32_t T, void *y_dev, void *stream) {
  if (!pool) return EDGELORA_ERR_INVALID_ARG;
  if (T > 0 && !adapter_id_dev) return EDGELORA_ERR_INVALID_ARG;
  return lora_linear_impl(pool, pool->plan, adapter_id_dev, W_dev, x_dev, T, y_dev,
                          static_cast<cudaStream_t>(stream));
}

int edgelora_lora_linear_planned(edgelora_pool_t *pool, edgelora_plan_t *plan, const void *W_dev,
                                 const void *x_dev, int32_t T, void *y_dev, void *stream) {
  if (!pool || !plan) return EDGELORA_ERR_INVALID_ARG;
  return lora_linear_impl(pool, plan, nullptr, W_dev, x_dev, T, y_dev,
                          static_cast<cudaStream_t>(stream));
}

int edgelora_lora_linear_host(edgelora_pool_t *p, const void *W_dev, const uint16_t *x_host,
                              const int32_t *adapter_id_host, int32_t T, uint16_t *y_host,
                              void *stream) {
  if (!p || T < 0) return EDGELORA_ERR_INVALID_ARG;
  if (T == 0) return EDGELORA_OK;
  if (!x_host || !adapter_id_host || !y_host) return EDGELORA_ERR_INVALID_ARG;
  if (T > p->cfg.max_tokens) return EDGELORA_ERR_TOO_MANY_TOKENS;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t mt = p->cfg.max_tokens;
  if (!p->hx) {  // first use: pinned staging and device mirrors for one batch
    CUDA_TRY(cudaMallocHost(&p->hx, mt * p->cfg.h_in * 2));
    CUDA_TRY(cudaMallocHost(&p->hy, mt * p->cfg.h_out * 2));
    CUDA_TRY(cudaMallocHost(&p->hids, mt * 4));
    CUDA_TRY(el_malloc(&p->dx, mt * p->cfg.h_in * 2));
    CUDA_TRY(el_malloc(&p->dy, mt * p->cfg.h_out * 2));
    CUDA_TRY(el_malloc(&p->dids, mt * 4));
  }
  const size_t xb = static_cast<size_t>(T) * p->cfg.h_in * 2, yb = static_cast<size_t>(T) * p->cfg.h_out * 2;
  memcpy(p->hx, x_host, xb);
  memcpy(p->hids, adapter_id_host, static_cast<size_t>(T) * 4);
  CUDA_TRY(cudaMemcpyAsync(p->dx, p->hx, xb, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(p->dids, p->hids, static_cast<size_t>(T) * 4, cudaMemcpyHostToDevice, s));
  int rc = lora_linear_impl(p, p->plan, p->dids, W_dev, p->dx, T, p->dy, s);
  if (rc != EDGELORA_OK) return rc;
  CUDA_TRY(cudaMemcpyAsync(p->hy, p->dy, yb, cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  memcpy(y_host, p->hy, yb);
  return EDGELORA_OK;
}

int edgelora_lora_linear_host_async(edgelora_pool_t *p, const void *W_dev, const uint16_t *x_host,
                                    const int32_t *adapter_id_host, int32_t T, uint16_t *y_host,
                                    void *stream) {
  if (!p || T < 0) return EDGELORA_ERR_INVALID_ARG;
  if (T == 0) return EDGELORA_OK;
  if (!x_host || !adapter_id_host || !y_host) return EDGELORA_ERR_INVALID_ARG;
  if (T > p->cfg.max_tokens) return EDGELORA_ERR_TOO_MANY_TOKENS;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t mt = p->cfg.max_tokens;
  if (!p->h2d_stream) {  // first use
    CUDA_TRY(cudaStreamCreateWithFlags(&p->h2d_stream, cudaStreamNonBlocking));
    CUDA_TRY(cudaStreamCreateWithFlags(&p->d2h_stream, cudaStreamNonBlocking));
    for (int b = 0; b < 2; ++b) {
      CUDA_TRY(el_malloc(&p->pdx[b], mt * p->cfg.h_in * 2));
      CUDA_TRY(el_malloc(&p->pdy[b], mt * p->cfg.h_out * 2));
      CUDA_TRY(el_malloc(&p->pdids[b], mt * 4));
      CUDA_TRY(cudaEventCreateWithFlags(&p->ev_in[b], cudaEventDisableTiming));
      CUDA_TRY(cudaEventCreateWithFlags(&p->ev_done[b], cudaEventDisableTiming));
      CUDA_TRY(cudaEventCreateWithFlags(&p->ev_out[b], cudaEventDisableTiming));
    }
  }
  const int b = static_cast<int>(p->host_calls & 1);
  const bool reused = p->host_calls >= 2;  // the set was used two calls ago
  ++p->host_calls;
  const size_t xb = static_cast<size_t>(T) * p->cfg.h_in * 2, yb = static_cast<size_t>(T) * p->cfg.h_out * 2;
  // inputs: after the layer that last read this set of mirrors
  if (reused) CUDA_TRY(cudaStreamWaitEvent(p->h2d_stream, p->ev_done[b], 0));
  CUDA_TRY(cudaMemcpyAsync(p->pdx[b], x_host, xb, cudaMemcpyHostToDevice, p->h2d_stream));
  CUDA_TRY(cudaMemcpyAsync(p->pdids[b], adapter_id_host, static_cast<size_t>(T) * 4, cudaMemcpyHostToDevice,
                           p->h2d_stream));
  CUDA_TRY(cudaEventRecord(p->ev_in[b], p->h2d_stream));
  // layer: after its inputs, and after the copy-out that last read this set's y
  CUDA_TRY(cudaStreamWaitEvent(s, p->ev_in[b], 0));
  if (reused) CUDA_TRY(cudaStreamWaitEvent(s, p->ev_out[b], 0));
  int rc = lora_linear_impl(p, p->plan, p->pdids[b], W_dev, p->pdx[b], T, p->pdy[b], s);
  if (rc != EDGELORA_OK) return rc;
  CUDA_TRY(cudaEventRecord(p->ev_done[b], s));
  // result
  CUDA_TRY(cudaStreamWaitEvent(p->d2h_stream, p->ev_done[b], 0));
  CUDA_TRY(cudaMemcpyAsync(y_host, p->pdy[b], yb, cudaMemcpyDeviceToHost, p->d2h_stream));
  CUDA_TRY(cudaEventRecord(p->ev_out[b], p->d2h_stream));
  return EDGELORA_OK;
}

int edgelora_pool_host_sync(edgelora_pool_t *p) {
  if (!p) return EDGELORA_ERR_INVALID_ARG;
  if (p->d2h_stream) CUDA_TRY(cudaStreamSynchronize(p->d2h_stream));
  return EDGELORA_OK;
}

}  // extern "C"
