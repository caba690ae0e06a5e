// Private to the library: the pool and plan objects behind the opaque handles of the C ABI, shared
// by the files that implement the host side (pool.cu, siteset.cu).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <utility>
#include <vector>

#include "internal.cuh"
#include "ptx.cuh"

namespace edgelora {

constexpr int kStagingBuffers = 4;

// text behind EDGELORA_ERR_CUDA for edgelora_strerror (per thread)
extern thread_local char g_last_error[256];
void set_last_cuda_error(cudaError_t e, const char *what);

struct TmapKey {
  const void *base;
  uint64_t d0, d1, d2;
  uint32_t b1, b0;  // box rows, box columns (which also say the swizzle)
  uint64_t s1, s2;  // byte strides of dimensions 1 and 2 (0 = dense)
  bool operator==(const TmapKey &o) const {
    return base == o.base && d0 == o.d0 && d1 == o.d1 && d2 == o.d2 && b1 == o.b1 && b0 == o.b0 && s1 == o.s1 &&
           s2 == o.s2;
  }
};
struct TmapEntry {
  TmapKey key;
  CUtensorMap map;
};

struct StagingBuf {
  uint8_t *host = nullptr;  // pinned: [A padded][B padded][SlotRow]
  cudaEvent_t done = nullptr;
  bool in_flight = false;
};

struct ProfRec {
  int kernel;
  cudaEvent_t start, stop;
};

}  // namespace edgelora

struct edgelora_plan {
  using PlanView = edgelora::PlanView;
  int32_t max_tokens = 0, n_slots = 0, last_T = 0;
  // The kernel that writes the plan lets its dependents start at once, and the decode kernels of a planned call read the
  // plan's ids before their dependency wait.  True until a planned decode call started behind that kernel: the first one
  // does, whatever overlap the pool allows, and those after it are behind it too.
  bool unread = false;
  void *block = nullptr;
  PlanView pv{};
};

struct edgelora_pool {
  using SlotRow = edgelora::SlotRow;
  using StagingBuf = edgelora::StagingBuf;
  using TmapEntry = edgelora::TmapEntry;
  using ProfRec = edgelora::ProfRec;
  edgelora_pool_config cfg{};
  int R_pad = 0, device = 0, sms = 0;
  bool owns_arena = false, a_q8 = false;  // a_q8: the A blocks are kept in Q8_0 (EDGELORA_FLAG_A_Q8)
  uint8_t *arena = nullptr;
  uint16_t *A_pool = nullptr, *B_pool = nullptr;
  size_t a_block = 0, b_block = 0;  // elements per slot
  SlotRow *slots_dev = nullptr;
  std::vector<SlotRow> slots_host;
  StagingBuf staging[edgelora::kStagingBuffers];
  int next_staging = 0;
  cudaStream_t side = nullptr;
  cudaEvent_t use_ev = nullptr;
  cudaEvent_t last_load = nullptr;  // the event of the staging buffer that the last load went through
  uint64_t load_seq = 0;
  std::vector<std::pair<cudaStream_t, uint64_t>> load_waited;  // per stream: last load it waited for
  bool use_recorded = false;
  edgelora_plan *plan = nullptr;
  float *zws = nullptr;
  int32_t *group_counters = nullptr;
  int32_t *tile_counters = nullptr, n_tile_counters = 0;  // arrivals per tile of the tensor-core shrink
  int opt_decode_splits = 0, opt_shrink_items = 0, opt_gather_splits = 0, opt_gather_min_t = 256, opt_shrink_depth = 0;
  uint32_t *status_dev = nullptr;
  std::vector<TmapEntry> tmaps;
  size_t tmap_next = 0;
  int opt_regime = 0, opt_profile = 0, opt_pdl = 1, opt_fused_decode = 1;
  struct {
    uint64_t key = 0;  // launch shape: K splits and shared memory
    int ctas = 0;      // the occupancy answer for it
  } fused_fits[8];
  int fused_next = 0;
  int tile_clusters[9] = {0};  // clusters of each size of the tile launch that the device holds at once; 0: not asked yet
  long long wait_cycles = edgelora::ptx::kWaitLimitCycles;
  int64_t last_info[8] = {0};
  int64_t total_launches = 0;
  // profiling
  std::vector<ProfRec> prof;
  size_t prof_used = 0;
  double prof_ms[5] = {0};
  int64_t prof_n[5] = {0};
  // host-buffer entry point
  uint16_t *hx = nullptr, *hy = nullptr, *dx = nullptr, *dy = nullptr;
  int32_t *hids = nullptr, *dids = nullptr;
  // pipelined host-buffer path: two sets of device mirrors, two copy streams, events per set
  uint16_t *pdx[2] = {nullptr, nullptr}, *pdy[2] = {nullptr, nullptr};
  int32_t *pdids[2] = {nullptr, nullptr};
  cudaStream_t h2d_stream = nullptr, d2h_stream = nullptr;
  cudaEvent_t ev_in[2] = {nullptr, nullptr}, ev_done[2] = {nullptr, nullptr}, ev_out[2] = {nullptr, nullptr};
  uint64_t host_calls = 0;
};


namespace edgelora {

// One linear site of a call: y = W x + s_a B_a A_a x over the batch of the call's plan.
struct SiteCall {
  edgelora_pool *p;
  const void *W;
  const uint16_t *x;
  void *y;
  // Two inputs of a set may lie at one address and still be read in rows of different widths.
  bool same_input(const SiteCall &o) const { return x == o.x && p->cfg.h_in == o.p->cfg.h_in; }
};

// How a call's first kernel stands to the work in front of it on the stream: as the pool's EDGELORA_OPT_PDL says;
// under that work's tail (the call reads nothing the call before it writes); or behind it, whatever the option says.
enum class Order { kPool, kIndependent, kAfter };

// The layer (see pool.cu).
int lora_linear_impl(edgelora_pool *p, edgelora_plan *plan, const int32_t *ids_dev, const void *W_dev,
                     const void *x_dev, int32_t T, void *y_dev, cudaStream_t stream, Order order = Order::kPool);
int prefill_sites(const SiteCall *sites, int n, edgelora_plan *plan, const int32_t *ids_dev, int32_t T,
                  cudaStream_t stream, bool pdl_first);
// Decode-sized batches: shrink and base product of a run of sites (at most kDecSites on at most kDecInputs inputs, no
// pool twice) in one launch each.  ids_dev: the caller's ids; the plan is published.  ws: see DecodeWorkspace.
struct DecodeWorkspace {
  float *partial = nullptr;      // two planes [N][128] per CTA
  int32_t *arrivals = nullptr;   // [CTAs][4]
  int32_t ctas = 0;              // one per SM, or as many as the set's sites have work for
};
// The CTAs of a set of these pools, and the fp32 values of their planes.
int32_t decode_workspace_ctas(edgelora_pool *const *pools, int32_t n, int32_t max_tokens);
size_t decode_workspace_planes(int32_t ctas, int32_t max_tokens);
int decode_sites(const SiteCall *sites, int n, edgelora_plan *plan, const int32_t *ids_dev, int32_t T,
                 const DecodeWorkspace &ws, cudaStream_t stream, bool pdl_first);
int wait_for_loads(edgelora_pool *p, cudaStream_t stream, bool capturing);

}  // namespace edgelora
