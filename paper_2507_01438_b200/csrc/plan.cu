// Routing plan (paper Section 3.4: requests needing the same adapter form a u-batch; Section 4.3:
// adapter ids are mapped to sample indices, results return to their original positions).
//
// One CTA turns adapter_id[T] into
//   ids_valid   the ids with out-of-range values replaced by -1 (status bit raised),
//   segments    maximal runs of equal id in token order,
//   groups      tokens ordered by (id, token): ids ascending with -1 first, token order kept,
//   short lists the groups restricted to tokens the gather-by-token shrink handles,
//   sgmv tiles  in batches above kDecodeMaxT tokens, for runs of >= kSegMin tokens on a real
//               adapter: 128-token tiles of the run (work list of the segment shrink),
//   tile lists  the distinct ids >= 0 inside every 256-token tile (the LoRA K blocks of that tile).
// Tokens of one run stay together in the group order, so the runs are sorted, not the tokens, by the
// unique keys ((id + 1) << 16 | run index) in shared memory: exact and the same on every launch.
// Batches up to 4096 tokens keep everything but the outputs in shared memory (plan_small).
#include "internal.cuh"
#include "launch.cuh"
#include "ptx.cuh"

namespace edgelora {

constexpr int kPlanThreads = 1024;

// Exclusive prefix sum over i in [0, n) of value(i), one element per thread per round;
// consume(i, prefix) is called for every i.  Returns the total.  `wt` is shared memory [34].
template <typename Value, typename Consume>
__device__ __forceinline__ int scan_rounds(int n, int *wt, Value value, Consume consume) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int base = 0;
  for (int i0 = 0; i0 < n; i0 += kPlanThreads) {
    const int i = i0 + tid;
    const int v = i < n ? value(i) : 0;
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += o;
    }
    if (lane == 31) wt[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      const int w = wt[lane];
      int wi = w;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, wi, d);
        if (lane >= d) wi += o;
      }
      wt[lane] = wi - w;
      if (lane == 31) wt[32] = wi;
    }
    __syncthreads();
    if (i < n) consume(i, base + wt[warp] + incl - v);
    base += wt[32];
    __syncthreads();
  }
  return base;
}

// The distinct ids >= 0 inside every 256-token tile, in order of first appearance (the LoRA K blocks of that tile
// in the base-product kernel).  One warp per tile; `first` has a bit per token, set for the heads of runs whose id does
// not occur earlier in their tile.  A tile's first token is a first appearance in any case.
__device__ __forceinline__ void list_tiles(const int32_t *valid, int32_t T, const PlanView &pv, const uint32_t *first) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n_mt = (T + kListTile - 1) / kListTile;
  for (int m = warp; m < n_mt; m += kPlanThreads / 32) {
    int32_t id[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int t = m * kListTile + q * 32 + lane;
      id[q] = t < T ? valid[t] : -1;
    }
    int base = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      uint32_t bits = m * kListTile + q * 32 < T ? first[m * 8 + q] : 0u;
      if (q == 0) bits |= __shfl_sync(0xffffffffu, id[0], 0) >= 0 ? 1u : 0u;
      if ((bits >> lane) & 1u) pv.mt_list[m * kListTile + base + __popc(bits & ((1u << lane) - 1u))] = id[q];
      base += __popc(bits);
    }
    if (lane == 0) pv.mt_count[m] = base;
  }
}
// Marks the head of a run (first token t0, id >= 0) for list_tiles.  prev_end: where the run in front of it with the same
// id ends (0: there is none); in the order of the runs by (id, run index) that is the neighbour.
__device__ __forceinline__ void mark_first(uint32_t *first, int t0, int prev_end) {
  if (prev_end <= (t0 & ~(kListTile - 1))) atomicOr(&first[t0 >> 5], 1u << (t0 & 31));
}

// Batches up to kPlanSmallT tokens: the plan is worked out in shared memory.  The general form below keeps its
// intermediate arrays in global memory and goes through them in about thirty barrier-separated passes, each a round trip
// to L2; here each thread looks after T / 1024 consecutive tokens and n_segs / 1024 consecutive places of the order of
// the runs, and the four prefix sums over the runs are one scan of four packed 16-bit fields.  Per build, back to back:
// 8 runs in 512 tokens 4.4 us (general form 11), 66 runs in 2112 tokens 5.6 (21), 2048 runs in 2048 tokens 17 (39), 4096 in
// 4096 34 (76).  Up to kCountRuns runs are ordered by counting smaller keys, more of them by a sorting network: 512 runs
// in 1024 tokens 9.4 us counted, 10.7 sorted; 1024 runs 11.8 sorted, 20 and more counted.
constexpr int kPlanSmallT = 4096;
constexpr int kPlanTok = kPlanSmallT / kPlanThreads;  // tokens per thread, consecutive
constexpr int kCountRuns = 512;
struct PlanSmall {
  int32_t *ids, *seg_start, *seg_id;
  uint32_t *key;             // (id + 1) << 16 | run: of every run, then in order
  int32_t *out, *out_short;  // by run: where it begins in perm and perm_short (-1: nowhere)
  static __host__ __device__ int32_t stride(int32_t T) { return (T + 4) & ~3; }  // T + 1 entries each
  static __host__ __device__ size_t bytes(int32_t T) { return 6 * sizeof(int32_t) * stride(T); }
  __device__ PlanSmall(uint32_t *mem, int32_t T) {
    const int32_t n = stride(T);
    ids = reinterpret_cast<int32_t *>(mem);
    seg_start = ids + n;
    seg_id = seg_start + n;
    key = reinterpret_cast<uint32_t *>(seg_id + n);
    out = seg_id + 2 * n;
    out_short = out + n;
  }
};

// Exclusive prefix sum over the block (one synchronisation; wt must not be in use by an earlier scan).
__device__ __forceinline__ unsigned long long scan_block(unsigned long long v, unsigned long long *wt,
                                                         unsigned long long &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned long long o = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) wt[warp] = incl;
  __syncthreads();
  unsigned long long w = wt[lane];  // every warp adds up the 32 warps' sums for itself
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned long long o = __shfl_up_sync(0xffffffffu, w, d);
    if (lane >= d) w += o;
  }
  total = __shfl_sync(0xffffffffu, w, 31);
  const unsigned long long before = __shfl_sync(0xffffffffu, w, max(warp - 1, 0));
  return (warp > 0 ? before : 0ull) + incl - v;
}

// Sorts n keys (a power of two, at least 32) in shared memory, ascending; the caller synchronises before and after.
// A warp's pairs of a step with j <= 32 lie in blocks of 64 keys that no other warp touches in such a step.
__device__ __forceinline__ void sort_keys(uint32_t *key, int n) {
  for (int k = 2; k <= n; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < (n >> 1); i += kPlanThreads) {
        const int lo = 2 * i - (i & (j - 1)), hi = lo + j;
        const uint32_t a = key[lo], b = key[hi];
        if ((a > b) == ((lo & k) == 0)) {
          key[lo] = b;
          key[hi] = a;
        }
      }
      if (j > 32 || (j == 1 && k >= 64)) __syncthreads();  // (j == 1: the next step is 2 k / 2 = k apart)
      else __syncwarp();
    }
  }
}

__device__ __forceinline__ void plan_small(const int32_t *__restrict__ ids, int32_t T, int32_t n_slots,
                                           const PlanView &pv, const PlanSmall &sh, uint32_t *first,
                                           unsigned long long (&wt)[2][kPlanThreads / 32]) {
  const int tid = threadIdx.x;
  // validate; segments = maximal runs of equal id in token order
  bool bad = false;
  int32_t id[kPlanTok];
#pragma unroll
  for (int q = 0; q < kPlanTok; ++q) {
    const int t = q * kPlanThreads + tid;
    if (t < T) {
      int32_t a = ids[t];
      if (a < -1 || a >= n_slots) {
        a = -1;
        bad = true;
      }
      sh.ids[t] = a;
      pv.ids_valid[t] = a;
    }
  }
  for (int i = tid; i < kPlanSmallT / 32; i += kPlanThreads) first[i] = 0;
  if (__syncthreads_or(bad ? 1 : 0) && tid == 0) atomicOr(pv.status, EDGELORA_STATUS_BAD_ADAPTER_ID);
  const int per = (T + kPlanThreads - 1) / kPlanThreads;  // tokens of this thread: [tid per, tid per + per)
  int heads = 0;
  uint32_t is_head = 0;
#pragma unroll
  for (int q = 0; q < kPlanTok; ++q) {
    const int t = tid * per + q;
    if (q < per && t < T) {
      id[q] = sh.ids[t];
      if (t == 0 || sh.ids[t - 1] != id[q]) {
        is_head |= 1u << q;
        ++heads;
      }
    }
  }
  unsigned long long total;
  int s = static_cast<int>(scan_block(heads, wt[0], total)) - 1;
  const int n_segs = static_cast<int>(total);
  const bool counted = n_segs <= kCountRuns;
  int npow2 = 32;
  while (!counted && npow2 < n_segs) npow2 <<= 1;
#pragma unroll
  for (int q = 0; q < kPlanTok; ++q) {
    const int t = tid * per + q;
    if (q < per && t < T) {
      if ((is_head >> q) & 1u) {
        ++s;
        sh.seg_start[s] = t;
        sh.seg_id[s] = id[q];
        sh.key[s] = (static_cast<uint32_t>(id[q] + 1) << 16) | static_cast<uint32_t>(s);
        pv.seg_start[s] = t;
        pv.seg_adapter[s] = id[q];
      }
      pv.tok_seg[t] = s;
    }
  }
  // (n_segs <= T and the network's next power of two may lie past the key array: out and out_short follow it, unused yet)
  for (int i = n_segs + tid; i < (counted ? (n_segs + 3) & ~3 : npow2); i += kPlanThreads) sh.key[i] = 0xFFFFFFFFu;
  if (tid == 0) {
    sh.seg_start[n_segs] = T;
    pv.seg_start[n_segs] = T;
    pv.counts[1] = n_segs;
  }
  __syncthreads();

  // the runs ordered by (id, run index): -1 first, token order kept.  Keys are unique.
  if (counted) {
    const uint32_t key = tid < n_segs ? sh.key[tid] : 0u;
    int place = 0;
    if (tid < n_segs)
      for (int i = 0; i < n_segs; i += 4) {
        const uint4 k = *reinterpret_cast<const uint4 *>(&sh.key[i]);
        place += (k.x < key) + (k.y < key) + (k.z < key) + (k.w < key);
      }
    __syncthreads();
    if (tid < n_segs) sh.key[place] = key;
  } else {
    sort_keys(sh.key, npow2);
  }
  __syncthreads();

  // one scan: tokens and short tokens (runs the gather-by-token shrink handles: every run of a small batch,
  // otherwise those below kSegMin) and group heads in the order of the runs, segment tiles in token order
  const bool all_short = T <= kDecodeMaxT;
  const int rper = (n_segs + kPlanThreads - 1) / kPlanThreads;  // places, and runs, of this thread: [tid rper, ...)
  auto len_of = [&](int r) { return sh.seg_start[r + 1] - sh.seg_start[r]; };
  auto short_of = [&](int len) { return (all_short || len < kSegMin) ? len : 0; };
  auto id_at = [&](int i) { return static_cast<int32_t>(sh.key[i] >> 16) - 1; };
  auto head_at = [&](int i) { return (i == 0 || (sh.key[i - 1] >> 16) != (sh.key[i] >> 16)) ? 1 : 0; };
  auto tiles_of = [&](int r) {
    const int len = len_of(r);
    return (!all_short && sh.seg_id[r] >= 0 && len >= kSegMin) ? (len + kTileM - 1) / kTileM : 0;
  };
  auto pack = [](int len, int sh_len, int head, int tiles) {
    return static_cast<unsigned long long>(len) | (static_cast<unsigned long long>(sh_len) << 16) |
           (static_cast<unsigned long long>(head) << 32) | (static_cast<unsigned long long>(tiles) << 48);
  };
  unsigned long long mine = 0;
  for (int q = 0; q < rper; ++q) {
    const int i = tid * rper + q;
    if (i < n_segs) {
      const int len = len_of(static_cast<int>(sh.key[i] & 0xFFFFu));
      mine += pack(len, short_of(len), head_at(i), tiles_of(i));
    }
  }
  unsigned long long pre = scan_block(mine, wt[1], total);
  const int n_groups = static_cast<int>((total >> 32) & 0xFFFF), n_short = static_cast<int>((total >> 16) & 0xFFFF);
  const int has_base = id_at(0) < 0 ? 1 : 0;  // the group of id -1 comes first
  for (int q = 0; q < rper; ++q) {
    const int i = tid * rper + q;
    if (i >= n_segs) break;
    const int r = static_cast<int>(sh.key[i] & 0xFFFFu), len = len_of(r), my_short = short_of(len), my_id = id_at(i);
    const int head = head_at(i), n_tiles = tiles_of(i);
    const int p_len = static_cast<int>(pre & 0xFFFF), p_short = static_cast<int>((pre >> 16) & 0xFFFF);
    const int g = static_cast<int>((pre >> 32) & 0xFFFF) + head - 1, p_tiles = static_cast<int>(pre >> 48);
    pre += pack(len, my_short, head, n_tiles);
    sh.out[r] = p_len;
    sh.out_short[r] = my_short > 0 ? p_short : -1;
    if (my_id >= 0) mark_first(first, sh.seg_start[r], head ? 0 : sh.seg_start[(sh.key[i - 1] & 0xFFFFu) + 1]);
    if (head) {
      pv.group_start[g] = p_len;
      pv.gs_short[g] = p_short;
      pv.group_adapter[g] = my_id;
      if (my_id >= 0) pv.lg_adapter[g - has_base] = my_id;
      if (g == has_base) pv.counts[6] = n_short - p_short;
    }
    for (int k = 0; k < n_tiles; ++k) {  // 128-token tiles of the (long) run i
      const int tile = p_tiles + k;
      if (tile < pv.max_sgmv_tiles) {
        pv.sgmv_tiles[4 * tile + 0] = sh.seg_start[i] + k * kTileM;
        pv.sgmv_tiles[4 * tile + 1] = min(kTileM, len_of(i) - k * kTileM);
        pv.sgmv_tiles[4 * tile + 2] = sh.seg_id[i];
        pv.sgmv_tiles[4 * tile + 3] = 0;
      }
    }
  }
  if (tid == 0) {
    pv.group_start[n_groups] = T;
    pv.gs_short[n_groups] = n_short;
    pv.counts[0] = n_groups;
    pv.counts[2] = min(static_cast<int>(total >> 48), pv.max_sgmv_tiles);
    pv.counts[3] = n_short;
    pv.counts[4] = n_groups - has_base;
    pv.counts[5] = 0;
    if (n_groups == has_base) pv.counts[6] = 0;
  }
  __syncthreads();
  // groups: the runs in order, concatenated (s is the run of this thread's last token)
#pragma unroll
  for (int q = kPlanTok - 1; q >= 0; --q) {
    const int t = tid * per + q;
    if (q < per && t < T) {
      const int off = t - sh.seg_start[s], pos = sh.out[s] + off;
      if (EL_CHECK(pv.status, s >= 0 && s < n_segs && pos >= 0 && pos < T, 30)) pv.perm[pos] = t;
      if (sh.out_short[s] >= 0 && EL_CHECK(pv.status, sh.out_short[s] + off < T, 31)) pv.perm_short[sh.out_short[s] + off] = t;
      if ((is_head >> q) & 1u) --s;
    }
  }
  list_tiles(sh.ids, T, pv, first);
}

__global__ void __launch_bounds__(kPlanThreads, 1)
plan_kernel(const int32_t *__restrict__ ids, int32_t T, int32_t n_slots, PlanView pv) {
  extern __shared__ __align__(16) uint32_t keys[];  // one key per run, padded to a power of two; or the small form's arrays
  __shared__ int wt[34];
  __shared__ unsigned long long wt_small[2][kPlanThreads / 32];
  __shared__ uint32_t first[kMaxTokensLimit / 32];  // see list_tiles
  const int tid = threadIdx.x;

  ptx::pdl_launch_dependents();
  ptx::pdl_wait_prior_grids();  // earlier kernels on the stream may still read the plan arrays
  if (T <= kPlanSmallT) {
    plan_small(ids, T, n_slots, pv, PlanSmall(keys, T), first, wt_small);
    return;
  }

  // 1. validate
  bool bad = false;
  for (int i = tid; i < kMaxTokensLimit / 32; i += kPlanThreads) first[i] = 0;
  for (int t = tid; t < T; t += kPlanThreads) {
    int32_t a = ids[t];
    if (a < -1 || a >= n_slots) {
      a = -1;
      bad = true;
    }
    pv.ids_valid[t] = a;
  }
  if (__syncthreads_or(bad ? 1 : 0) && tid == 0) atomicOr(pv.status, EDGELORA_STATUS_BAD_ADAPTER_ID);

  // 2. segments = maximal runs of equal id in token order
  auto is_head = [&](int t) { return (t == 0 || pv.ids_valid[t] != pv.ids_valid[t - 1]) ? 1 : 0; };
  const int n_segs = scan_rounds(
      T, wt, is_head, [&](int t, int before) {
        const int head = is_head(t);
        const int s = before + head - 1;
        pv.tok_seg[t] = s;
        if (head) {
          pv.seg_start[s] = t;
          pv.seg_adapter[s] = pv.ids_valid[t];
        }
      });
  if (tid == 0) {
    pv.seg_start[n_segs] = T;
    pv.counts[1] = n_segs;
  }
  __syncthreads();

  // 3. runs ordered by (id, run index): -1 first, token order kept (runs are in token order)
  int npow2 = 32;
  while (npow2 < n_segs) npow2 <<= 1;
  for (int i = tid; i < npow2; i += kPlanThreads)
    keys[i] = i < n_segs ? ((static_cast<uint32_t>(pv.seg_adapter[i] + 1) << 16) | static_cast<uint32_t>(i))
                         : 0xFFFFFFFFu;
  __syncthreads();
  sort_keys(keys, npow2);
  __syncthreads();

  // 4. groups: the runs in sorted order, concatenated.  out_start[j] (in pv.scratch) is where the
  // j-th sorted run begins in perm; inv (borrowing pv.mt_list until step 8) maps a run to j.
  int32_t *out_start = pv.scratch, *inv = pv.mt_list, *gidx = pv.perm_short;  // gidx: until step 6
  auto run_of = [&](int j) { return static_cast<int>(keys[j] & 0xFFFFu); };
  auto run_len = [&](int j) {
    const int s = run_of(j);
    return pv.seg_start[s + 1] - pv.seg_start[s];
  };
  scan_rounds(n_segs, wt, run_len, [&](int j, int before) {
    out_start[j] = before;
    inv[run_of(j)] = j;
  });
  for (int t = tid; t < T; t += kPlanThreads) {
    const int s = pv.tok_seg[t];
    const int pos = out_start[inv[s]] + (t - pv.seg_start[s]);
    if (EL_CHECK(pv.status, s >= 0 && s < n_segs && pos >= 0 && pos < T, 30)) pv.perm[pos] = t;
  }
  auto is_ghead = [&](int j) { return (j == 0 || (keys[j] >> 16) != (keys[j - 1] >> 16)) ? 1 : 0; };
  const int has_base = (n_segs > 0 && (keys[0] >> 16) == 0) ? 1 : 0;  // the group of id -1 sorts first
  const int n_groups = scan_rounds(n_segs, wt, is_ghead, [&](int j, int before) {
    const int head = is_ghead(j);
    const int g = before + head - 1;
    gidx[j] = g;
    const int32_t a = static_cast<int32_t>(keys[j] >> 16) - 1;
    if (a >= 0) mark_first(first, pv.seg_start[run_of(j)], head ? 0 : pv.seg_start[run_of(j - 1) + 1]);
    if (head) {
      pv.group_start[g] = out_start[j];
      pv.group_adapter[g] = a;
      if (a >= 0) pv.lg_adapter[g - has_base] = a;
    }
  });
  if (tid == 0) {
    pv.group_start[n_groups] = T;
    pv.counts[0] = n_groups;
    pv.counts[4] = n_groups - has_base;
    pv.counts[5] = 0;
  }

  // 5. the same groups restricted to "short" tokens: every token of a small batch, otherwise the
  // tokens of runs shorter than kSegMin (long runs go to the segment shrink).  sstart[j] replaces
  // out_start[j] in pv.scratch.
  const bool all_short = T <= kDecodeMaxT;
  auto short_len = [&](int j) {
    const int len = run_len(j);
    return (all_short || len < kSegMin) ? len : 0;
  };
  const int n_short = scan_rounds(n_segs, wt, short_len, [&](int j, int before) {
    out_start[j] = before;
    if (is_ghead(j)) pv.gs_short[gidx[j]] = before;
  });
  // 6. (gidx is dead from here: perm_short takes its final content)
  for (int t = tid; t < T; t += kPlanThreads) {
    const int s = pv.tok_seg[t];
    const int len = pv.seg_start[s + 1] - pv.seg_start[s];
    const int pos = out_start[inv[s]] + (t - pv.seg_start[s]);
    if ((all_short || len < kSegMin) && EL_CHECK(pv.status, pos >= 0 && pos < T, 31)) pv.perm_short[pos] = t;
  }
  if (tid == 0) {
    pv.gs_short[n_groups] = n_short;
    pv.counts[3] = n_short;
    pv.counts[6] = n_short - pv.gs_short[has_base];  // (written behind the barriers of the scan; n_short when no id >= 0 is there)
  }

  // 7. 128-token tiles of the long runs (segment shrink work list), in token order
  auto run_tiles = [&](int s) {
    const int len = pv.seg_start[s + 1] - pv.seg_start[s];
    return (!all_short && pv.seg_adapter[s] >= 0 && len >= kSegMin) ? (len + kTileM - 1) / kTileM : 0;
  };
  const int n_tiles = scan_rounds(n_segs, wt, run_tiles, [&](int s, int before) {
    const int t0 = pv.seg_start[s];
    const int len = pv.seg_start[s + 1] - t0;
    const int nt = run_tiles(s);
    for (int i = 0; i < nt; ++i) {
      const int tile = before + i;
      if (tile < pv.max_sgmv_tiles) {
        pv.sgmv_tiles[4 * tile + 0] = t0 + i * kTileM;
        pv.sgmv_tiles[4 * tile + 1] = min(kTileM, len - i * kTileM);
        pv.sgmv_tiles[4 * tile + 2] = pv.seg_adapter[s];
        pv.sgmv_tiles[4 * tile + 3] = 0;
      }
    }
  });
  if (tid == 0) pv.counts[2] = min(n_tiles, pv.max_sgmv_tiles);
  __syncthreads();  // inv (in pv.mt_list) is dead from here

  // 8. the adapters of every 256-token tile
  list_tiles(pv.ids_valid, T, pv, first);
}

void launch_plan(const int32_t *ids, int32_t T, int32_t n_slots, const PlanView &pv, bool pdl,
                 cudaStream_t stream) {
  int npow2 = 32;  // the number of runs is only known on the device: size for the worst case
  while (npow2 < T) npow2 <<= 1;
  const size_t smem = T <= kPlanSmallT ? PlanSmall::bytes(T) : static_cast<size_t>(npow2) * 4;
  launch_ex(plan_kernel, dim3(1), dim3(kPlanThreads), smem, stream, pdl, 1, ids, T, n_slots, pv);
}

void init_plan_kernel() {
  cudaFuncSetAttribute(plan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       kMaxTokensLimit * 4);
}

}  // namespace edgelora
