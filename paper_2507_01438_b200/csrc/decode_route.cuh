// Routing helpers shared by the kernels that derive a decode batch's u-batches (paper Section 3.4)
// from the caller's ids inside the kernel: a CTA-wide prefix sum and the publication of the routing
// plan in its canonical form (the form the plan kernel writes for larger batches).
#pragma once
#include "internal.cuh"
#include "ptx.cuh"

namespace edgelora {

// Exclusive prefix sum of one int per thread over the first 256 threads of the CTA; `total` gets
// the sum.  Every thread of the CTA calls it (it synchronises the CTA); threads from 256 on pass 0
// and ignore the result.  wt: shared memory, 9 ints.
__device__ __forceinline__ int block_scan_256(int v, int *wt, int &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31 && warp < 8) wt[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const int w = lane < 8 ? wt[lane] : 0;
    int wi = w;
#pragma unroll
    for (int d = 1; d < 8; d <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, wi, d);
      if (lane >= d) wi += o;
    }
    if (lane < 8) wt[lane] = wi - w;
    if (lane == 7) wt[8] = wi;
  }
  __syncthreads();
  const int res = wt[warp < 8 ? warp : 8] + incl - v;
  total = wt[8];
  __syncthreads();
  return res;
}

// Writes the routing plan of a batch of T <= 256 tokens in canonical order (ids ascending, -1
// first; segments in token order).  Called by every thread of one CTA; thread t < T passes the
// validated id `a` of token t (-1 = no adapter), the others -1.  s_id[256], 16-byte aligned, holds those ids already;
// s_cnt[256] and s_wt[9] are scratch.  Everything is worked out in shared memory and registers
// first; the stores come after griddepcontrol.wait (earlier kernels on the stream may still read the
// plan).
__device__ __forceinline__ void publish_decode_plan(const PlanView &pv, int a, int T, int any_bad, int KS,
                                                    const int32_t *s_id, int32_t *s_cnt, int *s_wt) {
  const int tid = threadIdx.x;
  int rp = 0;  // position of token tid by (id, token); four ids per shared-memory load
  if (tid < T) {
    auto in_front = [&](int id, int u) { return static_cast<int>(id < a) | (static_cast<int>(id == a) & static_cast<int>(u < tid)); };
    const int full = T & ~3;
#pragma unroll 4
    for (int u = 0; u < full; u += 4) {
      const int4 w = *reinterpret_cast<const int4 *>(s_id + u);
      rp += in_front(w.x, u) + in_front(w.y, u + 1) + in_front(w.z, u + 2) + in_front(w.w, u + 3);
    }
    for (int u = full; u < T; ++u) rp += in_front(s_id[u], u);
  }
  __syncthreads();  // every thread is done with s_cnt as a counter
  if (tid < T) s_cnt[rp] = tid;  // s_cnt now holds the tokens in canonical order
  __syncthreads();
  int ida = -2, tok = 0;
  bool head = false;
  if (tid < T) {
    tok = s_cnt[tid];
    ida = s_id[tok];
    head = tid == 0 || s_id[s_cnt[tid - 1]] != ida;
  }
  int n_groups;
  const int gi = block_scan_256(head ? 1 : 0, s_wt, n_groups);
  const int has_base = (T > 0 && s_id[s_cnt[0]] < 0) ? 1 : 0;
  const bool shead = tid < T && (tid == 0 || s_id[tid - 1] != a);
  int n_segs;
  const int si = block_scan_256(shead ? 1 : 0, s_wt, n_segs);

  ptx::pdl_wait_prior_grids();
  if (any_bad && tid == 0) atomicOr(pv.status, EDGELORA_STATUS_BAD_ADAPTER_ID);
  if (tid < T) {
    pv.ids_valid[tid] = a;
    pv.perm[tid] = tok;
    pv.perm_short[tid] = tok;
    if (head) {
      pv.group_start[gi] = tid;
      pv.gs_short[gi] = tid;
      pv.group_adapter[gi] = ida;
      if (ida >= 0) pv.lg_adapter[gi - has_base] = pv.mt_list[gi - has_base] = ida;  // (all tokens are one tile of the list)
    }
    pv.tok_seg[tid] = si + (shead ? 1 : 0) - 1;
    if (shead) {
      pv.seg_start[si] = tid;
      pv.seg_adapter[si] = a;
    }
  }
  if (tid == 0) {
    pv.group_start[n_groups] = T;
    pv.gs_short[n_groups] = T;
    pv.seg_start[n_segs] = T;
    pv.counts[0] = n_groups;
    pv.counts[1] = n_segs;
    pv.counts[2] = 0;
    pv.counts[3] = T;
    pv.counts[4] = n_groups - has_base;
    pv.counts[5] = KS;
    pv.counts[6] = 0;
    pv.mt_count[0] = n_groups - has_base;
  }
}

// The u-batches of a decode batch, in shared memory: adapters in order of first appearance, the tokens of each in token
// order, and the tokens of an adapter in blocks.
struct Groups {
  alignas(16) int32_t id[kDecodeMaxT];  // validated id of each token
  int32_t adapter[kDecodeMaxT];  // of each group
  int32_t cnt[kDecodeMaxT];      // scratch: tokens of each group
  int32_t wt[9];                 // scratch of the prefix sums
  int32_t n_groups, n_blocks;
  int16_t start[kDecodeMaxT + 1];    // groups' first positions in tok
  int16_t block_pos[kDecodeMaxT];    // blocks' first positions in tok
  uint8_t tok[kDecodeMaxT], block_group[kDecodeMaxT];
  uint8_t group[kDecodeMaxT];        // of each token with an adapter
  int16_t pos[kDecodeMaxT];          // its position in tok
};
// Exclusive prefix sums of a value per element, elements i = k * kN + tid, over kN threads that meet on barrier kBar.
template <int kBar, int kN, int kPer>
__device__ __forceinline__ int32_t group_scan(const int32_t (&v)[kPer], int32_t *wt, int tid, int32_t (&out)[kPer]) {
  const int lane = tid & 31, warp = tid >> 5;
  int32_t incl[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    incl[k] = v[k];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int32_t o = __shfl_up_sync(0xffffffffu, incl[k], d);
      if (lane >= d) incl[k] += o;
    }
    if (lane == 31) wt[k * (kN / 32) + warp] = incl[k];
  }
  ptx::named_barrier<kBar, kN>();
  int32_t total = 0;
#pragma unroll
  for (int i = 0; i < kPer * kN / 32; ++i) {
#pragma unroll
    for (int k = 0; k < kPer; ++k)
      if (i == k * (kN / 32) + warp) out[k] = total + incl[k] - v[k];
    total += wt[i];
  }
  return total;
}
// kN threads (128 or 256, a multiple of 32) call it with their number `tid`; they meet on the named barrier kBar.  Blocks
// hold at most kBlockTok tokens.  Returns whether one of this thread's ids was out of range (-1 is kept for it).
template <int kBlockTok, int kBar, int kN>
__device__ __forceinline__ bool derive_groups(Groups &s, const int32_t *ids, int T, int32_t n_slots, int tid) {
  constexpr int kPer = kDecodeMaxT / kN;
  const auto sync = [] { ptx::named_barrier<kBar, kN>(); };
  int32_t a[kPer], pos[kPer], first[kPer], v[kPer], out[kPer];
  bool bad = false;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int t = k * kN + tid;
    a[k] = t < T ? ids[t] : -1;
    if (a[k] < -1 || a[k] >= n_slots) {
      a[k] = -1;
      bad = true;
    }
    s.id[t] = a[k];
    s.cnt[t] = 0;
  }
  sync();
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int t = k * kN + tid;
    pos[k] = 0;
    first[k] = t;
    if (a[k] >= 0) {  // earlier tokens on the same adapter, four ids per shared-memory load
      auto see = [&](int id, int u) {
        if (id == a[k]) {
          if (pos[k] == 0) first[k] = u;
          ++pos[k];
        }
      };
      const int full = t & ~3;
#pragma unroll 4
      for (int u = 0; u < full; u += 4) {
        const int4 w = *reinterpret_cast<const int4 *>(&s.id[u]);
        see(w.x, u);
        see(w.y, u + 1);
        see(w.z, u + 2);
        see(w.w, u + 3);
      }
      for (int u = full; u < t; ++u) see(s.id[u], u);
    }
    v[k] = a[k] >= 0 && pos[k] == 0 ? 1 : 0;
  }
  const int32_t G = group_scan<kBar, kN, kPer>(v, s.wt, tid, out);
#pragma unroll
  for (int k = 0; k < kPer; ++k)
    if (v[k]) {
      s.group[k * kN + tid] = static_cast<uint8_t>(out[k]);
      s.adapter[out[k]] = a[k];
    }
  sync();
#pragma unroll
  for (int k = 0; k < kPer; ++k)
    if (a[k] >= 0) {
      first[k] = s.group[first[k]];  // its group from here on
      atomicAdd(&s.cnt[first[k]], 1);
    }
  sync();
#pragma unroll
  for (int k = 0; k < kPer; ++k) {  // tokens in the low half, blocks in the high half
    const int g = k * kN + tid, n = g < G ? s.cnt[g] : 0;
    v[k] = n | ((n + kBlockTok - 1) / kBlockTok) << 16;
  }
  const int32_t total = group_scan<kBar, kN, kPer>(v, s.wt, tid, out);
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int g = k * kN + tid, start = out[k] & 0xFFFF, b0 = out[k] >> 16;
    if (g < G) s.start[g] = static_cast<int16_t>(start);
    for (int b = 0; b < v[k] >> 16; ++b) {
      s.block_group[b0 + b] = static_cast<uint8_t>(g);
      s.block_pos[b0 + b] = static_cast<int16_t>(start + b * kBlockTok);
    }
  }
  if (tid == 0) {
    s.start[G] = static_cast<int16_t>(total & 0xFFFF);
    s.n_groups = G;
    s.n_blocks = total >> 16;
  }
  sync();
#pragma unroll
  for (int k = 0; k < kPer; ++k)
    if (a[k] >= 0) {
      const int p = s.start[first[k]] + pos[k];
      s.tok[p] = static_cast<uint8_t>(k * kN + tid);
      s.pos[k * kN + tid] = static_cast<int16_t>(p);
      s.group[k * kN + tid] = static_cast<uint8_t>(first[k]);
    }
  sync();
  return bad;
}

}  // namespace edgelora
