// fb_gate_commit: in-order retirement with KV freeze and readiness-gated
// admission (Alg. 1 lines 7-12, Eq. 2-3, Eq. 6 for the committing block).
//
// One CTA per request.  Its first warp evaluates the block-level predicates from the
// per-slot counts, one window block per lane; all threads then copy the retiring blocks'
// window K/V rows into the request's pages with 16-byte accesses.  Requests are independent,
// so no inter-CTA ordering is needed.  The step counters: up to eight requests form one
// cluster whose first CTA adds up the others' contributions (no clearing before the
// launch); larger batches add with integer atomics onto a cleared array.  The
// batch-synchronous variant (fb_config.batch_sync) adds a single-CTA kernel in front that
// reduces the per-request results over the batch into two of the counters, which every CTA
// here reads, and clears the others.
// Bound by latency (two rounds of dependent loads): call with its state reset, 1 and 8 requests
// 8.3 -> 4.0 and 4.6 us (one thread walked the blocks, and a memset cleared the counters),
// 64 requests 9.5 -> 7.3.
#include <cooperative_groups.h>

#include "fb_common.cuh"

namespace fb {

constexpr int kGateThreads = 512;
constexpr int kGateCluster = 8;      // largest batch that runs as one cluster (the portable cluster size)

struct GateParams {
  const int32_t *n_live, *req_slot_begin, *slot_stats;
  int32_t *active, *prefix_len, *L, *R, *tokens;
  uint8_t* pe_done;
  const int32_t* page_table;
  const uint4 *k_win, *v_win;
  uint4 *k_pool, *v_pool;
  int32_t* n_committed;
  uint8_t* spawned;
  int32_t *counters, *status;
  int32_t max_requests, wmax, bl, max_blocks, mask_id, s_pe, n_kv_heads, head_dim, num_pages,
      max_pages_per_req;
  float theta_spawn;
  int32_t batch_sync;
  int32_t clustered;       // the whole grid is one cluster
};

// Post-edit forwards of a block after this one, which it went into with m0 masks.
__device__ __forceinline__ int post_edits(int before, int m0) { return min(before + (m0 == 0 ? 1 : 0), 255); }
// Locally finished (Sec. 2.1): no masks left (m1), and either a quiet post-edit forward or the S_pe
// budget is used up.
__device__ __forceinline__ bool finished(const GateParams& p, int m0, int m1, int n_updates, int pe) {
  return m1 == 0 && ((m0 == 0 && n_updates == 0) || pe >= p.s_pe);
}

// blocks of the finished prefix, before EOS is looked at (a window has at most 8: there is a zero bit)
__device__ __forceinline__ int leading_blocks(unsigned fin) { return __ffs(~fin) - 1; }

// What a request's own block counts say to the batch reduction (Alg. 1 l.7-9 before any batch rule):
// its window, the finished prefix c (stopping after a block that holds EOS), and whether retiring
// those c blocks ends the request.
struct ReqEval {
  int first, w, L, R, c;
  bool ok, ends;
};
__device__ __forceinline__ ReqEval eval_request(const GateParams& p, int r) {
  ReqEval e;
  e.first = p.req_slot_begin[r];
  e.w = p.req_slot_begin[r + 1] - e.first;
  e.L = p.L[r]; e.R = p.R[r];
  e.c = 0; e.ends = false;
  e.ok = !(e.w != e.R - e.L || e.w < 0 || e.w > p.wmax);
  if (!e.ok) return e;
  unsigned fin = 0, eos = 0;                         // bit s: window block s
  for (int s = 0; s < e.w; ++s) {
    const int32_t* st = p.slot_stats + (e.first + s) * FB_SLOT_STATS;
    const int m0 = st[FB_STAT_M0], pe = post_edits(p.pe_done[r * p.wmax + s], m0);
    fin |= (unsigned)finished(p, m0, st[FB_STAT_M1], st[FB_STAT_M2T] + st[FB_STAT_T2T], pe) << s;
    eos |= (unsigned)(st[FB_STAT_EOS] != 0) << s;
  }
  const int lead = leading_blocks(fin);
  const unsigned ending = eos & ((1u << lead) - 1u);
  e.c = ending ? __ffs(ending) : lead;
  e.ends = ending || e.L + e.c == p.max_blocks;
  return e;
}
// Eq. 2 on the frontier block as it went into this forward (m0 masks, rdy of them ready; an
// empty window counts as ready); Eq. 3 with the window bounds once the oldest block is L
__device__ __forceinline__ bool clears_gate(const GateParams& p, int m0, int rdy, int L, int R) {
  const float rho = m0 != 0 ? __fdiv_rn((float)rdy, (float)m0) : 1.0f;
  return rho >= p.theta_spawn && R - L < p.wmax && R < p.max_blocks;
}
__device__ __forceinline__ bool clears_gate(const GateParams& p, const ReqEval& e, int c) {
  const int32_t* st = p.slot_stats + (e.first + e.w - 1) * FB_SLOT_STATS;
  return e.w > 0 ? clears_gate(p, st[FB_STAT_M0], st[FB_STAT_RDY], e.L + c, e.R) : clears_gate(p, 0, 0, e.L + c, e.R);
}

// batch_sync: the two reductions over the decoding sequences (Sec. 3.2: finished.all(),
// min_b rho_b), one CTA, before any state is touched.  A sequence that ends with its own
// finished prefix never holds the others back beyond it; if every sequence ends, each
// retires its own prefix.
__global__ void __launch_bounds__(kGateThreads) gate_batch_reduce_kernel(const GateParams p) {
  pdl_wait();
  __shared__ int s_min, s_max, s_all;
  if (threadIdx.x == 0) { s_min = 0x7fffffff; s_max = 0; s_all = 1; }
  __syncthreads();
  for (int r = threadIdx.x; r < p.max_requests; r += kGateThreads) {
    if (p.active[r] != 1) continue;
    const ReqEval e = eval_request(p, r);
    if (!e.ok) { atomicMin(&s_min, 0); continue; }   // pack and state disagree: nothing retires
    if (e.ends) atomicMax(&s_max, e.c); else atomicMin(&s_min, e.c);
  }
  __syncthreads();
  const int C = s_min != 0x7fffffff ? s_min : s_max;
  int left = 0;
  for (int r = threadIdx.x; r < p.max_requests; r += kGateThreads) {
    if (p.active[r] != 1) continue;
    const ReqEval e = eval_request(p, r);
    if (!e.ok) { atomicAnd(&s_all, 0); continue; }
    const int c = min(e.c, C);
    if (e.ends && c == e.c) continue;                // done: no longer part of the batch
    left = 1;
    if (!clears_gate(p, e, c)) atomicAnd(&s_all, 0);
  }
  const int any_left = __syncthreads_or(left);
  if (threadIdx.x < FB_CT_LOCKSTEP_COMMIT) p.counters[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    p.counters[FB_CT_LOCKSTEP_COMMIT] = C;
    p.counters[FB_CT_LOCKSTEP_ADMIT] = any_left && s_all;
  }
}

__global__ void __launch_bounds__(kGateThreads) gate_commit_kernel(const GateParams p) {
  pdl_wait();
  const int r = blockIdx.x;
  const int tid = threadIdx.x;
  __shared__ int s_c, s_first, s_P, s_spawn, s_newR;
  __shared__ int s_ct[FB_CT_LOCKSTEP_COMMIT];          // this request's share of the step counters
  static_assert(FB_CT_LOCKSTEP_COMMIT == 8 && FB_CT_LOCKSTEP_ADMIT == 9, "the summed counters come first");
  if (tid < 32) {
    // everything that does not depend on another load, together
    const int active = p.active[r], first = p.req_slot_begin[r], w = p.req_slot_begin[r + 1] - first;
    const int L0 = p.L[r], R = p.R[r], P = p.prefix_len[r];
    const int cap = p.batch_sync ? p.counters[FB_CT_LOCKSTEP_COMMIT] : 0, admit = p.batch_sync ? p.counters[FB_CT_LOCKSTEP_ADMIT] : 0;
    const int n_live = r == 0 ? *p.n_live : 0;
    const bool ok = w == R - L0 && w >= 0 && w <= p.wmax;
    int c = 0, spawn = 0, done = 0, m2t = 0, t2t = 0;
    if (active == 1 && ok) {                           // (uniform over the warp)
      // lane s: window block s
      int m0 = 0, rdy = 0, m1 = 1, nupd = 0, pn = 0;
      bool eos = false;
      if (tid < w) {
        const int32_t* st = p.slot_stats + (first + tid) * FB_SLOT_STATS;
        m0 = st[FB_STAT_M0]; rdy = st[FB_STAT_RDY]; m2t = st[FB_STAT_M2T]; t2t = st[FB_STAT_T2T]; m1 = st[FB_STAT_M1];
        eos = st[FB_STAT_EOS] != 0;
        nupd = m2t + t2t;
        pn = post_edits(p.pe_done[r * p.wmax + tid], m0);
      }
      // Alg. 1 l.7-9: the finished prefix, stopping after a block with EOS
      const bool fin = tid < w && finished(p, m0, m1, nupd, pn);
      const int lead = leading_blocks(__ballot_sync(0xffffffffu, fin));
      const unsigned ends = __ballot_sync(0xffffffffu, eos && tid < lead);
      const int own = ends ? __ffs(ends) : lead;
      // batch_sync: the batch's retire count caps the sequence's own; a block holding EOS
      // terminates only if it is among the blocks that do retire
      c = p.batch_sync ? min(own, cap) : own;
      const int L = L0 + c;
      done = (c == own && ends) || L == p.max_blocks;
      const int fm0 = __shfl_sync(0xffffffffu, m0, max(w - 1, 0)), frdy = __shfl_sync(0xffffffffu, rdy, max(w - 1, 0));
      if (!done) spawn = p.batch_sync ? admit : (int)clears_gate(p, fm0, frdy, L, R);
      const int shifted = __shfl_sync(0xffffffffu, pn, (tid + c) & 31);
      if (tid < p.wmax) p.pe_done[r * p.wmax + tid] = (uint8_t)(tid + c < w ? shifted : 0);   // (an admitted block starts at 0)
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        m2t += __shfl_xor_sync(0xffffffffu, m2t, o);
        t2t += __shfl_xor_sync(0xffffffffu, t2t, o);
      }
      if (tid == 0) {
        p.L[r] = L;
        p.prefix_len[r] = P + c * p.bl;
        if (done) p.active[r] = 2;
        if (spawn) p.R[r] = R + 1;
      }
    } else if (active == 1 && tid == 0) {              // pack and state disagree: leave the request alone
      atomicOr(p.status, FB_ST_BAD_STATE);
    }
    if (tid == 0) {
      s_c = c; s_first = first; s_P = P; s_spawn = spawn; s_newR = R;
      p.n_committed[r] = c;
      p.spawned[r] = (uint8_t)spawn;
      const bool counts = active == 1 && ok;
      s_ct[FB_CT_BLOCKS] = c; s_ct[FB_CT_TOKENS] = c * p.bl; s_ct[FB_CT_SPAWNED] = spawn;
      s_ct[FB_CT_FINISHED] = counts && done; s_ct[FB_CT_M2T] = m2t; s_ct[FB_CT_T2T] = t2t;
      s_ct[FB_CT_LIVE_SLOTS] = n_live; s_ct[FB_CT_ACTIVE] = counts && !done;
    }
    __syncwarp();
    if (!p.clustered && tid < FB_CT_LOCKSTEP_COMMIT && s_ct[tid]) atomicAdd(&p.counters[tid], s_ct[tid]);
  }
  __syncthreads();
  // freeze KV of the retiring blocks: window rows -> absolute positions
  const int c = s_c, first = s_first, P = s_P;
  const int vec_per_head = p.head_dim / 8;                 // uint4 per (token, head)
  const int vec_per_tok = p.n_kv_heads * vec_per_head;
  // (window resident in the pages: nothing to copy, the prefix pointer has moved over it)
  const int total = p.k_win ? c * p.bl * vec_per_tok : 0;
  // four pieces per thread and pass, all loads issued before the first store (source and
  // destination never overlap: window tensors against the page pool)
  constexpr int kBatch = 4;
  for (int i0 = tid; i0 < total; i0 += kBatch * kGateThreads) {
    uint4 kv[kBatch], vv[kBatch];
    size_t dst[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const int i = i0 + j * kGateThreads;
      dst[j] = ~(size_t)0;
      if (i >= total) continue;
      const int tok = i / vec_per_tok, rem = i % vec_per_tok;
      const int h = rem / vec_per_head, v = rem % vec_per_head;
      const int apos = P + tok;
      const int pidx = apos / kPage;
      if (pidx >= p.max_pages_per_req) { atomicOr(p.status, FB_ST_BAD_PAGE); continue; }
      const int page = p.page_table[r * p.max_pages_per_req + pidx];
      if (page < 0 || page >= p.num_pages) { atomicOr(p.status, FB_ST_BAD_PAGE); continue; }
      const size_t src = (size_t)(first * p.bl + tok) * vec_per_tok + rem;
      dst[j] = (((size_t)page * p.n_kv_heads + h) * kPage + apos % kPage) * vec_per_head + v;
      kv[j] = p.k_win[src];
      vv[j] = p.v_win[src];
    }
#pragma unroll
    for (int j = 0; j < kBatch; ++j)
      if (dst[j] != ~(size_t)0) { p.k_pool[dst[j]] = kv[j]; p.v_pool[dst[j]] = vv[j]; }
  }
  // the admitted block starts fully masked
  if (s_spawn) {
    int32_t* nb = p.tokens + (size_t)r * p.max_blocks * p.bl + (size_t)s_newR * p.bl;
    for (int t = tid; t < p.bl; t += kGateThreads) nb[t] = p.mask_id;
  }
  if (p.clustered) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    if (r == 0 && tid < FB_STEP_COUNTERS) {
      int sum = 0;
      if (tid < FB_CT_LOCKSTEP_COMMIT) {
        for (int k = 0; k < (int)cluster.num_blocks(); ++k) sum += *cluster.map_shared_rank(&s_ct[tid], k);
        p.counters[tid] = sum;
      } else if (!p.batch_sync) {
        p.counters[tid] = 0;
      }
    }
    cluster.sync();                     // the contributions stay put until they have been read
  }
}

int launch_gate(fb_ctx* ctx, const fb_pack* pk, const int32_t* slot_stats, const fb_state* st,
                const void* k_win, const void* v_win, void* k_pool, void* v_pool, int32_t* n_committed,
                uint8_t* spawned, int32_t* step_counters, int32_t* status, cudaStream_t stream) {
  const fb_config& c = ctx->cfg;
  GateParams p;
  p.n_live = pk->n_live; p.req_slot_begin = pk->req_slot_begin; p.slot_stats = slot_stats;
  p.active = st->active; p.prefix_len = st->prefix_len; p.L = st->L; p.R = st->R; p.tokens = st->tokens;
  p.pe_done = st->pe_done; p.page_table = st->page_table;
  p.k_win = static_cast<const uint4*>(k_win); p.v_win = static_cast<const uint4*>(v_win);
  p.k_pool = static_cast<uint4*>(k_pool); p.v_pool = static_cast<uint4*>(v_pool);
  p.n_committed = n_committed; p.spawned = spawned; p.counters = step_counters; p.status = status;
  p.max_requests = c.max_requests; p.wmax = c.wmax; p.bl = c.block_len; p.max_blocks = c.max_blocks;
  p.mask_id = c.mask_id; p.s_pe = c.s_pe; p.n_kv_heads = c.n_kv_heads; p.head_dim = c.head_dim;
  p.num_pages = c.num_pages; p.max_pages_per_req = c.max_pages_per_req; p.theta_spawn = c.theta_spawn;
  p.batch_sync = c.batch_sync;
  p.clustered = c.max_requests <= kGateCluster;
  if (c.batch_sync) {
    if (int e = cuda_err(ctx, launch_pdl(gate_batch_reduce_kernel, 1, kGateThreads, 0, stream, p),
                         "gate_batch_reduce_kernel launch"))
      return e;
  } else if (!p.clustered) {
    if (int e = cuda_err(ctx, cudaMemsetAsync(step_counters, 0, FB_STEP_COUNTERS * sizeof(int32_t), stream),
                         "clear step counters"))
      return e;
  }
  return cuda_err(ctx, launch_pdl_cluster(gate_commit_kernel, c.max_requests, kGateThreads, 0, stream,
                                          p.clustered ? c.max_requests : 1, p),
                  "gate_commit_kernel launch");
}

}  // namespace fb
