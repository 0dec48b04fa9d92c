// fb_wavefront_attn: W-shaped block-causal GQA attention over the packed
// wavefronts (Sec. 3.1 "W-shaped block-causal attention"; Sec. 3.2 Eq. 5).
//
// Persistent, warp-specialised tcgen05 kernel, one CTA per SM:
//   warps 0, 2  TMA producers: Q tiles, K/V tiles of the paged prefix (page-table
//               lookups) and of the window tensors, 2-stage K and V rings, one
//               stage of each per warp
//   warp 1      MMA issuer: S = Q K^T and O += P V with tcgen05.mma, S/P and O
//               in TMEM, two Q tiles (A, B) ping-ponged so that the tensor pipe
//               works on one tile while the other is in softmax
//   warp 3      idle (it completes the control warpgroup, which gives its
//               registers to the softmax warpgroups with setmaxnreg)
//   warps 4-7   softmax of tile A, one thread per query row: its 128 scores are read
//               from TMEM at once, exp2 against a lazily re-based reference (only the
//               first tile of an item takes a max pass), P (bf16) written over the
//               last columns of S in TMEM; epilogue
//   warps 8-11  the same for tile B
// What bounds it: at full load the board's power limit (the SM clock falls from 1965
// to about 1450 MHz), so both fewer cycles and fewer instructions pay; below that,
// the chain S -> P -> P V -> next S of a tile (2600 to 2900 cycles against 2048 of
// MMA time and as many of MUFU time for the two tiles of a CTA).  Sustained, back to
// back, with the loop's former form and now: long-context workload 1259 -> 1165 us,
// 64 requests 458 -> 424 us, 128 requests 498 -> 469 us, long context in 8 bits 996 ->
// 880 us.
// A Q tile is 128 rows = (128/G tokens) x (G query heads of one KV head) of one
// slot.  A unit runs two Q tiles side by side: two tiles of one request and KV
// head, which share each K/V tile from shared memory, or the odd tile left
// over, run under two adjacent KV heads at once (two K/V streams, served in
// turn).  The mask is per tile: a tile of the frozen prefix is
// fully visible except the ragged last one; the window tile is visible up to
// (s+1)*bl keys for a query in window slot s.  Tiles nobody can see are never
// loaded (the work list only spans visible tiles), and ragged tiles run the
// MMAs on ceil(valid/16)*16 keys only.  With the window resident in the pages
// every key tile is a paged one over absolute positions.
// Work items are sorted longest first by the pack kernel (those of a single request, no more
// than SMs, come unit by unit) and drawn by the CTAs from a global ticket.
// Long key ranges are split across CTAs; partial (max, sum, O) go to the
// workspace and a second kernel merges them in a fixed order.
#include <cudaTypedefs.h>

#include "attn_common.cuh"

namespace fb {

// Largest of N scores held in registers.
template <int N>
__device__ __forceinline__ float max_cols(const uint32_t* s) {
  float m8[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) m8[t] = fmaxf(__uint_as_float(s[t]), __uint_as_float(s[8 + t]));
#pragma unroll
  for (int i = 16; i < N; i += 16)
#pragma unroll
    for (int t = 0; t < 8; ++t) m8[t] = max3(m8[t], __uint_as_float(s[i + t]), __uint_as_float(s[i + 8 + t]));
  return fmaxf(fmaxf(fmaxf(m8[0], m8[1]), fmaxf(m8[2], m8[3])), fmaxf(fmaxf(m8[4], m8[5]), fmaxf(m8[6], m8[7])));
}

// P of N scores against the reference behind mb = m_ref * sl2 - shift: packed into pk, the sum of
// the unrounded values returned; `most`: the largest of eight partial sums of N / 8 values each, a
// bound on every value that costs three instructions a row (8-bit P saturates, so it needs one:
// the largest value itself took one instruction per pair and 10 % of that kernel's time).  A masked
// score (-inf) comes out as exactly 0.  All exponentials run on the MUFU pipe: moving 1/16 to 1/4 of
// them to a polynomial on the FMA pipe shortens the loop in cycles by up to 2.5 %, but at full load
// this kernel runs at the board's power limit, where the ~13 extra instructions per pair cost more
// clock than that gains (long-context workload, sustained: 1164 us without against 1174 to 1205 with
// a polynomial share; 64 requests 424 against 426 to 439; 8-bit pages 883 against 883 to 896).
template <bool F8, int N>
__device__ __forceinline__ float exp_cols(const uint32_t* s, uint32_t* pk, float sl2, float mb, float& most) {
  const float2 sl2v = make_float2(sl2, sl2), nmb = make_float2(-mb, -mb);
  float2 acc[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  float2 prev = make_float2(0.f, 0.f);
#pragma unroll
  for (int i = 0; i < N; i += 2) {
    const int pr = i >> 1;
    const float2 x = __ffma2_rn(make_float2(__uint_as_float(s[i]), __uint_as_float(s[i + 1])), sl2v, nmb);
    const float2 pv = make_float2(ex2_approx(x.x), ex2_approx(x.y));
    acc[pr & 3] = __fadd2_rn(acc[pr & 3], pv);
    if constexpr (F8) {
      if (i & 2) pk[i >> 2] = pack_e4m3x4(prev.x, prev.y, pv.x, pv.y);
      prev = pv;
    } else {
      pk[pr] = pack_bf16x2(pv.x, pv.y);
    }
  }
  if constexpr (F8)
    most = fmaxf(max3(acc[0].x, acc[0].y, acc[1].x), max3(max3(acc[1].y, acc[2].x, acc[2].y), acc[3].x, acc[3].y));
  const float2 t = __fadd2_rn(__fadd2_rn(acc[0], acc[1]), __fadd2_rn(acc[2], acc[3]));
  return t.x + t.y;
}

// A key tile taken 32 columns at a time out of TMEM: ragged tiles (`limit` visible keys) and full
// tiles that broke the bound on their exponentials.  A max pass first; rows whose scores lie more
// than 2^8 above the reference, or that ask for it (`grow`), move it to their largest score and
// rescale O and the row sum (O is quiescent: the commit behind this S also covered the previous
// P V).  Then the exponentials, last columns first, since P goes over the last columns of S.
// Warp-wide: every lane takes part.  By value in and out, so that the caller's registers stay
// registers: l (.x) with the tile's weights added, the reference (.y).
template <int D, bool F8>
__device__ __noinline__ float2 tile_compact(uint32_t tS, uint32_t tO, int limit, bool first, bool grow, float sl2,
                                            float shift, float m_ref, float l) {
  constexpr int P_COL = F8 ? 96 : 64, P_STEP = F8 ? 8 : 16;
  const int nch = (limit + 31) >> 5;
  float mx = -INFINITY;
#pragma unroll 1
  for (int c = 0; c < nch; ++c) {
    uint32_t s[32];
    tmem_ld32(tS + 32 * c, s);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 32; ++i) s[i] = 32 * c + i < limit ? s[i] : __float_as_uint(-INFINITY);
    mx = fmaxf(mx, max_cols<32>(s));
  }
  if (first) {
    m_ref = mx;                       // nothing accumulated yet
  } else {
    const float xmax = fmaf(mx, sl2, shift - m_ref * sl2);
    grow = grow || xmax > kRescaleThreshold;
    if (__any_sync(0xffffffffu, grow)) {
      const float alpha = grow ? ex2_approx(shift - xmax) : 1.0f;
      if (grow) { m_ref += (xmax - shift) / sl2; l *= alpha; }
#pragma unroll 1
      for (int c = 0; c < D / 32; ++c) {
        uint32_t o[32];
        tmem_ld32(tO + c * 32, o);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
        tmem_st32(tO + c * 32, o);
      }
    }
  }
  const float mb = m_ref * sl2 - shift;
  float sum = 0.f;
#pragma unroll 1
  for (int c = nch - 1; c >= 0; --c) {
    uint32_t s[32], pk[16];
    tmem_ld32(tS + 32 * c, s);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 32; ++i) s[i] = 32 * c + i < limit ? s[i] : __float_as_uint(-INFINITY);
    float none;
    sum += exp_cols<F8, 32>(s, pk, sl2, mb, none);
    if constexpr (F8) tmem_st8(tS + P_COL + P_STEP * c, pk);
    else tmem_st16(tS + P_COL + P_STEP * c, pk);
  }
  tmem_st_wait();
  return make_float2(l + sum, m_ref);
}

// F8: the KV pages hold FP8 E4M3 bytes (window resident in the pages, D = 128).  Both products
// then run as kind::f8f6f4 MMAs: the softmax warps convert their Q tile to E4M3 once per item
// (per-row power-of-two scale, undone in the row's score factor together with the K scale of
// the KV head) and write P as E4M3; O is scaled by the V scale of the KV head at the end.
template <int D, bool F8>
__global__ void __launch_bounds__(kAttnThreads, 1)
wavefront_attn_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmKwin,
                      const __grid_constant__ CUtensorMap tmVwin, const __grid_constant__ CUtensorMap tmKpool,
                      const __grid_constant__ CUtensorMap tmVpool, const __grid_constant__ CUtensorMap tmOut,
                      const AttnParams p) {
  static_assert(!F8 || D == 128, "8-bit pages: head_dim 128 only (one 128-byte swizzle row per key)");
  constexpr int NH = D / 64;                 // 64-element halves of the head dim (bf16 tiles)
  constexpr int Q_TILE_BYTES = NH * 16384;   // one 128-row bf16 tile
  constexpr int NHKV = F8 ? 1 : NH;          // 16 KB blocks of a K/V tile
  constexpr int TILE_BYTES = NHKV * 16384;   // one 128-key K or V tile
  constexpr int PAGE_BYTES = NHKV * 8192;    // one 64-key page of it
  constexpr int KSTEPS = F8 ? D / 32 : D / 16;   // MMAs per Q K^T
  constexpr int P_COL = F8 ? 96 : 64;            // P overwrites the last columns of its tile's S
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem;                        // [2] tiles A, B (bf16, as loaded)
  uint8_t* sQ8 = sQ + 2 * Q_TILE_BYTES;      // [2] the same in E4M3 (F8 only)
  uint8_t* sK = sQ8 + (F8 ? 2 * 16384 : 0);  // [2] stages
  uint8_t* sV = sK + 2 * TILE_BYTES;         // [2] stages
  uint8_t* sOut = sV + 2 * TILE_BYTES;       // [8] output staging of the softmax warps
  uint64_t* bars = reinterpret_cast<uint64_t*>(sOut + 8 * kStageBytes);
  uint64_t* q_full = bars + 0;
  uint64_t* q_empty = bars + 1;
  uint64_t* k_full = bars + 2;    // [2]
  uint64_t* k_empty = bars + 4;   // [2]
  uint64_t* v_full = bars + 6;    // [2]
  uint64_t* v_empty = bars + 8;   // [2]
  uint64_t* s_full = bars + 10;   // [2] A, B
  uint64_t* p_full = bars + 12;   // [2] P handed over (4 softmax warps)
  uint64_t* o_full = bars + 14;   // [2]
  uint64_t* item_full = bars + 20;   // [2] next work item published by the producer
  uint64_t* item_empty = bars + 22;  // [2] ... and read by the second producer, the MMA warp and the 8 softmax warps
  int* s_item = reinterpret_cast<int*>(bars + 28);                     // [2][kItemWords] published item records
  uint64_t* drain = bars + 25;       // give-up path only: everything the MMA warp has issued is complete
  uint64_t* q8_full = bars + 26;     // [2] F8: tile X converted to E4M3 by its 128 softmax threads
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 18);
  volatile int* abortf = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long LIM = p.wait_cycles;

  if (tid == 0) {
    *abortf = 0;
    mbar_init(q_full, 1); mbar_init(q_empty, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&k_full[i], 1); mbar_init(&k_empty[i], 1);
      mbar_init(&v_full[i], 1); mbar_init(&v_empty[i], 1);
      mbar_init(&s_full[i], 1); mbar_init(&p_full[i], 4); mbar_init(&o_full[i], 1);
      mbar_init(&item_full[i], 1); mbar_init(&item_empty[i], 10);
    }
    mbar_init(drain, 1);
    mbar_init(&q8_full[0], 128); mbar_init(&q8_full[1], 128);
    fence_mbar_init();
    tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmKwin); tma_prefetch_desc(&tmVwin);
    tma_prefetch_desc(&tmKpool); tma_prefetch_desc(&tmVpool); tma_prefetch_desc(&tmOut);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // The work list (and everything else) of the previous kernels is complete.  Without an early start
  // of the next kernel: where no merge stands between, the row pass came up under this kernel's
  // division of the SM and read at 0.9 of its rate (attention + row pass, 36 requests of 100 tokens, 6912
  // rows: 352 us, the two alone 14 + 309, now 325; a step of 24 short requests with four layers and
  // their scatters 319 -> 290).  Where a merge follows it makes no difference (8 requests 23.4 / 23.2).
  pdl_wait_only();

  // The control warpgroup (warps 0-3) hands registers to the softmax
  // warpgroups.  All four warps of a warpgroup execute the same setmaxnreg
  // instruction, and each role's code is dominated by its warpgroup's one.
  // Registers only move inside the CTA: what the two softmax warpgroups take
  // (2 x 128 x (200 - 168)) must not exceed what the control warpgroup gives up
  // (128 x (168 - 104)), or setmaxnreg.inc blocks for good.  (Cycles per launch on the long-context
  // workload, bf16 / 8-bit pages: 88 / 208 registers 1.478 M / 1.364 M, 104 / 200 1.464 M / 1.344 M,
  // 120 / 192 1.477 M / 1.361 M, 136 / 184 1.483 M / 1.413 M.)
  if (warp < 4) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
  if (warp == 0 || warp == 2) {
    // ----------------------------------------------------------- producers
    // Warp 0 owns K/V stage 0, warp 2 owns stage 1; warp 0 also draws the work
    // items and loads Q.  A unit whose tiles share K/V takes the stages in turn
    // (rr_k, rr_v), so each warp issues every other tile; a unit with two K/V
    // streams gives stage X to tile X, so each warp feeds one stream.  The MMA
    // warp follows the same rule.  The whole warp runs the loop converged and
    // one elected lane issues the copies: operands of the TMA / MMA
    // instructions then live in uniform registers (issuing from a single
    // diverged lane costs ~200 cycles each).
    const bool leader = elect_one();
    const int mine = warp >> 1;                    // the stage this warp fills
    int q_uses = 0, kfill = 0, vfill = 0, rr_k = 0, rr_v = 0;
    bool ok = true;
    // Page ids of the current request: lane i of pc_cur holds entry 32 * pc_blk + i of its
    // page-table row, pc_next the following 32 (loaded ahead), so a K/V tile costs two
    // shuffles instead of two dependent global loads.
    int pc_blk = 0, pc_cur = 0, pc_next = 0;
    auto load_pages = [&](int req, int blk) -> int {
      const int e = blk * 32 + lane;
      return e < p.max_pages_per_req ? __ldg(&p.page_table[(size_t)req * p.max_pages_per_req + e]) : -1;
    };
    // key tile j of the item, K or V of KV head kvh, into this warp's stage
    auto load_kv = [&](const ItemU& g, int kvh, int j, bool isV) -> bool {
      const int fill = isV ? vfill : kfill;
      uint64_t* full = isV ? &v_full[mine] : &k_full[mine];
      uint64_t* empty = isV ? &v_empty[mine] : &k_empty[mine];
      uint8_t* dst = (isV ? sV : sK) + mine * TILE_BYTES;
      const int gj = g.jb + j;
      const bool paged = gj < g.npt;
      const int npg = (gj * kTileN + kPage < g.prefix_len + (p.resident ? max(g.winA, g.winB) : 0)) ? 2 : 1;
      int page[2] = {0, 0};
      if (paged) {
        // the window of 64 cached entries moves on once V has reached its second half
        if (isV && ((gj * 2) >> 5) >= pc_blk + 1) {
          pc_cur = pc_next; ++pc_blk;
          pc_next = load_pages(g.req, pc_blk + 1);
        }
#pragma unroll
        for (int pg = 0; pg < 2; ++pg) {
          const int pidx = gj * 2 + pg, blk = pidx >> 5;
          int v = __shfl_sync(0xffffffffu, blk == pc_blk ? pc_cur : pc_next, pidx & 31);
          if (blk != pc_blk && blk != pc_blk + 1)                  // outside the window (not expected)
            v = pidx < p.max_pages_per_req ? __ldg(&p.page_table[(size_t)g.req * p.max_pages_per_req + pidx]) : -1;
          page[pg] = pg < npg ? v : 0;
        }
      }
      if (fill > 0 && !warp_wait(empty, (fill - 1) & 1, abortf, LIM)) return false;
      if (paged) {
#pragma unroll
        for (int pg = 0; pg < 2; ++pg) {
          if (page[pg] < 0 || page[pg] >= p.num_pages) { if (leader) atomicOr(p.status, FB_ST_BAD_PAGE); page[pg] = 0; }
        }
        if (leader) {
          mbar_arrive_expect_tx(full, npg * PAGE_BYTES);
          for (int pg = 0; pg < npg; ++pg) {
            const int y = (page[pg] * p.n_kv_heads + kvh) * kPage;
            for (int h = 0; h < NHKV; ++h)
              tma_load_2d(dst + h * 16384 + pg * 8192, isV ? &tmVpool : &tmKpool, full, h * 64, y);
          }
        }
      } else if (leader) {
        mbar_arrive_expect_tx(full, TILE_BYTES);
        const int row0 = g.win_row0 + (gj - g.npt) * kTileN;
        for (int h = 0; h < NH; ++h)
          tma_load_3d(dst + h * 16384, isV ? &tmVwin : &tmKwin, full, h * 64, kvh, row0);
      }
      __syncwarp();
      if (isV) ++vfill; else ++kfill;
      return true;
    };
    // Work items are handed out in the list's order through a global ticket; warp 0
    // draws the ticket and publishes the item to the other roles.
    for (int k = 0; ok; ++k) {
      ItemU g;
      bool more;
      if (warp == 0) {
        if (k >= 2 && !warp_wait(&item_empty[k & 1], ((k >> 1) - 1) & 1, abortf, LIM)) { ok = false; break; }
        int idx = blockIdx.x;        // the first round needs no ticket
        if (k > 0) {
          if (lane == 0) idx = gridDim.x + atomicAdd(&p.hdr->ticket, 1);
          idx = uni(idx);
        }
        // the record goes to shared memory: the other roles would each pay two dependent
        // global loads (~1300 cycles per item) for it
        more = publish_item(p, idx, &p.hdr->n_items, s_item + (k & 1) * kItemWords, lane, [&](int req, int jb) {
          pc_blk = (jb * 2) >> 5;
          pc_cur = load_pages(req, pc_blk);
          pc_next = load_pages(req, pc_blk + 1);
        });
        if (lane == 0) mbar_arrive(&item_full[k & 1]);
        load_item_uniform(s_item + (k & 1) * kItemWords, p, g);
        __syncwarp();
        if (!more) break;
      } else {
        if (!warp_wait(&item_full[k & 1], (k >> 1) & 1, abortf, LIM)) { ok = false; break; }
        more = load_item_uniform(s_item + (k & 1) * kItemWords, p, g);
        __syncwarp();
        if (lane == 0) mbar_arrive(&item_empty[k & 1]);
        if (!more) break;
        pc_blk = (g.jb * 2) >> 5;
        pc_cur = load_pages(g.req, pc_blk);
        pc_next = load_pages(g.req, pc_blk + 1);
      }
      if (g.n <= 0) continue;
      if (warp == 0) {
        if (q_uses > 0 && !warp_wait(q_empty, (q_uses - 1) & 1, abortf, LIM)) { ok = false; break; }
        ++q_uses;
        if (leader) {
          mbar_arrive_expect_tx(q_full, ((g.nA > 0) + (g.nB > 0)) * Q_TILE_BYTES);
          if (g.nA > 0)
            for (int h = 0; h < NH; ++h)
              tma_load_3d(sQ + h * 16384, &tmQ, q_full, h * 64, g.kvhA * p.group, g.rowA);
          if (g.nB > 0)
            for (int h = 0; h < NH; ++h)
              tma_load_3d(sQ + Q_TILE_BYTES + h * 16384, &tmQ, q_full, h * 64, g.kvhB * p.group, g.rowB);
        }
        __syncwarp();
      }
      if (!g.dual()) {
        // K runs one tile ahead of V; this warp takes the tiles that fall on its stage
        if ((rr_k++ & 1) == mine && !load_kv(g, g.kvhA, 0, false)) { ok = false; break; }
        for (int j = 0; j < g.n; ++j) {
          if (j + 1 < g.n && (rr_k++ & 1) == mine && !load_kv(g, g.kvhA, j + 1, false)) { ok = false; break; }
          if ((rr_v++ & 1) == mine && !load_kv(g, g.kvhA, j, true)) { ok = false; break; }
        }
      } else {
        const int kvh = mine ? g.kvhB : g.kvhA;
        if (!load_kv(g, kvh, 0, false)) { ok = false; break; }
        for (int j = 0; j < g.n; ++j) {
          if (!load_kv(g, kvh, j, true)) { ok = false; break; }
          if (j + 1 < g.n && !load_kv(g, kvh, j + 1, false)) { ok = false; break; }
        }
      }
    }
    // The last CTA to draw its last ticket re-arms the counter, so that the same work list can be
    // run again (also after a launch that gave up half way through its items).
    if (warp == 0 && lane == 0 && atomicAdd(&p.hdr->done, 1) == (int)gridDim.x - 1) { p.hdr->ticket = 0; p.hdr->done = 0; }
  } else if (warp == 1) {
    // ---------------------------------------------------------- MMA issuer
    // The tensor pipe takes 64 cycles per MMA and queues about 250 cycles of work behind the
    // issuing thread.  The K and V waits of a key tile come before the wait for P, which is
    // the last thing to arrive: behind it they would sit in the S -> P -> P V -> next S chain
    // that bounds a tile (measured: +3 to 5 % on the whole kernel).
    const bool leader = elect_one();
    int q_cnt = 0, q8A = 0, q8B = 0, cntPA = 0, cntPB = 0;
    bool ok = LIM >= 0;
    if (!ok) *abortf = 1;
    auto wait = [&](uint64_t* bar, uint32_t parity) { return warp_wait_ready(bar, parity, abortf, LIM); };
    // All descriptors are built once; a k-step only adds a constant to the
    // address field (low word, no carry: shared-memory addresses fit the
    // 14-bit field).
    const uint32_t idesc_pv = F8 ? umma_idesc_e4m3(128, D, 0, 1) : umma_idesc_bf16(128, D, 0, 1);
    const uint32_t idesc_qk_full = F8 ? umma_idesc_e4m3(128, kTileN, 0, 0) : umma_idesc_bf16(128, kTileN, 0, 0);
    constexpr int QOP_BYTES = F8 ? 16384 : Q_TILE_BYTES;       // the Q tile the MMAs read
    const uint64_t dQ0 = smem_desc_sw128(smem_u32(F8 ? sQ8 : sQ), 16, 1024);
    const uint64_t dK0 = smem_desc_sw128(smem_u32(sK), 16, 1024);
    const uint64_t dV0 = smem_desc_sw128(smem_u32(sV), 16384, 1024);
    // S_X = Q_X K^T over `ncols` keys of K stage `st`; X is 0 (tile A) or 1 (tile B)
    auto issue_qk = [&](const int X, int st, int ncols) {
      const uint32_t idesc = ncols == kTileN ? idesc_qk_full
                             : (F8 ? umma_idesc_e4m3(128, ncols, 0, 0) : umma_idesc_bf16(128, ncols, 0, 0));
      const uint64_t qa = dQ0 + (uint32_t)((X * QOP_BYTES) >> 4), kb = dK0 + (uint32_t)((st * TILE_BYTES) >> 4);
      const uint32_t d = tmem + X * 128;
      if (leader) {
#pragma unroll
        for (int ks = 0; ks < KSTEPS; ++ks) {          // 32 bytes of the 128-byte row per step
          const uint32_t off = ((ks >> 2) * 16384 + (ks & 3) * 32) >> 4;
          if (F8) umma_ss_f8(d, qa + off, kb + off, idesc, ks > 0 ? 1u : 0u);
          else umma_ss(d, qa + off, kb + off, idesc, ks > 0 ? 1u : 0u);
        }
        umma_commit(&s_full[X]);
      }
      __syncwarp();
    };
    // O_X (+)= P_X V over the first `nks` k-steps of V stage `st`; P_X is read from TMEM.  A step
    // is 16 keys (bf16) or 32 keys (E4M3): 8 TMEM columns of P and 2 KB / 4 KB of V rows.
    constexpr int PV_STEPS = F8 ? 4 : 8, PV_STEP_BYTES = F8 ? 4096 : 2048;
    auto issue_pv = [&](const int X, int st, int nks, bool acc) {
      const uint64_t vb = dV0 + (uint32_t)((st * TILE_BYTES) >> 4);
      const uint32_t d = tmem + 256 + X * 128, a = tmem + X * 128 + P_COL;
      if (leader) {
#pragma unroll
        for (int ks = 0; ks < PV_STEPS; ++ks)
          if (ks < nks) {
            if (F8) umma_ts_f8(d, a + ks * 8, vb + (uint32_t)((ks * PV_STEP_BYTES) >> 4), idesc_pv, (acc || ks > 0) ? 1u : 0u);
            else umma_ts(d, a + ks * 8, vb + (uint32_t)((ks * PV_STEP_BYTES) >> 4), idesc_pv, (acc || ks > 0) ? 1u : 0u);
          }
      }
      __syncwarp();
    };
    // k-steps of P V that cover the first `lim` keys of a tile
    auto pv_steps = [&](int lim) { return F8 ? (lim + 31) >> 5 : round16(lim) >> 4; };
    auto commit = [&](uint64_t* bar) { if (leader) umma_commit(bar); __syncwarp(); };
    // fills consumed from each K / V stage (see the producer)
    int kuse0 = 0, kuse1 = 0, vuse0 = 0, vuse1 = 0, rr_k = 0, rr_v = 0;
    auto wait_k = [&](int st) -> bool {
      const int use = st ? kuse1 : kuse0;
      if (st) ++kuse1; else ++kuse0;
      return wait(&k_full[st], use & 1);
    };
    auto wait_v = [&](int st) -> bool {
      const int use = st ? vuse1 : vuse0;
      if (st) ++vuse1; else ++vuse0;
      return wait(&v_full[st], use & 1);
    };
    for (int k = 0; ok; ++k) {
      if (!wait(&item_full[k & 1], (k >> 1) & 1)) { ok = false; break; }
      ItemU g;
      const bool more = load_item_uniform(s_item + (k & 1) * kItemWords, p, g);
      __syncwarp();
      if (lane == 0) mbar_arrive(&item_empty[k & 1]);
      if (!more) break;
      if (g.n <= 0) continue;
      const int nA = g.nA, nB = g.nB, n = g.n;
      if (F8) {     // the tiles in E4M3, written by the softmax warps
        if (nA > 0 && !wait(&q8_full[0], q8A & 1)) { ok = false; break; }
        if (nB > 0 && !wait(&q8_full[1], q8B & 1)) { ok = false; break; }
        q8A += nA > 0; q8B += nB > 0;
        fence_proxy_async_smem();
      } else if (!wait(q_full, q_cnt & 1)) { ok = false; break; }
      ++q_cnt;
      if (!g.dual()) {
        // ---- tiles A and B share every K/V tile
        int st = rr_k++ & 1;
        if (!wait_k(st)) { ok = false; break; }
        tc_fence_after();
        if (nA > 0) issue_qk(0, st, round16(g.limit(0, g.winA, p.resident)));
        if (nB > 0) issue_qk(1, st, round16(g.limit(0, g.winB, p.resident)));
        commit(&k_empty[st]);
        if (n == 1) commit(q_empty);               // Q is free once its last QK has run
        for (int j = 0; j < n; ++j) {
          const int sv = rr_v++ & 1;
          const int st1 = rr_k & 1;                // stage of K(j+1), if there is one
          if (!wait_v(sv)) { ok = false; break; }
          // K(j+1) has normally landed by now: taking its barrier here keeps the wait
          // off the P V -> next Q K^T stretch that the softmax warps are waiting for
          if (j + 1 < n) { ++rr_k; if (!wait_k(st1)) { ok = false; break; } }
          // tile A: O_A += P_A(j) V(j), then S_A(j+1) so that softmax A can go on
          if (j < nA) {
            const int nks = pv_steps(g.limit(j, g.winA, p.resident));
            if (!wait(&p_full[0], cntPA & 1)) { ok = false; break; }
            ++cntPA;
            tc_fence_after();
            issue_pv(0, sv, nks, j > 0);
          }
          if (j + 1 < nA) {
            tc_fence_after();
            issue_qk(0, st1, round16(g.limit(j + 1, g.winA, p.resident)));
          } else if (j + 1 == nA) {
            // its epilogue does not wait for tile B.  Call in us, waiting / not: one request of 64 tokens 10.0 / 9.5, 24
            // requests 161.3 / 159.7, 48 short ones 50.6 / 49.0, 8 requests in 8 bits 36.2 / 35.2.  (In the branch that
            // only the last key tile takes: a test of its own between P V and the next Q K^T costs 8-bit pages 1 % of
            // long items, 16 long contexts 1026 -> 1034 a step, here 1025.)
            commit(&o_full[0]);
          }
          // tile B
          if (j < nB) {
            const int nks = pv_steps(g.limit(j, g.winB, p.resident));
            if (!wait(&p_full[1], cntPB & 1)) { ok = false; break; }
            ++cntPB;
            tc_fence_after();
            issue_pv(1, sv, nks, j > 0);
          }
          commit(&v_empty[sv]);
          if (j + 1 < nB) {
            tc_fence_after();
            issue_qk(1, st1, round16(g.limit(j + 1, g.winB, p.resident)));
          } else if (j + 1 == nB) {
            commit(&o_full[1]);
          }
          if (j + 1 < n) {
            commit(&k_empty[st1]);
            if (j + 2 == n) commit(q_empty);
          }
        }
      } else {
        // ---- one Q tile under two KV heads: stream X owns K stage X and V stage X
        // (nA == nB == n, and both tiles see the same keys)
        if (!wait_k(0)) { ok = false; break; }
        tc_fence_after();
        issue_qk(0, 0, round16(g.limit(0, g.winA, p.resident)));
        commit(&k_empty[0]);
        if (!wait_k(1)) { ok = false; break; }
        tc_fence_after();
        issue_qk(1, 1, round16(g.limit(0, g.winB, p.resident)));
        commit(&k_empty[1]);
        if (n == 1) commit(q_empty);
        // The streams do not depend on each other but run alike: taken in turn.  (Serving whichever
        // tile's P is ready first means polling.)
        for (int j = 0; j < n && ok; ++j) {
#pragma unroll 1
          for (int X = 0; X < 2; ++X) {
            if (!wait_v(X)) { ok = false; break; }
            if (!wait(&p_full[X], (X ? cntPB : cntPA) & 1)) { ok = false; break; }
            if (X) ++cntPB; else ++cntPA;
            tc_fence_after();
            issue_pv(X, X, pv_steps(g.limit(j, g.winA, p.resident)), j > 0);
            commit(&v_empty[X]);
            if (j + 1 < n) {
              // this stream's next K tile could only be requested when its last Q K^T had
              // finished, one softmax ago: give it the time of the P V as well
              if (!wait_k(X)) { ok = false; break; }
              tc_fence_after();
              issue_qk(X, X, round16(g.limit(j + 1, g.winA, p.resident)));
              commit(&k_empty[X]);
              if (j + 2 == n && X == 1) commit(q_empty);
            } else {
              commit(&o_full[X]);
            }
          }
        }
      }
    }
  }
  } else {
    // ------------------------------------------------- softmax + epilogue
    // Four warps per Q tile, one thread per query row (its TMEM lane).  Every wait is
    // taken by the whole warp with one outcome (warp_wait): tcgen05.ld / st below are
    // warp-wide and must never run with part of a warp gone.
    asm volatile("setmaxnreg.inc.sync.aligned.u32 200;");
    const int X = (warp - 4) >> 2;                 // 0: tile A, 1: tile B
    const int quad = warp & 3;                     // TMEM lane quadrant of this warp
    const int row = quad * 32 + lane;              // query row of the tile
    const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
    const uint32_t tS = tmem + lane_base + X * 128;
    const uint32_t tO = tmem + lane_base + 256 + X * 128;
    float sl2 = p.scale_log2;          // F8: per item and row (K scale of the KV head, Q scale of the row)
    float out_scale = 1.0f;            // F8: V scale of the KV head
    constexpr float kShift = F8 ? kF8PShift : 0.f;
    int cntS = 0, cntO = 0, qcnt = 0;
    bool ok = LIM >= 0;
    if (!ok) *abortf = 1;
    for (int k = 0; ok; ++k) {
      if (!warp_wait_ready(&item_full[k & 1], (k >> 1) & 1, abortf, LIM)) { ok = false; break; }
      // The record stays in shared memory until this warp is done with the item and is read
      // where it is needed: its words would only take registers from the key loop.
      const volatile int* rec = s_item + (k & 1) * kItemWords;
      auto release = [&]() { __syncwarp(); if (lane == 0) mbar_arrive(&item_empty[k & 1]); };
      if (!rec[kRecMore]) { release(); break; }
      // key tiles this item has for tile X, and for both (none: the item is passed over by all roles)
      const int slotB = rec[kRecSlot + 1], span = rec[kRecJe];
      const int nA = max(0, min(span, rec[kRecNvis]) - rec[kRecJb]);
      const int nB = slotB >= 0 ? max(0, min(span, rec[kRecNvis + 1]) - rec[kRecJb]) : 0;
      const int nMine = X == 0 ? nA : nB;
      const int q_par = qcnt & 1;        // phase of q_full that carries this item's Q tiles
      if (max(nA, nB) > 0) ++qcnt;
      if (nMine == 0) { release(); continue; }
      if constexpr (F8) {
        // This thread's Q row, bf16 -> E4M3 with the power of two that brings its largest
        // magnitude into [128, 256) (exact), into the tile the MMAs read.  The 128-byte swizzle
        // puts 16-byte piece c of row r at piece c ^ (r & 7) of its 128-byte line.
        if (!warp_wait(q_full, q_par, abortf, LIM)) { ok = false; break; }
        const uint8_t* src = sQ + X * Q_TILE_BYTES + (row >> 3) * 1024 + (row & 7) * 128;
        uint4 qv[16];
#pragma unroll
        for (int c = 0; c < 16; ++c)
          qv[c] = *reinterpret_cast<const uint4*>(src + (c >> 3) * 16384 + (((c & 7) ^ (row & 7)) << 4));
        uint32_t am = 0;                 // largest |x| as bf16 bits (sign cleared: integer order = magnitude order)
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const uint32_t w[4] = {qv[c].x, qv[c].y, qv[c].z, qv[c].w};
#pragma unroll
          for (int i = 0; i < 4; ++i) am = max(am, max(w[i] & 0x7fffu, (w[i] >> 16) & 0x7fffu));
        }
        int kq = 134 - (int)(am >> 7);   // biased exponent of the bf16 -> 2^kq * amax in [128, 256)
        kq = am < 0x80u ? 0 : min(max(kq, -100), 100);      // zero / subnormal rows: no scaling
        const float f = __int_as_float((kq + 127) << 23);
        uint8_t* dst = sQ8 + X * 16384 + (row >> 3) * 1024 + (row & 7) * 128;
#pragma unroll
        for (int c8 = 0; c8 < 8; ++c8) {
          const uint4 a = qv[2 * c8], b = qv[2 * c8 + 1];
          const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
          uint32_t o[4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            o[i] = pack_e4m3x4(__uint_as_float(w[2 * i] << 16) * f, __uint_as_float(w[2 * i] & 0xffff0000u) * f,
                               __uint_as_float(w[2 * i + 1] << 16) * f, __uint_as_float(w[2 * i + 1] & 0xffff0000u) * f);
          *reinterpret_cast<uint4*>(dst + ((c8 ^ (row & 7)) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
        }
        fence_proxy_async_smem();
        mbar_arrive(&q8_full[X]);
        const int kvh = (rec[kRecKvh] >> (16 * X)) & 0xffff;
        sl2 = p.scale_log2 * __ldg(&p.k_scale[kvh]) * __int_as_float((127 - kq) << 23);
        out_scale = __ldg(&p.v_scale[kvh]);
      }
      float m_ref = -INFINITY, l = 0.f;
      for (int j = 0; j < nMine;) {
        // Tiles [j, full_end) are full: the whole prefix but its last tile, whole tiles of the window.
        // They run in a loop of their own, without a call or a limit in it.
        const int jb = rec[kRecJb], npt = rec[kRecNpt], winX = rec[kRecWin + X], prefix = rec[kRecPrefix] + (p.resident ? winX : 0);
        const int full_end = min(nMine, (jb + j < npt ? prefix / kTileN : npt + winX / kTileN) - jb);
        bool redo = false, grow = false;
        for (; j < full_end; ++j) {
          if (!warp_wait_ready(&s_full[X], cntS & 1, abortf, LIM)) { ok = false; break; }
          ++cntS;
          tc_fence_after();
          // The whole row of S is read at once and the exponentials are taken against the running
          // reference m_ref, which is only re-based when they grow past 2^8 (lazy rescale), so the
          // common tile needs no separate max pass; the first tile of an item has no reference
          // yet and takes one.  P goes over the last columns of S while the sum is still being
          // formed: what it overwrites is kept in registers (s + P_COL) and the rest stays in
          // TMEM, so the rare tile that has to be redone can be, and the check costs nothing on
          // the way to the hand-off.
          uint32_t s[128], pk[32];
          tmem_ld32(tS, s); tmem_ld32(tS + 32, s + 32); tmem_ld32(tS + 64, s + 64); tmem_ld32(tS + 96, s + 96);
          tmem_ld_wait();
          if (j == 0) m_ref = max_cols<128>(s);
          const float mb = m_ref * sl2 - kShift;
          float tile_sum, most;
          if constexpr (F8) {
            tile_sum = exp_cols<true, 128>(s, pk, sl2, mb, most);
            tmem_st32(tS + P_COL, pk);
            grow = !(most <= kGrowSum);
          } else {
            uint32_t pk2[32];
            tile_sum = exp_cols<false, 64>(s, pk, sl2, mb, most);
            tmem_st32(tS + P_COL, pk);
            tile_sum += exp_cols<false, 64>(s + 64, pk2, sl2, mb, most);
            tmem_st32(tS + P_COL + 32, pk2);
            grow = !(tile_sum <= kGrowSum);
          }
          tmem_st_wait();
          if (__any_sync(0xffffffffu, grow)) {
            // rare: put S back as it was and take the tile again, re-based
#pragma unroll
            for (int c = P_COL; c < 128; c += 32) tmem_st32(tS + c, s + c);
            tmem_st_wait();
            redo = true;
            break;
          }
          l += tile_sum;
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&p_full[X]);
        }
        if (!ok || j >= nMine) break;
        // a ragged tile, or one that has to be taken again
        if (!redo) {
          if (!warp_wait_ready(&s_full[X], cntS & 1, abortf, LIM)) { ok = false; break; }
          ++cntS;
          tc_fence_after();
        }
        const int jj = rec[kRecJb] + j, np = rec[kRecNpt], wx = rec[kRecWin + X];
        const int limit = redo ? kTileN
                          : jj < np ? rec[kRecPrefix] + (p.resident ? wx : 0) - jj * kTileN : wx - (jj - np) * kTileN;
        const float2 r = tile_compact<D, F8>(tS, tO, min(limit, kTileN), j == 0, redo && grow, sl2, kShift, m_ref, l);
        l = r.x; m_ref = r.y;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_full[X]);
        ++j;
      }
      if (!ok) break;
      if (!warp_wait_ready(&o_full[X], cntO & 1, abortf, LIM)) { ok = false; break; }
      ++cntO;
      tc_fence_after();
      if (rec[kRecChunks] <= 1) {
        // 64 columns of the warp's 32 rows at a time through its staging area (swizzled like the
        // tiles: 16-byte piece c of row r at c ^ (r & 7)) and out as one box of whole lines.  Plain
        // stores from the lanes' rows kept the softmax warps for 4,000 cycles per item.
        const int row0 = quad * 32, kvh = (rec[kRecKvh] >> (16 * X)) & 0xffff;
        const int y = kvh * p.group + row0 % p.group, z = rec[kRecSlot + X] * p.bl + rec[kRecT0 + X] + row0 / p.group;
        uint8_t* stage = sOut + (warp - 4) * kStageBytes;
        const float inv = out_scale / l;
        // (a loop: straight code that runs once an item is bound by fetching its instructions.  Call in us, straight /
        // loop: 48 short requests 50.0 / 49.0, four KV heads 32.5 / 31.4; long items and single requests alike.)
#pragma unroll 1
        for (int h = 0; h < NH; ++h) {
          uint32_t o[64];
          tmem_ld32(tO + h * 64, o);
          tmem_ld32(tO + h * 64 + 32, o + 32);
          if (lane == 0) bulk_wait_read();           // the staging area's previous contents are out
          __syncwarp();
          tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            uint32_t v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
              v[i] = pack_bf16x2(__uint_as_float(o[8 * c + 2 * i]) * inv, __uint_as_float(o[8 * c + 2 * i + 1]) * inv);
            *reinterpret_cast<uint4*>(stage + lane * 128 + ((c ^ (lane & 7)) << 4)) = make_uint4(v[0], v[1], v[2], v[3]);
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) { tma_store_3d(&tmOut, stage, h * 64, y, z); bulk_commit(); }
        }
      } else {
        const size_t tile = (size_t)(rec[kRecPartBase] + rec[kRecChunk]) * 2 + X;
        // the reference the exponentials were taken against, and the sum (the merge divides by
        // it: the V scale goes in here)
        reinterpret_cast<float2*>(p.part_ml)[tile * kTileM + row] = make_float2(m_ref * sl2 - kShift, l / out_scale);
#pragma unroll 1
        for (int c = 0; c < D / 32; ++c) {
          uint32_t o[32];
          tmem_ld32(tO + c * 32, o);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 4; ++i) st_global_v8(part_o_at<D>(p.part_o, tile, row, 4 * c + i), o + 8 * i);
        }
      }
      tc_fence_before();
      release();
    }
    if (lane == 0) bulk_wait_done();
  }
  // ---------------------------------------------------------------- teardown
  tc_fence_before();
  __syncthreads();
  if (*abortf) {
    // A bounded wait gave up.  Nothing may still be running on this CTA's shared memory or
    // TMEM when they are handed on: (1) the MMA warp commits everything it has issued to a
    // barrier of its own and waits for it (bounded by a fixed number of polls: an MMA batch
    // takes microseconds); (2) bulk copies the producers have issued land within
    // microseconds as well, the CTA sleeps for 640 us before it leaves.
    if (tid == 0) atomicOr(p.status, FB_ST_DEV_TIMEOUT);
    if (warp == 1) {
      if (elect_one()) umma_commit(drain);
      __syncwarp();
      for (int i = 0; i < 4096 && !mbar_test(drain, 0); ++i) __nanosleep(200);
    }
    for (int i = 0; i < 64; ++i) __nanosleep(10000);
    __syncthreads();
  }
  if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem, 512); }
}

// Merge of the split-KV partials (deterministic: a fixed order of additions).  A warp takes 8
// columns of 32 / W rows; its lanes are W groups that share the pieces of a row (group g takes
// pieces g, g + W, ...), so that up to 4 W pieces are in flight together and every access is a run
// of at least 256 bytes.  Each lane carries a running maximum along, the groups meet by shuffles.
// A CTA keeps its rows and columns and goes over every G-th unit, picking the split ones 32 at a
// time; it returns at once when no unit was split.
// Bound by the partials' way through the L2 (12 to 19 MB written on one SM and read on another) and
// by the latency of a round of such loads, 2 to 3 us, so W grows with the longest split of the
// batch, up to the point where the CTAs no longer run together.  Attention call in us with W = 1 / 2 / 4,
// taken when ranges were cut for two items an SM: one request of 3,000 tokens (then 6 pieces a unit)
// 20.9 / 19.3 / 20.1, 28,000 tokens (12 pieces) 84 / 76 / 65, 8 requests (3 pieces, 40 units) 23.6 /
// 26.9 / 29; with a warp per row over a row-major layout these took 23.1, 97 and 26.4.  Of the calls with
// the split chosen by estimate (18.3, 55, 23.1; the first in 12 pieces a unit, W = 4) the merge is 6, 10
// and 6 us, an empty one 2.
constexpr int kCombineThreads = 256, kCombineCtasPerSm = 8, kCombineDepth = 4, kCombineMostCtas = 1024, kCombineMaxWays = 4;
template <int D>
__global__ void __launch_bounds__(kCombineThreads, 3) attn_combine_kernel(const AttnParams p) {
  // Not followed early: the row pass of a small batch, one wave of large CTAs, would be dealt to the
  // SMs unevenly around the merge's last CTAs (a step of 4 requests, 384 rows: 69.4 -> 62.7 us; 8
  // requests with four layers 170.0 -> 167.3; where nothing follows in one wave there is no difference).
  pdl_wait_only();
  // (the CTA-pair kernel's list: its ticket is re-armed here, for a further run of the same list)
  if (blockIdx.x == 0 && threadIdx.x == 0) p.hdr->ticket = 0;
  const int n_parts = p.hdr->n_parts, n_units = p.hdr->n_units, longest = p.hdr->max_chunks;
  if (n_parts == 0) return;
  int W = 1;
  while (W < kCombineMaxWays && W * kCombineDepth < longest && 2 * W * n_units * (D / 8) <= kCombineMostCtas) W *= 2;
  const int per_unit = W * (D / 8), G = gridDim.x / per_unit;           // (the grid is a multiple of 4 D / 8)
  const int sub = blockIdx.x % per_unit, cols = sub % (D / 8);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rpw = 32 / W, way = lane / rpw;                             // rows per warp, this lane's group
  const int first_row = ((sub / (D / 8)) * 8 + warp) * rpw;             // of the unit's 256
  const int X = first_row >= kTileM, row = first_row % kTileM + lane % rpw;
  for (int u0 = blockIdx.x / per_unit; u0 < n_units; u0 += 32 * G) {
    // lane i holds what matters of the i-th of the CTA's next 32 units
    const int mine = u0 + lane * G;
    int u_slot = -1, u_kvh = 0, u_t0 = 0, u_nt = 1, u_nch = 0, u_nvis = 0, u_part = 0;
    if (mine < n_units) {
      const int4* up = reinterpret_cast<const int4*>(&p.units[mine]);
      const int4 a = up[0], b = up[1], c = up[2];
      u_slot = X == 0 ? a.z : a.w; u_kvh = X == 0 ? a.y & 0xffff : a.y >> 16;
      u_t0 = X == 0 ? b.x : b.y; u_nt = b.z; u_nch = b.w;
      u_nvis = X == 0 ? c.x : c.y; u_part = c.z;
    }
    unsigned todo = __ballot_sync(0xffffffffu, u_nch > 1 && u_slot >= 0);
    for (; todo; todo &= todo - 1) {
      const int src = __ffs(todo) - 1;
      const int slot = __shfl_sync(0xffffffffu, u_slot, src), kvh = __shfl_sync(0xffffffffu, u_kvh, src);
      const int t0 = __shfl_sync(0xffffffffu, u_t0, src), nt = __shfl_sync(0xffffffffu, u_nt, src);
      const int nch = __shfl_sync(0xffffffffu, u_nch, src), nvis = __shfl_sync(0xffffffffu, u_nvis, src);
      const int part_base = __shfl_sync(0xffffffffu, u_part, src);
      // chunks that hold keys visible to this tile: those that start before tile nvis
      const int nc = min(nch, (int)(((long long)nvis * nch + nt - 1) / nt));
      const size_t tile0 = (size_t)part_base * 2 + X;                 // chunk c: + 2 c
      const float2* ml = reinterpret_cast<const float2*>(p.part_ml) + tile0 * kTileM + row;
      float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      float M = -INFINITY, L = 0.f;
      for (int c0 = way; c0 < nc; c0 += kCombineDepth * W) {
        float2 w[kCombineDepth];
        float v[kCombineDepth][8];
#pragma unroll
        for (int k = 0; k < kCombineDepth; ++k) {
          const int c = c0 + k * W;
          w[k] = make_float2(-INFINITY, 0.f);
#pragma unroll
          for (int i = 0; i < 8; ++i) v[k][i] = 0.f;
          if (c < nc) {
            ld_global_v8(v[k], part_o_at<D>(p.part_o, tile0 + 2 * c, row, cols));
            w[k] = ml[(size_t)c * 2 * kTileM];
          }
        }
        float m = M;
#pragma unroll
        for (int k = 0; k < kCombineDepth; ++k) m = fmaxf(m, w[k].x);
        const float f = M == -INFINITY ? 0.f : ex2_approx(M - m);
        M = m;
        L *= f;
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] *= f;
#pragma unroll
        for (int k = 0; k < kCombineDepth; ++k) {
          const float wk = ex2_approx(w[k].x - M);                      // a piece that is not there: 2^-inf = 0
          L += wk * w[k].y;
#pragma unroll
          for (int i = 0; i < 8; ++i) acc[i] += wk * v[k][i];
        }
      }
      for (int o = rpw; o < 32; o <<= 1) {
        const float m2 = __shfl_xor_sync(0xffffffffu, M, o), m = fmaxf(M, m2);   // group 0 holds piece 0: finite in pairs with it
        const float f = M == -INFINITY ? 0.f : ex2_approx(M - m), f2 = m2 == -INFINITY ? 0.f : ex2_approx(m2 - m);
        M = m;
        L = L * f + __shfl_xor_sync(0xffffffffu, L, o) * f2;
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] = acc[i] * f + __shfl_xor_sync(0xffffffffu, acc[i], o) * f2;
      }
      if (way == 0) {
        const float inv = 1.0f / L;
        const int grow_ = slot * p.bl + t0 + row / p.group;
        const int head = kvh * p.group + row % p.group;
        *reinterpret_cast<uint4*>(p.out + ((size_t)grow_ * p.n_q_heads + head) * D + cols * 8) =
            make_uint4(pack_bf16x2(acc[0] * inv, acc[1] * inv), pack_bf16x2(acc[2] * inv, acc[3] * inv),
                       pack_bf16x2(acc[4] * inv, acc[5] * inv), pack_bf16x2(acc[6] * inv, acc[7] * inv));
      }
    }
  }
}

// ------------------------------------------------------------------- host
int ensure_device(fb_ctx* ctx) {
  int dev = 0;
  if (int e = cuda_err(ctx, cudaGetDevice(&dev), "cudaGetDevice")) return e;
  if (ctx->dev_ready && ctx->device == dev) return FB_OK;
  // first use, or the caller moved the context to another device: set up again there and
  // forget the cached tensor maps
  ctx->dev_ready = false;
  for (auto& mp : ctx->map_ptrs) mp = nullptr;
  // (two attributes, not cudaGetDeviceProperties, which takes milliseconds: this is on the path of
  // a new context's first step)
  int major = 0, sms = 0;
  if (int e = cuda_err(ctx, cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev), "cudaDeviceGetAttribute")) return e;
  if (int e = cuda_err(ctx, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "cudaDeviceGetAttribute")) return e;
  if (major != 10) return set_err(ctx, FB_ERR_UNSUPPORTED, "the attention kernel needs an sm_100 device");
  ctx->num_sms = sms;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (int e = cuda_err(ctx, cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q),
                       "cudaGetDriverEntryPoint"))
    return e;
  if (!fn || q != cudaDriverEntryPointSuccess)
    return set_err(ctx, FB_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
  ctx->encode_fn = fn;
  const int smem64 = kSmem64, smem128 = kSmem128;
  if (int e = cuda_err(ctx, cudaFuncSetAttribute(wavefront_attn_kernel<64, false>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, smem64), "smem attr"))
    return e;
  if (int e = cuda_err(ctx, cudaFuncSetAttribute(wavefront_attn_kernel<128, false>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, smem128), "smem attr"))
    return e;
  if (int e = cuda_err(ctx, cudaFuncSetAttribute(wavefront_attn_kernel<128, true>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemF8), "smem attr"))
    return e;
  if (int e = lm_head_device_setup(ctx)) return e;
  if (int e = attn_pair_device_setup(ctx)) return e;
  ctx->device = dev;
  ctx->dev_ready = true;
  return FB_OK;
}

static int encode(fb_ctx* ctx, CUtensorMap* m, const void* base, int rank, const cuuint64_t* dims,
                  const cuuint64_t* strides, const cuuint32_t* box,
                  CUtensorMapDataType dtype = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16) {
  cuuint32_t es[3] = {1, 1, 1};
  auto fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled>(ctx->encode_fn);
  CUresult r = fn(m, dtype, rank, const_cast<void*>(base), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return set_err(ctx, FB_ERR_CUDA, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
  return FB_OK;
}

void fill_attn_params(fb_ctx* ctx, AttnParams& p, const int32_t* page_table, void* out, void* ws, int32_t* status,
                      int list) {
  const fb_config& c = ctx->cfg;
  uint8_t* w = static_cast<uint8_t*>(ws);
  p.hdr = reinterpret_cast<SchedHeader*>(w + ctx->ws.l[list].header);
  p.items = reinterpret_cast<const AttnItem*>(w + ctx->ws.l[list].items);
  p.units = reinterpret_cast<const AttnUnit*>(w + ctx->ws.l[list].units);
  p.page_table = page_table;
  p.out = static_cast<__nv_bfloat16*>(out);
  p.part_ml = reinterpret_cast<float*>(w + ctx->ws.l[list].part_ml);
  p.part_o = reinterpret_cast<float*>(w + ctx->ws.l[list].part_o);
  p.max_items = ctx->ws.l[list].max_items; p.max_units = ctx->ws.l[list].max_units;
  p.status = status;
  p.bl = c.block_len; p.n_q_heads = c.n_q_heads; p.n_kv_heads = c.n_kv_heads; p.group = ctx->group;
  p.max_pages_per_req = c.max_pages_per_req; p.num_pages = c.num_pages;
  p.resident = c.window_in_pages;
  p.k_scale = nullptr; p.v_scale = nullptr;
  p.scale_log2 = ctx->sm_scale * kLog2eF;
  p.wait_cycles = ctx->wait_cycles;
}

int launch_attn_combine(fb_ctx* ctx, const AttnParams& p, int list, cudaStream_t stream) {
  if (list == 0 && ctx->ws.l[0].max_parts == 0) return FB_OK;      // this context never splits a key range
  const int per_unit = kCombineMaxWays * ctx->cfg.head_dim / 8;
  const int groups = max(1, min(ctx->ws.l[list].max_units, kCombineCtasPerSm * ctx->num_sms / per_unit));
  if (ctx->cfg.head_dim == 64)
    return cuda_err(ctx, launch_pdl(attn_combine_kernel<64>, groups * per_unit, kCombineThreads, 0, stream, p),
                    "attn_combine_kernel launch");
  return cuda_err(ctx, launch_pdl(attn_combine_kernel<128>, groups * per_unit, kCombineThreads, 0, stream, p),
                  "attn_combine_kernel launch");
}

// q and out have one shape; Q is loaded as whole tiles, the output leaves 32 rows at a time
static int encode_q_out(fb_ctx* ctx, const void* q, const void* out) {
  const fb_config& c = ctx->cfg;
  const cuuint64_t rows = (cuuint64_t)c.max_requests * c.wmax * c.block_len, D = c.head_dim;
  cuuint64_t dims[3] = {D, (cuuint64_t)c.n_q_heads, rows};
  cuuint64_t str[2] = {D * 2, (cuuint64_t)c.n_q_heads * D * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)ctx->group, (cuuint32_t)ctx->tokens_per_tile};
  if (int e = encode(ctx, &ctx->tm_q, q, 3, dims, str, box)) return e;
  cuuint32_t obox[3] = {64, (cuuint32_t)(ctx->group < 32 ? ctx->group : 32), (cuuint32_t)(ctx->group < 32 ? 32 / ctx->group : 1)};
  return encode(ctx, &ctx->tm_out, out, 3, dims, str, obox);
}

int launch_attn(fb_ctx* ctx, const fb_pack* pk, const void* q, const void* k_win, const void* v_win,
                const void* k_pool, const void* v_pool, const int32_t* page_table, void* out, void* ws,
                int32_t* status, cudaStream_t stream) {
  (void)pk;
  if (int e = ensure_device(ctx)) return e;
  const fb_config& c = ctx->cfg;
  const cuuint64_t rows = (cuuint64_t)c.max_requests * c.wmax * c.block_len;
  const cuuint64_t D = c.head_dim;
  const void* ptrs[6] = {q, k_win, v_win, k_pool, v_pool, out};
  if (ctx->maps_f8 || memcmp(ptrs, ctx->map_ptrs, sizeof(ptrs)) != 0) {
    if (int e = encode_q_out(ctx, q, out)) return e;
    {
      cuuint64_t dims[3] = {D, (cuuint64_t)c.n_kv_heads, rows};
      cuuint64_t str[2] = {D * 2, (cuuint64_t)c.n_kv_heads * D * 2};
      cuuint32_t box[3] = {64, 1, 128};
      // window resident in the pages: no window tensors; the two maps are never used then
      if (int e = encode(ctx, &ctx->tm_kwin, k_win ? k_win : k_pool, 3, dims, str, box)) return e;
      if (int e = encode(ctx, &ctx->tm_vwin, v_win ? v_win : v_pool, 3, dims, str, box)) return e;
      cuuint32_t half[3] = {64, 1, 64};       // the CTA-pair kernel: each CTA takes 64 of a tile's 128 window keys
      if (int e = encode(ctx, &ctx->tm_kwin_half, k_win ? k_win : k_pool, 3, dims, str, half)) return e;
    }
    {
      cuuint64_t dims[2] = {D, (cuuint64_t)c.num_pages * c.n_kv_heads * kPage};
      cuuint64_t str[1] = {D * 2};
      cuuint32_t box[2] = {64, 64};
      if (int e = encode(ctx, &ctx->tm_kpool, k_pool, 2, dims, str, box)) return e;
      if (int e = encode(ctx, &ctx->tm_vpool, v_pool, 2, dims, str, box)) return e;
    }
    memcpy(ctx->map_ptrs, ptrs, sizeof(ptrs));
    ctx->maps_f8 = false;
  }
  AttnParams p;
  fill_attn_params(ctx, p, page_table, out, ws, status, 0);
  const int grid = ctx->num_sms;
  if (c.head_dim == 64) {
    if (int e = cuda_err(ctx, launch_pdl(wavefront_attn_kernel<64, false>, grid, kAttnThreads, kSmem64, stream, ctx->tm_q,
                                         ctx->tm_kwin, ctx->tm_vwin, ctx->tm_kpool, ctx->tm_vpool, ctx->tm_out, p),
                         "wavefront_attn_kernel launch"))
      return e;
    return launch_attn_combine(ctx, p, 0, stream);
  }
  // quads first (the CTA-pair kernel), then everything else
  if (ctx->pair_on)
    if (int e = launch_attn_pair(ctx, page_table, out, ws, status, stream)) return e;
  if (int e = cuda_err(ctx, launch_pdl(wavefront_attn_kernel<128, false>, grid, kAttnThreads, kSmem128, stream, ctx->tm_q,
                                       ctx->tm_kwin, ctx->tm_vwin, ctx->tm_kpool, ctx->tm_vpool, ctx->tm_out, p),
                       "wavefront_attn_kernel launch"))
    return e;
  return launch_attn_combine(ctx, p, 0, stream);
}

// Attention over 8-bit pages (window resident in the pages, head_dim 128): the pools are E4M3
// bytes, one (page, KV head) is a 64 x 128-byte tile = one TMA box.
int launch_attn_fp8(fb_ctx* ctx, const fb_pack* pk, const void* q, const void* k_pool8, const void* v_pool8,
                    const float* k_scale, const float* v_scale, const int32_t* page_table, void* out, void* ws,
                    int32_t* status, cudaStream_t stream) {
  (void)pk;
  if (int e = ensure_device(ctx)) return e;
  const fb_config& c = ctx->cfg;
  const void* ptrs[6] = {q, nullptr, nullptr, k_pool8, v_pool8, out};
  if (!ctx->maps_f8 || memcmp(ptrs, ctx->map_ptrs, sizeof(ptrs)) != 0) {
    if (int e = encode_q_out(ctx, q, out)) return e;
    cuuint64_t dims[2] = {128, (cuuint64_t)c.num_pages * c.n_kv_heads * kPage};
    cuuint64_t str[1] = {128};
    cuuint32_t box[2] = {128, 64};
    if (int e = encode(ctx, &ctx->tm_kpool, k_pool8, 2, dims, str, box, CU_TENSOR_MAP_DATA_TYPE_UINT8)) return e;
    if (int e = encode(ctx, &ctx->tm_vpool, v_pool8, 2, dims, str, box, CU_TENSOR_MAP_DATA_TYPE_UINT8)) return e;
    ctx->tm_kwin = ctx->tm_kpool; ctx->tm_vwin = ctx->tm_vpool;        // never used: every key tile is a paged one
    memcpy(ctx->map_ptrs, ptrs, sizeof(ptrs));
    ctx->maps_f8 = true;
  }
  AttnParams p;
  fill_attn_params(ctx, p, page_table, out, ws, status, 0);
  p.k_scale = k_scale; p.v_scale = v_scale;
  if (int e = cuda_err(ctx, launch_pdl(wavefront_attn_kernel<128, true>, ctx->num_sms, kAttnThreads, (size_t)kSmemF8, stream,
                                       ctx->tm_q, ctx->tm_kwin, ctx->tm_vwin, ctx->tm_kpool, ctx->tm_vpool, ctx->tm_out, p),
                       "wavefront_attn_kernel (8-bit pages) launch"))
    return e;
  return launch_attn_combine(ctx, p, 0, stream);
}

}  // namespace fb
