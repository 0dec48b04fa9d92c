// fb_pack_wavefronts: Heterogeneous Wavefront Packing (Sec. 3.2, Eq. 4).
//
// One launch.  Blocks 0..nb-1 compact the live blocks of all decoding
// requests into slots and gather tokens / position ids; the last two blocks
// build the two attention work lists (units, key-axis chunks, longest first but for one request's few)
// from the same per-request state: list 0 for the one-CTA kernel, list 1 (four
// Q tiles of one request and KV head at a time) for the CTA-pair kernel.
// Everything is integer work on a few KB.
#include "fb_common.cuh"

namespace fb {

// Threads per block: bound by latency (dependent loads, block barriers), so small batches take small blocks
// (1024 threads do not fit their tables into static shared memory).  Call in us, back to back:
//   requests        1    2    4    8    9   16   24   32   64  128
//   128 threads   4.4  4.8  5.0  5.8
//   256           4.4  4.7  5.1  5.7  5.5  5.9  6.2  8.0  7.6 10.7
//   512           4.4  5.2  5.6  6.3  6.0  6.4  6.6  7.4  7.7 10.8
// The line lies at 8 because build_sched changes its way there: every warp for itself up to 8 requests, a thread a
// request above (16 requests 6.9 the first way, 6.4 the other; 24: 7.8, 6.6; 32: 10.6, 7.4).
constexpr int kPackThreads = 512, kPackThreadsSmall = 256, kPackSmallRequests = 8;
constexpr int kSlotsPerBlock = 32;
constexpr int kPackLongPages = 1 << 20;   // (kLong: with two pages a key tile, ranges stay below 2^20 key tiles here)
constexpr int kCostBins = 1024;
constexpr int kUnitInfo = 1024;       // units whose geometry stays in shared memory between the two passes over items

struct PackParams {
  const int32_t *active, *prefix_len, *L, *R, *tokens;
  int32_t *n_live, *slot_req, *slot_s, *slot_pos0, *slot_kv_len, *slot_flags, *req_slot_begin, *qtok, *pos;
  int32_t* status;
  SchedHeader* hdr[2];
  AttnItem* items[2];
  AttnUnit* units[2];
  int32_t max_items[2], max_units[2], max_parts[2], target_items[2];
  int32_t pair_on;
  int32_t max_requests, wmax, bl, max_slots, max_blocks, mask_id, n_kv_heads;
  int32_t tiles_per_slot, tokens_per_tile, min_chunk_tiles;
  int32_t auto_split, auto_min_chunk;
  int32_t resident;   // window K/V live in the pages: key tiles follow absolute positions
  int32_t n_gather_blocks;
};

// live-block count of request r, sanitised to [0, wmax]; the loads do not wait for one another
__device__ __forceinline__ int live_blocks(const PackParams& p, int r, int32_t* status) {
  const int active = p.active[r], L = p.L[r], R = p.R[r];
  if (active != 1) return 0;
  int w = R - L;
  if (L < 0 || R > p.max_blocks || w < 0 || w > p.wmax) {
    if (status) atomicOr(status, FB_ST_BAD_STATE);
    w = w < 0 ? 0 : (w > p.wmax ? p.wmax : w);
    if (L < 0 || L + w > p.max_blocks) w = 0;
  }
  return w;
}

// Exclusive block scan of N values per thread: excl = prefix, tot = block sum.  All threads must
// call; `sh` [N * T / 32] must not be in use by an earlier scan (one barrier inside).
template <int T, int N>
__device__ __forceinline__ void block_excl_scan(const int (&v)[N], int (&excl)[N], int (&tot)[N], int* sh) {
  constexpr int NW = T / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x[N];
#pragma unroll
  for (int n = 0; n < N; ++n) x[n] = v[n];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1)
#pragma unroll
    for (int n = 0; n < N; ++n) {
      const int y = __shfl_up_sync(0xffffffffu, x[n], o);
      if (lane >= o) x[n] += y;
    }
  if (lane == 31)
#pragma unroll
    for (int n = 0; n < N; ++n) sh[n * NW + warp] = x[n];
  __syncthreads();
#pragma unroll
  for (int n = 0; n < N; ++n) {
    int w = lane < NW ? sh[n * NW + lane] : 0;       // every warp scans the warp sums
#pragma unroll
    for (int o = 1; o < NW; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    tot[n] = __shfl_sync(0xffffffffu, w, NW - 1);
    const int before = __shfl_sync(0xffffffffu, w, warp == 0 ? 0 : warp - 1);
    excl[n] = x[n] - v[n] + (warp == 0 ? 0 : before);
  }
}

// Sort key of a work item: its key-tile iterations; an iteration with two Q
// tiles takes about 7/6 of one with a single tile (measured).
__device__ __forceinline__ int item_cost(int nA, int nB) {
  const int n = max(nA, nB), both = min(nA, nB);
  return (6 * n + both + 1) >> 1;
}

__device__ __forceinline__ ReqGeom geom_of(const PackParams& p, int w, int prefix_len, int list) {
  return req_geom_of(w, prefix_len, p.tiles_per_slot, p.bl, p.n_kv_heads, p.resident, list, p.pair_on);
}
__device__ __forceinline__ ReqGeom req_geom(const PackParams& p, int r, int list) {
  const int P = p.prefix_len[r];
  const int w = live_blocks(p, r, nullptr);      // (bad states are reported once, by the gather blocks)
  return geom_of(p, w, w ? P : 0, list);
}

// a / d for 0 <= a, 0 < d with a quotient below 2^20: a reciprocal (inv_of(d)) off by a few units in the last
// place puts the product within one of the quotient, the remainder says which way.  The list is built by
// chains of such quotients; a hardware-less integer division is four times as long.  Quotients that count key
// tiles may be larger where a page table reaches that far: there the estimate is off by several (up to four at
// 2^24), and kLong divides.  (Divided in here whenever the estimate is large, the code of the division alone
// costs ordinary lists 0.3 to 0.7 us; as a kernel of its own, nothing.)
__device__ __forceinline__ float inv_of(int d) { return __fdividef(1.0f, (float)d); }
template <bool kLong = false>
__device__ __forceinline__ int quot(int a, int d, float inv) {
  if (kLong) return a / d;
  const int q = (int)((float)a * inv), r = a - q * d;
  return q + (r >= d) - (r < 0);
}

// unit record of two Q tiles qa, qb (absolute tile indices of the request; qb < 0: none) under
// KV heads hA, hB
__device__ __forceinline__ AttnUnit make_unit(const PackParams& p, const ReqGeom& q, int req, int first, int qa, int qb,
                                              int hA, int hB, float inv_tps) {
  AttnUnit un;
  un.req = req;
  un.kvh = hA | (hB << 16);
  const int sA = quot(qa, p.tiles_per_slot, inv_tps);
  un.slotA = first + sA;
  un.t0A = (qa - sA * p.tiles_per_slot) * p.tokens_per_tile;
  un.winA = (sA + 1) * p.bl;
  un.nvisA = p.resident ? (q.P + un.winA + kTileN - 1) / kTileN : q.npt + (un.winA + kTileN - 1) / kTileN;
  if (qb >= 0) {
    const int sB = quot(qb, p.tiles_per_slot, inv_tps);
    un.slotB = first + sB;
    un.t0B = (qb - sB * p.tiles_per_slot) * p.tokens_per_tile;
    un.winB = (sB + 1) * p.bl;
    un.nvisB = p.resident ? (q.P + un.winB + kTileN - 1) / kTileN : q.npt + (un.winB + kTileN - 1) / kTileN;
  } else {
    un.slotB = -1; un.t0B = 0; un.winB = 0; un.nvisB = 0;
  }
  un.n_tiles = q.nt; un.n_chunks = 0; un.part_base = -1;
  un.prefix_len = q.P; un.npt = q.npt; un.win_row0 = first * p.bl;
  return un;
}

// `list` 0: pairs of tiles and leftover tiles, one record per scheduling unit.  `list` 1: quads,
// two records per scheduling unit (2u for the first CTA of the pair, 2u + 1 for the second), both
// cut into the same chunks; an item names record 2u.
//
// Bound by the chain of dependent steps in one block.  Up to kPackSmallRequests every warp holds all of them, a
// lane each, and forms sums, split and bases for itself, without a barrier; above, a thread holds a request.
// Call in us, back to back, before and with this, the quotients by reciprocal and the unit records in registers: one
// request of 3,000 tokens 5.7 / 4.0, 8 requests 6.0 / 5.2, 24 requests 7.4 / 6.4, 64 requests 9.3 / 7.6, in 8 bits
// 9.6 / 7.8, 128 requests 13.3 / 10.6, 600 requests 46 / 37.  Steps with the first two: a toy request 23.5 / 21.8, one
// request with four layers 105.8 / 102.4, a 28,000-token one 83.1 / 80.2.
template <int T, bool kLong>
__device__ void build_sched(const PackParams& p, const int list) {
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int NW = T / 32;
  const int mult = list + 1;            // unit records (and partial-result ranges) per scheduling unit
  SchedHeader* const hdr = p.hdr[list];
  AttnItem* const items = p.items[list];
  AttnUnit* const units = p.units[list];
  const int max_items = p.max_items[list], max_units = p.max_units[list], max_parts = p.max_parts[list];
  __shared__ int sh_scan[3 * NW], sh_scan2[NW], sh_scan3[NW];
  __shared__ int bins[kCostBins];
  __shared__ int sh_total, sh_units, sh_chunks, sh_longest;
  __shared__ SplitStat sh_stat[kSplitCandidates];
  static_assert(kSplitCandidates == 32, "one lane per candidate");
  __shared__ SplitRule sh_rule;
  __shared__ int s_ub[T], s_pb[T], s_first[T], s_wb[T], s_w[T], s_P[T];
  __shared__ int4 s_info[kUnitInfo];
  __shared__ int s_req[kUnitInfo];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float inv_tps = inv_of(p.tiles_per_slot);

  // Record of unit `ul` of a request of list 0.  Full pairs first, numbered h * nfull + pr: the pairs of one
  // (request, KV head) are adjacent, are handed out back to back and so share their K/V through L2.  Then the
  // leftover tile, one unit per two KV heads.
  auto unit_record = [&](const ReqGeom& q, int req, int first, int ul) {
    const bool full = ul < q.nfull * p.n_kv_heads;
    const int hf = q.nfull > 1 ? quot(ul, q.nfull, inv_of(q.nfull)) : ul;
    const int h = full ? hf : 2 * (ul - q.nfull * p.n_kv_heads);
    const int qa = q.tile0 + (full ? 2 * (ul - hf * q.nfull) : q.ntq - 1);
    const bool two = !full && h + 1 < p.n_kv_heads;
    return make_unit(p, q, req, first, qa, full ? qa + 1 : two ? qa : -1, h, two ? h + 1 : h, inv_tps);
  };
  // the last k < n with base[k] <= i (requests without units share their successor's base and are skipped by "last")
  auto owner = [](const int* base, int n, int i) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (base[mid] <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
  };
  // One request, no more items than SMs: its pieces are alike and each CTA gets one or none, so nothing is sorted.
  // (Not for several requests: with the longest pieces first, the two SMs of a pair get a long and a short one;
  // 8 requests with four layers 167 us a step sorted, 169 without.)  A unit's pieces side by side: with the same keys of
  // all units side by side instead, one request of 3,000 tokens and four layers takes 1 % longer.
  auto one_request = [&](const SplitRule& rule, int k, int n_items) {
    const ReqGeom q = geom_of(p, s_w[k], s_P[k], list);
    const int nc = req_split(rule, s_wb[k], q.nunits, q.nt).nch_c;
    const float inv = inv_of(max(nc, 1));
    for (int i = tid; i < n_items; i += T) {
      const int u = quot(i, nc, inv), c = i - u * nc;
      if (c == 0) {
        AttnUnit un = unit_record(q, k, s_first[k], u);
        un.n_chunks = nc;
        un.part_base = nc > 1 ? i : -1;
        units[u] = un;
      }
      AttnItem it; it.unit = u; it.chunk = c; it.jb = quot<kLong>(c * q.nt, nc, inv); it.je = quot<kLong>((c + 1) * q.nt, nc, inv);
      it.req = k; it.pad[0] = it.pad[1] = it.pad[2] = 0;
      items[i] = it;
    }
  };
  auto write_header = [&](int n_items, int unit_total, int part_total, int total_tiles, int ct, int most) {
    if (tid != 0) return;
    hdr->n_items = min(n_items, max_items);
    hdr->n_units = min(mult * unit_total, max_units);
    hdr->chunk_tiles = ct;
    hdr->n_parts = mult * part_total;
    hdr->total_tiles = total_tiles;
    hdr->ticket = 0; hdr->done = 0; hdr->max_chunks = most;
    if (n_items > max_items || mult * unit_total > max_units || mult * part_total > max_parts)
      atomicOr(p.status, FB_ST_BAD_STATE);
  };
  // The units of the `n` requests from r0 on, whose geometry and bases are in the tables: unit record, cost
  // histogram of its items.  A unit cut into many pieces is given to several threads.
  auto write_units = [&](const SplitRule& rule, int r0, int n, int tu, int unit_run, int most) {
    int shift = 0;
    while (shift < 5 && (1 << shift) < most && (tu << (shift + 1)) <= T) ++shift;
    for (int j = tid; j < tu << shift; j += T) {
      const int i = j >> shift, c0 = j & ((1 << shift) - 1);
      const int k = owner(s_ub, n, i), ul = i - s_ub[k];
      const int u = unit_run + i;
      if (mult * (u + 1) > max_units) continue;
      const ReqGeom q = geom_of(p, s_w[k], s_P[k], list);
      const ReqSplit qs = req_split(rule, s_wb[k], q.nunits, q.nt);
      const int first = s_first[k], nc = qs.chunks(ul);
      // (records in registers: an array of them indexed in a loop lives in local memory)
      AttnUnit un, un1;
      if (list == 0) {
        un = unit_record(q, r0 + k, first, ul);
      } else {
        // quad qd of KV head h: tiles 4 qd + r and 4 qd + 2 + r belong to CTA r of the pair
        const int h = ul / q.nquad, qd = ul % q.nquad;
        un = make_unit(p, q, r0 + k, first, 4 * qd, 4 * qd + 2, h, h, inv_tps);
        un1 = make_unit(p, q, r0 + k, first, 4 * qd + 1, 4 * qd + 3, h, h, inv_tps);
      }
      int nch = nc;
      const int pb = nc > 1 ? mult * (s_pb[k] + qs.part_off(ul)) : -1;
      // the workspace is sized for the bound on the split pieces (split_rule); a unit that
      // would still fall outside it is dropped and FB_ST_BAD_STATE is raised below
      if (nc > 1 && pb + mult * nc > max_parts) nch = 0;
      int nvA = un.nvisA, nvB = un.nvisB;
      un.n_chunks = nch;
      un.part_base = nc > 1 ? pb : -1;
      if (c0 == 0) units[mult * u] = un;
      if (list == 1) {
        un1.n_chunks = nch;
        un1.part_base = nc > 1 ? pb + nc : -1;
        if (c0 == 0) units[2 * u + 1] = un1;
        nvA = max(nvA, un1.nvisA); nvB = max(nvB, un1.nvisB);
      }
      if (c0 == 0 && u < kUnitInfo) { s_info[u] = make_int4(nvA, nvB, q.nt, nch); s_req[u] = r0 + k; }
      const float inv = inv_of(nc);
      for (int c = c0; c < nch; c += 1 << shift) {
        const int jb = quot<kLong>(c * q.nt, nc, inv), je = quot<kLong>((c + 1) * q.nt, nc, inv);
        const int cost = item_cost(max(0, min(je, nvA) - jb), max(0, min(je, nvB) - jb));
        atomicAdd(&bins[min(cost, kCostBins - 1)], 1);
      }
    }
  };
  // Behind the units: descending exclusive offsets over the cost bins (thread t owns the bins
  // kCostBins - 1 - kBinsPer * t and below: largest cost first), the header, the items, longest first.
  auto write_items = [&](int unit_total, int part_total, int total_tiles, int ct, int most) {
    constexpr int kBinsPer = kCostBins / T;
    static_assert(kBinsPer * T == kCostBins && kBinsPer >= 1, "whole bins per thread");
    int c[kBinsPer], sum = 0;
#pragma unroll
    for (int j = 0; j < kBinsPer; ++j) { c[j] = bins[kCostBins - 1 - (kBinsPer * tid + j)]; sum += c[j]; }
    int bpre[1], btot[1];
    block_excl_scan<T, 1>({sum}, bpre, btot, sh_scan3);
    int base = bpre[0];
    const int total_items = btot[0];
#pragma unroll
    for (int j = 0; j < kBinsPer; ++j) { bins[kCostBins - 1 - (kBinsPer * tid + j)] = base; base += c[j]; }
    write_header(total_items, unit_total, part_total, total_tiles, ct, most);
    __syncthreads();
    const int n_sched = min(unit_total, max_units / mult);
    int shift = 0;
    while (shift < 5 && (1 << shift) < most && (n_sched << (shift + 1)) <= T) ++shift;
    for (int j = tid; j < n_sched << shift; j += T) {
      const int u = j >> shift;
      int nvA, nvB, nt, nch, req;
      if (u < kUnitInfo) {
        req = s_req[u];
        const int4 f = s_info[u];
        nvA = f.x; nvB = f.y; nt = f.z; nch = f.w;
      } else {
        const AttnUnit un = units[mult * u];
        nvA = un.nvisA; nvB = un.nvisB; nt = un.n_tiles; nch = un.n_chunks; req = un.req;
        if (mult == 2) { const AttnUnit u1 = units[2 * u + 1]; nvA = max(nvA, u1.nvisA); nvB = max(nvB, u1.nvisB); }
      }
      const float inv = inv_of(max(nch, 1));
      for (int c = j & ((1 << shift) - 1); c < nch; c += 1 << shift) {
        const int jb = quot<kLong>(c * nt, nch, inv), je = quot<kLong>((c + 1) * nt, nch, inv);
        const int cost = item_cost(max(0, min(je, nvA) - jb), max(0, min(je, nvB) - jb));
        const int at = atomicAdd(&bins[min(cost, kCostBins - 1)], 1);
        if (at < max_items) {
          AttnItem it; it.unit = mult * u; it.chunk = c; it.jb = jb; it.je = je;
          it.req = req; it.pad[0] = it.pad[1] = it.pad[2] = 0;
          items[at] = it;
        }
      }
    }
  };
  auto most_chunks = [](const ReqSplit& sp, int nunits) {
    return nunits ? max(sp.ufine > 0 ? sp.nch_c : 0, sp.ufine < nunits ? sp.nch_f : 0) : 0;
  };
  // the candidate of this lane, and the best of all: the least (estimate, candidate)
  auto best_candidate = [&](const SplitStat& st, int ct) {
    const float e = lane > 0 && ct < p.auto_min_chunk ? -1.f : split_estimate(st, max_parts);
    // (non-negative floats order like their bits; nothing to do at all: candidate 0)
    const unsigned mine = e >= 0.f ? __float_as_uint(e) : 0xffffffffu, least = __reduce_min_sync(kAll, mine);
    return __shfl_sync(kAll, ct, __ffs(__ballot_sync(kAll, mine == least)) - 1);
  };
  auto add_request = [&](SplitStat& st, int nt, int pairs, int nunits, int ct, float inv_ct) {
    const int nch = quot(nt + ct - 1, ct, inv_ct), len = quot<kLong>(nt + nch - 1, nch, inv_of(nch));
    split_stat_add_pieces(st, nt, pairs, nunits, nch, len);
  };

  for (int i = tid; i < kCostBins; i += T) bins[i] = 0;
  if (p.max_requests <= kPackSmallRequests) {
    // ---- every warp for itself: lane r is request r
    const ReqGeom g = lane < p.max_requests ? req_geom(p, lane, list) : ReqGeom{};
    const int nunits = g.nt ? g.nunits : 0, pairs = g.nfull * p.n_kv_heads;
    const int total = __reduce_add_sync(kAll, nunits * g.nt), n_units = __reduce_add_sync(kAll, nunits);
    const int longest = __reduce_max_sync(kAll, g.nt);
    SplitRule rule;
    if (list == 0 && p.auto_split) {
      int chosen = max(longest, 1);
      if (split_worth_estimating(total, n_units, longest)) {
        const int ct = max(split_candidate(lane, longest), 1);
        const float inv_ct = inv_of(ct);
        SplitStat st{};
        for (unsigned todo = __ballot_sync(kAll, nunits > 0); todo; todo &= todo - 1) {
          const int r = __ffs(todo) - 1;
          add_request(st, __shfl_sync(kAll, g.nt, r), __shfl_sync(kAll, pairs, r), __shfl_sync(kAll, nunits, r), ct, inv_ct);
        }
        chosen = best_candidate(st, ct);
      }
      rule = split_auto(total, n_units, chosen, p.min_chunk_tiles);
    } else {
      rule = split_rule(total, n_units, p.target_items[list], p.min_chunk_tiles);
    }
    int v[3] = {nunits * g.nt, nunits, g.w}, x[3] = {v[0], v[1], v[2]};
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const int y = __shfl_up_sync(kAll, x[i], o);
        if (lane >= o) x[i] += y;
      }
    const ReqSplit sp = req_split(rule, x[0] - v[0], nunits, g.nt);
    const int parts = sp.parts(nunits), most = __reduce_max_sync(kAll, most_chunks(sp, nunits));
    const int n_items = __reduce_add_sync(kAll, sp.items(nunits));
    int xp = parts;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kAll, xp, o);
      if (lane >= o) xp += y;
    }
    if (warp == 0) {
      s_ub[lane] = x[1] - v[1]; s_pb[lane] = xp - parts; s_first[lane] = x[2] - v[2];
      s_wb[lane] = x[0] - v[0]; s_w[lane] = g.w; s_P[lane] = g.P;
    }
    const int part_total = __shfl_sync(kAll, xp, 31);
    __syncthreads();                    // the tables are there, the bins are clear
    const unsigned with_work = __ballot_sync(kAll, nunits > 0);
    if (list == 0 && __popc(with_work) == 1 && rule.fine_from == 0x7fffffff && n_items <= min(kSms, max_items) &&
        n_units <= max_units && part_total <= max_parts) {
      write_header(n_items, n_units, part_total, total, rule.ct, most);
      one_request(rule, __ffs(with_work) - 1, n_items);
      return;
    }
    write_units(rule, 0, p.max_requests, n_units, 0, most);
    __syncthreads();
    write_items(n_units, part_total, total, rule.ct, most);
    return;
  }
  // ---- a thread per request, T at a time
  if (tid == 0) { sh_total = 0; sh_units = 0; sh_chunks = 0; sh_longest = 0; }
  if (tid < kSplitCandidates) sh_stat[tid] = SplitStat{};
  // phase 1: total key-tile work, longest key range -> chunk length.  The requests' geometry is
  // loaded once where one pass over the requests holds all of them.
  const bool one_pass = p.max_requests <= T;
  ReqGeom g0{};
  int mine = 0, mine_units = 0, mine_longest = 0;
  for (int r = tid; r < p.max_requests; r += T) {
    const ReqGeom g = req_geom(p, r, list);
    mine += g.nunits * g.nt;
    mine_units += g.nt ? g.nunits : 0;
    mine_longest = max(mine_longest, g.nt);
    g0 = g;
  }
  s_w[tid] = g0.w; s_P[tid] = g0.P;
  mine = __reduce_add_sync(kAll, mine); mine_units = __reduce_add_sync(kAll, mine_units);
  mine_longest = __reduce_max_sync(kAll, mine_longest);
  __syncthreads();
  if (lane == 0 && mine_units) {
    atomicAdd(&sh_total, mine); atomicAdd(&sh_units, mine_units); atomicMax(&sh_longest, mine_longest);
  }
  __syncthreads();
  if (list == 0 && p.auto_split && !split_worth_estimating(sh_total, sh_units, sh_longest)) {
    if (tid == 0) sh_rule = split_auto(sh_total, sh_units, max(sh_longest, 1), p.min_chunk_tiles);
  } else if (list == 0 && p.auto_split) {
    // every lane a candidate chunk length, the requests dealt to the warps
    const int ct = max(split_candidate(lane, sh_longest), 1);
    const float inv_ct = inv_of(ct);
    SplitStat st{};
    for (int r = warp; r < p.max_requests; r += NW) {
      const ReqGeom g = one_pass ? geom_of(p, s_w[r], s_P[r], list) : req_geom(p, r, list);
      if (g.nt > 0) add_request(st, g.nt, g.nfull * p.n_kv_heads, g.nunits, ct, inv_ct);
    }
    if (st.items) {
      atomicAdd(&sh_stat[lane].work, st.work); atomicAdd(&sh_stat[lane].items, st.items);
      atomicAdd(&sh_stat[lane].parts, st.parts); atomicMax(&sh_stat[lane].longest, st.longest);
    }
    __syncthreads();
    if (tid < 32) {
      const int chosen = best_candidate(sh_stat[lane], ct);
      if (lane == 0) sh_rule = split_auto(sh_total, sh_units, chosen, p.min_chunk_tiles);
    }
  } else if (tid == 0) {
    sh_rule = split_rule(sh_total, sh_units, p.target_items[list], p.min_chunk_tiles);
  }
  __syncthreads();
  const SplitRule rule = sh_rule;
  // phase 2 + 3: per-request bases (scan over up to T requests at a time), then the units of
  // these requests
  int unit_run = 0, part_run = 0, slot_run = 0, work_run = 0;
  for (int r0 = 0; r0 < p.max_requests; r0 += T) {
    const int r = r0 + tid;
    ReqGeom g{};
    if (one_pass) g = g0;
    else if (r < p.max_requests) g = req_geom(p, r, list);
    const int nunits = g.nt ? g.nunits : 0;
    int pre[3], tot[3];
    block_excl_scan<T, 3>({nunits * g.nt, nunits, g.w}, pre, tot, sh_scan);
    const int wbase = work_run + pre[0];
    const ReqSplit rs = req_split(rule, wbase, nunits, g.nt);
    const int most = __reduce_max_sync(kAll, most_chunks(rs, nunits));
    if (lane == 0) atomicMax(&sh_chunks, most);
    int ppre[1], ptot[1];
    block_excl_scan<T, 1>({rs.parts(nunits)}, ppre, ptot, sh_scan2);
    s_ub[tid] = pre[1]; s_pb[tid] = part_run + ppre[0]; s_first[tid] = slot_run + pre[2]; s_wb[tid] = wbase;
    if (!one_pass) { s_w[tid] = g.w; s_P[tid] = g.P; }
    __syncthreads();
    write_units(rule, r0, min(T, p.max_requests - r0), tot[1], unit_run, sh_chunks);
    unit_run += tot[1]; part_run += ptot[0]; slot_run += tot[2]; work_run += tot[0];
    __syncthreads();                      // the tables are overwritten next
  }
  write_items(unit_run, part_run, sh_total, rule.ct, sh_chunks);
}

template <int T, bool kLong>
__global__ void __launch_bounds__(T) pack_kernel(const PackParams p) {
  // Not followed early: the attention's CTAs, which take an SM each, would move in while the list is
  // still being built.  Steps with and without that, in us: one request with four layers 105 -> 102,
  // 28,000 tokens 83 -> 81, 8 requests 79 -> 77.5, 24 requests 311.5 -> 308.5.
  pdl_wait_only();
  if ((int)blockIdx.x >= p.n_gather_blocks) { build_sched<T, kLong>(p, (int)blockIdx.x - p.n_gather_blocks); return; }
  __shared__ int sh_scan[T / 32];
  __shared__ int s_req[kSlotsPerBlock], s_idx[kSlotsPerBlock], s_w[kSlotsPerBlock];
  const int tid = threadIdx.x;
  const int slot0 = blockIdx.x * kSlotsPerBlock;
  if (tid < kSlotsPerBlock) s_req[tid] = -1;
  __syncthreads();
  int run = 0;
  for (int r0 = 0; r0 < p.max_requests; r0 += T) {
    const int r = r0 + tid;
    const int w = r < p.max_requests ? live_blocks(p, r, p.status) : 0;
    int pre[1], tot[1];
    if (r0) __syncthreads();              // the scan's scratch of the previous round has been read
    block_excl_scan<T, 1>({w}, pre, tot, sh_scan);
    const int begin = run + pre[0];
    run += tot[0];
    if (r < p.max_requests) {
      if (blockIdx.x == 0) p.req_slot_begin[r] = begin;
      for (int s = 0; s < w; ++s) {
        const int slot = begin + s;
        if (slot >= slot0 && slot < slot0 + kSlotsPerBlock) {
          s_req[slot - slot0] = r; s_idx[slot - slot0] = s; s_w[slot - slot0] = w;
        }
      }
    }
  }
  if (blockIdx.x == 0 && tid == 0) { p.req_slot_begin[p.max_requests] = run; *p.n_live = run; }
  __syncthreads();
  // all slots of this block at once: one thread per (slot, token)
  for (int i = tid; i < kSlotsPerBlock * p.bl; i += T) {
    const int k = i / p.bl, t = i % p.bl;
    const int slot = slot0 + k;
    if (slot >= p.max_slots) break;
    const int r = s_req[k];
    if (r < 0) {
      if (t == 0) {
        p.slot_req[slot] = -1; p.slot_s[slot] = 0; p.slot_pos0[slot] = 0; p.slot_kv_len[slot] = 0;
        p.slot_flags[slot] = 0;
      }
      p.qtok[slot * p.bl + t] = p.mask_id; p.pos[slot * p.bl + t] = 0;
      continue;
    }
    const int s = s_idx[k], w = s_w[k];
    const int P = p.prefix_len[r], g = p.L[r] + s;
    const int pos0 = P + s * p.bl;
    if (t == 0) {
      p.slot_req[slot] = r; p.slot_s[slot] = s; p.slot_pos0[slot] = pos0;
      p.slot_kv_len[slot] = P + (s + 1) * p.bl;
      p.slot_flags[slot] = (s == 0 ? FB_FLAG_OLDEST : 0) | (s == w - 1 ? FB_FLAG_FRONTIER : 0);
    }
    p.qtok[slot * p.bl + t] = p.tokens[(size_t)r * p.max_blocks * p.bl + (size_t)g * p.bl + t];  // Eq. 4: qtok = x[b, o_b + ...]
    p.pos[slot * p.bl + t] = pos0 + t;                                                           //        pos  = o_b + ...
  }
}

int launch_pack(fb_ctx* ctx, const fb_state* st, const fb_pack* out, void* ws, int32_t* status,
                cudaStream_t stream) {
  const fb_config& c = ctx->cfg;
  PackParams p;
  p.active = st->active; p.prefix_len = st->prefix_len; p.L = st->L; p.R = st->R; p.tokens = st->tokens;
  p.n_live = out->n_live; p.slot_req = out->slot_req; p.slot_s = out->slot_s; p.slot_pos0 = out->slot_pos0;
  p.slot_kv_len = out->slot_kv_len; p.slot_flags = out->slot_flags; p.req_slot_begin = out->req_slot_begin;
  p.qtok = out->qtok; p.pos = out->pos; p.status = status;
  uint8_t* w = static_cast<uint8_t*>(ws);
  for (int l = 0; l < 2; ++l) {
    p.hdr[l] = reinterpret_cast<SchedHeader*>(w + ctx->ws.l[l].header);
    p.items[l] = reinterpret_cast<AttnItem*>(w + ctx->ws.l[l].items);
    p.units[l] = reinterpret_cast<AttnUnit*>(w + ctx->ws.l[l].units);
    p.max_items[l] = ctx->ws.l[l].max_items; p.max_units[l] = ctx->ws.l[l].max_units;
    p.max_parts[l] = ctx->ws.l[l].max_parts;
  }
  p.target_items[0] = ctx->target_items;
  p.target_items[1] = ctx->target_items > 1 ? ctx->target_items / 2 : 1;
  p.pair_on = ctx->pair_on;
  p.max_requests = c.max_requests; p.wmax = c.wmax; p.bl = c.block_len;
  p.max_slots = c.max_requests * c.wmax; p.max_blocks = c.max_blocks; p.mask_id = c.mask_id;
  p.n_kv_heads = c.n_kv_heads; p.tiles_per_slot = ctx->tiles_per_slot;
  p.tokens_per_tile = ctx->tokens_per_tile;
  p.min_chunk_tiles = ctx->min_chunk_tiles;
  p.auto_split = ctx->auto_split; p.auto_min_chunk = ctx->auto_min_chunk;
  p.resident = ctx->cfg.window_in_pages;
  p.n_gather_blocks = (p.max_slots + kSlotsPerBlock - 1) / kSlotsPerBlock;
  // one more block per work list in use (the CTA-pair kernel's list only when that kernel is on)
  const int grid = p.n_gather_blocks + 1 + (p.pair_on ? 1 : 0);
  // (a prefix that its row of the page table does not hold is a bad state, reported by the attention)
  const bool small = p.max_requests <= kPackSmallRequests, far = c.max_pages_per_req >= kPackLongPages;
  const int threads = small ? kPackThreadsSmall : kPackThreads;
  auto* const kernel = small ? (far ? pack_kernel<kPackThreadsSmall, true> : pack_kernel<kPackThreadsSmall, false>)
                             : (far ? pack_kernel<kPackThreads, true> : pack_kernel<kPackThreads, false>);
  return cuda_err(ctx, launch_pdl(kernel, grid, threads, 0, stream, p), "pack_kernel launch");
}

}  // namespace fb
