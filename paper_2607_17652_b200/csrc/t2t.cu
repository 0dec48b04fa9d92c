// fb_t2t_step: the token-to-token step over the logits (Sec. 2.1, Eq. 1; the
// counts of Eq. 2).
//
// Kernel 1 (bandwidth-bound): one CTA per live row, or a cluster of up to eight CTAs per
// row when the batch has few rows, streams the row's bf16 logits once with 16-byte loads
// (the next batch of loads in flight while the current one is absorbed) and keeps, per
// thread, a running (max, first index of the max, sum of exp relative to that max); a
// warp-shuffle + shared-memory reduction merges them with the lowest-index rule.
// Output: top-1 token and its softmax probability 1 / sum exp(z - max).
// Kernel 2 (tiny): one warp per slot applies Eq. 1 to the slot's bl positions,
// updates the tokens in place and produces the per-block counts.
#include <cfloat>

#include <cooperative_groups.h>

#include "fb_common.cuh"

namespace fb {

constexpr int kRowUnroll = 4;   // 16-byte loads per thread and batch, two batches in flight
constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ uint4 ld_stream16(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ float fast_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// What a logit adds to the sum of a thread that has no maximum yet: nothing if it is -inf, but a NaN
// (the maximum passes it by) makes the sum NaN for good.
__device__ __forceinline__ float no_max_term(float z) { return z == -INFINITY ? 0.f : z; }

struct RowAcc {
  float m;    // running max
  float s;    // sum of exp(z - m)
  int idx;    // first index where z == m
};

__device__ __forceinline__ void merge(RowAcc& a, const RowAcc& b) {
  // lowest index wins ties; sums are rescaled to the larger max
  if (b.m > a.m || (b.m == a.m && b.idx < a.idx)) {
    const float sc = a.m == -INFINITY ? 0.f : fast_ex2((a.m - b.m) * kLog2e);
    a.s = a.s * sc + b.s; a.m = b.m; a.idx = b.idx;
  } else {
    const float sc = b.m == -INFINITY ? 0.f : fast_ex2((b.m - a.m) * kLog2e);
    a.s += b.s * sc;
  }
}

__device__ __forceinline__ void absorb8(RowAcc& a, const uint4 v, int base) {
  float z[8] = {bf16_lo(v.x), bf16_hi(v.x), bf16_lo(v.y), bf16_hi(v.y),
                bf16_lo(v.z), bf16_hi(v.z), bf16_lo(v.w), bf16_hi(v.w)};
  float cm = fmaxf(fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3])), fmaxf(fmaxf(z[4], z[5]), fmaxf(z[6], z[7])));
  if (cm > a.m) {                       // rare after the first few chunks
    a.s *= a.m == -INFINITY ? 0.f : fast_ex2((a.m - cm) * kLog2e);   // (0 * NaN stays NaN)
    a.m = cm;
    int k = 7;
#pragma unroll
    for (int i = 6; i >= 0; --i) k = z[i] == cm ? i : k;
    a.idx = base + k;
  }
  float acc = 0.f;
  if (a.m == -INFINITY) {                // no maximum so far
#pragma unroll
    for (int i = 0; i < 8; ++i) acc += no_max_term(z[i]);
    a.s += acc;
    return;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) acc += fast_ex2((z[i] - a.m) * kLog2e);
  a.s += acc;
}

__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// Two 16-byte pieces at once (`base` < `base2`: their first vocabulary indices): the maximum of the
// 16 logits on the packed values, the exponentials with packed fp32 arithmetic into two sums.
// The difference to the maximum comes first, then the scaling: the maximum's own term is exactly 1 and
// the sum never below it.  One fused multiply-add z log2(e) - m log2(e) leaves the rounding error of
// the product m log2(e) in the exponent of every term (1e-6 at m = 28).  The separate multiply shows in
// neither large nor small passes (call in us, without / with: 5120 rows 255.0 / 255.1, 640 rows 56.3 /
// 56.3, 64 rows 17.4 / 17.4, events around it and a cold L2) and costs whole steps 0.1 to 0.7 %.
__device__ __forceinline__ void absorb16(RowAcc& a, float2& s2, const uint4 v, const uint4 w, int base, int base2) {
  const uint32_t q[8] = {v.x, v.y, v.z, v.w, w.x, w.y, w.z, w.w};
  const uint32_t mm = max_bf16x2(max_bf16x2(max_bf16x2(q[0], q[1]), max_bf16x2(q[2], q[3])),
                                 max_bf16x2(max_bf16x2(q[4], q[5]), max_bf16x2(q[6], q[7])));
  const float cm = fmaxf(bf16_lo(mm), bf16_hi(mm));
  if (cm > a.m) {                       // rare after the first few pieces
    const float f = a.m == -INFINITY ? 0.f : fast_ex2((a.m - cm) * kLog2e);
    s2.x *= f; s2.y *= f;
    a.m = cm;
#pragma unroll
    for (int i = 7; i >= 0; --i) {
      const int at = (i < 4 ? base : base2) + 2 * (i & 3);
      if (bf16_hi(q[i]) == cm) a.idx = at + 1;
      if (bf16_lo(q[i]) == cm) a.idx = at;
    }
  }
  if (a.m == -INFINITY) {                // no maximum so far
#pragma unroll
    for (int i = 0; i < 8; ++i) s2.x += no_max_term(bf16_lo(q[i])) + no_max_term(bf16_hi(q[i]));
    return;
  }
  const float2 nm2 = make_float2(-a.m, -a.m), l2 = make_float2(kLog2e, kLog2e);
  float2 t = make_float2(0.f, 0.f);      // a sum of its own first: short chains of roundings
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float2 x = __fmul2_rn(__fadd2_rn(make_float2(bf16_lo(q[i]), bf16_hi(q[i])), nm2), l2);
    t = __fadd2_rn(t, make_float2(fast_ex2(x.x), fast_ex2(x.y)));
  }
  s2 = __fadd2_rn(s2, t);
}

template <int T>
__global__ void __launch_bounds__(T)
t2t_rows_kernel(const uint4* __restrict__ logits, const int32_t* __restrict__ n_live, int bl, int nvec,
                int32_t* __restrict__ argmax, float* __restrict__ conf, int32_t* __restrict__ status) {
  pdl_wait_then_release();          // (the update is next)
  // a cluster of cl CTAs shares one row: CTA `rank` streams the rank-th piece of it and rank 0
  // merges the pieces through distributed shared memory (cl == 1: the whole row, no exchange)
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int cl = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int row = blockIdx.x / cl;
  const int tid = threadIdx.x;
  if (row >= *n_live * bl) {            // padding slot: no bytes read (the whole cluster leaves)
    if (tid == 0 && rank == 0) { argmax[row] = -1; conf[row] = 0.f; }
    return;
  }
  constexpr int U = kRowUnroll, kStep = U * T;
  const int seg = (nvec + cl - 1) / cl;
  const int vbeg = min(nvec, rank * seg), vend = min(nvec, vbeg + seg);
  const uint4* p = logits + (size_t)row * nvec;
  RowAcc a{-INFINITY, 0.f, 0x7fffffff};
  float2 s2 = make_float2(0.f, 0.f);
  const int full = (vend - vbeg) / kStep;         // whole batches
  uint4 v[2][U];
  if (full > 0) {
#pragma unroll
    for (int u = 0; u < U; ++u) v[0][u] = ld_stream16(p + vbeg + tid + u * T);
  }
  int k = 0;
  for (; k + 2 <= full; k += 2) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (k + h + 1 < full) {
#pragma unroll
        for (int u = 0; u < U; ++u) v[h ^ 1][u] = ld_stream16(p + vbeg + (k + h + 1) * kStep + tid + u * T);
      }
#pragma unroll
      for (int u = 0; u < U; u += 2) {
        const int i = vbeg + (k + h) * kStep + tid + u * T;
        absorb16(a, s2, v[h][u], v[h][u + 1], i * 8, (i + T) * 8);
      }
    }
  }
  if (k < full) {
#pragma unroll
    for (int u = 0; u < U; u += 2) {
      const int i = vbeg + k * kStep + tid + u * T;
      absorb16(a, s2, v[0][u], v[0][u + 1], i * 8, (i + T) * 8);
    }
  }
  a.s = s2.x + s2.y;
  for (int i = vbeg + full * kStep + tid; i < vend; i += T) absorb8(a, ld_stream16(p + i), i * 8);
  // warp reduce
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    RowAcc b;
    b.m = __shfl_xor_sync(0xffffffffu, a.m, o);
    b.s = __shfl_xor_sync(0xffffffffu, a.s, o);
    b.idx = __shfl_xor_sync(0xffffffffu, a.idx, o);
    merge(a, b);
  }
  __shared__ RowAcc sh[T / 32];
  if ((tid & 31) == 0) sh[tid >> 5] = a;
  __syncthreads();
  RowAcc b{-INFINITY, 0.f, 0x7fffffff};
  auto warp_merge = [&](int from) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      if (o > from) continue;
      RowAcc c;
      c.m = __shfl_xor_sync(0xffffffffu, b.m, o);
      c.s = __shfl_xor_sync(0xffffffffu, b.s, o);
      c.idx = __shfl_xor_sync(0xffffffffu, b.idx, o);
      merge(b, c);
    }
  };
  if (tid < 32) {
    if (tid < T / 32) b = sh[tid];
    warp_merge(16);
  }
  if (cl > 1) {                          // uniform over the cluster
    __shared__ RowAcc part;
    if (tid == 0) part = b;
    cluster.sync();
    if (rank == 0 && tid < 32) {
      b = tid < cl ? *cluster.map_shared_rank(&part, tid) : RowAcc{-INFINITY, 0.f, 0x7fffffff};
      warp_merge(4);                     // cl <= 8
    }
    cluster.sync();                      // the pieces stay put until rank 0 has read them
    if (rank != 0) return;
  }
  if (tid == 0) {
    const float pr = 1.0f / b.s;         // the max itself contributes exp(0) = 1 exactly: b.s >= 1
    if (!(b.s >= 1.0f) || !(pr == pr) || b.s > FLT_MAX) {
      atomicOr(status, FB_ST_NAN_LOGIT);
      argmax[row] = b.idx == 0x7fffffff ? 0 : b.idx;
      conf[row] = 0.f;
    } else {
      argmax[row] = b.idx;
      conf[row] = pr;
    }
  }
}

struct UpdParams {
  const int32_t *n_live, *slot_req, *slot_s, *L;
  int32_t* tokens;
  const int32_t* argmax;
  const float* conf;
  uint8_t* action;
  int32_t* slot_stats;
  int32_t max_slots, bl, max_blocks, mask_id, eos_id;
  float tau_mask, tau_edit;
  int32_t delta_literal, force_progress;
};

__global__ void __launch_bounds__(128) t2t_update_kernel(const UpdParams p) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int slot = blockIdx.x * 4 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  // The kernel before is the row pass or the merge of the LM head, of the same call, and releases this one when it
  // has waited itself: slots and state are older and read ahead of the wait, the first 32 tokens of the block too.
  // What is left behind it is one round of loads.  Both kernels in us, back to back, before / with it: V = 1024: 24
  // requests 8.5 / 7.8, 64 requests 12.7 / 11.9, 128 requests 21.5 / 20.5; V = 8,000: 64 requests 23.0 / 21.7; V = 151,552:
  // one request 10.4 / 9.9, 64 requests 246.0 / 245.7.
  int n_live = 0, r = 0, s0 = 0, g = 0, x0 = 0;
  int32_t* tok = p.tokens;
  if (slot < p.max_slots) {
    n_live = __ldcg(p.n_live); r = __ldcg(p.slot_req + slot); s0 = __ldcg(p.slot_s + slot);
    if (slot < n_live) {
      g = __ldcg(p.L + r) + s0;
      tok += (size_t)r * p.max_blocks * p.bl + (size_t)g * p.bl;
      if (lane < p.bl) x0 = __ldcg(tok + lane);
    }
  }
  pdl_wait_only();
  if (slot >= p.max_slots) return;
  if (slot >= n_live) {
    for (int t = lane; t < p.bl; t += 32) p.action[slot * p.bl + t] = 0;
    if (lane < FB_SLOT_STATS) p.slot_stats[slot * FB_SLOT_STATS + lane] = 0;
    return;
  }
  int m0 = 0, rdy = 0, m2t = 0, t2t = 0, m1 = 0, eos = 0;
  float bestp = -1.f;                               // most confident mask this lane left in place
  int bestt = 0x7fffffff;
  for (int t = lane; t < p.bl; t += 32) {
    const int i = slot * p.bl + t;
    int x = t == lane ? x0 : tok[t];
    const int xh = p.argmax[i];
    const float pr = p.conf[i];
    uint8_t act = FB_ACT_NONE;
    if (x == p.mask_id) {                         // Gamma of Eq. 1: strict >
      m0++;
      rdy += pr >= p.tau_mask;                    // Eq. 2 numerator: >=
      // Delta as printed has no "revealed" condition: with delta_literal a mask whose
      // prediction is not [M] itself is updated once p > tau_edit as well
      if (pr > p.tau_mask || (p.delta_literal && x != xh && pr > p.tau_edit)) { x = xh; act = FB_ACT_M2T; m2t++; }
      else if (pr > bestp) { bestp = pr; bestt = t; }
    } else if (x != xh && pr > p.tau_edit) {      // Delta of Eq. 1, revealed only
      x = xh; act = FB_ACT_T2T; t2t++;
    }
    if (act) tok[t] = x;
    p.action[i] = act;
    m1 += x == p.mask_id;
    eos |= x == p.eos_id;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    m0 += __shfl_xor_sync(0xffffffffu, m0, o);
    rdy += __shfl_xor_sync(0xffffffffu, rdy, o);
    m2t += __shfl_xor_sync(0xffffffffu, m2t, o);
    t2t += __shfl_xor_sync(0xffffffffu, t2t, o);
    m1 += __shfl_xor_sync(0xffffffffu, m1, o);
    eos |= __shfl_xor_sync(0xffffffffu, eos, o);
  }
  // forced progress: the oldest block went in with masks and Eq. 1 revealed none -> its most
  // confident masked position (lowest position on ties) is revealed
  if (p.force_progress && s0 == 0 && m0 > 0 && m2t == 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float op = __shfl_xor_sync(0xffffffffu, bestp, o);
      const int ot = __shfl_xor_sync(0xffffffffu, bestt, o);
      if (op > bestp || (op == bestp && ot < bestt)) { bestp = op; bestt = ot; }
    }
    const int xh = p.argmax[slot * p.bl + bestt];
    if (lane == 0) { tok[bestt] = xh; p.action[slot * p.bl + bestt] = FB_ACT_FORCED; }
    m2t = 1; m1 -= xh != p.mask_id; eos |= xh == p.eos_id;
  }
  if (lane == 0) {
    int32_t* s = p.slot_stats + slot * FB_SLOT_STATS;
    s[FB_STAT_M0] = m0; s[FB_STAT_RDY] = rdy; s[FB_STAT_M2T] = m2t; s[FB_STAT_T2T] = t2t; s[FB_STAT_M1] = m1;
    s[FB_STAT_EOS] = eos;
  }
}

// Threads that share a row (in CTAs of up to 512, a cluster of up to eight).  A pass is fastest
// with about 1,000 threads an SM: fewer do not cover the load latency, more only add merging.
// That is about 180,000 threads over the slot capacity (live rows are typically two thirds of
// it), rounded to a power of two, and no more threads than the row has pairs of pieces.
// Measured, V = 151,552, call time in us (live rows of capacity: 128x1 / 256x1 / 512x1 / 512x2 /
// 512x4 threads x CTAs per row; in front the former 128 threads, a pair of CTAs below 2048 rows):
//     64 of    64:  30.4 |  27.0   21.4   17.8   13.5    9.9
//     96 of   128:  33.8 |  47.9   31.8   19.0   13.0   14.1
//    640 of  1024:  47.3 |  60.7   43.0   42.5   51.3   68.7
//   3072 of  4608:   160 |   155    159    170    212    307
//   5120 of  8192:   259 |   252    262    279    351    511
// Many short rows: there the machine is full with any number of threads a row, and the fewer there
// are the less is merged and the longer each one streams; what speaks for more is the tail, in which
// the last rows run alone (their time is nvec / threads).  So 64 threads from rows = 2 nvec on, a warp
// from 6 nvec on.  us, 128 / 64 / 32 threads (in front the former two CTAs or 128 threads):
//   9600 of 12800, V =  2,048:  25.2 |  27.3   20.2   17.8
//                       8,000:  58.9 |  50.9   40.2   37.4
//                      24,000:   101 |  91.7   83.0   84.1
//                      64,000 (6400 live):  141 |   136    137    154
//   6144 of  8192, V = 16,000:  54.3 |  48.5   43.8   43.6
//                      32,000:  78.3 |  75.2   75.3   82.6
//   2304 of  3072, V =  4,096:  11.0 |  10.8    9.4   10.8
struct RowShape { int threads, ctas; };
static RowShape row_shape(int rows, int nvec) {
  const int floor_ = rows < 2048 ? 256 : 128;
  int w = 128;
  while (w < 4096 && (long long)w * 1448 / 1024 * rows < 180000) w *= 2;   // nearest power of two (in the log)
  w = w < floor_ ? floor_ : w;
  while (w > 128 && 2 * w > nvec) w /= 2;
  if (rows >= 2048 && 2ll * nvec <= rows) w = rows >= 4096 && 6ll * nvec <= rows ? 32 : 64;
  RowShape s;
  s.threads = w < 512 ? w : 512;
  s.ctas = w / s.threads;
  return s;
}

int launch_t2t(fb_ctx* ctx, const fb_pack* pk, const void* logits, const fb_state* st, int32_t* argmax,
               float* conf, uint8_t* action, int32_t* slot_stats, int32_t* status, cudaStream_t stream) {
  const fb_config& c = ctx->cfg;
  const int max_slots = c.max_requests * c.wmax;
  const int rows = max_slots * c.block_len;
  const RowShape shape = row_shape(rows, c.vocab / 8);
  const int T = shape.threads, cl = shape.ctas;
  auto launch = [&](auto kernel, int threads) {
    return cuda_err(ctx, launch_pdl_cluster(kernel, rows * cl, threads, 0, stream, cl,
                                            static_cast<const uint4*>(logits), pk->n_live, c.block_len,
                                            c.vocab / 8, argmax, conf, status),
                    "t2t_rows_kernel launch");
  };
  const int e = T == 32    ? launch(t2t_rows_kernel<32>, 32)
                : T == 64  ? launch(t2t_rows_kernel<64>, 64)
                : T == 128 ? launch(t2t_rows_kernel<128>, 128)
                : T == 256 ? launch(t2t_rows_kernel<256>, 256)
                           : launch(t2t_rows_kernel<512>, 512);
  if (e) return e;
  return launch_t2t_update(ctx, pk, st, argmax, conf, action, slot_stats, stream);
}

// Eq. 1 and the block counts from (argmax, conf), whoever produced them.
int launch_t2t_update(fb_ctx* ctx, const fb_pack* pk, const fb_state* st, const int32_t* argmax, const float* conf,
                      uint8_t* action, int32_t* slot_stats, cudaStream_t stream) {
  const fb_config& c = ctx->cfg;
  const int max_slots = c.max_requests * c.wmax;
  UpdParams u;
  u.n_live = pk->n_live; u.slot_req = pk->slot_req; u.slot_s = pk->slot_s; u.L = st->L; u.tokens = st->tokens;
  u.argmax = argmax; u.conf = conf; u.action = action; u.slot_stats = slot_stats;
  u.max_slots = max_slots; u.bl = c.block_len; u.max_blocks = c.max_blocks; u.mask_id = c.mask_id;
  u.eos_id = c.eos_id; u.tau_mask = c.tau_mask; u.tau_edit = c.tau_edit;
  u.delta_literal = c.delta_literal; u.force_progress = c.force_progress;
  return cuda_err(ctx, launch_pdl(t2t_update_kernel, (max_slots + 3) / 4, 128, 0, stream, u), "t2t_update_kernel launch");
}

}  // namespace fb
