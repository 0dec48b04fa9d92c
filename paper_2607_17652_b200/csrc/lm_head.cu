// fb_lm_head_t2t: the T2T row pass taken straight from the LM head.  z = x W^T
// (hidden states x [rows, hidden], head weights W [V, hidden], bf16, fp32
// accumulation on the tensor cores) is never written: the epilogue of every
// 128 x 256 output tile reduces its rows to (max, sum of exponentials, first
// index of the max), a second kernel merges the tiles of a row, and the Eq. 1
// update runs on the result as in fb_t2t_step.  What the fused form saves is
// the 2 V bytes per row that the stand-alone row pass has to read.
//
// Persistent, warp-specialised tcgen05 GEMM, one CTA per SM, 256 threads:
//   warp 0      TMA producer: A tile (128 rows of x) and B tile (256 rows of W)
//               per 64-element slice of the hidden dimension, 4 stages
//   warp 1      MMA issuer: 4 x tcgen05.mma (M 128, N 256, K 16) per stage into
//               one of two 256-column accumulators in TMEM
//   warps 4-7   epilogue: one thread per output row, 32 columns at a time
// Tiles are taken vocabulary-major (all row tiles of one 256-token slice of W
// next to each other), so W streams from HBM once and x stays in L2.
//
// Two forms.  One CTA per tile as above, or (kPair) a cluster of two CTAs per 256 rows: one MMA spans both
// (M 256, cta_group::2), each CTA holds its own 128 rows of x and half of the slice of W, and its
// accumulator is its own 128 rows again, so the epilogue is the same.  A stage is 32 KB for as many
// operations as 48 KB before, six stages fit, and a CTA reads 8 KB instead of 12 KB of shared memory
// per MMA.  What bounds the product is the board's power limit, which is where the saved traffic shows:
// a step of 64 requests (5,120 rows, V = 151,552, hidden 2048), back to back, 2781 -> 2616 us.
// Where which one runs: lm_forms.h, by what the context can hold on the host and by the live rows on the device.
#include <cudaTypedefs.h>

#include <cfloat>

#include "fb_common.cuh"
#include "lm_forms.h"
#include "ptx_sm100.cuh"

namespace fb {

constexpr int kLmThreads = 256;
constexpr int kLmBK = 64, kLmStages = 4;
constexpr int kLmABytes = kLmBM * kLmBK * 2, kLmBBytes = kLmBN * kLmBK * 2;
constexpr int kLmStageBytes = kLmABytes + kLmBBytes;                 // 48 KB
constexpr int kLmPairStages = 6, kLmPairStageBytes = kLmABytes + kLmBBytes / 2;   // 32 KB a CTA
constexpr int kLmSmem = kLmStages * kLmStageBytes + 2048;            // + barriers + 1 KB alignment slack
static_assert(kLmPairStages * kLmPairStageBytes == kLmStages * kLmStageBytes, "one shared-memory size for both forms");
constexpr float kLmLog2e = 1.4426950408889634f;

struct LmParams {
  const int32_t* n_live;
  float4* part;          // [n_tiles_n][rows_pad] (max, sum exp, first index of the max as bits, -)
  int32_t* status;
  int32_t bl, vocab, hidden, n_tiles_n, rows_pad;
  int32_t both;          // both forms are launched ...
  unsigned long long pairs_mask;   // ... and lm_pairs_of says which one works
  long long wait_cycles;
};

// 32 more columns of a row: running maximum with its first index, sum of exponentials relative to it
// (an equal later maximum keeps the first index; all -inf adds nothing, a NaN makes the sum NaN).
__device__ __forceinline__ void absorb32(const uint32_t* v, int col, float& mx, float& sum, int& arg) {
  float m4[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) m4[t] = fmaxf(__uint_as_float(v[t]), __uint_as_float(v[4 + t]));
#pragma unroll
  for (int i = 8; i < 32; i += 8)
#pragma unroll
    for (int t = 0; t < 4; ++t) m4[t] = max3(m4[t], __uint_as_float(v[i + t]), __uint_as_float(v[i + 4 + t]));
  const float cm = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
  if (cm > mx) {
    int first = 31;
#pragma unroll
    for (int j = 30; j >= 0; --j) first = __uint_as_float(v[j]) == cm ? j : first;
    sum *= ex2_approx((mx - cm) * kLmLog2e);                          // 0 * 2^-inf = 0 at the first maximum
    mx = cm; arg = col + first;
  }
  if (mx == -INFINITY) {                // (the maximum passes NaN by)
#pragma unroll
    for (int j = 0; j < 32; ++j) sum += __uint_as_float(v[j]) == -INFINITY ? 0.f : __uint_as_float(v[j]);
    return;
  }
  // difference first, then the scaling: the maximum's own term is exactly 1 (see absorb16 in t2t.cu)
  const float2 nm2 = make_float2(-mx, -mx), l2 = make_float2(kLmLog2e, kLmLog2e);
  float2 s4[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
  for (int j = 0; j < 32; j += 2) {
    const float2 x = __fmul2_rn(__fadd2_rn(make_float2(__uint_as_float(v[j]), __uint_as_float(v[j + 1])), nm2), l2);
    s4[(j >> 1) & 3] = __fadd2_rn(s4[(j >> 1) & 3], make_float2(ex2_approx(x.x), ex2_approx(x.y)));
  }
  const float2 t = __fadd2_rn(__fadd2_rn(s4[0], s4[1]), __fadd2_rn(s4[2], s4[3]));
  sum += t.x + t.y;
}

template <bool kPair>
__global__ void __launch_bounds__(kLmThreads, 1)
lm_head_stats_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
                     const LmParams p) {
  constexpr int kStages = kPair ? kLmPairStages : kLmStages, kStageBytes = kPair ? kLmPairStageBytes : kLmStageBytes;
  // Where both forms are launched, the pairs' grid comes second.  It is started when the first one is through (turned
  // down), or from its first moment on (at work: the CTAs find room as the first one's leave, and what is turned down is
  // gone when that ends).  Either way the first has waited for everything older, so the pairs may read n_live (past the
  // L1) ahead of their own wait.  Turned down, they let the merge start, and one CTA waits for the first grid all the
  // same: the merge waits for this grid alone.
  const bool second = p.both && kPair;
  if (!second) pdl_wait_only();
  const int live_rows = __ldcg(p.n_live) * p.bl;
  const int m_tiles = (live_rows + kLmBM - 1) / kLmBM;          // row tiles that hold live rows
  const bool wanted = !p.both || lm_pairs_of(p.pairs_mask, m_tiles) == kPair;
  if (p.both && wanted != kPair) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (second && (wanted || blockIdx.x == 0)) pdl_wait_only();
  if (!wanted) return;                                          // (the whole grid)
  extern __shared__ uint8_t smem_raw[];
  // (a pair's CTAs lay their shared memory out alike: the MMA's descriptors are offsets in both)
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
  uint64_t* full = bars;                    // [kStages] stage filled (TMA bytes); pair: the first CTA's, for both
  uint64_t* empty = bars + 6;               // [kStages] stage consumed (MMA commit); pair: in both
  uint64_t* acc_full = bars + 12;           // [2] accumulator complete (MMA commit); pair: in both
  uint64_t* acc_empty = bars + 14;          // [2] accumulator read out (4 epilogue warps; pair: the first CTA's, 8)
  uint64_t* drain = bars + 16;              // give-up path only
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 17);
  volatile int* abortf = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long LIM = p.wait_cycles;
  const int rank = kPair ? (int)cluster_ctarank() : 0;
  const bool first = rank == 0;             // issues the MMAs
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    return __all_sync(0xffffffffu, kPair ? mbar_wait_cluster(bar, parity, abortf, LIM) : mbar_wait(bar, parity, abortf, LIM));
  };
  if (tid == 0) {
    *abortf = 0;
    for (int i = 0; i < kStages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], kPair ? 8 : 4); }
    mbar_init(drain, 1);
    fence_mbar_init();
    tma_prefetch_desc(&tmX); tma_prefetch_desc(&tmW);
  }
  if (warp == 1) {
    if constexpr (kPair) { tmem_alloc_pair(tmem_slot, 512); tmem_relinquish_pair(); }
    else { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (kPair) cluster_sync_all();  // both CTAs' barriers are there before either signals the other's
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int m_steps = kPair ? (m_tiles + 1) / 2 : m_tiles;
  const int n_tiles = m_steps * p.n_tiles_n;
  const int t0 = kPair ? blockIdx.x / 2 : blockIdx.x, t_step = kPair ? gridDim.x / 2 : gridDim.x;
  const int k_blocks = p.hidden / kLmBK;

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    const bool leader = elect_one();
    int fill = 0;
    bool ok = true;
    for (int t = t0; t < n_tiles && ok; t += t_step) {
      const int n = t / m_steps, m = (t % m_steps) * (kPair ? 2 : 1) + rank;
      for (int kb = 0; kb < k_blocks; ++kb, ++fill) {
        const int st = fill % kStages, round = fill / kStages;
        if (round > 0 && !wait(&empty[st], (round - 1) & 1)) { ok = false; break; }
        if (leader) {
          uint8_t* a = smem + st * kStageBytes;
          if constexpr (kPair) {
            if (first) mbar_arrive_expect_tx(&full[st], 2 * kStageBytes);
            const uint32_t bar = mapa_u32(&full[st], 0);
            tma_load_2d_pair(a, &tmX, bar, kb * kLmBK, m * kLmBM);
            tma_load_2d_pair(a + kLmABytes, &tmW, bar, kb * kLmBK, n * kLmBN + rank * (kLmBN / 2));
          } else {
            mbar_arrive_expect_tx(&full[st], kStageBytes);
            tma_load_2d(a, &tmX, &full[st], kb * kLmBK, m * kLmBM);
            tma_load_2d(a + kLmABytes, &tmW, &full[st], kb * kLmBK, n * kLmBN);
          }
        }
        __syncwarp();
      }
    }
  } else if (warp == 1 && first) {
    // ---------------------------------------------------------- MMA issuer
    const bool leader = elect_one();
    const uint32_t idesc = umma_idesc_bf16(kPair ? 2 * kLmBM : kLmBM, kLmBN, 0, 0);
    const uint64_t dA0 = smem_desc_sw128(smem_u32(smem), 16, 1024);
    const uint64_t dB0 = smem_desc_sw128(smem_u32(smem + kLmABytes), 16, 1024);
    int fill = 0, i = 0;
    bool ok = true;
    for (int t = t0; t < n_tiles && ok; t += t_step, ++i) {
      const int b = i & 1;
      if (i >= 2 && !wait(&acc_empty[b], ((i >> 1) - 1) & 1)) { ok = false; break; }
      tc_fence_after();
      for (int kb = 0; kb < k_blocks; ++kb, ++fill) {
        const int st = fill % kStages, round = fill / kStages;
        if (!wait(&full[st], round & 1)) { ok = false; break; }
        tc_fence_after();
        if (leader) {
          const uint32_t so = (uint32_t)((st * kStageBytes) >> 4);
#pragma unroll
          for (int ks = 0; ks < kLmBK / 16; ++ks) {
            const uint64_t da = dA0 + so + (uint32_t)((ks * 32) >> 4), db = dB0 + so + (uint32_t)((ks * 32) >> 4);
            const uint32_t acc = (kb > 0 || ks > 0) ? 1u : 0u;
            if constexpr (kPair) umma_ss_pair(tmem + b * kLmBN, da, db, idesc, acc);
            else umma_ss(tmem + b * kLmBN, da, db, idesc, acc);
          }
          if constexpr (kPair) {
            umma_commit_pair(&empty[st], true);
            if (kb == k_blocks - 1) umma_commit_pair(&acc_full[b], true);
          } else {
            umma_commit(&empty[st]);
            if (kb == k_blocks - 1) umma_commit(&acc_full[b]);
          }
        }
        __syncwarp();
      }
    }
  } else if (warp >= 4) {
    // ------------------------------------------------------------ epilogue
    const int quad = warp & 3;
    const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
    int i = 0;
    bool ok = true;
    for (int t = t0; t < n_tiles && ok; t += t_step, ++i) {
      const int n = t / m_steps, m = (t % m_steps) * (kPair ? 2 : 1) + rank, b = i & 1;
      if (!wait(&acc_full[b], (i >> 1) & 1)) { ok = false; break; }   // one outcome per warp
      tc_fence_after();
      const uint32_t tacc = tmem + lane_base + b * kLmBN;
      const int col0 = n * kLmBN;
      float mx = -INFINITY, sum = 0.f;
      int arg = 0x7fffffff;
      uint32_t buf[2][32];
      tmem_ld32(tacc, buf[0]);
#pragma unroll
      for (int c = 0; c < kLmBN / 32; ++c) {
        const uint32_t* v = buf[c & 1];
        tmem_ld_wait();
        if (c + 1 < kLmBN / 32) tmem_ld32(tacc + (c + 1) * 32, buf[(c + 1) & 1]);
        const int valid = p.vocab - (col0 + c * 32);                 // columns of this chunk inside the vocabulary
        if (valid >= 32) {
          absorb32(v, col0 + c * 32, mx, sum, arg);
        } else if (valid > 0) {                                      // (the last tile: columns past the vocabulary count as -inf)
          uint32_t z[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) z[j] = j < valid ? v[j] : __float_as_uint(-INFINITY);
          absorb32(z, col0 + c * 32, mx, sum, arg);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (first) mbar_arrive(&acc_empty[b]);
        else mbar_arrive_cluster_relaxed(mapa_u32(&acc_empty[b], 0));   // (what it hands back is tensor memory)
      }
      const int row = m * kLmBM + quad * 32 + lane;
      if (row < live_rows)
        p.part[(size_t)n * p.rows_pad + row] = make_float4(mx, sum, __int_as_float(arg), 0.f);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*abortf) {
    // give-up path: the MMA warp waits for everything it has issued (own barrier, bounded
    // polls), copies in flight land while the CTA sleeps, then TMEM and shared memory go back
    if (tid == 0) atomicOr(p.status, FB_ST_DEV_TIMEOUT);
    if (warp == 1 && first) {
      if (elect_one()) { if constexpr (kPair) umma_commit_pair(drain, false); else umma_commit(drain); }
      __syncwarp();
      for (int i = 0; i < 4096 && !mbar_test(drain, 0); ++i) __nanosleep(200);
    }
    for (int i = 0; i < 64; ++i) __nanosleep(10000);
    __syncthreads();
  }
  if constexpr (kPair) cluster_sync_all();  // neither CTA leaves while the other may still signal it or read its shared memory
  if (warp == 1) {
    tc_fence_after();
    if constexpr (kPair) tmem_dealloc_pair(tmem, 512); else tmem_dealloc(tmem, 512);
  }
}

// Tiles of a row -> top-1 token (lowest index on ties) and its confidence 1 / sum exp(z - max).
// A CTA takes 32 rows, one per lane, so that a tile's results are read as whole lines; its 32 warps
// take the tiles in turn and meet in shared memory (5120 rows of 592 tiles: 41 us with a warp per row
// that read 16 bytes of a line, now about 10).
constexpr int kLmMergeWarps = 32;
__global__ void __launch_bounds__(32 * kLmMergeWarps) lm_head_merge_kernel(const LmParams p, int32_t* argmax, float* conf,
                                                                          int max_rows) {
  pdl_wait_then_release();          // (the update is next)
  __shared__ float s_m[kLmMergeWarps][32], s_s[kLmMergeWarps][32];
  __shared__ int s_a[kLmMergeWarps][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, row = blockIdx.x * 32 + lane;
  const int live = *p.n_live * p.bl;
  if (blockIdx.x * 32 >= live) {                    // (the whole CTA)
    if (warp == 0 && row < max_rows) { argmax[row] = -1; conf[row] = 0.f; }
    return;
  }
  float M = -INFINITY, S = 0.f;
  int arg = 0x7fffffff;
  auto add = [&](float m, float s, int a) {         // tiles come in ascending order: an equal maximum keeps the first index
    if (m > M) { S = S * (M == -INFINITY ? 0.f : ex2_approx((M - m) * kLmLog2e)) + s; M = m; arg = a; }
    else S += m == -INFINITY ? s : s * ex2_approx((m - M) * kLmLog2e);      // (no maximum: s is 0 or NaN)
  };
  if (row < live) {
    constexpr int kDepth = 4;
    for (int n0 = warp; n0 < p.n_tiles_n; n0 += kDepth * kLmMergeWarps) {
      float4 q[kDepth];
#pragma unroll
      for (int k = 0; k < kDepth; ++k) q[k] = p.part[(size_t)min(n0 + k * kLmMergeWarps, p.n_tiles_n - 1) * p.rows_pad + row];
#pragma unroll
      for (int k = 0; k < kDepth; ++k)
        if (n0 + k * kLmMergeWarps < p.n_tiles_n) add(q[k].x, q[k].y, __float_as_int(q[k].z));
    }
  }
  s_m[warp][lane] = M; s_s[warp][lane] = S; s_a[warp][lane] = arg;
  __syncthreads();
  if (warp != 0 || row >= max_rows) return;
  if (row >= live) { argmax[row] = -1; conf[row] = 0.f; return; }
  for (int k = 1; k < kLmMergeWarps; ++k) {
    const float m = s_m[k][lane], s = s_s[k][lane];
    const int a = s_a[k][lane];
    if (m == M && m != -INFINITY) { S += s; arg = min(arg, a); }
    else add(m, s, a);
  }
  if (!(S >= 1.0f) || S > FLT_MAX || arg == 0x7fffffff) {
    atomicOr(p.status, FB_ST_NAN_LOGIT);
    argmax[row] = arg == 0x7fffffff ? 0 : arg;
    conf[row] = 0.f;
  } else {
    argmax[row] = arg;
    conf[row] = 1.0f / S;
  }
}

static int lm_rows_pad(const fb_config& c) {
  const int rows = c.max_requests * c.wmax * c.block_len;
  return (rows + kLmBM - 1) / kLmBM * kLmBM;
}

size_t lm_head_workspace_bytes(const fb_ctx* ctx) {
  const fb_config& c = ctx->cfg;
  const size_t n_tiles_n = (c.vocab + kLmBN - 1) / kLmBN;
  return n_tiles_n * (size_t)lm_rows_pad(c) * sizeof(float4);
}

// per-device kernel attribute (called from ensure_device with that device current)
int lm_head_device_setup(fb_ctx* ctx) {
  if (int e = cuda_err(ctx, cudaFuncSetAttribute(lm_head_stats_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 kLmSmem), "smem attr"))
    return e;
  return cuda_err(ctx, cudaFuncSetAttribute(lm_head_stats_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            kLmSmem), "smem attr");
}

int launch_lm_head(fb_ctx* ctx, const fb_pack* pk, const void* x, const void* w, int hidden, const fb_state* st,
                   int32_t* argmax, float* conf, uint8_t* action, int32_t* slot_stats, void* ws, int32_t* status,
                   cudaStream_t stream) {
  if (int e = ensure_device(ctx)) return e;
  const fb_config& c = ctx->cfg;
  const int rows = c.max_requests * c.wmax * c.block_len;
  auto fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled>(ctx->encode_fn);
  CUtensorMap tmX, tmW;
  const cuuint32_t es[2] = {1, 1};
  {
    const cuuint64_t dims[2] = {(cuuint64_t)hidden, (cuuint64_t)rows};
    const cuuint64_t str[1] = {(cuuint64_t)hidden * 2};
    const cuuint32_t box[2] = {kLmBK, kLmBM};
    if (fn(&tmX, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(x), dims, str, box, es,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return set_err(ctx, FB_ERR_CUDA, "cuTensorMapEncodeTiled failed for x");
  }
  auto encode_w = [&](CUtensorMap& map, cuuint32_t box_rows) {
    const cuuint64_t dims[2] = {(cuuint64_t)hidden, (cuuint64_t)c.vocab};
    const cuuint64_t str[1] = {(cuuint64_t)hidden * 2};
    const cuuint32_t box[2] = {kLmBK, box_rows};
    if (fn(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(w), dims, str, box, es,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return set_err(ctx, FB_ERR_CUDA, "cuTensorMapEncodeTiled failed for w");
    return (int)FB_OK;
  };
  if (int e = encode_w(tmW, kLmBN)) return e;
  LmParams p;
  p.n_live = pk->n_live;
  p.part = static_cast<float4*>(ws);
  p.status = status;
  p.bl = c.block_len; p.vocab = c.vocab; p.hidden = hidden;
  p.n_tiles_n = (c.vocab + kLmBN - 1) / kLmBN;
  p.rows_pad = lm_rows_pad(c);
  p.wait_cycles = ctx->wait_cycles;
  // (both forms, since the live rows are only known on the device)
  p.both = lm_both_forms((rows + kLmBM - 1) / kLmBM, p.n_tiles_n, hidden, ctx->num_sms);
  p.pairs_mask = p.both ? lm_pairs_mask(p.n_tiles_n, hidden, ctx->num_sms) : 0;
  if (int e = cuda_err(ctx, launch_pdl(lm_head_stats_kernel<false>, ctx->num_sms, kLmThreads, kLmSmem, stream, tmX, tmW, p),
                       "lm_head_stats_kernel launch"))
    return e;
  if (p.both) {
    CUtensorMap tmWHalf;
    if (int e = encode_w(tmWHalf, kLmBN / 2)) return e;
    if (int e = cuda_err(ctx, launch_pdl_cluster(lm_head_stats_kernel<true>, ctx->num_sms / 2 * 2, kLmThreads, kLmSmem, stream, 2,
                                                 tmX, tmWHalf, p), "lm_head_stats_kernel (pairs) launch"))
      return e;
  }
  if (int e = cuda_err(ctx, launch_pdl(lm_head_merge_kernel, (rows + 31) / 32, 32 * kLmMergeWarps, 0, stream, p, argmax, conf, rows),
                       "lm_head_merge_kernel launch"))
    return e;
  return launch_t2t_update(ctx, pk, st, argmax, conf, action, slot_stats, stream);
}

}  // namespace fb
