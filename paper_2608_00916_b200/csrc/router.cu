// Router on the tensor cores: logits = x W_r (+ b_r), softmax statistics, top-k, gates, and the permutation's per-tile
// histogram, in one kernel.  x and W_r are bf16 (an fp32 W_r comes as three exact bf16 terms), so that a bf16 MMA with fp32
// accumulation is an fp32 contraction up to summation order.
//
// CL CTAs share the 128 tokens of a tile.  W_r^T is the M operand (128 experts, twice above 128 of them), tokens are N.  The K blocks
// are summed in four chains (fewer below four K blocks), each in an accumulator of its own, and the chains in their order: the
// tensor core drops what lies below the last place of an accumulator, so that the error grows with the length of a chain (rms
// 2.1e-6 with one chain, 0.5e-6 with four at d 2048 and unit-variance logits).
// The order of the sums depends on d alone, so that a token's logits, and with them its experts, are the same bits whatever the
// number of tokens of the call selects.  Two ways to share the work:
//   by chains (SPLIT: four CTAs, four chains, up to 128 experts): each CTA sums one chain for all 128 tokens, fetching a quarter of
//     W_r and of the tokens' columns, and sends the sums through the cluster to the CTA that routes the token
//   by tokens: each CTA contracts the 128 / CL tokens that it routes, and fetches all of W_r
// What bounds it: up to some ten thousand tokens the latency of fetching W_r and the tokens through one SM each and of routing,
// hence the split; from there on the stream of x from HBM.  At d 2048 and 128 experts the sums of a tile are complete 3.8 us after
// the kernel's first instruction by chains, and 2.9 us later where they are routed, 9.0 us by tokens; the kernel takes 11.6 and
// 14.6 us at 241 tokens (scoring 221.8 -> 219.6 us with the tables' share, see place_kernel).  With one CTA per tile the
// accumulators fill tensor memory, so that an SM holds one CTA: 42 -> 56 us at 24576 tokens, 49 -> 60 at 32768 against one chain and
// two CTAs.
//
// Three steps between barriers.  (1) A warp per token: bias, softmax and its column sums; a lane holds NV / 4 groups of four
// columns.  (2) A thread per token: top-k as a three-level tournament, groups of four columns, supers of four groups, the maxima
// of the supers in registers; a round takes the largest super (lowest among equals), the group and the column in it, removes the
// column and repairs the maxima above it, which is the rule "largest, lowest index among equals" because the levels partition the
// columns in order.  (3) The picks and gates leave as whole lines.
//
// A CTA routes a handful of tokens and every instruction of that arrives cold, about 450 cycles for each eight of them.  So
// while the operands are on their way the waiting warps run the steps once on whatever shared memory holds, each warp one
// step, so that the code is fetched side by side; what this first pass stores is overwritten by the same threads.
#include <string.h>

#include <algorithm>

#include "common.cuh"
#include "ptx.cuh"
#include "tensor_maps.cuh"

namespace moe {

constexpr int RO_TOK = 128;                    // tokens of a tile (the permutation's token tile as well)
constexpr int RO_WARPS = 12;                   // routing warps
constexpr int RO_THREADS = 64 + 32 * RO_WARPS;  // warps: 0 TMA producer, 1 MMA issuer, 2.. routing
constexpr int RO_BK = 64;
constexpr int RO_CHUNK_BYTES = 64 * RO_BK * 2;   // 8 KB per 64 columns of W_r and K block
constexpr int RO_MAX_STAGES = 16;
constexpr int RO_CHAINS = 4;  // partial sums of a logit
// Bytes of the operand stages by tokens.  Every CTA fetches all of W_r, and waits for latency more than for bandwidth, so the copies in
// flight count: 100 -> 200 KB at d 2048 and 128 experts 20 -> 19 us at 128 tokens, 26 -> 23 at 8192, 35 -> 31 at 16384 (one chain).
// By chains the sums of all chains (67 KB) lie behind the stages: other CTAs send them while this one still contracts.
constexpr int RO_RING = 200 * 1024, RO_SPLIT_RING = 128 * 1024;
static_assert(RO_TOK == TOK_TILE, "the histogram written here is the permutation's");

struct RouterParams {
  CUtensorMap map_x, map_w0, map_w1, map_w2;
  int32_t* status;
  float* row_gate;       // cleared here: pad rows must read 0
  int64_t rows;
  const float* bias;     // [E] or null
  float* logits;         // [T, E] saved logits
  float* logits_out;     // optional copy for the caller
  int32_t *idx, *idx_out;
  float *gates, *gates_out;
  float* psum_part;      // [CTAs with tokens, E] column sums of p
  int32_t* tile_counts;  // [tiles, E] picks of every 128-token tile
  int64_t T;
  int E, k;
  int k_blocks, k_total, chains;  // K blocks of one bf16 term of W_r, and of all terms; chains they are summed in
  int w_chunks, whole_chunks;  // 64-column chunks of W_r; E is a multiple of 64, so they are one copy
  int stages;
  uint32_t w_bytes, stage_bytes;  // of a stage: W_r, and with the tokens
};

__device__ __forceinline__ void st_cluster_f32(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void red_cluster_add(uint32_t addr, int v) {
  asm volatile("red.relaxed.cluster.shared::cluster.add.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ float4 lds_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts_f4(uint32_t addr, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ float max4(float4 v) { return fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)); }
// index (0..3) of the first component equal to m
__device__ __forceinline__ int first_eq4(float4 v, float m) { return v.x == m ? 0 : (v.y == m ? 1 : (v.z == m ? 2 : 3)); }
__device__ __forceinline__ float4 without(float4 v, int i, float by) {
  return make_float4(i == 0 ? by : v.x, i == 1 ? by : v.y, i == 2 ? by : v.z, i == 3 ? by : v.w);
}
// The caller's copy of the logits, whose alignment nothing checks
__device__ __forceinline__ void store_caller(float* out, float4 v) {
  if ((reinterpret_cast<uintptr_t>(out) & 15u) == 0) {
    *reinterpret_cast<float4*>(out) = v;
  } else {
    out[0] = v.x;
    out[1] = v.y;
    out[2] = v.z;
    out[3] = v.w;
  }
}
__device__ __forceinline__ int lds_int(uint32_t addr) {
  int v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float warp_max(float v) {  // NaN is dropped
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, off));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
  return v;
}

// A NaN logit counts as -inf in the selection, and every token gets k distinct experts whatever its logits are (the
// permutation indexes its tables with the picks): once nothing larger than -inf is left, the lowest index that is not among
// the j picks so far is taken.  picks: the token's picks {exponential, column}, `pitch` bytes apart.
__device__ __forceinline__ int lowest_untaken(int j, uint32_t picks, uint32_t pitch) {
  int e = 0;
#pragma unroll 1
  for (int q = 0; q < j;) {
    if (lds_int(picks + q * pitch + 4) == e) {
      ++e;
      q = 0;
    } else {
      ++q;
    }
  }
  return e;
}

// Top-k of one token: `row` its logits (missing columns are -inf), `maxima` the maxima of its groups, both in shared memory and
// used up.  Leaves the picks and returns 1 / sum of their exponentials.
template <int SUPERS>
__device__ __forceinline__ float select_topk(int k, uint32_t row, uint32_t maxima, uint32_t picks, uint32_t pick_pitch, int* s_hist,
                                             int count) {
  float sm[SUPERS];
#pragma unroll
  for (int q = 0; q < SUPERS; ++q) sm[q] = max4(lds_f4(maxima + q * 16));
  float vmax = 0.f, zs = 0.f;
#pragma unroll 1
  for (int j = 0; j < k; ++j) {
    float best = sm[0];
#pragma unroll
    for (int q = 1; q < SUPERS; ++q) best = fmaxf(best, sm[q]);
    int s = SUPERS - 1;
#pragma unroll
    for (int q = SUPERS - 2; q >= 0; --q) s = (sm[q] == best) ? q : s;
    const float4 g4 = lds_f4(maxima + s * 16);
    const int gi = first_eq4(g4, best), g = s * 4 + gi;
    const float4 v4 = lds_f4(row + g * 16);
    const int ci = first_eq4(v4, best);
    int col = g * 4 + ci;
    if (!(best > -INFINITY)) col = lowest_untaken(j, picks, pick_pitch);
    if (j == 0) vmax = best;
    const float ex = expf(best - vmax);
    zs += ex;
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(picks + j * pick_pitch), "r"(__float_as_uint(ex)), "r"(col) : "memory");
    atomicAdd(&s_hist[col], count);  // the tile's histogram (integer adds: order-free)
    const float4 nv = without(v4, ci, -INFINITY);
    sts_f4(row + g * 16, nv);
    const float4 ng = without(g4, gi, max4(nv));
    sts_f4(maxima + s * 16, ng);
    const float ns = max4(ng);
#pragma unroll
    for (int q = 0; q < SUPERS; ++q) sm[q] = (q == s) ? ns : sm[q];
  }
  return 1.f / zs;
}

__device__ __forceinline__ void routing_sync() { asm volatile("bar.sync 1, %0;" ::"n"(32 * RO_WARPS) : "memory"); }

template <int CL, int NV, bool SPLIT>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(RO_THREADS, 1)
    router_cluster_kernel(const __grid_constant__ RouterParams p) {
  static_assert(!SPLIT || (CL == RO_CHAINS && NV == 4));
  constexpr int MINE = RO_TOK / CL;             // this CTA's tokens of the tile
  constexpr int N = SPLIT ? RO_TOK : MINE;      // tokens it contracts
  constexpr uint32_t ACCS = NV / 4, TMEM_COLS = RO_CHAINS * ACCS * MINE;  // per chain an accumulator for each 128 experts, a column per token
  extern __shared__ unsigned char ro_smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * RO_MAX_STAGES + 1];  // full, empty, accumulator complete
  __shared__ uint32_t tmem_base_slot;
  __shared__ int s_hist[32 * NV];
  __shared__ __align__(16) float s_psum[RO_WARPS][32 * NV];
  __shared__ __align__(16) float s_first[40 * NV + 4];  // a row, its maxima and a pick for the first pass of the selection
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = CL > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  const int tile = blockIdx.x / CL;
  const int64_t first = static_cast<int64_t>(tile) * RO_TOK + rank * MINE, left = p.T - first;
  const int tokens = left < MINE ? static_cast<int>(left) : MINE;  // of which are there (may be negative)
  // K blocks it contracts: its chain, or all of them
  const int k_begin = SPLIT ? p.k_total * rank / RO_CHAINS : 0, k_end = SPLIT ? p.k_total * (rank + 1) / RO_CHAINS : tokens > 0 ? p.k_total : 0;
  const int k_blocks = k_end - k_begin;
  const uint32_t smem_base = (smem_u32(ro_smem_raw) + 1023u) & ~1023u;
  const uint32_t bar0 = smem_u32(bars);
  const uint32_t acc_bar = bar0 + 8u * (2 * RO_MAX_STAGES);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (RO_MAX_STAGES + s); };

  if (tid == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(acc_bar, 1);
    fence_mbar_init();
    tma_prefetch_desc(&p.map_x);
    tma_prefetch_desc(&p.map_w0);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&tmem_base_slot), TMEM_COLS);
    tmem_relinquish();
  }
  for (int i = tid; i < 32 * NV; i += RO_THREADS) s_hist[i] = 0;
  chain_wait();  // everything above touches only this CTA's own state
  init_status_block(p.status, blockIdx.x == 0 && tid == 0);  // long before a wait of this kernel can run out
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (CL > 1) cluster_arrive();  // the counts are cleared: waited for where they are added to
  const uint32_t tmem_base = tmem_base_slot;

  if (warp == 0) {
    if (elect_one()) {  // TMA producer
      int s = 0;
      uint32_t phase = 0, it = 0;
      bool ok = true;
      // (what this thread takes to refill a stage counts like latency: no divisions and no choice of maps in the loop)
      const int token0 = SPLIT ? tile * RO_TOK : static_cast<int>(first);
      int seg = k_begin / p.k_blocks, kk = (k_begin - seg * p.k_blocks) * RO_BK;
      for (int left_kb = k_blocks; left_kb > 0 && ok; ++seg, kk = 0) {
        const CUtensorMap* const mw = seg == 0 ? &p.map_w0 : (seg == 1 ? &p.map_w1 : &p.map_w2);
        const int kk_end = min(p.k_blocks * RO_BK, kk + left_kb * RO_BK);
        left_kb -= (kk_end - kk) / RO_BK;
#pragma unroll 1
        for (; kk < kk_end; kk += RO_BK, ++it) {
          const uint32_t sW = smem_base + s * p.stage_bytes, bar = full_bar(s);
          if (!mbar_wait(empty_bar(s), phase ^ 1u)) {
            ok = false;
            break;
          }
          mbar_expect_tx(bar, p.stage_bytes);
          if (p.whole_chunks) {
            tma_load_4d(sW, mw, bar, 0, kk, 0, 0);
          } else {  // E is not a multiple of 64: a box per chunk, the last one clipped
#pragma unroll 1
            for (int c = 0; c < p.w_chunks; ++c) tma_load_3d(sW + c * RO_CHUNK_BYTES, mw, bar, c * 64, kk, 0);
          }
          tma_load_2d(sW + p.w_bytes, &p.map_x, bar, kk, token0);
          if (++s == p.stages) {
            s = 0;
            phase ^= 1u;
          }
        }
      }
      chain_next();
      if (!ok) {  // gave up: the copies in flight land in this CTA's shared memory before it leaves (bounded again)
        record_status(p.status, DEV_TIMEOUT, 3100);
        const uint32_t n = static_cast<uint32_t>(p.stages);
        for (uint32_t i = it > n ? it - n : 0; i < it; ++i) mbar_wait(full_bar(i % n), (i / n) & 1u);
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {  // MMA issuer
      // (experts beyond the chunks of W_r are whatever lies behind them; their accumulator lanes are not read)
      constexpr uint32_t idesc = umma_idesc(128, N, 1, 0);
      const uint64_t descW = smem_desc(smem_base, RO_CHUNK_BYTES, 1024);
      const uint64_t descX = smem_desc(smem_base + p.w_bytes, 0, 1024);
      int s = 0;
      uint32_t phase = 0;
      bool ok = true;
      // chain c: K blocks c k_total / chains and on
      int chain = 0, first_kb = 0, next_kb = SPLIT ? k_blocks : p.k_total / p.chains;
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (kb == next_kb) {
          ++chain;
          first_kb = kb;
          next_kb = p.k_total * (chain + 1) / p.chains;
        }
        if (!mbar_wait(full_bar(s), phase)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t off = (static_cast<uint64_t>(s) * p.stage_bytes) >> 4;
#pragma unroll
        for (int ks = 0; ks < RO_BK / 16; ++ks)
#pragma unroll
          for (uint32_t h = 0; h < ACCS; ++h)
            umma_bf16(tmem_base + (chain * ACCS + h) * N, descW + off + ((h * 2 * RO_CHUNK_BYTES + ks * 2048) >> 4), descX + off + (ks * 32 >> 4), idesc,
                      kb != first_kb || ks != 0 ? 1u : 0u);
        umma_commit(empty_bar(s));
        if (++s == p.stages) {
          s = 0;
          phase ^= 1u;
        }
      }
      if (!ok) record_status(p.status, DEV_TIMEOUT, 3200);
      // also after giving up: the MMAs issued so far finish before the waiting warps go on and the tensor memory is freed
      if (k_blocks > 0)
        umma_commit(acc_bar);
      else
        mbar_arrive(acc_bar);
      if (!ok) mbar_wait(acc_bar, 0u);
    }
  } else {
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * (RO_WARPS * 32) + (tid - 64); i < p.rows;
         i += static_cast<int64_t>(gridDim.x) * (RO_WARPS * 32))
      p.row_gate[i] = 0.f;
  }

  // the logits of this CTA's tokens, over the operand stages; SPLIT: behind them, a buffer for the sums of each chain
  const uint32_t part = smem_base + (SPLIT ? p.stages * p.stage_bytes : 0u);
  constexpr uint32_t PITCH = 32 * NV * 4 + 16;  // rows 16 bytes apart in the banks
  constexpr uint32_t CHAIN_BYTES = MINE * PITCH;
  if (warp >= 2) {
    constexpr uint32_t MAX_PITCH = 32 * (NV / 4) * 4 + 16;
    const uint32_t maxima = part + (SPLIT ? RO_CHAINS : 1) * CHAIN_BYTES;  // of the groups of four columns
    const uint32_t picks = maxima + MINE * MAX_PITCH;           // {exponential, column}: k rows of MINE (and one, in other banks)
    const uint32_t pick_pitch = MINE * 8 + 8, recip = picks + p.k * pick_pitch;  // 1 / sum of the exponentials
    const int w = warp - 2, E = p.E, k = p.k;
    float acc[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) acc[q] = 0.f;
#pragma unroll 1
    for (int pass = w % 3;; pass = 3) {  // 0, 1, 2: that step only, before there is anything to route; 3: all of them
      const bool all = pass == 3;
      if (all || pass == 0) {
#pragma unroll 1
        for (int i = w; i < (all ? tokens : w + 1); i += RO_WARPS) {
          const uint32_t mrow = maxima + i * MAX_PITCH;
          float v[NV];
          float vmax = -INFINITY;
#pragma unroll
          for (int q = 0; q < NV / 4; ++q) {
            const int col = 4 * (lane + 32 * q);
            const uint32_t a = part + i * PITCH + col * 4;
            float4 sum = lds_f4(a);
            if (SPLIT) {
#pragma unroll
              for (int c = 1; c < RO_CHAINS; ++c) {
                const float4 next = lds_f4(a + c * CHAIN_BYTES);
                sum = make_float4(sum.x + next.x, sum.y + next.y, sum.z + next.z, sum.w + next.w);
              }
            }
            if (col < E) {  // E is a multiple of 8: the four columns exist or do not
              if (p.bias) {  // by words: it may lie anywhere in a buffer of parameters
                const float* const b = p.bias + col;
                sum = make_float4(sum.x + b[0], sum.y + b[1], sum.z + b[2], sum.w + b[3]);
              }
              if (i < tokens) {
                const int64_t at = (first + i) * E + col;
                *reinterpret_cast<float4*>(p.logits + at) = sum;
                if (p.logits_out) store_caller(p.logits_out + at, sum);
              }
            } else {
              sum = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            }
            if (all) sts_f4(a, sum);
            v[4 * q] = sum.x;
            v[4 * q + 1] = sum.y;
            v[4 * q + 2] = sum.z;
            v[4 * q + 3] = sum.w;
            const float m = max4(sum);
            if (all) asm volatile("st.shared.f32 [%0], %1;" ::"r"(mrow + (lane + 32 * q) * 4), "f"(m) : "memory");
            vmax = fmaxf(vmax, m);
          }
          vmax = warp_max(vmax);
          float z = 0.f;
#pragma unroll
          for (int q = 0; q < NV; ++q) {
            v[q] = expf(v[q] - vmax);
            z += v[q];
          }
          const float rz = 1.f / warp_sum(z);
#pragma unroll
          for (int q = 0; q < NV; ++q) acc[q] = fmaf(v[q], rz, acc[q]);
        }
      }
      if (all) routing_sync();
      const int t = tid - 64;
      if (all ? t < tokens : pass == 1) {
        const uint32_t scratch = smem_u32(s_first);
        const float rz = select_topk<2 * NV>(all ? k : 1, all ? part + t * PITCH : scratch,
                                             all ? maxima + t * MAX_PITCH : scratch + 32 * NV * 4,
                                             all ? picks + t * 8 : scratch + 40 * NV * 4, pick_pitch, s_hist, all ? 1 : 0);
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(all ? recip + t * 4 : scratch + 40 * NV * 4 + 8), "f"(rz) : "memory");
      }
      if (all) routing_sync();
      if (all || pass == 2) {
#pragma unroll 1
        for (int i = t; i < tokens * k; i += 32 * RO_WARPS) {
          const int tok = i / k, j = i - tok * k;
          uint32_t exb, col;
          asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(exb), "=r"(col) : "r"(picks + j * pick_pitch + tok * 8) : "memory");
          const float g = __uint_as_float(exb) * __int_as_float(lds_int(recip + tok * 4));
          const int64_t at = first * k + i;
          p.idx[at] = static_cast<int32_t>(col);
          p.gates[at] = g;
          p.idx_out[at] = static_cast<int32_t>(col);
          p.gates_out[at] = g;
          if (!all) break;
        }
      }
      if (all) break;
      // logits: tensor memory (lane = expert, column = token) -> shared memory (the operand stages have all been consumed)
      const bool ok = mbar_wait(acc_bar, 0u);
      if (!ok && lane == 0) record_status(p.status, DEV_TIMEOUT, 3300);
      tc_fence_after();
      const int ew = warp & 3;
      if constexpr (SPLIT) {
        // the chain's sums of every token go to the CTA that routes it
        cluster_wait();  // all four run
        if (ok)
#pragma unroll 1
          for (int c = w >> 2; c < RO_TOK / 16; c += RO_WARPS / 4) {
            const int e = ew * 32 + lane, tok0 = c * 16;
            uint32_t r[16];
            tmem_ld16(tmem_base + (static_cast<uint32_t>(ew * 32) << 16) + tok0, r);
            tmem_ld_wait();
            const uint32_t to = mapa_shared(part + rank * CHAIN_BYTES + (tok0 % MINE) * PITCH + e * 4, tok0 / MINE);
            if (e < E)
#pragma unroll
              for (int i = 0; i < 16; ++i) st_cluster_f32(to + i * PITCH, __uint_as_float(r[i]));
          }
        tc_fence_before();
        cluster_sync_diverged();  // the sums of all chains are there
      } else if (ok && tokens > 0) {
#pragma unroll 1
        for (int c = w >> 2; c < static_cast<int>(ACCS) * (MINE / 16); c += RO_WARPS / 4) {
          const int e = c / (MINE / 16) * 128 + ew * 32 + lane, tok0 = c % (MINE / 16) * 16;
          uint32_t r[RO_CHAINS][16];
#pragma unroll
          for (int q = 0; q < RO_CHAINS; ++q)
            if (q < p.chains) tmem_ld16(tmem_base + (static_cast<uint32_t>(ew * 32) << 16) + q * (ACCS * MINE) + c * 16, r[q]);
          tmem_ld_wait();
          float sum[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) sum[i] = __uint_as_float(r[0][i]);
#pragma unroll
          for (int q = 1; q < RO_CHAINS; ++q)
            if (q < p.chains)
#pragma unroll
              for (int i = 0; i < 16; ++i) sum[i] += __uint_as_float(r[q][i]);
          if (e < E)
#pragma unroll
            for (int i = 0; i < 16; ++i) asm volatile("st.shared.f32 [%0], %1;" ::"r"(part + (tok0 + i) * PITCH + e * 4), "f"(sum[i]) : "memory");
        }
      }
      if (!SPLIT) {
        tc_fence_before();
        routing_sync();
      }
#pragma unroll
      for (int q = 0; q < NV; ++q) acc[q] = 0.f;
    }
#pragma unroll
    for (int q = 0; q < NV; ++q) s_psum[w][4 * (lane + 32 * (q / 4)) + q % 4] = acc[q];
    routing_sync();
    if (CL > 1 && !SPLIT) cluster_wait();  // the tile's first CTA has cleared its counts
    const int e = tid - 64;
    if (e < E) {
      float s = 0.f;
#pragma unroll 4
      for (int u = 0; u < RO_WARPS; ++u) s += s_psum[u][e];
      if (tokens > 0) p.psum_part[static_cast<int64_t>(blockIdx.x) * E + e] = s;
      if (CL > 1 && rank != 0 && tokens > 0) red_cluster_add(mapa_shared(smem_u32(&s_hist[e]), 0), s_hist[e]);
      if (CL == 1) p.tile_counts[static_cast<int64_t>(tile) * E + e] = s_hist[e];
    }
  } else if (CL > 1) {
    cluster_wait();
    if (SPLIT) cluster_sync_diverged();
  }
  if (CL > 1)
    cluster_sync_diverged();  // the counts of the tile are complete
  else
    block_sync_diverged();  // tensor memory has been read
  if (CL > 1 && rank == 0 && tid >= 64 && tid - 64 < p.E) p.tile_counts[static_cast<int64_t>(tile) * p.E + tid - 64] = s_hist[tid - 64];
  if (warp == 1) {
    __syncwarp();  // freeing tensor memory takes the whole warp
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

// CTAs per token tile: as many as have an SM each, and more than one wave of them only where there is no choice.  Clusters of four
// do not fill the chip (they lie within a part of it), so they go up to eight ninths of the SMs.  Router stage, us, with one / two /
// four at d 2048 and 128 experts: 128 tokens 25 / 23 / 20, 4096 (128 CTAs of four) 26 / 24 / 21, 4737 (152) 26 / 24 / 35, 8192 27 / 25 / 35,
// 9472 (148 CTAs of two) 29 / 26 / 49, 9473 29 / 39 / 49, 16384 33 / 45 / 65, 32768 59 / 85 / 129.  Above 128 experts one CTA's accumulators
// do not fit: 256 experts, two / four: 28 / 25 at 128 tokens, 29 / 25 at 4096, 29 / 43 at 4737, 54 / 82 at 16384.  With few experts the rows
// of W_r are short and come slowly however few they are, and all CTAs ask for the same lines, so that two are worse than one: d 4096
// and 8 experts 32 / 33 at 4737, 37 / 43 at 8192, 39 / 46 at 9472; d 256 and 8 experts 19 / 18 at 4737, 20 / 20 at 8192.
// One CTA per tile in the persistent GEMM template, four warps routing: 27 at 128 to 4096 tokens, 28 at 8192, 32 at 16384, 54 at 32768.
int router_cluster(const Shape& s, int sm_count, int64_t T) {
  const int64_t tiles = (T + RO_TOK - 1) / RO_TOK;
  if (tiles * 4 * 9 <= sm_count * 8) return 4;
  return s.E <= 128 && (s.E < 32 || tiles * 2 > sm_count) ? 1 : 2;
}

template <int CL, int NV, bool SPLIT = false>
static moe_status launch_one(moe_ctx_impl* ctx, RouterParams& p, int tiles, cudaStream_t st) {
  auto* const kernel = router_cluster_kernel<CL, NV, SPLIT>;
  // the stages (and what an MMA reads behind an odd number of chunks), and over them what the routing needs: the logits of the
  // CTA's tokens, the maxima of their groups, and {pick, column} and 1 / sum for k picks
  constexpr size_t mine = RO_TOK / CL;
  auto routing = [](int k) {
    return (SPLIT ? RO_CHAINS : 1) * mine * (128 * NV + 16) + mine * (32 * NV + 16) + k * (mine * 8 + 8) + mine * 4;
  };
  auto smem_of = [](size_t ring, size_t over) { return (SPLIT ? ring + over : ring > over ? ring : over) + 1024; };
  constexpr int ring = SPLIT ? RO_SPLIT_RING : RO_RING;
  p.w_bytes = p.w_chunks * RO_CHUNK_BYTES;
  p.stage_bytes = p.w_bytes + (SPLIT ? RO_TOK : mine) * RO_BK * 2;
  p.stages = std::min<int>(ring / p.stage_bytes, RO_MAX_STAGES);
  const size_t smem = smem_of(p.stages * p.stage_bytes + (p.w_chunks & 1) * RO_CHUNK_BYTES, routing(p.k));
  constexpr int slot = SPLIT ? 3 : (CL == 1 ? 0 : CL == 2 ? 1 : 2) + (NV == 4 ? 0 : 4);
  if (!(ctx->router_attr & (1u << slot))) {  // per device (the context is bound to one), and for every context on it: the most of all
    const size_t most = smem_of(ring + RO_CHUNK_BYTES, routing(MAX_K));
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(most)) != cudaSuccess)
      return MOE_ERR_CUDA;
    ctx->router_attr |= 1u << slot;
  }
  launch_kernel(kernel, tiles * CL, RO_THREADS, smem, st, p);
  return cudaGetLastError() == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
}

moe_status launch_router_tc(moe_ctx_impl* ctx, int64_t T, const WsLayout& L, char* ws, const GemmIO& io, cudaStream_t st) {
  const Shape& s = ctx->s;
  void* fn = ctx->encode_fn;
  RouterParams p;
  memset(&p, 0, sizeof(p));
  p.E = s.E;
  p.k = s.k;
  p.T = T;
  p.w_chunks = (s.E + 63) / 64;
  p.whole_chunks = s.E % 64 == 0;
  auto map_w = [&](CUtensorMap* m, const uint16_t* w) {  // W_r as a one-slab tensor of weights
    return p.whole_chunks ? map_mn(fn, m, w, 1, s.d, s.E, p.w_chunks) : map_3d(fn, m, w, 1, s.d, s.E, 64);
  };
  p.k_blocks = s.d / RO_BK;
  p.k_total = p.k_blocks * (io.W_r_mid ? 3 : 1);
  p.chains = p.k_total >= RO_CHAINS ? RO_CHAINS : p.k_total >= 2 ? 2 : 1;
  const int cl = router_cluster(s, ctx->sm_count, T);
  const bool split = cl == RO_CHAINS && s.E <= 128 && p.chains == RO_CHAINS;
  bool ok = map_2d(fn, &p.map_x, io.x, T, s.d, split ? RO_TOK : RO_TOK / cl) && map_w(&p.map_w0, io.W_r);
  if (io.W_r_mid) ok = ok && map_w(&p.map_w1, io.W_r_mid) && map_w(&p.map_w2, io.W_r_lo);
  if (!ok) return MOE_ERR_CUDA;
  p.status = reinterpret_cast<int32_t*>(ws + L.status);
  p.row_gate = reinterpret_cast<float*>(ws + L.row_gate);
  p.rows = L.rows_alloc;
  p.bias = io.b_r;
  p.logits = reinterpret_cast<float*>(ws + L.logits);
  p.logits_out = io.logits_out;
  p.idx = reinterpret_cast<int32_t*>(ws + L.idx);
  p.gates = reinterpret_cast<float*>(ws + L.gates);
  p.idx_out = io.idx_out;
  p.gates_out = io.gates_out;
  p.psum_part = reinterpret_cast<float*>(ws + L.psum_part);
  p.tile_counts = reinterpret_cast<int32_t*>(ws + L.tile_counts);
  const int tiles = static_cast<int>((T + RO_TOK - 1) / RO_TOK);
  if (s.E <= 128) {
    switch (cl) {
      case 4: return split ? launch_one<4, 4, true>(ctx, p, tiles, st) : launch_one<4, 4>(ctx, p, tiles, st);
      case 2: return launch_one<2, 4>(ctx, p, tiles, st);
      default: return launch_one<1, 4>(ctx, p, tiles, st);
    }
  }
  return cl == 4 ? launch_one<4, 8>(ctx, p, tiles, st) : launch_one<2, 8>(ctx, p, tiles, st);
}

}  // namespace moe
