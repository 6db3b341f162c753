// Grouped GEMMs of the MoE layer on tcgen05 tensor cores (sm_100a).
//
// One persistent, warp-specialised kernel template serves the six contractions of the layer:
//   F3  [hg|hu] = xp  W_gate[e] | W_up[e]          + SwiGLU epilogue (writes hg, hu and act = gate silu(hg) hu)
//   F4  o       = act W_down[e]
//   B2  da      = dy_rows W_down[e]^T               + SwiGLU-backward epilogue (reads hg, hu; writes dhg, dhu, dg partials)
//   B4  dxp     = dhg W_gate[e]^T + dhu W_up[e]^T   (one accumulator, two K segments)
//   B3  dW_down[e]          = act_e^T dy_rows_e     (K = rows of expert e, one CTA owns a whole output tile)
//   B5  dW_gate[e]|dW_up[e] = xp_e^T [dhg_e|dhu_e]
// and the two contractions of the router's backward pass, whose operands are bf16 (or fp32 split exactly into two bf16
// terms), so that a bf16 MMA with fp32 accumulation is an fp32 contraction up to summation order:
//   DX  dxr    = dl_hi W_r^T + dl_lo W_r^T          (router term of dx; the unpermute kernel adds the dxp rows)
//   DWR dW_r partial[s] = x_s^T (dl_hi + dl_lo)_s   (token slices s; partials are summed by a small kernel)
// Tiles are 128 x 256 with K steps of 64; operands arrive by TMA into 128-byte-swizzled shared memory (4 stages),
// the accumulator lives in tensor memory (2 x 256 columns, so the epilogue of one tile overlaps the main loop
// of the next).  Operand major-ness replaces every transpose: row-major [rows, K] is a K-major operand,
// row-major [K, cols] is an MN-major operand, and the UMMA instruction takes either.
// Row buffers are expert-major with each expert's segment padded to 128 rows of zeros, so an M tile never
// straddles two experts and the ragged K of the weight gradients needs no masking.
// Warp roles: warp 0 TMA producer, warp 1 MMA issuer (owns the TMEM allocation), warps 2..9 epilogue.  The expert-LoRA
// variant runs on the same template (launch_lora_gemm at the end of this file); the router's forward pass is in router.cu.
// Every mbarrier wait is bounded; on a timeout the kernel records it in the status word and leaves.
#include <math.h>

#include "gemm_common.cuh"
#include "tensor_maps.cuh"

namespace moe {

// Block `worker` of `workers`
template <int KIND, Accumulate ACC>
__device__ __forceinline__ void grouped_gemm(const GemmParams& p, const int worker, const int workers) {
  using TR = Traits<KIND>;
  constexpr int EPI_WARPS = 8;
  extern __shared__ __align__(1024) unsigned char gemm_smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t smem_base = smem_u32(gemm_smem_raw);
  // barriers: full, empty, accumulator full / empty, drain (failure path); behind them the base of the accumulators
  constexpr int BARS = STAGES * STAGE_BYTES + EPI_BYTES, TMEM_SLOT = BARS + 8 * (2 * STAGES + 5);
  const uint32_t bar0 = smem_base + BARS;
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
  auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * STAGES + a); };
  auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * STAGES + 2 + a); };

  constexpr bool teams = EpilogueTeams<KIND, ACC>::value;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull_bar(a), 1);
      mbar_init(tempty_bar(a), (teams ? 16 : 32) * EPI_WARPS);
    }
    mbar_init(bar0 + 8u * (2 * STAGES + 4), 1);
    fence_mbar_init();
    tma_prefetch_desc(&p.mapA0);
    tma_prefetch_desc(&p.mapB0);
  }
  if (warp == 1) {
    tmem_alloc(smem_base + TMEM_SLOT, TMEM_COLS);
    tmem_relinquish();
  }
  // Row GEMMs of the experts wait for the kernel before them in front of their rows (chain_warp).  Not dgrad-down, whose epilogue needs all
  // registers (with it 8 bytes of them go to memory): alone 36.4 -> 35.4 us at d 768, f 2048 and 125 rows per expert, 64.4 -> 62.1 at 500 rows, where
  // steps take 150.5 -> 150.2 and 355.5 -> 352.2.
  constexpr bool PRELOAD = !TR::WGRAD && !TR::STATIC_M && KIND != GEMM_B2;
  if (!PRELOAD && !p.ready) chain_wait();  // everything above touches only this CTA's own state
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *reinterpret_cast<const volatile uint32_t*>(gemm_smem_raw + TMEM_SLOT);
  const int ntiles = total_tiles<KIND>(p);

  // The producer and the MMA issuer are one thread each.  What they do per K block (a wait, a few copies or four MMAs, a
  // commit) has to fit well inside the 512 cycles that the tensor core needs for it; run by a whole warp with one lane
  // enabled, with a division for the stage index, it took 400 - 700 cycles and set the pace of every kernel here.  With the
  // issuer alone run by a whole warp gate/up at 1024 rows per expert takes 757 us instead of 688.
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (elect_one()) {
      RingPos pos;
      uint32_t it = 0;
      bool ok = true;
      RoleClock clk(p.timers);
      int kb = 0;  // the first K block of the first tile that is not on its way yet
      Tile tl = {};
      if (PRELOAD) {
        const bool any = worker < ntiles;
        if (any) tl = get_tile<KIND>(p, worker);
        const int pre = any ? min(STAGES, p.k_blocks) : 0;
        for (int i = 0; i < pre; ++i) {
          mbar_expect_tx(full_bar(i), p.stage_tx);
          issue_loads<KIND, 2>(p, tl, i, 0, smem_base + i * STAGE_BYTES + A_BYTES, full_bar(i));
        }
        if (!p.ready) chain_wait();
        for (; kb < pre; ++kb, ++it) {
          issue_loads<KIND, 1>(p, tl, kb, smem_base + kb * STAGE_BYTES, 0, full_bar(kb));
          pos.next(STAGES);
        }
      }
      for (int rd = 0; rd * workers < ntiles && ok; ++rd, kb = 0) {
        const int t = tile_of_round<KIND>(rd, worker, workers);
        if (t >= ntiles) continue;
        if (!PRELOAD || rd) tl = get_tile<KIND>(p, t);
        for (; kb < tl.nkb; ++kb, ++it) {
          clk.start();
          if (!mbar_wait(empty_bar(pos.s), pos.phase ^ 1u)) {
            ok = false;
            break;
          }
          clk.add(0);
          const uint32_t sA = smem_base + pos.s * STAGE_BYTES;
          mbar_expect_tx(full_bar(pos.s), p.stage_tx);
          issue_loads<KIND>(p, tl, kb, sA, sA + A_BYTES, full_bar(pos.s));
          pos.next(STAGES);
        }
      }
      clk.report(0, 1);  // total; waiting for a free stage
      // Not earlier without next_early: blocks of the next kernel that only wait would sit beside the main loop.  A trigger comes after
      // a wait everywhere (chain_warp): a `ready` block without tiles, or whose K loop fits the ring, gets here while its predecessor runs.
      if (p.ready) chain_wait();
      chain_next();
      if (!ok) {
        // gave up: the copies already issued still land in this CTA's shared memory - wait for them (bounded again)
        // before the CTA may exit
        record_status(p.status, DEV_TIMEOUT, 100 + KIND);
        for (uint32_t i = it > static_cast<uint32_t>(STAGES) ? it - STAGES : 0; i < it; ++i)
          mbar_wait(full_bar(i % STAGES), (i / STAGES) & 1u);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (elect_one()) {
      const uint32_t idesc = umma_idesc(BM, p.mma_n, TR::A_MN, TR::B_MN);
      constexpr uint32_t A_KSTEP = TR::A_MN ? 2048 : 32, B_KSTEP = TR::B_MN ? 2048 : 32;  // bytes per K = 16
      const uint64_t descA = smem_desc(smem_base, TR::A_MN ? CHUNK_BYTES : 0, 1024);
      const uint64_t descB = smem_desc(smem_base + A_BYTES, TR::B_MN ? CHUNK_BYTES : 0, 1024);
      RingPos pos;
      uint32_t tc = 0;
      bool ok = true;
      RoleClock clk(p.timers);
      for (int rd = 0; rd * workers < ntiles && ok; ++rd) {
        const int t = tile_of_round<KIND>(rd, worker, workers);
        if (t >= ntiles) continue;
        const Tile tl = get_tile<KIND>(p, t);
        if (tl.nkb == 0) continue;
        const int acc = tc & 1;
        const uint32_t aph = (tc >> 1) & 1u;
        ++tc;
        clk.start();
        if (!mbar_wait(tempty_bar(acc), aph ^ 1u)) {
          ok = false;
          break;
        }
        clk.add(0);
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * ACC_COLS;
        // Asking for the next stage before this one's MMAs are issued lets a copy that has landed be seen early; where none
        // has, try_wait may hold the thread for a moment.  With it, without it and with test_wait in its place the row GEMMs at
        // 62 to 1024 rows per expert take the same time, within 1 %.
        bool ready = false;  // the stage about to be used was already seen full
        for (int kb = 0; kb < tl.nkb; ++kb) {
          clk.start();
          if (!ready && !mbar_wait(full_bar(pos.s), pos.phase)) {
            ok = false;
            break;
          }
          clk.add(1);
          tc_fence_after();
          const uint64_t off = (pos.s * STAGE_BYTES) >> 4;
          const uint32_t done = empty_bar(pos.s);
          pos.next(STAGES);
          ready = kb + 1 < tl.nkb && mbar_try_wait(full_bar(pos.s), pos.phase);
          const int nks = kb == tl.nkb - 1 ? tl.klast : BK / 16;
#pragma unroll
          for (int ks = 0; ks < BK / 16; ++ks)
            if (ks < nks)
              umma_bf16(d_tmem, descA + off + (ks * A_KSTEP >> 4), descB + off + (ks * B_KSTEP >> 4), idesc,
                        (kb | ks) != 0 ? 1u : 0u);
          umma_commit(done);
        }
        if (ok) umma_commit(tfull_bar(acc));
      }
      clk.report(2, 3, 4);  // total; waiting for a drained accumulator; waiting for operands
      if (!ok) {
        // gave up: let every MMA issued so far finish (bounded) before the tensor memory is freed
        record_status(p.status, DEV_TIMEOUT, 200 + KIND);
        umma_commit(bar0 + 8u * (2 * STAGES + 4));
        mbar_wait(bar0 + 8u * (2 * STAGES + 4), 0u);
      }
    }
  } else if (warp < 2 + EPI_WARPS) {
    // ------------------------------------------------------------------ epilogue (128 TMEM lanes; two warps per
    // lane quadrant, each draining half of the tile's columns, or every other tile: EpilogueTeams)
    const int ew = warp & 3;           // TMEM lane quadrant this warp may read
    const int half = (warp - 2) >> 2;  // which half of the columns
    EpiStage es{smem_base + STAGES * STAGE_BYTES + (warp - 2) * (EPI_UNITS * EPI_UNIT_BYTES), 0u};
    uint32_t tc = 0;
    bool ok = true;
    if (PRELOAD && !p.ready) chain_wait();  // for what it reads itself
    auto clocked = [&]() { return p.timers && threadIdx.x == 64; };  // asked again each time: a flag would cost a register
    if (clocked()) sum_cycles(p.timers + 5, false);  // total
    for (int rd = 0; rd * workers < ntiles && ok; ++rd) {
      const int t = tile_of_round<KIND>(rd, worker, workers);
      if (t >= ntiles) continue;
      const Tile tl = get_tile<KIND>(p, t);
      const int rin = ew * 32 + lane;  // row inside the tile
      if (tl.nkb == 0) {
        // weight gradient of an expert without tokens: zeros
        if (half != 0) continue;
        if (KIND == GEMM_DWR) {
          const int m = tl.m0 + rin;
          if (m < p.M_total)
            for (int col = tl.n0; col < min(tl.n0 + 128, p.N_total); col += 4)
              *reinterpret_cast<float4*>(p.outf + (static_cast<int64_t>(tl.e) * p.M_total + m) * p.N_total + col) =
                  make_float4(0.f, 0.f, 0.f, 0.f);
        } else if (TR::WGRAD) {
          wgrad_zero_fill<KIND>(p, tl.e, tl.m0 + rin, tl.n0);
        }
        continue;
      }
      const int acc = tc & 1;
      const uint32_t aph = (tc >> 1) & 1u;
      ++tc;
      if (teams && acc != half) continue;  // the other team's tile
      epilogue_prefetch<KIND, ACC>(p, static_cast<int64_t>(tl.row0) + rin, tl.n0, teams || half == 0, tl.e, tl.m0 + rin);
      if (clocked()) sum_cycles(p.timers + 6, false);  // waiting for a finished accumulator
      if (!mbar_wait(tfull_bar(acc), aph)) {
        ok = false;
        break;
      }
      if (clocked()) sum_cycles(p.timers + 6, true);
      tc_fence_after();
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(ew * 32) << 16) + acc * ACC_COLS;
      const int64_t row = static_cast<int64_t>(tl.row0) + rin;
      int part = teams ? 0 : half;  // which half of the columns
      const int last = teams ? 1 : half;
      auto release = [&]() {
        if (part != last) return;
        tc_fence_before();
        mbar_arrive(tempty_bar(acc));
      };
      if (KIND == GEMM_DWR) {
        // fp32 partial of dW_r for this token slice: hi and lo halves of dl share one accumulator pair
        const int m = tl.m0 + rin;
#pragma unroll 1
        for (int c = 2 * half; c < 2 * half + 2; ++c) {
          uint32_t rh[32], rl[32];
          tmem_ld32(taddr + c * 32, rh);
          tmem_ld32(taddr + 128 + c * 32, rl);
          tmem_ld_wait();
          const int col = tl.n0 + c * 32;
          if (m < p.M_total) {
            float* dst = p.outf + (static_cast<int64_t>(tl.e) * p.M_total + m) * p.N_total + col;
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
              if (col + i >= p.N_total) continue;
              float4 v = make_float4(
                  __uint_as_float(rh[i]) + __uint_as_float(rl[i]), __uint_as_float(rh[i + 1]) + __uint_as_float(rl[i + 1]),
                  __uint_as_float(rh[i + 2]) + __uint_as_float(rl[i + 2]), __uint_as_float(rh[i + 3]) + __uint_as_float(rl[i + 3]));
              if (p.acc_fp32) {
                const float4 old = *reinterpret_cast<const float4*>(dst + i);
                v = make_float4(old.x + v.x, old.y + v.y, old.z + v.z, old.w + v.w);
              }
              *reinterpret_cast<float4*>(dst + i) = v;
            }
          }
        }
      } else {
#pragma unroll 1
        for (; part <= last; ++part)
          expert_epilogue<KIND, ACC>(p, tl.e, row, (TR::WGRAD ? tl.m0 : tl.row0) + ew * 32, tl.n0, taddr, true,
                                     TR::WGRAD          ? p.M_total - (tl.m0 + ew * 32)
                                     : KIND == GEMM_DX ? static_cast<int>(p.T - tl.row0 - ew * 32)
                                     : p.clip_rows     ? tl.valid - ew * 32
                                                       : 32,
                                     es, lane, part, release);
      }
      if (KIND == GEMM_DWR) release();
    }
    if (clocked()) {
      sum_cycles(p.timers + 5, true);
      atomicAdd(p.timers + 7, 1ull);  // CTAs counted
    }
    if (!ok && lane == 0) {
      record_status(p.status, DEV_TIMEOUT, 300 + KIND);
    }
  } else {
    chain_warp(p.next_early);
  }

  // 31 lanes of the producer's and the issuer's warps have passed by their roles: the barrier takes threads one by one.  (A
  // warp barrier in front of an aligned one changes the code of the roles' loops: dgrad gate/up on pairs 656 -> 664 us.)
  tc_fence_before();
  block_sync_diverged();
  if (warp == 1) {
    __syncwarp();  // freeing tensor memory takes the whole warp
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

template <int KIND, Accumulate ACC = Accumulate::NONE>
__global__ void __launch_bounds__(GEMM_THREADS, 1) grouped_gemm_kernel(const __grid_constant__ GemmParams p) {
  grouped_gemm<KIND, ACC>(p, blockIdx.x, gridDim.x);
}

// The two contractions over dl side by side: the first `dx_blocks` blocks DX, the others DWR.  Both are a launch and the latency of a
// tile or two up to some thousand tokens, and equal in work beyond (with an fp32 router weight DX has three segments to DWR's two).  One
// after the other -> together, us a step: the smallest shape (d 256, f 512, 8 experts, 256 tokens) 66.2 -> 64.7; 1000 tokens and more at
// d 2048 alike (0.998, 0.997).  The launches alone, between events, with dwr_reduce_kernel: 25 -> 26 at 1000 tokens, 34 -> 33 at 4096, 73 -> 69 at
// 16384, with an fp32 weight 27 -> 26, 36 -> 33, 81 -> 86.
__global__ void __launch_bounds__(GEMM_THREADS, 1)
    router_gradient_kernel(const __grid_constant__ GemmParams dx, const __grid_constant__ GemmParams dwr, int dx_blocks) {
  const int block = blockIdx.x;
  if (block < dx_blocks)
    grouped_gemm<GEMM_DX, Accumulate::NONE>(dx, block, dx_blocks);
  else
    grouped_gemm<GEMM_DWR, Accumulate::NONE>(dwr, block - dx_blocks, gridDim.x - dx_blocks);
}

// ------------------------------------------------------------------------------------------ host side
template <int KIND, Accumulate ACC = Accumulate::NONE>
static moe_status launch_kind(moe_ctx_impl* ctx, const GemmParams& p, cudaStream_t st) {
  auto* const kernel = grouped_gemm_kernel<KIND, ACC>;
  unsigned char* const done = &ctx->attr_done[ACC == Accumulate::LOAD_ADD ? 2 : 0][KIND];
  if (!*done) {  // per device: the context is bound to one
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(GEMM_SMEM)) != cudaSuccess)
      return MOE_ERR_CUDA;
    *done = 1;
  }
  launch_kernel(kernel, ctx->sm_count, GEMM_THREADS, GEMM_SMEM, st, p);
  return cudaGetLastError() == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;  // reported here, and not by the next call once more
}

// Row tiles (or pairs) walked together inside a column tile: 1 while the expert's weights are few column tiles wide (they
// stay in L2 between row tiles: Qwen3-30B-A3B shape), 16 for wide experts (coarse shape: at 112 column tiles an expert's
// gate and up slabs are 235 MB and were read from DRAM once per row pair).  A group ends with its expert (expert_tile_order): a
// step at that shape then reads 1.9 GB less for gate/up, 4 GB less for dgrad gate/up and takes, with 512 / 1024 / 4096 rows per
// expert and the weight gradients in groups as well, 4640 -> 4275, 8130 -> 7590 and 31200 -> 28600 us (at the power cap, where a
// byte from DRAM costs what 110 flops do).  MOE_ROW_GROUP overrides (measurements).
int row_group_for(int n_tiles, const moe_ctx_impl* ctx) {
  if (ctx->row_group_override > 0) return ctx->row_group_override;
  return n_tiles > 12 ? 16 : 1;
}

// The same for a weight gradient on CTA pairs: 256-row tiles of the output walked together inside a column tile.  With column
// tiles fastest every row tile reads the operand of the columns (`columns` wide, the expert's rows long) from DRAM again once
// that operand has outgrown L2; walked in groups, row and column operands are shared by the pairs that run at the same time.
// wgrad gate/up at d 4096, f 14336, 4096 rows per expert: 25.9 -> 6.6 GB read, 6013 -> 5110 us; at 1024 rows (59 MB) 2.34 -> 0.56 GB,
// 1426 -> 1285 us, a step 6414 -> 6275 at 768 rows, 4616 -> 4547 at 512 (29 MB).  With 15 MB (256 rows, one-CTA tiles) nothing is read
// twice either way and rows of adjacent columns leave together: 662 -> 704 us in groups.  Hence above 24 MB, and where there are more
// column tiles than a group has rows.
static int wgrad_group_for(int n_tiles, double rows_per_expert, int64_t columns, const moe_ctx_impl* ctx) {
  if (ctx->row_group_override > 0) return ctx->row_group_override;
  return n_tiles > 16 && rows_per_expert * static_cast<double>(columns) * 2.0 >= 24e6 ? 16 : 1;
}

// Whether the pairs of a GEMM keep step (Pace): where L2 does not hold what they share - the weights of wide experts, which row GEMMs
// walk in groups, or the operands of one expert's weight gradient (24 MB as above) - and tiles are long, from 32 K blocks (about
// 14 us) on: a round begins with a question that takes 1 us.  MOE_ROW_GROUP=1 lets all pairs run freely (measurements).
static bool keeps_step(int row_group, bool wgrad, double k_blocks, double operand_bytes, const moe_ctx_impl* ctx) {
  return ctx->row_group_override != 1 && k_blocks >= 32.0 && (wgrad ? operand_bytes >= 24e6 : row_group > 1);
}

// Forward-only calls leave pad rows alone (nothing reads them afterwards), which at few rows per expert is most of what
// the activations move: scoring 241 tokens (15 rows per expert) 296 -> 268 us, 2048 tokens 367 -> 356 us.  Below 192
// rows per expert most tiles are partial as well, and A comes in groups of 32 rows of which the empty ones are not read:
// 268 -> 263 us and 356 -> 354 us.  Above, the extra copy instructions cost more than the reads they save (with them at
// 1024 rows per expert 1437 -> 1557 us).
static void clip_pads(GemmParams* p, bool forward_only, double rows_per_expert) {
  p->clip_rows = forward_only ? 1 : 0;
  p->part_rows = forward_only && rows_per_expert < 192.0 ? 1 : 0;
}

// One launch of an expert / router contraction.  `pair`: CTA-pair kernel.  `part`: 0 = the whole tile list; row GEMMs
// of the mixed schedule: 1 = the pair kernel over complete pairs of row blocks only, 2 = the one-CTA kernel over the
// leftover blocks.
// `only`: DX, DWR - leaves the parameters there and launches nothing.
static moe_status launch_gemm_variant(moe_ctx_impl* ctx, GemmKind kind, int64_t T, const WsLayout& L, char* ws,
                                      const GemmIO& io, cudaStream_t st, bool pair, int part, GemmParams* only = nullptr) {
  const uint16_t *W_gate = io.W_gate, *W_up = io.W_up, *W_down = io.W_down;
  uint16_t *dW_gate = io.dW_gate, *dW_up = io.dW_up, *dW_down = io.dW_down;
  const Shape& s = ctx->s;
  const int d = s.d, f = s.f, E = s.E;
  const int64_t R = L.rows_max;
  const double rows_per_expert = static_cast<double>(T) * s.k / E;
  void* fn = ctx->encode_fn;
  uint16_t* xp = reinterpret_cast<uint16_t*>(ws + L.xp);
  uint16_t* hg = reinterpret_cast<uint16_t*>(ws + L.hg);
  uint16_t* hu = reinterpret_cast<uint16_t*>(ws + L.hu);
  uint16_t* act = reinterpret_cast<uint16_t*>(ws + L.act);
  uint16_t* o = reinterpret_cast<uint16_t*>(ws + L.o);
  uint16_t* dhg = reinterpret_cast<uint16_t*>(ws + L.dhg);
  uint16_t* dhu = reinterpret_cast<uint16_t*>(ws + L.dhu);
  uint16_t* dxp = reinterpret_cast<uint16_t*>(ws + L.dxp);
  GemmParams p;
  memset(&p, 0, sizeof(p));
  p.sched = reinterpret_cast<const int32_t*>(ws + L.sched);
  p.tile_expert = reinterpret_cast<const int32_t*>(ws + L.tile_expert);
  p.pad_offsets = reinterpret_cast<const int32_t*>(ws + L.pad_offsets);
  p.counts = reinterpret_cast<const int32_t*>(ws + L.counts);
  p.pair_tab = reinterpret_cast<const int32_t*>(ws + L.pair_tab);
  p.expert_order = reinterpret_cast<const int32_t*>(ws + L.expert_order);
  p.timers = ctx->gemm_timers ? reinterpret_cast<unsigned long long*>(ws + L.timers) + 8 * kind : nullptr;
  if (part == 1) {
    p.pair_tab = reinterpret_cast<const int32_t*>(ws + L.fpair_tab);
    p.pair_count_slot = 3;
  } else {
    p.pair_count_slot = 2;
  }
  p.oob_row = static_cast<int>(R);
  p.tile_list = part == 2 ? reinterpret_cast<const int32_t*>(ws + L.single_tab) : nullptr;
  p.status = reinterpret_cast<int32_t*>(ws + L.status);
  p.E = E;
  if ((kind == GEMM_B3 || kind == GEMM_B5) && io.e_count > 0) {  // one group of experts, in index order
    p.E = io.e_count;
    p.e_first = io.e_first;
    p.expert_grouped = 1;
  }
  p.ready = io.ready ? 1 : 0;
  p.next_early = io.next_early ? 1 : 0;
  p.mma_n = BN;
  p.stage_tx = STAGE_BYTES;
  p.nseg = (kind == GEMM_B4 || kind == GEMM_DX) ? 2 : 1;
  p.k_blocks1 = 0;
  p.out_scale = 1.f;
  auto on_pairs = [&]() {
    const bool wgrad = kind == GEMM_B3 || kind == GEMM_B5;
    const double blocks = wgrad ? rows_per_expert / BK : p.k_blocks * p.nseg;
    const double operands = rows_per_expert * 2.0 * (kind == GEMM_B5 ? d + 2.0 * f : d + static_cast<double>(f));
    if (part == 0 && keeps_step(p.row_group, wgrad, blocks, operands, ctx)) p.pace = reinterpret_cast<int32_t*>(ws + L.pace) + kind * PACE_SLOTS;
    return launch_pair_gemm(ctx, kind, p, st);
  };
  bool ok = true;
  switch (kind) {
    case GEMM_F3:
      ok = map_2d(fn, &p.mapA0, xp, R, d, 128) && map_2d(fn, &p.mapS0, xp, R, d, 32) &&
           map_mn(fn, &p.mapB0, W_gate, E, d, f, 2) && map_mn(fn, &p.mapB1, W_up, E, d, f, 2);
      p.mapA1 = p.mapA0;
      clip_pads(&p, !io.save_preactivations, rows_per_expert);
      p.n_tiles = (f + 127) / 128;
      p.k_blocks = d / BK;
      p.N_total = f;
      p.out0 = hg; p.out1 = hu; p.out2 = act;
      p.ld_out = f;
      p.row_gate = reinterpret_cast<const float*>(ws + L.row_gate);
      p.save_pre = io.save_preactivations ? 1 : 0;
      if (!ok) return MOE_ERR_CUDA;
      p.row_group = row_group_for(p.n_tiles, ctx);
      return pair ? on_pairs() : launch_kind<GEMM_F3>(ctx, p, st);
    case GEMM_F4:
      ok = map_2d(fn, &p.mapA0, act, R, f, 128) && map_2d(fn, &p.mapS0, act, R, f, 32) &&
           map_mn(fn, &p.mapB0, W_down, E, f, d, pair ? 2 : 4);
      p.mapA1 = p.mapA0; p.mapB1 = p.mapB0;
      clip_pads(&p, !io.save_preactivations, rows_per_expert);
      p.n_tiles = (d + 255) / 256;
      p.k_blocks = f / BK;
      p.N_total = d;
      p.out0 = o;
      p.ld_out = d;
      if (!ok) return MOE_ERR_CUDA;
      p.row_group = row_group_for(p.n_tiles, ctx);
      return pair ? on_pairs() : launch_kind<GEMM_F4>(ctx, p, st);
    case GEMM_B2:
      ok = map_2d(fn, &p.mapA0, o, R, d, 128) && map_3d(fn, &p.mapB0, W_down, E, f, d, pair ? 128 : 256);
      p.mapA1 = p.mapA0; p.mapB1 = p.mapB0;
      p.n_tiles = (f + 255) / 256;
      p.k_blocks = d / BK;
      p.N_total = f;
      p.in0 = hg; p.in1 = hu;
      p.out0 = dhg; p.out1 = dhu;
      p.ld_out = f;
      p.row_gate = reinterpret_cast<const float*>(ws + L.row_gate);
      p.outf = reinterpret_cast<float*>(ws + L.dg_part);
      p.rows_max = L.rows_max;
      if (!ok) return MOE_ERR_CUDA;
      p.row_group = row_group_for(p.n_tiles, ctx);
      return pair ? on_pairs() : launch_kind<GEMM_B2>(ctx, p, st);
    case GEMM_B4:
      ok = map_2d(fn, &p.mapA0, dhg, R, f, 128) && map_2d(fn, &p.mapA1, dhu, R, f, 128) &&
           map_3d(fn, &p.mapB0, W_gate, E, d, f, pair ? 128 : 256) &&
           map_3d(fn, &p.mapB1, W_up, E, d, f, pair ? 128 : 256);
      p.n_tiles = (d + 255) / 256;
      p.k_blocks = f / BK;
      p.N_total = d;
      p.out0 = dxp;
      p.ld_out = d;
      if (!ok) return MOE_ERR_CUDA;
      p.row_group = row_group_for(p.n_tiles, ctx);
      return pair ? on_pairs() : launch_kind<GEMM_B4>(ctx, p, st);
    case GEMM_B3:
      ok = map_mn_rows(fn, &p.mapA0, act, R, f, 2) && map_mn_rows(fn, &p.mapB0, o, R, d, pair ? 2 : 4);
      p.mapA1 = p.mapA0; p.mapB1 = p.mapB0;
      p.m_tiles = pair ? (f + 255) / 256 : (f + 127) / 128;
      p.n_tiles = (d + 255) / 256;
      p.M_total = f;
      p.N_total = d;
      p.out0 = dW_down;
      p.accf0 = io.dW_down_acc;
      p.acc_fp32 = io.dW_down_acc != nullptr;
      p.row_group = wgrad_group_for(p.n_tiles, rows_per_expert, d, ctx);
      p.ld_out = d;
      p.expert_stride = static_cast<int64_t>(f) * d;
      if (!ok) return MOE_ERR_CUDA;
      return pair         ? on_pairs()
             : p.acc_fp32 ? launch_kind<GEMM_B3, Accumulate::LOAD_ADD>(ctx, p, st)
                          : launch_kind<GEMM_B3>(ctx, p, st);
    case GEMM_B5:
      ok = map_mn_rows(fn, &p.mapA0, xp, R, d, 2) && map_mn_rows(fn, &p.mapB0, dhg, R, f, 2) &&
           map_mn_rows(fn, &p.mapB1, dhu, R, f, 2);
      p.mapA1 = p.mapA0;
      p.m_tiles = pair ? (d + 255) / 256 : (d + 127) / 128;
      p.n_tiles = (f + 127) / 128;
      p.M_total = d;
      p.N_total = f;
      p.out0 = dW_gate; p.out1 = dW_up;
      p.accf0 = io.dW_gate_acc; p.accf1 = io.dW_up_acc;
      p.acc_fp32 = io.dW_gate_acc != nullptr;
      p.row_group = wgrad_group_for(p.n_tiles, rows_per_expert, 2 * f, ctx);
      p.ld_out = f;
      p.expert_stride = static_cast<int64_t>(d) * f;
      if (!ok) return MOE_ERR_CUDA;
      return pair         ? on_pairs()
             : p.acc_fp32 ? launch_kind<GEMM_B5, Accumulate::LOAD_ADD>(ctx, p, st)
                          : launch_kind<GEMM_B5>(ctx, p, st);
    case GEMM_DX:
      // dxr[T,d] = dl_hi W_r^T + dl_lo W_r^T
      ok = map_2d(fn, &p.mapA0, ws + L.dl_hi, T, E, 128) && map_2d(fn, &p.mapA1, ws + L.dl_lo, T, E, 128) &&
           map_3d(fn, &p.mapB0, io.W_r, 1, d, E, 256);
      p.mapB1 = p.mapB0;
      if (io.W_r_mid) {  // fp32 router weight: dl_hi W_hi^T + dl_lo W_hi^T + dl_hi W_mid^T (the rest is below 2^-17)
        ok = ok && map_2d(fn, &p.mapA2, ws + L.dl_hi, T, E, 128) && map_3d(fn, &p.mapB2, io.W_r_mid, 1, d, E, 256);
        p.nseg = 3;
      }
      p.static_m_tiles = static_cast<int>((T + BM - 1) / BM);
      p.n_tiles = (d + 255) / 256;
      p.k_blocks = (E + BK - 1) / BK;
      p.N_total = d;
      p.T = T;
      p.out0 = reinterpret_cast<uint16_t*>(ws + L.dxr);
      p.ld_out = d;
      if (!ok) return MOE_ERR_CUDA;
      if (only) {
        *only = p;
        return MOE_OK;
      }
      return launch_kind<GEMM_DX>(ctx, p, st);
    case GEMM_DWR: {
      // partial[s][d,E] = x_s^T (dl_hi + dl_lo)_s over token slices of split_rows tokens
      p.whole_chunks = E % 64 == 0;
      ok = map_mn_rows(fn, &p.mapA0, io.x, T, d, 2) &&
           (p.whole_chunks ? map_mn_rows(fn, &p.mapB0, ws + L.dl_hi, T, E, 2) && map_mn_rows(fn, &p.mapB1, ws + L.dl_lo, T, E, 2)
                           : map_2d(fn, &p.mapB0, ws + L.dl_hi, T, E, 64) && map_2d(fn, &p.mapB1, ws + L.dl_lo, T, E, 64));
      p.mapA1 = p.mapA0;
      // (few tokens, io.dW_r: one slice, straight into dW_r)
      const int slices = io.dW_r ? 1 : DWR_SPLIT;
      const int64_t per = ((T + slices - 1) / slices + BK - 1) / BK * BK;
      p.split_rows = static_cast<int>(per);
      p.rows_total = static_cast<int>((T + BK - 1) / BK * BK);
      p.E = slices;  // slices play the role of experts in the tile list
      p.m_tiles = (d + 127) / 128;
      p.n_tiles = (E + 127) / 128;
      p.M_total = d;
      p.N_total = E;
      p.outf = io.dW_r ? io.dW_r : reinterpret_cast<float*>(ws + L.dwr_part);
      p.acc_fp32 = io.dW_r && io.dW_r_accumulate;
      if (!ok) return MOE_ERR_CUDA;
      if (only) {
        *only = p;
        return MOE_OK;
      }
      return launch_kind<GEMM_DWR>(ctx, p, st);
    }
    default:
      break;
  }
  (void)T;
  return MOE_ERR_INVALID_ARG;
}

// Expected number of `size`-row tiles of an expert when the loads scatter around `mean` like independent picks
// (variance = mean): sum over j of P(load > j size); from eight tiles on the last one is half full on average.
static double expected_tiles(double mean, double size) {
  if (mean >= 8.0 * size) return mean / size + 0.5;
  const double sd = sqrt(mean > 1.0 ? mean : 1.0);
  double n = 1.0;
  for (int j = 1; j < 16; ++j) n += 0.5 * erfc((j * size - mean) / (sd * 1.4142135623730951));
  return n;
}

// Tile shape per GEMM.  A CTA pair (256 x 256 tile, each CTA staging its rows of A and half of B) moves a third
// less operand data from L2 per flop than a one-CTA 128 x 256 tile, and the L2 -> SM feed is what limits these
// kernels.  Row GEMMs pair two 128-row blocks of ONE expert, so an expert with an odd block count pays for a block it does not
// have: a block on pairs costs less than a one-CTA block (0.76 - 0.81 at 256 and 300 rows, 0.85 - 0.87 from 512 on), but there
// are more of them.  Whether pairs win therefore oscillates with the rows per expert, and the rule compares the expected
// numbers of blocks, for experts loaded alike, under a threshold of 0.80 that is fitted to where the sign changes (it puts
// the lines at 131, 263 and 368 rows).  Measured at
// d 2048, f 768, 128 experts (one-CTA -> pair, us; gate/up, down, dgrad gate/up): 62 rows per expert 162 -> 167, 81 -> 84,
// 156 -> 161; 128: 176 -> 177, 89 -> 91, 167 -> 168; 256: 230 -> 223, 131 -> 124, 232 -> 216; 300: 267 -> 274, 151 -> 156,
// 265 -> 270; 512: 380 -> 358, 221 -> 208, 396 -> 375; 768: 535 -> 494, 310 -> 283, 559 -> 522; 1024: 689 -> 635, 400 -> 360,
// 727 -> 670.  A few wide experts (d 4096, f 14336, 8 experts) leave a last round of pairs nearly empty at 512 and 768
// rows, which the rule does not see: 865 -> 905, 432 -> 494, 891 -> 1070 at 512; 256: 522 -> 542, 308 -> 282, 643 -> 548;
// 1024: 1524 -> 1494, 796 -> 754, 1698 -> 1611; 4096: 6604 -> 6187, 3138 -> 3065, 7312 -> 6943.
// The dgrad-down GEMM is held by its epilogue (it reads hg and hu) rather than by the feed and gains less: 112 -> 125 at 62
// rows, 127 -> 136 at 128, 166 -> 167 at 256, 181 -> 204 at 300, 248 -> 247 at 512, 333 -> 336 at 768, 418 -> 415 at 1024, 615 ->
// 591 at 1536, 811 -> 788 at 2048; wide experts 301 -> 313 at 256, 510 -> 473 at 512, 702 -> 705 at 768, 881 -> 843 at 1024,
// 3681 -> 3227 at 4096: pairs from 768 rows on, where the two are equal (reached by widths below d 1024 or f 512 and by wide experts
// only: the rest take the tokens as N, see below).
// Half-empty pairs are better than complete pairs plus the leftover blocks in a second, one-CTA launch
// (MOE_FLAG_HYBRID_TILES: 4.22 ms a step against 4.17 at 1024 rows per expert).
// Weight gradients pair along the weight dimension without leftovers, but their K loop is the expert's row count, and
// with few K blocks the output leaves as fast as HBM takes it (tile-shaped stores reach 6 TB/s here) only from one-CTA
// tiles, whose two CTAs do not have to meet.  One-CTA -> pairs, us, wgrad-down / gate/up at d 2048, f 768, 128 experts: 89 / 167 ->
// 104 / 196 at 62 rows, 132 / 257 -> 139 / 272 at 256, 146 / 293 -> 147 / 302 at 312, 163 / 332 -> 158 / 323 at 375, 181 / 377 -> 171 /
// 352 at 437, 202 / 419 -> 186 / 384 at 512, 342 / 691 -> 289 / 621 at 1024; d 1024, f 768, 64 experts 47 / 76 -> 47 / 78 at 312, 51 / 85 ->
// 51 / 82 at 375; d 4096, f 14336, 8 experts 265 / 569 -> 273 / 604 at 256, 294 / 661 -> 296 / 644 at 312, 339 / 780 -> 327 / 715 at 375.
// The line stands at 384.  When they accumulate in fp32 it lies higher (see Accumulate).
static bool row_gemm_on_pairs(const moe_ctx_impl* ctx, GemmKind kind, double rows_per_expert) {
  if (ctx->tile_mode != 0) return ctx->tile_mode == 1;
  if (kind == GEMM_B4 && ctx->b4_pair_override >= 0) return ctx->b4_pair_override != 0;
  if (kind == GEMM_B2) return rows_per_expert >= 768.0;
  return 0.80 * 2.0 * expected_tiles(rows_per_expert, 2 * BM) < expected_tiles(rows_per_expert, BM);
}

// Row GEMMs with the tokens as the N operand (gemm_tokens.cu): no padding rows in the MMAs, but longer epilogues (the results
// have to be transposed), so the K loop must be long, and where an expert's rows fill the other tiles anyway there is nothing
// to gain.  The other tiles begin to need a second block of 128 rows where the experts average 120, and that is the main line.
// Pairs or one-CTA tiles, whichever the rule above takes -> tokens, us, at d 2048, f 768, 128 experts:
//   rows        8           32          64          96          120         128         256         512         640
//   gate/up     165 -> 154  165 -> 158  165 -> 162  163 -> 160  167 -> 164  174 -> 169  220 -> 207  348 -> 316  418 -> 386
//   down        81 -> 80    81 -> 82    81 -> 84    81 -> 82    85 -> 88    91 -> 91    121 -> 120  198 -> 200  235 -> 239
//   dgrad-down  111 -> 91   111 -> 96   111 -> 102  112 -> 106  124 -> 115  127 -> 118  168 -> 147  251 -> 221  301 -> 258
//   dgrad-g/u   156 -> 150  156 -> 152  156 -> 156  155 -> 155  164 -> 158  171 -> 161  215 -> 196  360 -> 323  437 -> 396
// (the down GEMM ties by stage, but whole calls gain by it at 128 and 256 rows: scoring 2048 tokens 311, 312 -> 306, 307, a training
// step of 4096 1426, 1434 -> 1399, 1431; 1024, 2048, 4096 rows: gate/up 629 -> 592, 1198 -> 1157, 2399 -> 2385, dgrad-g/u 670 -> 624, 1228 -> 1174, 2362 -> 2370) and at
// d 4096, f 14336, 8 experts, whose row tiles are walked in groups:
//   rows        8           64          96          128         256         512         640           768           1536
//   gate/up     341 -> 327  342 -> 330  342 -> 345  362 -> 356  507 -> 457  795 -> 766  999 -> 917    1161 -> 1077  2092 -> 2137
//   down        147 -> 150  148 -> 153  147 -> 158  222 -> 163  280 -> 260  485 -> 475  556 -> 532    642 -> 679    1097 -> 1170
//   dgrad-down  213 -> 176  214 -> 186  214 -> 199  233 -> 211  321 -> 282  492 -> 417  545 -> 508    643 -> 588    1166 -> 1164
//   dgrad-g/u   313 -> 306  314 -> 312  314 -> 328  462 -> 333  541 -> 502  936 -> 942  1115 -> 1151  1295 -> 1428  2224 -> 2438
// Between, at 64 / 96 / 128 / 256 / 640 / 2048 rows:
//   gate/up     d 3072, f 1536: 121 -> 124, 121 -> 126, 146 -> 130, 162 -> 151, 306 -> 276, 862 -> 831; d 4096, f 3072: 156 -> 161, 156 ->
//               167, 167 -> 175, 239 -> 218, 426 -> 393, 1203 -> 1166; d 2048, f 512: 65 -> 68, 66 -> 69, 72 -> 72, 92 -> 90, 146 -> 139;
//               d 1024, f 512: 40 -> 44, 39 -> 44, 44 -> 48, 56 -> 57, 88 -> 94, 211 -> 240; f 1536: 53 -> 57, 54 -> 58, 57 -> 62, 70 -> 75
//   down        d 2048, f 512: 35 -> 41, 35 -> 40, 40 -> 43, 56 -> 58, 94 -> 103; d 1024, f 768: 31 -> 34, 30 -> 33, 33 -> 35, 42 -> 44, 66 -> 67;
//               f 1536: 30 -> 32, 30 -> 32, 37 -> 33, 41 -> 41, 65 -> 62, 159 -> 154; d 2048, f 1536: 79 -> 78, 78 -> 78, 90 -> 83, 110 -> 103, 222
//               -> 213, 592 -> 595; d 3072, f 1536: 60 -> 63, 60 -> 64, 74 -> 66, 87 -> 81, 167 -> 155, 441 -> 435
//   dgrad-down  faster from d 1024, f 512 on (72 -> 74 there at 512, f 4096 412 -> 378 at 2048); at narrower widths a gain where its other form is slow
//               to start: d 128, f 512 19 -> 13, 19 -> 14, 19 -> 17 at 16, 64, 120; d 768, f 768 23 -> 19, 23 -> 21, 25 -> 26; d 256, f 1024 33 ->
//               25, 33 -> 30, 44 -> 39 (33 -> 35 at 96); d 64, f 64 13 -> 11, 13 -> 13, 13 -> 15: up to 96 rows
//   dgrad-g/u   d 1024, f 512: 41 -> 42, 40 -> 44, 46 -> 45, 54 -> 52, 81 -> 77, 210 -> 204; f 768: 55 -> 56, 55 -> 58, 60 -> 58, 72 -> 68; f 1536: 56
//               -> 54, 56 -> 57, 68 -> 59, 72 -> 70; d 1536, f 1024: 60 -> 55, 60 -> 56, 59 -> 58; d 3072, f 1536: 123 -> 122, 123 -> 126, 150 ->
//               130, 163 -> 150, 316 -> 285, 882 -> 857; d 4096, f 3072: 156 -> 157, 155 -> 164, 177 -> 170, 235 -> 216, 452 -> 417, 1229 -> 1220
static bool row_gemm_by_tokens(const moe_ctx_impl* ctx, GemmKind kind, double rows) {
  const int d = ctx->s.d, f = ctx->s.f;
  if (ctx->tile_mode != 0 || (kind == GEMM_B4 && ctx->b4_pair_override >= 0)) return false;
  if (d < 1024 || f < 512) return kind == GEMM_B2 && rows < 96.0;
  switch (kind) {
    case GEMM_F3:
      return d >= 2048 && (rows < 48.0 || rows >= 120.0 || (d < 3072 && f >= 768)) && rows < (f <= 1536 ? 3072.0 : 1536.0);
    case GEMM_F4: return (f >= 1536 || (d >= 2048 && f >= 768)) && rows >= 120.0 && rows < 640.0;
    case GEMM_B2: return f <= 3072 || rows < 1536.0;
    case GEMM_B4:
      return (rows >= 120.0 || (static_cast<int64_t>(d) * f >= 1 << 20 && (rows < 80.0 || d < 3072))) && rows < (d <= 3072 ? 3072.0 : 640.0);
    default: return false;
  }
}

moe_status launch_grouped_gemm(moe_ctx_impl* ctx, GemmKind kind, int64_t T, const WsLayout& L, char* ws,
                               const GemmIO& io, cudaStream_t st) {
  const bool row_kind = kind == GEMM_F3 || kind == GEMM_F4 || kind == GEMM_B2 || kind == GEMM_B4;
  const bool wgrad_kind = kind == GEMM_B3 || kind == GEMM_B5;
  const double rows_per_expert = static_cast<double>(T) * ctx->s.k / ctx->s.E;
  if (wgrad_kind) {
    const double line = io.dW_down_acc ? 704.0 : 384.0;
    const bool pair = ctx->tile_mode == 1 || ctx->tile_mode == 3 || (ctx->tile_mode == 0 && rows_per_expert >= line);
    return launch_gemm_variant(ctx, kind, T, L, ws, io, st, pair, 0);
  }
  if (!row_kind) return launch_gemm_variant(ctx, kind, T, L, ws, io, st, false, 0);
  if (row_gemm_by_tokens(ctx, kind, rows_per_expert)) return launch_token_gemm(ctx, kind, L, ws, io, nullptr, rows_per_expert < 80.0, st);
  const bool pair = row_gemm_on_pairs(ctx, kind, rows_per_expert);
  if (ctx->tile_mode != 3) return launch_gemm_variant(ctx, kind, T, L, ws, io, st, pair, 0);
  const moe_status rc = launch_gemm_variant(ctx, kind, T, L, ws, io, st, true, 1);
  if (rc != MOE_OK) return rc;
  return launch_gemm_variant(ctx, kind, T, L, ws, io, st, false, 2);
}

moe_status launch_router_gradient(moe_ctx_impl* ctx, int64_t T, const WsLayout& L, char* ws, const GemmIO& io, cudaStream_t st) {
  GemmParams dx, dwr;
  moe_status rc = launch_gemm_variant(ctx, GEMM_DX, T, L, ws, io, st, false, 0, &dx);
  if (rc == MOE_OK) rc = launch_gemm_variant(ctx, GEMM_DWR, T, L, ws, io, st, false, 0, &dwr);
  if (rc != MOE_OK) return rc;
  unsigned char* const done = &ctx->attr_done[2][GEMM_DX];  // (no other kernel of that family is of this kind)
  if (!*done) {
    if (cudaFuncSetAttribute(router_gradient_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(GEMM_SMEM)) != cudaSuccess)
      return MOE_ERR_CUDA;
    *done = 1;
  }
  launch_kernel(router_gradient_kernel, ctx->sm_count, GEMM_THREADS, GEMM_SMEM, st, dx, dwr, ctx->sm_count / 2);
  return cudaGetLastError() == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
}

// The expert GEMM that an operation of the expert-LoRA variant is, with its low-rank segment (-1: a skinny one).
static int lora_row_gemm(LoraOp op) {
  switch (op) {
    case LORA_F3: return GEMM_F3;
    case LORA_F4: return GEMM_F4;
    case LORA_B2: return GEMM_B2;
    case LORA_B4: return GEMM_B4;
    default: return -1;
  }
}

// Backward operations of the expert-LoRA variant (see launch_lora_gemm below, which prepares `p`).
static moe_status launch_lora_gemm_bwd(moe_ctx_impl* ctx, LoraOp op, const WsLayout& L, char* ws, const GemmIO& io,
                                       const LoraArgs& lo, GemmParams p, bool pair, cudaStream_t st) {
  const Shape& s = ctx->s;
  const int d = s.d, f = s.f, E = s.E, r = lo.rank;
  const int64_t R = L.rows_max;
  void* fn = ctx->encode_fn;
  auto B16 = [&](size_t off) { return reinterpret_cast<uint16_t*>(ws + off); };
  uint16_t *xp = B16(L.xp), *hg = B16(L.hg), *hu = B16(L.hu), *act = B16(L.act), *dyr = B16(L.o), *dhg = B16(L.dhg),
           *dhu = B16(L.dhu), *dxp = B16(L.dxp), *u = B16(L.lora_u), *v = B16(L.lora_v), *w = B16(L.lora_w),
           *z = B16(L.lora_z);
  const uint32_t skinny_tx = A_BYTES + CHUNK_BYTES;
  const int nb = pair ? 128 : 256;  // rows of a K-major B box
  bool ok = true;
  switch (op) {
    case LORA_W:  // w[R,64] = s dy_rows B2[e]^T      (B4 kind, one segment, K-major B of 64 rows)
      ok = map_2d(fn, &p.mapA0, dyr, R, d, 128) && map_3d(fn, &p.mapB0, lo.B2, E, r, d, 64);
      p.mapA1 = p.mapA0; p.mapB1 = p.mapB0;
      p.n_tiles = 1;
      p.k_blocks = d / BK;
      p.nseg = 1;
      p.mma_n = 64; p.stage_tx = skinny_tx;
      p.N_total = 64;
      p.out0 = w;
      p.ld_out = 64;
      p.out_scale = lo.scale;
      if (!ok) return MOE_ERR_CUDA;
      return launch_kind<GEMM_B4>(ctx, p, st);
    case LORA_Z:  // z[R,64] = s (dhg B1g[e]^T + dhu B1u[e]^T)   (B4 kind, two segments)
      ok = map_2d(fn, &p.mapA0, dhg, R, f, 128) && map_2d(fn, &p.mapA1, dhu, R, f, 128) &&
           map_3d(fn, &p.mapB0, lo.B1g, E, r, f, 64) && map_3d(fn, &p.mapB1, lo.B1u, E, r, f, 64);
      p.n_tiles = 1;
      p.k_blocks = f / BK;
      p.nseg = 2;
      p.mma_n = 64; p.stage_tx = skinny_tx;
      p.N_total = 64;
      p.out0 = z;
      p.ld_out = 64;
      p.out_scale = lo.scale;
      if (!ok) return MOE_ERR_CUDA;
      return launch_kind<GEMM_B4>(ctx, p, st);
    case LORA_B2:  // da = dy_rows Wd^T + w A2^T, SwiGLU-backward epilogue
      ok = map_2d(fn, &p.mapA0, dyr, R, d, 128) && map_3d(fn, &p.mapB0, io.W_down, E, f, d, nb) &&
           map_2d(fn, &p.mapA2, w, R, 64, 128) && map_3d(fn, &p.mapB2, lo.A2, E, f, r, nb);
      p.mapA1 = p.mapA0; p.mapB1 = p.mapB0;
      p.n_tiles = (f + 255) / 256;
      p.k_blocks = d / BK;
      p.k_blocks1 = 1;
      p.N_total = f;
      p.in0 = hg; p.in1 = hu;
      p.out0 = dhg; p.out1 = dhu;
      p.ld_out = f;
      p.outf = reinterpret_cast<float*>(ws + L.dg_part);
      p.rows_max = L.rows_max;
      if (!ok) return MOE_ERR_CUDA;
      return pair ? launch_pair_gemm(ctx, GEMM_B2, p, st) : launch_kind<GEMM_B2>(ctx, p, st);
    case LORA_B4:  // dxp = dhg Wg^T + dhu Wu^T + z A1^T
      ok = map_2d(fn, &p.mapA0, dhg, R, f, 128) && map_2d(fn, &p.mapA1, dhu, R, f, 128) &&
           map_3d(fn, &p.mapB0, io.W_gate, E, d, f, nb) && map_3d(fn, &p.mapB1, io.W_up, E, d, f, nb) &&
           map_2d(fn, &p.mapA2, z, R, 64, 128) && map_3d(fn, &p.mapB2, lo.A1, E, d, r, nb);
      p.n_tiles = (d + 255) / 256;
      p.k_blocks = f / BK;
      p.nseg = 2;
      p.k_blocks1 = 1;
      p.N_total = d;
      p.out0 = dxp;
      p.ld_out = d;
      if (!ok) return MOE_ERR_CUDA;
      return pair ? launch_pair_gemm(ctx, GEMM_B4, p, st) : launch_kind<GEMM_B4>(ctx, p, st);
    case LORA_DB2:  // dB2[e][r,d] = v_e^T dy_rows_e      (B3 kind, M = rank)
      ok = map_mn_rows(fn, &p.mapA0, v, R, 64, 2) && map_mn_rows(fn, &p.mapB0, dyr, R, d, 4);
      p.mapA1 = p.mapA0; p.mapB1 = p.mapB0;
      p.m_tiles = 1;
      p.n_tiles = (d + 255) / 256;
      p.M_total = r;
      p.N_total = d;
      p.out0 = lo.dB2;
      p.ld_out = d;
      p.expert_stride = static_cast<int64_t>(r) * d;
      if (!ok) return MOE_ERR_CUDA;
      return launch_kind<GEMM_B3>(ctx, p, st);
    case LORA_DA2:  // dA2[e][f,r] = act_e^T w_e           (B3 kind, N = rank)
    case LORA_DA1:  // dA1[e][d,r] = xp_e^T z_e
      ok = map_mn_rows(fn, &p.mapA0, op == LORA_DA2 ? act : xp, R, op == LORA_DA2 ? f : d, 2) &&
           map_mn_rows(fn, &p.mapB0, op == LORA_DA2 ? w : z, R, 64, 1);
      p.mapA1 = p.mapA0; p.mapB1 = p.mapB0;
      p.M_total = op == LORA_DA2 ? f : d;
      p.m_tiles = (p.M_total + 127) / 128;
      p.n_tiles = 1;
      p.mma_n = 64; p.stage_tx = skinny_tx;
      p.N_total = r;
      p.out0 = op == LORA_DA2 ? lo.dA2 : lo.dA1;
      p.ld_out = r;
      p.expert_stride = static_cast<int64_t>(p.M_total) * r;
      if (!ok) return MOE_ERR_CUDA;
      return launch_kind<GEMM_B3>(ctx, p, st);
    case LORA_DB1:  // dB1g[e] | dB1u[e] [r,f] = u_e^T [dhg_e | dhu_e]   (B5 kind, M = rank)
      ok = map_mn_rows(fn, &p.mapA0, u, R, 64, 2) && map_mn_rows(fn, &p.mapB0, dhg, R, f, 2) &&
           map_mn_rows(fn, &p.mapB1, dhu, R, f, 2);
      p.mapA1 = p.mapA0;
      p.m_tiles = 1;
      p.n_tiles = (f + 127) / 128;
      p.M_total = r;
      p.N_total = f;
      p.out0 = lo.dB1g; p.out1 = lo.dB1u;
      p.ld_out = f;
      p.expert_stride = static_cast<int64_t>(r) * f;
      if (!ok) return MOE_ERR_CUDA;
      return launch_kind<GEMM_B5>(ctx, p, st);
    default:
      break;
  }
  return MOE_ERR_INVALID_ARG;
}

// ------------------------------------------------------------------------------------------ expert LoRA
// The adapted layer reuses the kernels above with different operands: the low-rank path enters each row GEMM as one
// extra 64-deep K segment ([xp | u] [[W]; [B1]], ...), the four 64-wide row buffers u, v, w, z come from skinny
// instances (N = 64) of the F4 / B4 kinds, and the adapter gradients from instances of the B3 / B5 kinds whose M or
// N is the rank.  The four large ones take the tile shape the plain layer would
// (rank 16, 8192 tokens, 512 rows per expert: a step 2132 -> 2079 us), the others one-CTA tiles.  On row tiles they
// walk in plain column order, also those of wide experts, with the tokens as N as the plain layer does (row_group_for): adapters
// on such experts have not been timed.
moe_status launch_lora_gemm(moe_ctx_impl* ctx, LoraOp op, int64_t T, const WsLayout& L, char* ws, const GemmIO& io,
                            const LoraArgs& lo, cudaStream_t st) {
  const Shape& s = ctx->s;
  const int d = s.d, f = s.f, E = s.E, r = lo.rank;
  const int64_t R = L.rows_max;
  void* fn = ctx->encode_fn;
  auto B16 = [&](size_t off) { return reinterpret_cast<uint16_t*>(ws + off); };
  uint16_t *xp = B16(L.xp), *hg = B16(L.hg), *hu = B16(L.hu), *act = B16(L.act), *o = B16(L.o), *dhg = B16(L.dhg),
           *dhu = B16(L.dhu), *dxp = B16(L.dxp), *u = B16(L.lora_u), *v = B16(L.lora_v), *w = B16(L.lora_w),
           *z = B16(L.lora_z);
  GemmParams p;
  memset(&p, 0, sizeof(p));
  p.sched = reinterpret_cast<const int32_t*>(ws + L.sched);
  p.tile_expert = reinterpret_cast<const int32_t*>(ws + L.tile_expert);
  p.pad_offsets = reinterpret_cast<const int32_t*>(ws + L.pad_offsets);
  p.counts = reinterpret_cast<const int32_t*>(ws + L.counts);
  p.pair_tab = reinterpret_cast<const int32_t*>(ws + L.pair_tab);
  p.pair_count_slot = 2;
  p.oob_row = static_cast<int>(R);
  p.expert_order = reinterpret_cast<const int32_t*>(ws + L.expert_order);
  p.status = reinterpret_cast<int32_t*>(ws + L.status);
  p.E = E;
  p.ready = io.ready ? 1 : 0;
  p.next_early = io.next_early ? 1 : 0;
  p.mma_n = BN;
  p.stage_tx = STAGE_BYTES;
  p.nseg = 1;
  p.out_scale = 1.f;
  p.row_gate = reinterpret_cast<const float*>(ws + L.row_gate);
  const uint32_t skinny_tx = A_BYTES + CHUNK_BYTES;  // a 128 x 64 A tile and one 64 x 64 B tile
  const int kind = lora_row_gemm(op);
  const double rows_per_expert = static_cast<double>(T) * s.k / E;
  if (kind >= 0 && row_gemm_by_tokens(ctx, static_cast<GemmKind>(kind), rows_per_expert))
    return launch_token_gemm(ctx, static_cast<GemmKind>(kind), L, ws, io, &lo, rows_per_expert < 80.0, st);
  const bool pair = kind >= 0 && row_gemm_on_pairs(ctx, static_cast<GemmKind>(kind), rows_per_expert);
  if (kind >= 0 && ctx->gemm_timers) p.timers = reinterpret_cast<unsigned long long*>(ws + L.timers) + 8 * kind;
  bool ok = true;
  switch (op) {
    case LORA_U:  // u[R,64] = s xp A1[e]            (F4 kind, N = 64)
    case LORA_V:  // v[R,64] = s act A2[e]
      ok = map_2d(fn, &p.mapA0, op == LORA_U ? xp : act, R, op == LORA_U ? d : f, 128) &&
           map_mn(fn, &p.mapB0, op == LORA_U ? lo.A1 : lo.A2, E, op == LORA_U ? d : f, r, 1);
      p.mapA1 = p.mapA0; p.mapB1 = p.mapB0;
      p.n_tiles = 1;
      p.k_blocks = (op == LORA_U ? d : f) / BK;
      p.mma_n = 64; p.stage_tx = skinny_tx;
      p.N_total = 64;
      p.out0 = op == LORA_U ? u : v;
      p.ld_out = 64;
      p.out_scale = lo.scale;
      if (!ok) return MOE_ERR_CUDA;
      return launch_kind<GEMM_F4>(ctx, p, st);
    case LORA_F3:  // [hg|hu] = xp [Wg|Wu] + u [B1g|B1u]
      ok = map_2d(fn, &p.mapA0, xp, R, d, 128) && map_mn(fn, &p.mapB0, io.W_gate, E, d, f, 2) &&
           map_mn(fn, &p.mapB1, io.W_up, E, d, f, 2) && map_2d(fn, &p.mapA2, u, R, 64, 128) &&
           map_mn(fn, &p.mapB2, lo.B1g, E, r, f, 2) && map_mn(fn, &p.mapB3, lo.B1u, E, r, f, 2);
      p.mapA1 = p.mapA0;
      p.n_tiles = (f + 127) / 128;
      p.k_blocks = d / BK;
      p.k_blocks1 = 1;
      p.N_total = f;
      p.out0 = hg; p.out1 = hu; p.out2 = act;
      p.ld_out = f;
      p.save_pre = 1;
      if (!ok) return MOE_ERR_CUDA;
      return pair ? launch_pair_gemm(ctx, GEMM_F3, p, st) : launch_kind<GEMM_F3>(ctx, p, st);
    case LORA_F4:  // o = act Wd + v B2
      ok = map_2d(fn, &p.mapA0, act, R, f, 128) && map_mn(fn, &p.mapB0, io.W_down, E, f, d, pair ? 2 : 4) &&
           map_2d(fn, &p.mapA2, v, R, 64, 128) && map_mn(fn, &p.mapB2, lo.B2, E, r, d, pair ? 2 : 4);
      p.mapA1 = p.mapA0; p.mapB1 = p.mapB0;
      p.n_tiles = (d + 255) / 256;
      p.k_blocks = f / BK;
      p.k_blocks1 = 1;
      p.N_total = d;
      p.out0 = o;
      p.ld_out = d;
      if (!ok) return MOE_ERR_CUDA;
      return pair ? launch_pair_gemm(ctx, GEMM_F4, p, st) : launch_kind<GEMM_F4>(ctx, p, st);
    default:
      break;
  }
  return launch_lora_gemm_bwd(ctx, op, L, ws, io, lo, p, pair, st);
}

}  // namespace moe
