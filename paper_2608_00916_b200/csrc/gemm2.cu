// The six expert contractions on CTA pairs (cluster of 2, tcgen05 cta_group::2).
//
// Why pairs: with one CTA per 128 x 256 tile every SM stages 48 KB of operands per 64-deep K step, and the profile
// of that kernel shows the tensor pipe about half busy with no memory unit saturated - the four-stage ring cannot
// keep enough bytes in flight.  A pair computes a 256 x 256 tile: each CTA stages its own 128 rows of A and only
// HALF of B (128 of the 256 columns); the MMA reads both halves from the two CTAs' shared memories.  Per SM that is
// 32 KB per K step for the same MMA time, and the ring grows to six stages.
//
// Protocol (leader = cluster rank 0).  Both producers issue their own TMA loads, all credited to the LEADER's full
// barrier (the leader's producer posts the expected byte count of both CTAs).  The leader's MMA thread issues
// tcgen05.mma.cta_group::2 and commits to the empty / accumulator-full barriers of BOTH CTAs.  The epilogue warps of
// both CTAs drain their own tensor memory (their 128 rows) and arrive on the leader's accumulator-empty barrier.
// Tensor memory is allocated and freed by one warp of each CTA; cluster barriers bracket the kernel so that no CTA
// leaves while its partner may still touch its shared memory, barriers or tensor memory.
//
// Row GEMMs pair two consecutive 128-row blocks of ONE expert; an expert with an odd number of blocks gets a pair
// whose second half is empty: that CTA stages its half of B, and for A it issues the same TMA copy at a row beyond
// the end of the row buffer, which the copy engine fills with zeros without touching memory - so the unavoidable MMA
// over the empty half multiplies zeros (its power draw depends on the operand data, and the step is power-bound) -
// and nothing of its accumulator half is read or stored.  Weight gradients pair along M.
#include "gemm_common.cuh"

namespace moe {

constexpr int STAGES2 = 6;
constexpr int GEMM2_THREADS = 352;  // warps: 0 TMA producer, 1 MMA issuer, 2..9 epilogue (two per TMEM lane quadrant), 10 chain
constexpr int BH_BYTES = 128 * BK * 2;              // this CTA's half of B: 16 KB
constexpr int STAGE2_BYTES = A_BYTES + BH_BYTES;    // 32 KB
static_assert(ring_fits(STAGES2, STAGE2_BYTES));
constexpr size_t GEMM2_SMEM = static_cast<size_t>(STAGES2) * STAGE2_BYTES + EPI_BYTES + BARS_BYTES;

struct Tile2 {
  int e, row0, m0, n0, nkb;
  int klast;    // K = 16 steps issued in the last K block
  int valid;    // row GEMMs: rows of this CTA's 128 that exist (clip_rows: that are routed rows)
  bool write;   // this CTA's 128 rows exist (false: the empty half of an odd expert's last pair)
  bool full;    // both halves of the pair exist
};

template <int KIND>
__device__ __forceinline__ int total_tiles2(const GemmParams& p) {
  if (Traits<KIND>::WGRAD) return p.E * p.m_tiles * p.n_tiles;  // m_tiles = 256-row pairs of the output
  return p.sched[p.pair_count_slot] * p.n_tiles;                // number of row-block pairs in the table in use
}

template <int KIND>
__device__ __forceinline__ Tile2 get_tile2(const GemmParams& p, int t, int rank) {
  Tile2 tl;
  tl.klast = BK / 16;
  if (Traits<KIND>::WGRAD) {
    const int per = p.m_tiles * p.n_tiles;
    const int slot = t / per;
    tl.e = p.expert_grouped ? p.e_first + slot : p.expert_order[slot];  // else: longest K loops first
    const int rem = t - slot * per;
    int mt, nt;
    row_tile_order(rem, p.n_tiles, p.row_group, p.m_tiles, mt, nt);
    tl.m0 = mt * 2 * BM + rank * BM;
    tl.n0 = nt * Traits<KIND>::N_SPAN;
    tl.row0 = p.pad_offsets[tl.e];
    tl.nkb = (p.counts[tl.e] + BK - 1) / BK;  // the rest of the 128-row padding is zeros
    tl.klast = last_k_steps(p.counts[tl.e]);
    tl.valid = BM;
    tl.write = true;
    tl.full = true;
  } else {
    int pr, nt;
    if (p.row_group > 1 && p.pair_count_slot == 2) {
      const int q = t / p.n_tiles;
      const int4 at = *reinterpret_cast<const int4*>(p.pair_tab + 4 * q);
      const int row0 = p.pad_offsets[at.x], rows = p.pad_offsets[at.x + 1] - row0;
      expert_tile_order(t, p.n_tiles, p.row_group, q - (at.y - row0) / (2 * BM), (rows + 2 * BM - 1) / (2 * BM), pr, nt);
    } else {
      row_tile_order(t, p.n_tiles, p.row_group, p.sched[p.pair_count_slot], pr, nt);
    }
    const int4 info = *reinterpret_cast<const int4*>(p.pair_tab + 4 * pr);  // expert, first row, blocks (1 or 2)
    tl.e = info.x;
    tl.row0 = info.y + rank * BM;
    tl.write = rank < info.z;
    tl.valid = !tl.write ? 0 : p.clip_rows ? rows_in_tile(p, tl.e, tl.row0) : BM;
    tl.full = info.z == 2;
    tl.m0 = 0;
    tl.n0 = nt * Traits<KIND>::N_SPAN;
    tl.nkb = p.k_blocks * p.nseg + p.k_blocks1;
  }
  return tl;
}

// Loads of one K block for the CTA of rank `rank`: its rows of A and its 128-column half of B (PART as in issue_loads).
template <int KIND, int PART = 3>
__device__ __forceinline__ void issue_loads2(const GemmParams& p, const Tile2& tl, int kb, int rank, uint32_t sA,
                                             uint32_t sB, uint32_t bar) {
  constexpr bool A = (PART & 1) != 0, B = (PART & 2) != 0;
  if (!Traits<KIND>::WGRAD && PART == 3 && kb >= p.k_blocks * p.nseg) {  // extra K segment of the low-rank adapter path
    const int kk = kb - p.k_blocks * p.nseg;
    tma_load_2d_pair(sA, &p.mapA2, bar, kk * BK, tl.write ? tl.row0 : p.oob_row);
    if (KIND == GEMM_F3)
      tma_load_4d_pair(sB, rank ? &p.mapB3 : &p.mapB2, bar, 0, kk * BK, tl.n0 / 64, tl.e);
    else if (KIND == GEMM_F4)
      tma_load_4d_pair(sB, &p.mapB2, bar, 0, kk * BK, tl.n0 / 64 + rank * 2, tl.e);
    else
      tma_load_3d_pair(sB, &p.mapB2, bar, kk * BK, tl.n0 + rank * 128, tl.e);
    return;
  }
  if (KIND == GEMM_F3) {
    if (A) load_a_rows<true>(p, sA, bar, kb * BK, tl.row0, tl.valid);
    const CUtensorMap* mb = rank ? &p.mapB1 : &p.mapB0;  // leader: gate columns, partner: the matching up columns
    if (B) tma_load_4d_pair(sB, mb, bar, 0, kb * BK, tl.n0 / 64, tl.e);
  } else if (KIND == GEMM_F4) {
    if (A) load_a_rows<true>(p, sA, bar, kb * BK, tl.row0, tl.valid);
    if (B) tma_load_4d_pair(sB, &p.mapB0, bar, 0, kb * BK, tl.n0 / 64 + rank * 2, tl.e);
  } else if (KIND == GEMM_B2) {
    if (A) tma_load_2d_pair(sA, &p.mapA0, bar, kb * BK, tl.write ? tl.row0 : p.oob_row);
    if (B) tma_load_3d_pair(sB, &p.mapB0, bar, kb * BK, tl.n0 + rank * 128, tl.e);
  } else if (KIND == GEMM_B4) {
    const int seg = kb / p.k_blocks, kk = kb - seg * p.k_blocks;
    if (A) tma_load_2d_pair(sA, seg ? &p.mapA1 : &p.mapA0, bar, kk * BK, tl.write ? tl.row0 : p.oob_row);
    if (B) tma_load_3d_pair(sB, seg ? &p.mapB1 : &p.mapB0, bar, kk * BK, tl.n0 + rank * 128, tl.e);
  } else if (KIND == GEMM_B3) {
    const int row = tl.row0 + kb * BK;
    tma_load_3d_pair(sA, &p.mapA0, bar, 0, row, tl.m0 / 64);
    tma_load_3d_pair(sB, &p.mapB0, bar, 0, row, tl.n0 / 64 + rank * 2);
  } else {  // GEMM_B5
    const int row = tl.row0 + kb * BK;
    const CUtensorMap* mb = rank ? &p.mapB1 : &p.mapB0;  // leader: dhg columns, partner: dhu columns
    tma_load_3d_pair(sA, &p.mapA0, bar, 0, row, tl.m0 / 64);
    tma_load_3d_pair(sB, mb, bar, 0, row, tl.n0 / 64);
  }
}

// The bound of 512 threads keeps the weight gradients at 128 registers: blocks of the bandwidth-bound kernels of the chain have to
// fit beside them.
// PACED: the pairs keep step (Pace).  A kernel of its own: the question at every K block whether the end of a tile is near costs the copy
// thread time where tiles are short, also when no counters are given - F4 of 12 K blocks at d 2048, f 768 2 % (388 -> 396 us at 1024 rows per
// expert, 723 -> 739 at 2048), the weight gradients 1 %; as two loops with the question between them F4 takes 6 % longer.
template <int KIND, bool PACED>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(Traits<KIND>::WGRAD ? 512 : GEMM2_THREADS, 1)
    grouped_gemm_pair_kernel(const __grid_constant__ GemmParams p) {
  using TR = Traits<KIND>;
  extern __shared__ __align__(1024) unsigned char gemm2_smem_raw[];

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const bool leader = rank == 0;
  const uint32_t smem_base = smem_u32(gemm2_smem_raw);
  // barriers: full, empty, accumulator full / empty, drain (failure path); behind them the base of the accumulators
  constexpr int BARS = STAGES2 * STAGE2_BYTES + EPI_BYTES, TMEM_SLOT = BARS + 8 * (2 * STAGES2 + 5);
  const uint32_t bar0 = smem_base + BARS;
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES2 + s); };
  auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * STAGES2 + a); };
  auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * STAGES2 + 2 + a); };

  constexpr bool teams = EpilogueTeams<KIND, Accumulate::REDUCE>::value;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES2; ++s) {
      mbar_init(full_bar(s), 1);   // used in the leader only: its producer's arrive + the bytes of both CTAs
      mbar_init(empty_bar(s), 1);  // one commit from the leader's MMA thread
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull_bar(a), 1);   // one commit from the leader's MMA thread
      mbar_init(tempty_bar(a), teams ? 8 : 16);  // used in the leader only: 8 epilogue warps of each CTA, or 4
    }
    mbar_init(bar0 + 8u * (2 * STAGES2 + 4), 1);
    fence_mbar_init();
    tma_prefetch_desc(&p.mapA0);
    tma_prefetch_desc(&p.mapB0);
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_base + TMEM_SLOT, TMEM_COLS);
    tmem_relinquish_pair();
  }
  constexpr bool PRELOAD = !TR::WGRAD;  // as in gemm.cu
  if (!PRELOAD && !p.ready) chain_wait();  // everything above touches only this CTA's own state
  tc_fence_before();
  cluster_sync_all();  // barriers of both CTAs are initialised before anyone signals across the pair
  tc_fence_after();
  const uint32_t tmem_base = *reinterpret_cast<const volatile uint32_t*>(gemm2_smem_raw + TMEM_SLOT);
  const int ntiles = total_tiles2<KIND>(p);
  const int cid = blockIdx.x >> 1, nclusters = gridDim.x >> 1;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (both CTAs; one thread)
    if (elect_one()) {
      RingPos pos;
      uint32_t it = 0;
      bool ok = true;
      RoleClock clk(leader ? p.timers : nullptr);
      int kb = 0;  // the first K block of the first tile that is not on its way yet
      Pace pace(PACED && leader ? p.pace : nullptr, nclusters);
      if (PRELOAD) {
        const Tile2 tl = cid < ntiles ? get_tile2<KIND>(p, cid, rank) : Tile2{};
        const int pre = cid < ntiles ? min(STAGES2, p.k_blocks) : 0;
        for (int i = 0; i < pre; ++i) {
          if (leader) mbar_expect_tx(full_bar(i), 2 * STAGE2_BYTES);
          issue_loads2<KIND, 2>(p, tl, i, rank, 0, smem_base + i * STAGE2_BYTES + A_BYTES, mapa_shared(full_bar(i), 0));
        }
        if (!p.ready) chain_wait();
        for (; kb < pre; ++kb, ++it) {
          issue_loads2<KIND, 1>(p, tl, kb, rank, smem_base + kb * STAGE2_BYTES, 0, mapa_shared(full_bar(kb), 0));
          pos.next(STAGES2);
        }
      }
      for (int rd = 0; rd * nclusters < ntiles && ok; ++rd, kb = 0) {
        const int t = tile_of_round<KIND>(rd, cid, nclusters);
        if (t >= ntiles) continue;
        const Tile2 tl = get_tile2<KIND>(p, t, rank);
        int mark = 0;
        if (PACED) {
          pace.begin(rd);
          mark = max(tl.nkb - PACE_MARGIN, kb);
          if (tl.nkb <= kb) pace.near_end(rd);
        }
        for (; kb < tl.nkb; ++kb, ++it) {
          if (PACED && kb == mark) pace.near_end(rd);
          clk.start();
          if (!mbar_wait(empty_bar(pos.s), pos.phase ^ 1u)) {
            ok = false;
            break;
          }
          clk.add(0);
          if (leader) mbar_expect_tx(full_bar(pos.s), 2 * STAGE2_BYTES);
          const uint32_t sA = smem_base + pos.s * STAGE2_BYTES;
          issue_loads2<KIND>(p, tl, kb, rank, sA, sA + A_BYTES, mapa_shared(full_bar(pos.s), 0));
          pos.next(STAGES2);
        }
      }
      clk.report(0, 1);
      if (p.ready) chain_wait();  // as in gemm.cu
      chain_next();
      if (!ok) {
        // gave up: the leader waits (bounded) for the copies of BOTH CTAs that were already issued - they are all credited
        // to its full barriers - so that neither CTA exits with copies in flight (the cluster barrier below holds the
        // partner until then)
        record_status(p.status, DEV_TIMEOUT, 1100 + KIND);
        if (leader)
          for (uint32_t i = it > static_cast<uint32_t>(STAGES2) ? it - STAGES2 : 0; i < it; ++i)
            mbar_wait(full_bar(i % STAGES2), (i / STAGES2) & 1u);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (leader CTA only; one thread)
    if (leader && elect_one()) {
      constexpr uint32_t idesc = umma_idesc(2 * BM, BN, TR::A_MN, TR::B_MN);
      constexpr uint32_t A_KSTEP = TR::A_MN ? 2048 : 32, B_KSTEP = TR::B_MN ? 2048 : 32;
      const uint64_t descA = smem_desc(smem_base, TR::A_MN ? CHUNK_BYTES : 0, 1024);
      const uint64_t descB = smem_desc(smem_base + A_BYTES, TR::B_MN ? CHUNK_BYTES : 0, 1024);
      RingPos pos;
      uint32_t tc = 0;
      bool ok = true;
      RoleClock clk(p.timers);
      for (int rd = 0; rd * nclusters < ntiles && ok; ++rd) {
        const int t = tile_of_round<KIND>(rd, cid, nclusters);
        if (t >= ntiles) continue;
        const Tile2 tl = get_tile2<KIND>(p, t, rank);
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
        bool ready = false;  // the stage about to be used was already seen full
        for (int kb = 0; kb < tl.nkb; ++kb) {
          clk.start();
          if (!ready && !mbar_wait(full_bar(pos.s), pos.phase)) {
            ok = false;
            break;
          }
          clk.add(1);
          tc_fence_after();
          const uint64_t off = (pos.s * STAGE2_BYTES) >> 4;
          const uint32_t done = empty_bar(pos.s);
          pos.next(STAGES2);
          ready = kb + 1 < tl.nkb && mbar_try_wait(full_bar(pos.s), pos.phase);
          const int nks = kb == tl.nkb - 1 ? tl.klast : BK / 16;
#pragma unroll
          for (int ks = 0; ks < BK / 16; ++ks)
            if (ks < nks)
              umma_bf16_pair(d_tmem, descA + off + (ks * A_KSTEP >> 4), descB + off + (ks * B_KSTEP >> 4), idesc,
                             (kb | ks) != 0 ? 1u : 0u);
          umma_commit_pair_both(done);  // the stage is free in both CTAs once these MMAs have read it
        }
        if (ok) umma_commit_pair_both(tfull_bar(acc));
      }
      clk.report(2, 3, 4);
      if (!ok) {
        // gave up: let every MMA issued so far finish (bounded) before the pair's tensor memory is freed
        record_status(p.status, DEV_TIMEOUT, 1200 + KIND);
        umma_commit_pair_both(bar0 + 8u * (2 * STAGES2 + 4));
        mbar_wait(bar0 + 8u * (2 * STAGES2 + 4), 0u);
      }
    }
  } else if (warp < 10) {
    // ------------------------------------------------------------------ epilogue (8 warps per CTA, own 128 rows:
    // two warps per TMEM lane quadrant, each draining half of the tile's columns, or every other tile: EpilogueTeams)
    const int ew = warp & 3;
    const int half = (warp - 2) >> 2;
    EpiStage es{smem_base + STAGES2 * STAGE2_BYTES + (warp - 2) * (EPI_UNITS * EPI_UNIT_BYTES), 0u};
    uint32_t tc = 0;
    bool ok = true;
    if (PRELOAD && !p.ready) chain_wait();  // for what it reads itself
    const bool clocked = p.timers && leader && threadIdx.x == 64;
    if (clocked) sum_cycles(p.timers + 5, false);  // total
    for (int rd = 0; rd * nclusters < ntiles && ok; ++rd) {
      const int t = tile_of_round<KIND>(rd, cid, nclusters);
      if (t >= ntiles) continue;
      const Tile2 tl = get_tile2<KIND>(p, t, rank);
      const int rin = ew * 32 + lane;
      if (tl.nkb == 0) {
        if (TR::WGRAD && half == 0) wgrad_zero_fill<KIND>(p, tl.e, tl.m0 + rin, tl.n0);
        continue;
      }
      const int acc = tc & 1;
      const uint32_t aph = (tc >> 1) & 1u;
      ++tc;
      if (teams && acc != half) continue;  // the other team's tile
      epilogue_prefetch<KIND, Accumulate::REDUCE>(p, static_cast<int64_t>(tl.row0) + rin, tl.n0, tl.write && half == 0);
      if (clocked) sum_cycles(p.timers + 6, false);  // waiting for a finished accumulator
      if (!mbar_wait(tfull_bar(acc), aph)) {
        ok = false;
        break;
      }
      if (clocked) sum_cycles(p.timers + 6, true);
      tc_fence_after();
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(ew * 32) << 16) + acc * ACC_COLS;
      const int last = teams ? 1 : half;
#pragma unroll 1
      for (int part = teams ? 0 : half; part <= last; ++part)
        expert_epilogue<KIND, Accumulate::REDUCE>(
            p, tl.e, static_cast<int64_t>(tl.row0) + rin, (TR::WGRAD ? tl.m0 : tl.row0) + ew * 32, tl.n0, taddr, tl.write,
            TR::WGRAD ? p.M_total - (tl.m0 + ew * 32) : p.clip_rows ? tl.valid - ew * 32 : 32, es, lane, part, [&]() {
              if (part != last) return;
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive_cluster(mapa_shared(tempty_bar(acc), 0));
            });
    }
    if (clocked) {
      sum_cycles(p.timers + 5, true);
      atomicAdd(p.timers + 7, 1ull);  // CTAs counted
    }
    if (!ok && lane == 0) {
      record_status(p.status, DEV_TIMEOUT, 1300 + KIND);
    }
  } else {
    chain_warp(p.next_early);
  }

  tc_fence_before();
  cluster_sync_diverged();  // the partner has stopped using this CTA's shared memory, barriers and tensor memory
  if (warp == 1) {
    __syncwarp();  // freeing tensor memory takes the whole warp
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, TMEM_COLS);
  }
}

template <int KIND, bool PACED>
static moe_status launch_pair_kernel(moe_ctx_impl* ctx, const GemmParams& p, cudaStream_t st) {
  auto* const kernel = grouped_gemm_pair_kernel<KIND, PACED>;
  unsigned char* const done = &ctx->attr_done[PACED ? 4 : 1][KIND];
  if (!*done) {  // per device: the context is bound to one
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(GEMM2_SMEM)) != cudaSuccess)
      return MOE_ERR_CUDA;
    *done = 1;
  }
  const int grid = ctx->sm_count & ~1;  // whole pairs
  launch_kernel(kernel, grid, GEMM2_THREADS, GEMM2_SMEM, st, p);
  return cudaGetLastError() == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
}

template <int KIND>
static moe_status launch_pair_kind(moe_ctx_impl* ctx, const GemmParams& p, cudaStream_t st) {
  return p.pace ? launch_pair_kernel<KIND, true>(ctx, p, st) : launch_pair_kernel<KIND, false>(ctx, p, st);
}

moe_status launch_pair_gemm(moe_ctx_impl* ctx, GemmKind kind, const GemmParams& p, cudaStream_t st) {
  switch (kind) {
    case GEMM_F3: return launch_pair_kind<GEMM_F3>(ctx, p, st);
    case GEMM_F4: return launch_pair_kind<GEMM_F4>(ctx, p, st);
    case GEMM_B2: return launch_pair_kind<GEMM_B2>(ctx, p, st);
    case GEMM_B3: return launch_pair_kind<GEMM_B3>(ctx, p, st);
    case GEMM_B4: return launch_pair_kind<GEMM_B4>(ctx, p, st);
    case GEMM_B5: return launch_pair_kind<GEMM_B5>(ctx, p, st);
    default: return MOE_ERR_INVALID_ARG;
  }
}

}  // namespace moe
