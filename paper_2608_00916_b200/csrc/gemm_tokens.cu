// Row GEMMs with the weights as the M operand and the tokens as the N operand, on CTA pairs (tcgen05 cta_group::2):
// F3, F4, B2 and B4 of gemm.cu's list.
//
// Why: the kernels of gemm.cu and gemm2.cu take 128 or 256 rows of one expert as M, and an expert's last tile is padding on
// average half of that: at 256 rows per expert a pair tile computes 384 rows, at 1024 rows 1152.  N comes in steps of 16, so
// here an expert's rows are cut into equal tiles of at most 256 tokens, the last one shorter: the MMAs, the copies of the rows
// and the epilogue shrink with them.
//
// What bounds it: up to 256 rows per expert HBM (the weights once, the rows once), beyond that the path between L2 and the SMs,
// which carries about 75 bytes of operand copies or 30 bytes of stores a cycle and SM: 29 KB per K block take 390 cycles, the
// MMAs over 208 tokens 416.  Tiles of 512 rows of weights x 128 tokens (two accumulators each) moved 40 KB for 416 cycles of MMA
// and took 20 us more at 256 to 1024 rows.
//
// Tile: 256 rows of weights x n tokens.  F3 takes 64 gate and 64 up columns into each CTA, the other kinds 128 features.  Per
// K block a CTA stages its 128 weight rows (16 KB) and half of the tokens (n / 2 rows, up to 16 KB); six stages.  Two
// accumulators of 256 columns let the epilogue of a tile overlap the main loop of the next.  The protocol between the two
// CTAs is that of gemm2.cu.
//
// Epilogue: a TMEM lane is a feature and a column a token, so results are transposed on their way out: tcgen05.ld in the
// 16 x 256-bit shape leaves them in the register layout of 8 x 8 matrices, stmatrix.trans writes those token by token, and
// the four warps of a group (one per lane quadrant) store whole row segments of 128 (F3) or 256 bytes, 16 tokens at a time.
// In F3 a feature's gate value is in lane quadrant 0 or 1 and its up value in 2 or 3, at the same place of the register
// layout: the two warps swap halves through shared memory, and each finishes eight of the 16 tokens.  In B2 hg and hu come
// the other way, through the same staging units and ldmatrix.trans.
#include <string.h>

#include "gemm_common.cuh"
#include "tensor_maps.cuh"

namespace moe {

constexpr int TK_MAX_STAGES = 8;
// Epilogue groups of four warps, a lane quadrant each.  With two, and the gates of a unit fetched in that unit, dgrad-down was
// held by its epilogue (3300 cycles a unit): 154 / 249 / 318 / 414 us at 256 / 512 / 768 / 1024 rows per expert against 146 / 229 /
// 302 / 375.
constexpr int TK_GROUPS = 3;
constexpr int TK_THREADS = 96 + 128 * TK_GROUPS;  // warps: 0 TMA producer, 1 MMA issuer, 2.. epilogue, the last one chain (chain_warp)
// Tiles hold up to 256 tokens, a stage 16 KB of weights and up to 16 KB of tokens, and the ring six of them; with few rows per
// expert (p.small) up to 128 tokens, so that eight stages fit (and the host has half as many maps to encode, 0.65 us each).
// Gate/up and dgrad-down, us, six stages -> eight: 154 / 93 -> 153 / 91 at 4 rows per expert, 158 / 101 -> 159 / 101 at 62, 160 / 106 ->
// 166 / 107 at 94 (a second tile per expert), at d 4096, f 14336 340 / 190 -> 331 / 184 at 64, 357 / 211 -> 368 / 215 at 128: below 80.
constexpr int TK_RING_BYTES = 6 * 32768;
// Staging of an epilogue group, 16 tokens: hg, hu and act at 2 KB and 4 KB of values on their way between the gate and the up
// warps (F3), hg and hu at 4 KB and 256 bytes of dg partials (B2), two buffers of 4 KB (F4, B4).
constexpr int TK_SWAP = 6144, TK_DG = 8192, TK_EPI_BYTES = 10240;
constexpr size_t TK_SMEM = static_cast<size_t>(TK_RING_BYTES) + TK_GROUPS * TK_EPI_BYTES + 1024;

struct TokenGemmParams {
  CUtensorMap a0, a1;      // weights: F3 gate and up, B4 gate and up (its two K segments), F4 and B2 down
  CUtensorMap ax0, ax1;    // the same for the extra K segment of the low-rank adapters
  CUtensorMap b[2][8];     // rows of segment 0, of segment 1 (B4); boxes of 16, 32, .. 128 rows (small: .. 64)
  CUtensorMap bx;          // rows of the extra segment; 128 rows (small: 64)
  const int32_t *sched, *pair_tab, *tile_expert, *pad_offsets, *counts;
  int32_t* status;
  unsigned long long* timers;
  int n_tiles;             // weight tiles
  int ready, next_early;   // as in GemmParams
  int row_group;
  int k_blocks, nseg, k_blocks1;
  int N_total;             // features of the output
  uint16_t *out0, *out1, *out2;
  const uint16_t *in0, *in1;  // B2: hg, hu
  int64_t ld_out;
  const float* row_gate;   // F3, B2
  float* outf;             // B2: partial sums of dg, one slice per 128 features
  int64_t rows_max;
  int save_pre;            // F3: also store hg, hu
  int clip_rows;           // pad rows are not stored
  int small;               // few rows per expert
};

template <int KIND>
struct TokenTraits {
  static constexpr int A_MN = (KIND == GEMM_F3 || KIND == GEMM_F4) ? 1 : 0;
  static constexpr int SPAN = KIND == GEMM_F3 ? 64 : 128;  // features of the output in one CTA
};

struct TokenTile {
  int e, row0;  // expert, first row
  int n;        // tokens (a multiple of 16)
  int stored;   // of those, rows that are stored
  int zeros;    // pad rows after the tile that belong to nobody's tile and have to read zero
  int nt;       // weight tile
};

__device__ __forceinline__ int token_tiles(const TokenGemmParams& p) { return p.sched[p.small ? 0 : 2] * p.n_tiles; }

// An expert's rows are cut into as many tiles as it has pairs of 128-row blocks (small: blocks), all of one size but for the last.
__device__ __forceinline__ TokenTile get_token_tile(const TokenGemmParams& p, int t) {
  TokenTile tl;
  int ri, b, first;
  if (p.row_group > 1) {
    const int q = t / p.n_tiles, e = p.small ? p.tile_expert[q] : p.pair_tab[4 * q], most = p.small ? BM : 2 * BM;
    first = p.pad_offsets[e];
    b = p.small ? q - first / BM : (p.pair_tab[4 * q + 1] - first) / most;
    expert_tile_order(t, p.n_tiles, p.row_group, q - b, (p.pad_offsets[e + 1] - first + most - 1) / most, ri, tl.nt);
  } else {
    ri = t / p.n_tiles;
    tl.nt = t - ri * p.n_tiles;
  }
  if (p.small) {
    tl.e = p.tile_expert[ri];
    first = p.pad_offsets[tl.e];
    b = ri - first / BM;
  } else {
    const int4 info = *reinterpret_cast<const int4*>(p.pair_tab + 4 * ri);  // expert, first row of the pair
    tl.e = info.x;
    first = p.pad_offsets[tl.e];
    b = (info.y - first) / (2 * BM);
  }
  const int count = p.counts[tl.e], most = p.small ? BM : 2 * BM, tiles = (count + most - 1) / most;
  const int size = ((count + tiles - 1) / tiles + 15) & ~15, left = count - b * size;
  tl.n = min(size, (left + 15) & ~15);
  tl.row0 = first + b * size;
  tl.stored = p.clip_rows ? min(tl.n, left) : tl.n;
  tl.zeros = !p.clip_rows && b == tiles - 1 ? (count + ROW_PAD - 1) / ROW_PAD * ROW_PAD - (b * size + tl.n) : 0;
  return tl;
}

// 16 TMEM lanes x 16 columns: register 4 j + 2 i + b of a thread is lane 8 i + thread / 4, column 8 j + 2 (thread % 4) + b.
__device__ __forceinline__ void tmem_ld_16x16(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr)
               : "memory");
}
// Four 8 x 8 matrices, transposed: lane l names row l % 8 (a token) of matrix l / 8 (eight features).
__device__ __forceinline__ void stmatrix4_trans(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c),
               "r"(d)
               : "memory");
}
__device__ __forceinline__ void ldmatrix4_trans(uint32_t addr, uint32_t (&w)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ uint32_t pack_regs(uint32_t lo, uint32_t hi) { return pack_bf16x2(__uint_as_float(lo), __uint_as_float(hi)); }

// Staging units hold 16 token rows of PIECES 16-byte pieces.  Pieces are XORed with the token, so that neither the columns of
// pieces that matrices are written to nor the rows read back meet in a bank.  Address of a lane's row of the four matrices
// (32 features from piece `piece0`) of tokens 8 j .. 8 j + 7:
template <int PIECES>
__device__ __forceinline__ uint32_t matrix_row(uint32_t unit, int piece0, int j, int lane) {
  const int tok = 8 * j + (lane & 7);
  return unit + tok * (PIECES * 16) + (((piece0 + (lane >> 3)) ^ (tok & 7)) << 4);
}
// A warp's 32 features x 16 tokens (r: its two lane halves) as bf16
template <int PIECES>
__device__ __forceinline__ void stage_features(uint32_t unit, int piece0, const uint32_t (&r)[2][8], int lane) {
#pragma unroll
  for (int j = 0; j < 2; ++j)
    stmatrix4_trans(matrix_row<PIECES>(unit, piece0, j, lane), pack_regs(r[0][4 * j], r[0][4 * j + 1]),
                    pack_regs(r[0][4 * j + 2], r[0][4 * j + 3]), pack_regs(r[1][4 * j], r[1][4 * j + 1]),
                    pack_regs(r[1][4 * j + 2], r[1][4 * j + 3]));
}
// Four of the unit's 16 tokens (the warp's share) to global memory; `out`: first token, first feature of the unit.
template <int PIECES>
__device__ __forceinline__ void store_tokens(uint32_t unit, uint16_t* out, int64_t ld, int rows, int cols, int q, int lane) {
  constexpr int PER = 32 / PIECES;  // token rows per instruction
  const int cc = lane % PIECES;
#pragma unroll
  for (int i = 0; i < 4 / PER; ++i) {
    const int tok = 4 * q + PER * i + lane / PIECES;
    const uint4 v = ld_shared_v4(unit + tok * (PIECES * 16) + ((cc ^ (tok & 7)) << 4));
    if (tok < rows && cc * 8 < cols) *reinterpret_cast<uint4*>(out + tok * ld + cc * 8) = v;
  }
}

__device__ __forceinline__ void group_sync(int group) { asm volatile("bar.sync %0, 128;" ::"r"(1 + group) : "memory"); }
// Whether a bounded wait succeeded in all four warps of an epilogue group: they share barriers, so they go on or leave together.
__device__ __forceinline__ bool group_agrees(bool ok, int group) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.and.pred q, %2, 128, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(ok ? 1u : 0u), "r"(1 + TK_GROUPS + group)
      : "memory");
  return r != 0;
}

// Pad rows behind the expert's last tile.
template <int KIND>
__device__ __forceinline__ void zero_tokens(const TokenGemmParams& p, const TokenTile& tl, int f0, int cols, int thread) {
  constexpr int SPAN = TokenTraits<KIND>::SPAN;
  for (int i = thread; i < tl.zeros * (SPAN / 8); i += 128 * TK_GROUPS) {
    const int tok = i / (SPAN / 8), col = i % (SPAN / 8) * 8;
    if (col >= cols) continue;
    const int64_t at = (static_cast<int64_t>(tl.row0) + tl.n + tok) * p.ld_out + f0 + col;
    const uint4 z = make_uint4(0, 0, 0, 0);
    if (KIND != GEMM_F3 || p.save_pre) *reinterpret_cast<uint4*>(p.out0 + at) = z;
    if (KIND == GEMM_B2 || (KIND == GEMM_F3 && p.save_pre)) *reinterpret_cast<uint4*>(p.out1 + at) = z;
    if (KIND == GEMM_F3) *reinterpret_cast<uint4*>(p.out2 + at) = z;
  }
}

// B2: this thread's pieces of hg and hu of the 16 tokens from `row` (two each; zeros beyond the features).
__device__ __forceinline__ void fetch_pre(const TokenGemmParams& p, int64_t row, int f0, int cols, int q, int lane, uint4 (&v)[4]) {
  const bool in = (lane & 15) * 8 < cols;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int64_t at = (row + i * 8 + q * 2 + (lane >> 4)) * p.ld_out + f0 + (lane & 15) * 8;
    const uint16_t *qh = p.in0 + at, *qu = p.in1 + at;
    v[i] = in ? __ldg(reinterpret_cast<const uint4*>(qh)) : make_uint4(0, 0, 0, 0);
    v[2 + i] = in ? __ldg(reinterpret_cast<const uint4*>(qu)) : make_uint4(0, 0, 0, 0);
  }
}

// One tile.  Unit u of 16 tokens belongs to group u % TK_GROUPS.  A group's staging is written again once all of its warps have
// stored what they read from it: the barrier before a tile's first unit sees to that, and so does another one in front of
// each further unit, or (F4, B4) taking two buffers in turn.
template <int KIND, typename Release>
__device__ __forceinline__ void token_epilogue(const TokenGemmParams& p, const TokenTile& tl, int rank, uint32_t taddr,
                                               uint32_t staging, int group, int q, int lane, Release release) {
  constexpr int SPAN = TokenTraits<KIND>::SPAN, PIECES = SPAN / 8;
  const int f0 = tl.nt * (2 * SPAN) + rank * SPAN;
  const int cols = p.N_total - f0;
  const uint32_t lanes = taddr + (static_cast<uint32_t>(q * 32) << 16);
  const int units = tl.n >> 4;
  if (units <= group) release();
  const int side = q >> 1;  // F3: 0 gate, 1 up; it finishes tokens 8 side .. 8 side + 7
  const float* const gates = p.row_gate + tl.row0 + 8 * side + 2 * (lane & 3);
  float2 gate = make_float2(0.f, 0.f);  // of the next unit: fetched where it is used, it would hold every unit up
  if (KIND == GEMM_F3 && group < units) gate = *reinterpret_cast<const float2*>(gates + group * 16);
  int turn = 0;
#pragma unroll 1
  for (int u = group; u < units; u += TK_GROUPS, turn ^= 1) {
    const uint32_t buf = staging + (KIND == GEMM_F3 ? 0 : turn * 4096);
    uint32_t r[2][8];  // the warp's two lane halves
#pragma unroll
    for (int h = 0; h < 2; ++h) tmem_ld_16x16(lanes + (static_cast<uint32_t>(h * 16) << 16) + u * 16, r[h]);
    const int64_t row = tl.row0 + u * 16;
    const float2 gt = gate;
    if (KIND == GEMM_F3 && u + TK_GROUPS < units) gate = *reinterpret_cast<const float2*>(gates + (u + TK_GROUPS) * 16);
    tmem_ld_wait();
    if (u + TK_GROUPS >= units) release();
    const int rows = tl.stored - u * 16;
    if (rows <= 0 || cols <= 0) continue;  // the same for the whole group
    const int64_t at = row * p.ld_out + f0;
    if (KIND == GEMM_F3) {
      const int piece0 = (q & 1) * 4;
      if (u != group) group_sync(group);
      if (p.save_pre) stage_features<PIECES>(buf + side * 2048, piece0, r, lane);
      const uint32_t swap = staging + TK_SWAP + q * 1024 + lane * 16, theirs = staging + TK_SWAP + (q ^ 2) * 1024 + lane * 16;
#pragma unroll
      for (int h = 0; h < 2; ++h)
        st_shared_v4(swap + h * 512, side ? r[h][0] : r[h][4], side ? r[h][1] : r[h][5], side ? r[h][2] : r[h][6],
                     side ? r[h][3] : r[h][7]);
      group_sync(group);
      uint32_t w[4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint4 o = ld_shared_v4(theirs + h * 512);
        const uint32_t other[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          float a[2];
#pragma unroll
          for (int b = 0; b < 2; ++b) {
            const float own = __uint_as_float(side ? r[h][4 + 2 * i + b] : r[h][2 * i + b]), got = __uint_as_float(other[2 * i + b]);
            const float g = side ? got : own, up = side ? own : got;
            a[b] = (b ? gt.y : gt.x) * g * fast_sigmoid(g) * up;
          }
          w[2 * h + i] = pack_bf16x2(a[0], a[1]);
        }
      }
      stmatrix4_trans(matrix_row<PIECES>(buf + 4096, piece0, side, lane), w[0], w[1], w[2], w[3]);
      group_sync(group);
      if (p.save_pre) {
        store_tokens<PIECES>(buf, p.out0 + at, p.ld_out, rows, cols, q, lane);
        store_tokens<PIECES>(buf + 2048, p.out1 + at, p.ld_out, rows, cols, q, lane);
      }
      store_tokens<PIECES>(buf + 4096, p.out2 + at, p.ld_out, rows, cols, q, lane);
    } else {
      stage_features<PIECES>(buf, q * 4, r, lane);
      group_sync(group);
      store_tokens<PIECES>(buf, p.out0 + at, p.ld_out, rows, cols, q, lane);
    }
  }
  zero_tokens<KIND>(p, tl, f0, cols, (group * 4 + q) * 32 + lane);
}

// dgrad-down with the SwiGLU-backward epilogue.  hg and hu arrive a unit ahead of their use, as coalesced pieces, and are
// staged where the results will be; dg = <da, silu(hg) hu> is summed over the thread's features, over the lanes that hold the
// same token, and over the four warps of the group.
template <typename Release>
__device__ __forceinline__ void token_epilogue_b2(const TokenGemmParams& p, const TokenTile& tl, int rank, uint32_t taddr,
                                                  uint32_t staging, int group, int q, int lane, const uint4 (&first)[4],
                                                  Release release) {
  constexpr int PIECES = 16;
  const int f0 = tl.nt * 256 + rank * 128;
  const int cols = p.N_total - f0;
  const uint32_t lanes = taddr + (static_cast<uint32_t>(q * 32) << 16);
  const int units = tl.n >> 4;
  if (units <= group) release();
  uint4 next[4] = {first[0], first[1], first[2], first[3]};
  const float* const gates = p.row_gate + tl.row0 + 2 * (lane & 3);
  float2 ng[2] = {};  // gates of the next unit
  if (group < units) {
#pragma unroll
    for (int j = 0; j < 2; ++j) ng[j] = *reinterpret_cast<const float2*>(gates + group * 16 + 8 * j);
  }
#pragma unroll 1
  for (int u = group; u < units; u += TK_GROUPS) {
    const uint32_t buf = staging, dgs = staging + TK_DG;
    uint32_t r[2][8];
#pragma unroll
    for (int h = 0; h < 2; ++h) tmem_ld_16x16(lanes + (static_cast<uint32_t>(h * 16) << 16) + u * 16, r[h]);
    const int64_t row = tl.row0 + u * 16;
    const float2 gate[2] = {ng[0], ng[1]};
    if (cols > 0) {
      if (u != group) group_sync(group);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int tok = (i & 1) * 8 + q * 2 + (lane >> 4);
        st_shared_v4(buf + (i >> 1) * 4096 + tok * 256 + (((lane & 15) ^ (tok & 7)) << 4), next[i].x, next[i].y, next[i].z, next[i].w);
      }
      if (u + TK_GROUPS < units) {
        fetch_pre(p, row + 16 * TK_GROUPS, f0, cols, q, lane, next);
#pragma unroll
        for (int j = 0; j < 2; ++j) ng[j] = *reinterpret_cast<const float2*>(gates + (u + TK_GROUPS) * 16 + 8 * j);
      }
    }
    tmem_ld_wait();
    if (u + TK_GROUPS >= units) release();
    float* const dg_out = p.outf + static_cast<int64_t>(tl.nt * 2 + rank) * p.rows_max + row;
    if (cols <= 0) {  // the same for the whole group; its slice of dg is read all the same
      if (q == 0 && lane < 16) dg_out[lane] = 0.f;
      continue;
    }
    group_sync(group);
    float dg[4] = {0.f, 0.f, 0.f, 0.f};  // tokens 8 j + 2 (lane % 4) + b
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint32_t ah = matrix_row<PIECES>(buf, q * 4, j, lane), au = ah + 4096;
      uint32_t wh[4], wu[4];
      ldmatrix4_trans(ah, wh);
      ldmatrix4_trans(au, wu);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        float hg[2], hu[2], oh[2], ou[2];
        unpack_bf16x2(wh[m], hg[0], hg[1]);
        unpack_bf16x2(wu[m], hu[0], hu[1]);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const float sg = fast_sigmoid(hg[b]);
          const float da = __uint_as_float(r[m >> 1][4 * j + 2 * (m & 1) + b]);  // dy W_down^T without the gate
          dg[2 * j + b] = fmaf(da, hg[b] * sg * hu[b], dg[2 * j + b]);
          const float dag = (b ? gate[j].y : gate[j].x) * da;
          oh[b] = dag * hu[b] * sg * (1.f + hg[b] * (1.f - sg));
          ou[b] = dag * hg[b] * sg;
        }
        wh[m] = pack_bf16x2(oh[0], oh[1]);
        wu[m] = pack_bf16x2(ou[0], ou[1]);
      }
      __syncwarp();  // the warp's pieces have been read
      stmatrix4_trans(ah, wh[0], wh[1], wh[2], wh[3]);
      stmatrix4_trans(au, wu[0], wu[1], wu[2], wu[3]);
    }
#pragma unroll
    for (int off = 4; off < 32; off <<= 1)
#pragma unroll
      for (int i = 0; i < 4; ++i) dg[i] += __shfl_xor_sync(0xFFFFFFFFu, dg[i], off);
    if (lane < 4) {
#pragma unroll
      for (int j = 0; j < 2; ++j)
        asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(dgs + (q * 16 + 8 * j + 2 * lane) * 4), "f"(dg[2 * j]), "f"(dg[2 * j + 1])
                     : "memory");
    }
    group_sync(group);
    const int64_t at = row * p.ld_out + f0;
    store_tokens<PIECES>(buf, p.out0 + at, p.ld_out, 16, cols, q, lane);
    store_tokens<PIECES>(buf + 4096, p.out1 + at, p.ld_out, 16, cols, q, lane);
    if (q == 0 && lane < 16) {
      float s = 0.f;
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        float v;
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(dgs + (w * 16 + lane) * 4) : "memory");
        s += v;
      }
      dg_out[lane] = s;
    }
  }
  zero_tokens<GEMM_B2>(p, tl, f0, cols, (group * 4 + q) * 32 + lane);
}

template <int KIND>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TK_THREADS, 1)
    token_gemm_kernel(const __grid_constant__ TokenGemmParams p) {
  constexpr int A_MN = TokenTraits<KIND>::A_MN;
  extern __shared__ unsigned char tk_smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * TK_MAX_STAGES + 5];  // full, empty, accumulator full / empty, drain (failure path)
  __shared__ uint32_t tmem_base_slot;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const bool leader = rank == 0;
  const uint32_t smem_base = (smem_u32(tk_smem_raw) + 1023u) & ~1023u;
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (TK_MAX_STAGES + s); };
  auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * TK_MAX_STAGES + a); };
  auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * TK_MAX_STAGES + 2 + a); };

  if (threadIdx.x == 0) {
    for (int s = 0; s < TK_MAX_STAGES; ++s) {
      mbar_init(full_bar(s), 1);   // used in the leader only: its producer's arrive + the bytes of both CTAs
      mbar_init(empty_bar(s), 1);  // one commit from the leader's MMA thread
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull_bar(a), 1);    // one commit from the leader's MMA thread
      mbar_init(tempty_bar(a), 8 * TK_GROUPS);  // used in the leader only: the epilogue warps of both CTAs
    }
    mbar_init(bar0 + 8u * (2 * TK_MAX_STAGES + 4), 1);
    fence_mbar_init();
    tma_prefetch_desc(&p.a0);
    tma_prefetch_desc(&p.a1);
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(&tmem_base_slot), TMEM_COLS);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync_all();  // barriers of both CTAs are initialised before anyone signals across the pair
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;
  const int ntiles = token_tiles(p);
  const int cid = blockIdx.x >> 1, nclusters = gridDim.x >> 1;
  const uint32_t stages = p.small ? 8 : 6, stage_bytes = TK_RING_BYTES / stages;
  const int nkb = p.k_blocks * p.nseg + p.k_blocks1;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (both CTAs; one thread)
    if (elect_one()) {
      RingPos pos;
      uint32_t it = 0;
      bool ok = true;
      RoleClock clk(leader ? p.timers : nullptr);
      // The loop over the K blocks is kept short: what this thread takes to issue the copies of a stage that has become free
      // counts like latency.  With a division for the segment, the choice of the maps and the address of the barrier in it gate/up
      // took 343 us at 512 rows per expert (326 now) and 632 at 1024 (600), dgrad gate/up 664 at 1024 (638), scoring 241 tokens 230
      // (225).
      const uint32_t full0 = mapa_shared(full_bar(0), 0);
      auto load_weights = [&](const CUtensorMap* a0, const CUtensorMap* a1, int kk, int wx, int e, uint32_t sA, uint32_t bar) {
        if (KIND == GEMM_F3) {
          tma_load_4d_pair(sA, a0, bar, 0, kk, wx, e);
          tma_load_4d_pair(sA + CHUNK_BYTES, a1, bar, 0, kk, wx, e);
        } else if (KIND == GEMM_F4) {
          tma_load_4d_pair(sA, a0, bar, 0, kk, wx, e);
        } else {  // B2, B4: K-major weights
          tma_load_3d_pair(sA, a0, bar, kk, wx, e);
        }
      };
      auto weight_coord = [&](const TokenTile& tl) {
        return KIND == GEMM_F3 ? tl.nt * 2 + rank : KIND == GEMM_F4 ? tl.nt * 4 + rank * 2 : tl.nt * 256 + rank * 128;
      };
      auto token_box = [&](const TokenTile& tl) { return ((tl.n >> 1) + 15) / 16 - 1; };  // this CTA's tokens: 16 (box + 1) rows
      // The weights are the caller's: those of the first stages are fetched before the kernel in front of this one has completed,
      // the rows once it has (chain_warp).
      int kk = 0;  // of the first tile: where the loop takes over
      TokenTile tl = {};
      if (cid < ntiles) tl = get_token_tile(p, cid);
      {
        const int pre = cid < ntiles ? min(static_cast<int>(stages), p.k_blocks) : 0, box = token_box(tl);
        for (int i = 0; i < pre; ++i) {
          if (leader) mbar_expect_tx(full_bar(i), 2 * (A_BYTES + (box + 1) * 16 * BK * 2));
          load_weights(&p.a0, &p.a1, i * BK, weight_coord(tl), tl.e, smem_base + i * stage_bytes, full0 + 8u * i);
        }
        if (!p.ready) chain_wait();
        for (; it < static_cast<uint32_t>(pre); ++it, kk += BK) {
          tma_load_2d_pair(smem_base + it * stage_bytes + A_BYTES, &p.b[0][box], full0 + 8u * it, kk, tl.row0 + rank * (tl.n >> 1));
          pos.next(stages);
        }
      }
      for (int t = cid; t < ntiles && ok; t += nclusters) {
        if (t != cid) tl = get_token_tile(p, t);
        const int box = token_box(tl);  // (of the extra segment: all rows of the map's box)
        const int y = tl.row0 + rank * (tl.n >> 1);
        const int wx = weight_coord(tl);
        const int segs = p.nseg + (p.k_blocks1 ? 1 : 0);
#pragma unroll 1
        for (int seg = 0; seg < segs && ok; ++seg, kk = 0) {
          const bool extra = seg == p.nseg;
          const CUtensorMap* const a0 = extra ? &p.ax0 : KIND == GEMM_B4 && seg == 1 ? &p.a1 : &p.a0;
          const CUtensorMap* const a1 = extra ? &p.ax1 : &p.a1;  // F3: the up columns
          const CUtensorMap* const b = extra ? &p.bx : &p.b[KIND == GEMM_B4 ? seg : 0][box];
          const uint32_t tx = 2 * (extra ? stage_bytes : A_BYTES + (box + 1) * 16 * BK * 2);  // of both CTAs
          const int k_end = (extra ? p.k_blocks1 : p.k_blocks) * BK;
#pragma unroll 1
          for (; kk < k_end; kk += BK, ++it) {
            clk.start();
            if (!mbar_wait(empty_bar(pos.s), pos.phase ^ 1u)) {
              ok = false;
              break;
            }
            clk.add(0);
            if (leader) mbar_expect_tx(full_bar(pos.s), tx);
            const uint32_t sA = smem_base + pos.s * stage_bytes, bar = full0 + 8u * pos.s;
            load_weights(a0, a1, kk, wx, tl.e, sA, bar);
            tma_load_2d_pair(sA + A_BYTES, b, bar, kk, y);
            pos.next(stages);
          }
        }
      }
      clk.report(0, 1);
      if (p.ready) chain_wait();  // as in gemm.cu
      chain_next();
      if (!ok) {
        // gave up: the leader waits (bounded) for the copies of BOTH CTAs that were already issued, all credited to its full
        // barriers, so that neither CTA exits with copies in flight (the cluster barrier below holds the partner until then)
        record_status(p.status, DEV_TIMEOUT, 2100 + KIND);
        if (leader)
          for (uint32_t i = it > stages ? it - stages : 0; i < it; ++i) mbar_wait(full_bar(i % stages), (i / stages) & 1u);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (leader CTA only; one thread)
    if (leader && elect_one()) {
      constexpr uint32_t A_KSTEP = A_MN ? 2048 : 32;
      const uint64_t descA = smem_desc(smem_base, A_MN ? CHUNK_BYTES : 0, 1024);
      const uint64_t descB = smem_desc(smem_base + A_BYTES, 0, 1024);
      RingPos pos;
      uint32_t tc = 0;
      bool ok = true;
      RoleClock clk(p.timers);
      for (int t = cid; t < ntiles && ok; t += nclusters) {
        // Looked up in the tables, which lie in L1.  Handed over with the stages by the producer, the tile's tokens cost that thread a store and
        // this one a load per K block: 16384 tokens, forward 1346 -> 1360 us, training 3817 -> 3855; 2048 tokens, scoring 289 -> 292.
        const uint32_t idesc = umma_idesc(2 * BM, get_token_tile(p, t).n, A_MN, 0);
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
        for (int kb = 0; kb < nkb; ++kb) {
          clk.start();
          if (!ready && !mbar_wait(full_bar(pos.s), pos.phase)) {
            ok = false;
            break;
          }
          clk.add(1);
          tc_fence_after();
          const uint64_t off = (pos.s * stage_bytes) >> 4;
          const uint32_t done = empty_bar(pos.s);
          pos.next(stages);
          ready = kb + 1 < nkb && mbar_try_wait(full_bar(pos.s), pos.phase);
#pragma unroll
          for (int ks = 0; ks < BK / 16; ++ks)
            umma_bf16_pair(d_tmem, descA + off + (ks * A_KSTEP >> 4), descB + off + (ks * 32 >> 4), idesc, (kb | ks) != 0 ? 1u : 0u);
          umma_commit_pair_both(done);  // the stage is free in both CTAs once these MMAs have read it
        }
        if (ok) umma_commit_pair_both(tfull_bar(acc));
      }
      clk.report(2, 3, 4);
      if (!ok) {
        // gave up: let every MMA issued so far finish (bounded) before the pair's tensor memory is freed
        record_status(p.status, DEV_TIMEOUT, 2200 + KIND);
        umma_commit_pair_both(bar0 + 8u * (2 * TK_MAX_STAGES + 4));
        mbar_wait(bar0 + 8u * (2 * TK_MAX_STAGES + 4), 0u);
      }
    }
  } else if (warp < 2 + 4 * TK_GROUPS) {
    // ------------------------------------------------------------------ epilogue
    const int q = warp & 3;
    const int group = (warp - 2) >> 2;
    const uint32_t staging = smem_base + TK_RING_BYTES + group * TK_EPI_BYTES;
    uint32_t tc = 0;
    bool ok = true;
    if (!p.ready) chain_wait();  // for what it reads itself
    const bool clocked = p.timers && leader && threadIdx.x == 64;
    if (clocked) sum_cycles(p.timers + 5, false);  // total
    for (int t = cid; t < ntiles; t += nclusters) {
      const TokenTile tl = get_token_tile(p, t);
      const int acc = tc & 1;
      const uint32_t aph = (tc >> 1) & 1u;
      ++tc;
      uint4 pre[4];
      if constexpr (KIND == GEMM_B2) {
        const int f0 = tl.nt * 256 + rank * 128, cols = p.N_total - f0;
        // hg and hu come from DRAM: their lines are called into L2 while the main loop runs, the first unit's into registers
        for (int i = threadIdx.x - 64; i < tl.n * 2; i += 128 * TK_GROUPS) {
          const int64_t at = (static_cast<int64_t>(tl.row0) + (i >> 1)) * p.ld_out + f0 + (i & 1) * 64;
          if ((i & 1) * 64 >= cols) continue;
          asm volatile("prefetch.global.L2 [%0];" ::"l"(p.in0 + at));
          asm volatile("prefetch.global.L2 [%0];" ::"l"(p.in1 + at));
        }
        if (group < tl.n >> 4) fetch_pre(p, static_cast<int64_t>(tl.row0) + group * 16, f0, cols, q, lane, pre);
      }
      if (clocked) sum_cycles(p.timers + 6, false);  // waiting for a finished accumulator
      ok = group_agrees(mbar_wait(tfull_bar(acc), aph), group);
      if (clocked) sum_cycles(p.timers + 6, true);
      if (!ok) break;
      tc_fence_after();
      auto release = [&]() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(mapa_shared(tempty_bar(acc), 0));
      };
      const uint32_t taddr = tmem_base + acc * ACC_COLS;
      if constexpr (KIND == GEMM_B2)
        token_epilogue_b2(p, tl, rank, taddr, staging, group, q, lane, pre, release);
      else
        token_epilogue<KIND>(p, tl, rank, taddr, staging, group, q, lane, release);
    }
    if (clocked) {
      sum_cycles(p.timers + 5, true);
      atomicAdd(p.timers + 7, 1ull);  // CTAs counted
    }
    if (!ok && lane == 0) record_status(p.status, DEV_TIMEOUT, 2300 + KIND);
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

template <int KIND>
static moe_status launch_token_kind(moe_ctx_impl* ctx, const TokenGemmParams& p, cudaStream_t st) {
  if (!ctx->attr_done[3][KIND]) {  // per device: the context is bound to one
    if (cudaFuncSetAttribute(token_gemm_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(TK_SMEM)) !=
        cudaSuccess)
      return MOE_ERR_CUDA;
    ctx->attr_done[3][KIND] = 1;
  }
  launch_kernel(token_gemm_kernel<KIND>, ctx->sm_count & ~1, TK_THREADS, TK_SMEM, st, p);
  return cudaGetLastError() == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
}

moe_status launch_token_gemm(moe_ctx_impl* ctx, GemmKind kind, const WsLayout& L, char* ws, const GemmIO& io, const LoraArgs* lo,
                             bool small, cudaStream_t st) {
  const Shape& s = ctx->s;
  const int d = s.d, f = s.f, E = s.E, r = lo ? lo->rank : 0;
  const int64_t R = L.rows_max;
  void* fn = ctx->encode_fn;
  auto B16 = [&](size_t off) { return reinterpret_cast<uint16_t*>(ws + off); };
  auto rows = [&](CUtensorMap (&m)[8], const uint16_t* base, int64_t width) {
    for (int i = 0; i < (small ? 4 : 8); ++i)
      if (!map_2d(fn, &m[i], base, R, width, 16 * (i + 1))) return false;
    return true;
  };
  TokenGemmParams p;
  memset(&p, 0, sizeof(p));
  p.sched = reinterpret_cast<const int32_t*>(ws + L.sched);
  p.pair_tab = reinterpret_cast<const int32_t*>(ws + L.pair_tab);
  p.tile_expert = reinterpret_cast<const int32_t*>(ws + L.tile_expert);
  p.small = small ? 1 : 0;
  p.pad_offsets = reinterpret_cast<const int32_t*>(ws + L.pad_offsets);
  p.counts = reinterpret_cast<const int32_t*>(ws + L.counts);
  p.status = reinterpret_cast<int32_t*>(ws + L.status);
  p.timers = ctx->gemm_timers ? reinterpret_cast<unsigned long long*>(ws + L.timers) + 8 * (GEMM_KINDS + kind) : nullptr;
  p.ready = io.ready ? 1 : 0;
  p.next_early = io.next_early ? 1 : 0;
  p.nseg = 1;
  p.k_blocks1 = lo ? 1 : 0;
  bool ok = true;
  switch (kind) {
    case GEMM_F3:
      ok = map_mn(fn, &p.a0, io.W_gate, E, d, f, 1) && map_mn(fn, &p.a1, io.W_up, E, d, f, 1) && rows(p.b[0], B16(L.xp), d) &&
           (!lo || (map_mn(fn, &p.ax0, lo->B1g, E, r, f, 1) && map_mn(fn, &p.ax1, lo->B1u, E, r, f, 1) &&
                    map_2d(fn, &p.bx, B16(L.lora_u), R, 64, small ? 64 : 128)));
      p.n_tiles = (f + 127) / 128;
      p.k_blocks = d / BK;
      p.N_total = f;
      p.out0 = B16(L.hg); p.out1 = B16(L.hu); p.out2 = B16(L.act);
      p.row_gate = reinterpret_cast<const float*>(ws + L.row_gate);
      p.save_pre = io.save_preactivations ? 1 : 0;
      p.clip_rows = io.save_preactivations ? 0 : 1;
      break;
    case GEMM_F4:
      ok = map_mn(fn, &p.a0, io.W_down, E, f, d, 2) && rows(p.b[0], B16(L.act), f) &&
           (!lo || (map_mn(fn, &p.ax0, lo->B2, E, r, d, 2) && map_2d(fn, &p.bx, B16(L.lora_v), R, 64, small ? 64 : 128)));
      p.n_tiles = (d + 255) / 256;
      p.k_blocks = f / BK;
      p.N_total = d;
      p.out0 = B16(L.o);
      p.clip_rows = io.save_preactivations ? 0 : 1;
      break;
    case GEMM_B2:
      ok = map_3d(fn, &p.a0, io.W_down, E, f, d, 128) && rows(p.b[0], B16(L.o), d) &&
           (!lo || (map_3d(fn, &p.ax0, lo->A2, E, f, r, 128) && map_2d(fn, &p.bx, B16(L.lora_w), R, 64, small ? 64 : 128)));
      p.n_tiles = (f + 255) / 256;
      p.k_blocks = d / BK;
      p.N_total = f;
      p.in0 = B16(L.hg); p.in1 = B16(L.hu);
      p.out0 = B16(L.dhg); p.out1 = B16(L.dhu);
      p.row_gate = reinterpret_cast<const float*>(ws + L.row_gate);
      p.outf = reinterpret_cast<float*>(ws + L.dg_part);
      p.rows_max = L.rows_max;
      break;
    case GEMM_B4:
      ok = map_3d(fn, &p.a0, io.W_gate, E, d, f, 128) && map_3d(fn, &p.a1, io.W_up, E, d, f, 128) && rows(p.b[0], B16(L.dhg), f) &&
           rows(p.b[1], B16(L.dhu), f) &&
           (!lo || (map_3d(fn, &p.ax0, lo->A1, E, d, r, 128) && map_2d(fn, &p.bx, B16(L.lora_z), R, 64, small ? 64 : 128)));
      p.n_tiles = (d + 255) / 256;
      p.nseg = 2;
      p.k_blocks = f / BK;
      p.N_total = d;
      p.out0 = B16(L.dxp);
      break;
    default:
      return MOE_ERR_INVALID_ARG;
  }
  if (!ok) return MOE_ERR_CUDA;
  p.ld_out = p.N_total;
  p.row_group = row_group_for(p.n_tiles, ctx);
  switch (kind) {
    case GEMM_F3: return launch_token_kind<GEMM_F3>(ctx, p, st);
    case GEMM_F4: return launch_token_kind<GEMM_F4>(ctx, p, st);
    case GEMM_B2: return launch_token_kind<GEMM_B2>(ctx, p, st);
    default: return launch_token_kind<GEMM_B4>(ctx, p, st);
  }
}

}  // namespace moe
