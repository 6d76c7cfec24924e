// Tensor-core expert GEMMs for sm_100a: tcgen05.mma with TMEM accumulators, operands staged in
// shared memory by TMA, warp-specialised persistent CTAs (one per SM).
//
//   T_GATEUP  routed gate/up (Eq. 6): int8 tokens x 2-bit weights -> int32; epilogue applies
//             the dequantisation scales, SiLU and the gate*up product, writes h as bf16
//   T_DOWN    routed down (Eq. 5): int8 Q_a(h) x 2-bit weights -> int32 -> y fp32
//   B_GATEUP  shared expert gate/up (Eq. 2): bf16 x bf16 -> fp32 -> h_shared bf16
//   B_DOWN    shared expert down -> s fp32
//   Q8_*, Q4_* the same two with RTN INT8 / INT4 weight codes (Section 4.3): the codes travel to
//             shared memory as stored, the unpacker warps expand them to bf16 (exact: |q| <= 127)
//             in the swizzled operand layout, the MMA is the bf16 one and the epilogue multiplies
//             every output column by its row scale
//
// Tile: 128 token rows (UMMA M, one TMEM lane per row) x BN weight rows (UMMA N = 256; for a down
// projection the largest multiple of 32 up to 256 that divides its width, e.g. 224 for 896, and for a routed one of few row
// tiles the narrowest from 64 on whose tiles are no more than the SMs); K advances 128 bytes of the token
// operand per pipeline stage (128 int8 or 64 bf16), four K=32-byte MMAs per stage.
//
// Ternary weights travel as 2-bit codes all the way into shared memory (TMA box of 32 bytes per
// weight row and stage) and are expanded there to int8 by the unpacker warps, directly into the
// 128-byte-swizzled operand layout the MMA reads.  The stored code is code+1 in {0,1,2}, so the
// expansion is a shift and a mask ((w >> 2i) & 0x03030303); the weights enter the MMA as
// UNSIGNED int8 and the epilogue subtracts the token's row sum (sum_k q_k) to recover
// sum_k q_k * code_k exactly.  The shift/mask yields the 16 codes of a word in the order
// 0,4,8,12,1,5,...; the token operand is stored in the same order by the activation quantizer,
// and an integer dot product does not depend on the order of its terms.
//
// Warp roles: 0 TMA producer of the token operand (and of bf16 weights), 1 TMA producer of packed weights, 2 MMA issuer and
// TMEM owner, 4-11 two groups of unpackers that take alternate pipeline stages, 12 and up epilogue (eight or sixteen warps, an
// equal number per TMEM lane quarter, which share the tile's columns).  Kernels with nothing to expand have their epilogue from
// warp 4 on (see kEpiFirst, kEpiWarps).
// Pairs of CTAs (CG = 2, clusters of two; long prefills, see routed_ctas_per_tile): a tile is 256 token rows, 128 in either
// CTA, and cta_group::2 MMAs, issued by the first CTA, read half of the weight rows from each.  So either CTA fetches, expands and
// keeps 128 weight rows instead of 256 for the same MMA work (32 KB per stage instead of 48, six stages instead of three), and an
// SM's shared memory moves 72 KB per step instead of 112 in the 512 cycles that the step's MMAs take.  The second CTA's copies and
// announcements go to the first one's `full` barriers; commits arrive at both.  2048 x 11008, 8192 tokens, 16 experts, both builds in
// turn: routed gate/up 643 -> 477 us (3 100 TOP/s), routed down 315 -> 241.  Half of that is the issue loop (see issue_mmas).
//
// Two accumulator buffers of 256 TMEM columns let the epilogue of one tile overlap the MMAs of
// the next.  Every mbarrier wait is bounded; on expiry the CTA raises a status word and leaves.
#include <cuda.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "mote_common.cuh"
#include "mote_internal.h"
#include "ptx_sm100.cuh"

namespace mote {

using namespace ptx;

enum { MODE_T_GATEUP = 0, MODE_T_DOWN = 1, MODE_B_GATEUP = 2, MODE_B_DOWN = 3,
       MODE_Q8_GATEUP = 4, MODE_Q8_DOWN = 5, MODE_Q4_GATEUP = 6, MODE_Q4_DOWN = 7,
       MODE_T_GATEUP_SHORT = 8 };

constexpr int kBM = 128;
constexpr int kStageA = kBM * 128;             // 16 KB: 128 rows x 128 B
constexpr int kStageB = 256 * 128;             // 32 KB: up to 256 rows x 128 B
constexpr int kStagesTernary = 3, kStagesBf16 = 4, kStagesRtn = 3;
constexpr int kStagesPaired = 6;               // half the weight rows per CTA: 32 KB per stage
constexpr int kMaxStages = 6;
constexpr int kTmemCols = 512;
// Up to this K a tile's epilogue (7 000 cycles on eight warps) takes clearly longer than its MMAs (512 per 128 of K), so the ternary
// gate/up GEMM on pairs of CTAs has sixteen epilogue warps there, at 72 registers.  Where the MMAs hide eight warps' epilogue, the
// extra warps only take issue slots from the unpackers.  f = 4096, 4 experts, top-2, 4096 tokens, eight / sixteen warps: 74 / 68 us at
// K = 1024, 74 / 69 (1152), 77 / 72 (1280), 79 / 75 (1408), 80 / 78.5 (1536), 85 / 87 (1792), 92 / 95 (2048); 896 x 4864 80 / 74.5.
// The line was drawn between K = 896 and 2048; by these figures it could lie at 1536.
constexpr int kShortK = 1024;

struct UmmaArgs {
  const int4* tiles;        // [0] = {n_mtiles,0,0,0}; [1+i] = {expert, row0, rows, 0}
  int n_ntiles;             // tiles along the output columns
  int k_steps;              // pipeline stages along K (128 bytes of the token operand each)
  int k_splits;             // down projections: items per output tile, each over 1/k_splits of K (>= 1)
  int64_t split_stride;     // elements between the partial outputs of consecutive splits
  int bn;                   // weight rows per tile (UMMA N)
  int split_tail;           // down projections with bn = 256, k_splits = 1: see plan_items
  int n_out;                // output row length (f for gate/up, d for down)
  int b_rows_per_expert;    // rows of the weight tensor map per expert (0: shared expert)
  const float* beta;        // [rows]   (ternary modes)
  const int32_t* rowsum;    // [rows]
  const float* alpha0;      // [E]; RTN modes: [n_out] scale of every output column
  const float* alpha1;      // [E] (gate/up: alpha_up); RTN gate/up: [n_out] scales of the up matrix
  void* out;                // bf16 [rows, n_out] (gate/up) or fp32 [rows, n_out] (down)
  int32_t* tap0;            // optional int32 [rows, n_out]
  int32_t* tap1;
  uint32_t* beta_out_bits;  // gate/up of the routed experts: running max |h| per row (atomicMax on the bits)
  uint32_t* status;
  // shared down projection with the combine of Eq. 2 and Eq. 4 folded into its epilogue (comb_out != null):
  //   comb_out[t, :] = bf16( s[t, :] + sum_j comb_w[t, j] * comb_y[comb_perm[t*k + j], :] [+ comb_res[t, :]] )
  const float* comb_y; const float* comb_w; const int32_t* comb_perm; const uint16_t* comb_res; uint16_t* comb_out;
  int comb_k;
  int comb_wide;            // comb_res and comb_out are 32-byte aligned (the caller only promises 16): 32-byte accesses
};

struct __align__(8) PipeBarriers {
  uint64_t full[kMaxStages], empty[kMaxStages], full_p[kMaxStages], empty_p[kMaxStages], tmem_full[2], tmem_empty[2];
  uint32_t tmem_base;
  int abort_flag;
};

// CG: CTAs per tile (see the head of this file)
template <int MODE, int CG = 1>
struct ModeTraits {
  static constexpr bool kTernary = (MODE == MODE_T_GATEUP || MODE == MODE_T_DOWN || MODE == MODE_T_GATEUP_SHORT);
  static constexpr int kRtnBits = kTernary ? 0 : MODE >= MODE_Q4_GATEUP ? 4 : MODE >= MODE_Q8_GATEUP ? 8 : 0;
  static constexpr bool kRtn = kRtnBits != 0;
  static constexpr bool kUnpack = kTernary || kRtn;       // weights reach shared memory as codes
  static constexpr bool kGateUp = (MODE % 2 == 0);
  static constexpr int kStageB = mote::kStageB / CG;
  static constexpr int kStages = CG == 2 ? kStagesPaired : kTernary ? kStagesTernary : kRtn ? kStagesRtn : kStagesBf16;
  // code bytes per weight row and pipeline stage: 128 2-bit codes, 64 int8 codes or 64 4-bit codes
  static constexpr int kCodeRowBytes = kRtnBits == 8 ? 64 : 32;
  static constexpr int kStageP = 256 * kCodeRowBytes / CG;     // up to 256 rows, half of them per CTA of a pair
  static constexpr int kStagesP = CG == 2 ? kStagesPaired : kRtnBits == 8 ? 3 : 4;
  // gate/up epilogue: every epilogue warp stages 32 rows x kEpiCols bf16 (row pitch padded by 16 B)
  // and writes them out as whole row segments
  // (bf16 gate/up only.  For the ternary gate/up, whose epilogue competes with the unpackers for
  // issue slots, staging -- with plain stores or with a TMA store -- measured slower than letting
  // every thread write its own 32 bytes.)
  // bf16 weights need no unpackers, whose warps do the epilogue then.  The down projection, whose epilogue waits for the rows of
  // y that it combines, has sixteen: all CTAs are in it at once after the last round (2048 x 11008, 2048 tokens: 86 -> 83 us).
  static constexpr int kEpiFirst = kUnpack ? 12 : 4;
  static constexpr int kEpiWarps = (MODE == MODE_B_DOWN || MODE == MODE_T_GATEUP_SHORT) ? 16 : 8;
  static constexpr int kThreads = (kEpiFirst + kEpiWarps) * 32;
  static constexpr int kEpiCols = 32;
  static constexpr int kEpiPitch = kEpiCols * 2 + 16;
  static constexpr size_t kEpiStage = (kGateUp && !kTernary) ? size_t(8) * 32 * kEpiPitch : 0;
  static constexpr size_t kSmem = 1024 + size_t(kStages) * (kStageA + kStageB) +
                                  (kUnpack ? size_t(kStagesP) * kStageP : 0) + kEpiStage + sizeof(PipeBarriers);
};

// What a CTA of one GEMM (SMODE < 0) or of a pair of GEMMs lays out in shared memory.
template <int MODE, int SMODE, int CG>
struct PairTraits {
  static_assert(CG == 1, "pairs of GEMMs run on single CTAs");
  static constexpr int kStageB = mote::kStageB;
  using TR = ModeTraits<MODE>; using TS = ModeTraits<SMODE>;
  static constexpr bool kGateUp = TR::kGateUp, kUnpack = true;
  static constexpr int kEpiFirst = TR::kEpiFirst, kEpiWarps = TR::kEpiWarps, kThreads = TR::kThreads;
  static constexpr int kStages = kStagesTernary;
  static constexpr int kStageP = std::max(TR::kStageP, TS::kUnpack ? TS::kStageP : 0);
  static constexpr int kStagesP = TS::kRtnBits == 8 ? 3 : 4;
  static constexpr size_t kEpiStage = TS::kEpiStage;
  static constexpr size_t kSmem = 1024 + size_t(kStages) * (kStageA + kStageB) + size_t(kStagesP) * kStageP + kEpiStage + sizeof(PipeBarriers);
};
template <int MODE, int CG>
struct PairTraits<MODE, -1, CG> : ModeTraits<MODE, CG> {};

// Item order.  The CTAs of the grid work on neighbouring items at the same time, and the operand
// those items share is the one L2 serves to all of them from a single HBM read.
//   gate/up: row tile fastest -- concurrent items share the (small) weight tile; the token operand
//            (T x d) stays in L2 across column tiles;
//   down:    column tile fastest -- concurrent items share the token operand (P x f, larger than
//            L2 for long prefills), which is then read from HBM once instead of once per column tile.
// A down projection with few row tiles may split K over k_splits items per output tile (each
// writes its partial sums; the caller adds them in a fixed order): item = (row tile, split, column tile).
//
// The items of the last, partial round of the persistent grid would leave most SMs idle for a whole
// tile time (512 tiles on 148 CTAs: 3.46 rounds cost 4).  Where at most half of the CTAs have a
// tile left in that round, a down projection with 256-column tiles cuts each of those tiles into its
// two 128-column halves, one item each: the round then takes 0.57 of a tile time (the MMA pipe runs
// N = 128 at 0.87 of its N = 256 rate).  Items [0, n_whole) are whole tiles, [n_whole, n_items) halves.
// In a pair of GEMMs the shared expert's items follow the routed ones, so that round is not the last and nothing stands
// still either way; the rule is kept there because it came out no worse.  Of 104 short prefills (2048 x 11008, 1536 x 8960, 2048 x
// 5632 and narrower, 256 to 1408 tokens) cutting and not cutting agree within 1 % in 93, cutting is up to 6 % faster in eight (2048 x
// 11008, 4 experts: 161 / 170 us at 384 tokens, top-2, 214 / 224 at 896, top-1) and slower in three (16 experts, 960 tokens:
// 332 / 312; 2048 x 5632 203 / 192; INT8, 4 experts, 384 tokens 160 / 158).
struct ItemPlan { int n_items, n_whole; };
template <bool kGateUp>
__device__ __forceinline__ ItemPlan plan_items(const UmmaArgs& a, int n_mtiles, int workers) {
  ItemPlan p;
  p.n_items = p.n_whole = n_mtiles * a.n_ntiles * (kGateUp ? 1 : a.k_splits);
  if (!kGateUp && a.split_tail) {
    const int tail = p.n_items % workers;
    if (tail > 0 && 2 * tail <= workers) { p.n_whole = p.n_items - tail; p.n_items += tail; }
  }
  return p;
}
// half: -1 for a whole tile, else which 128-column half of tile (m_tile, n_tile) the item is
template <bool kGateUp>
__device__ __forceinline__ void decode_item(const UmmaArgs& a, int item, int n_mtiles, int n_whole, int4& tile,
                                            int& n_tile, int& half) {
  half = -1;
  if (!kGateUp && item >= n_whole) {
    const int j = item - n_whole;
    item = n_whole + (j >> 1);
    half = j & 1;
  }
  int m_tile;
  if (kGateUp) { m_tile = item % n_mtiles; n_tile = item / n_mtiles; }
  else { m_tile = item / (a.n_ntiles * a.k_splits); n_tile = item % a.n_ntiles; }
  tile = a.tiles[1 + m_tile];
}
// pipeline steps [kb, ke) of an item, and which split it is
template <bool kGateUp>
__device__ __forceinline__ int item_k_range(const UmmaArgs& a, int item, int& kb, int& ke) {
  if (kGateUp || a.k_splits <= 1) { kb = 0; ke = a.k_steps; return 0; }
  const int split = (item / a.n_ntiles) % a.k_splits;
  kb = split * a.k_steps / a.k_splits;
  ke = (split + 1) * a.k_steps / a.k_splits;
  return split;
}

// What a CTA does after one of its bounded waits has run out (abort flag raised in shared memory):
// give copies and MMAs still in flight time to land before shared memory and TMEM go away ...
__device__ __forceinline__ void drain_after_abort(volatile int* abort_flag) {
  if (*abort_flag) {
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
  }
}
// ... and raise the device status word the host reads with mote_device_status.
__device__ __forceinline__ void report_abort(volatile int* abort_flag, uint32_t* status) {
  if (*abort_flag) atomicExch(status, 1u);
}

// glu_h as ONE copy of code.  The gate/up epilogue recomputes about one element in a thousand with
// the pinned sequence, from a loop unrolled over sixteen elements: sixteen inlined copies of the
// division and the polynomial cost it instruction cache and scheduling freedom for nothing
// (8 % of the kernel at K = 896).
static __device__ __noinline__ float glu_h_rare(int acc_g, int acc_u, float c_g, float c_u) {
  return glu_h(acc_g, acc_u, c_g, c_u);
}

// ------------------------------------------------------------------------------------------------
// What the warps of a CTA do for one item, by role.  A ring of `n` stages is walked with the parity of its barriers'
// phase; false: a bounded wait ran out.
// ------------------------------------------------------------------------------------------------
struct RingPos {
  uint32_t stage = 0, phase = 0;
  __device__ __forceinline__ void next(uint32_t n) {
    if (++stage == n) { stage = 0; phase ^= 1; }
  }
};

// The weight rows of one stage that this CTA fetches.  One CTA per tile: gate rows and up rows, or the (up to) 256 rows of a
// down tile, as two boxes.  A pair: the first CTA the gate rows and the second the up rows, or either half of a down tile; there
// the box is half a tile, or 64 rows where a tile is 256 wide, since it may be cut into halves (weight_box_rows).
template <int MODE, int CG, typename Load>
__device__ __forceinline__ void load_weight_rows(const CUtensorMap& tm_b0, const CUtensorMap& tm_b1, const UmmaArgs& a, uint32_t dst,
                                                 int row_bytes, int b_row, int width, uint32_t rank, Load&& load) {
  using TR = ModeTraits<MODE, CG>;
  if (CG == 1) {
    load(dst, tm_b0, b_row);
    if (TR::kGateUp) load(dst + 128 * row_bytes, tm_b1, b_row);
    else if (width > 128) load(dst + 128 * row_bytes, tm_b1, b_row + 128);
  } else if (TR::kGateUp) {
    load(dst, rank ? tm_b1 : tm_b0, b_row);
  } else {
    b_row += (int)rank * (width / 2);
    load(dst, tm_b0, b_row);
    if (a.bn == 256 && width > 128) load(dst + 64 * row_bytes, tm_b0, b_row + 64);
  }
}

// the token operand, and the weights where they are bf16.  In a pair either CTA fetches its own 128 token rows and its half
// of the weight rows; all of it is counted on the first CTA's barrier, where the MMA issuer waits.
template <int MODE, int S, int CG>
__device__ __forceinline__ bool load_operands(const CUtensorMap& tm_a, const CUtensorMap& tm_b0, const CUtensorMap& tm_b1,
                                              const UmmaArgs& a, int item, int n_mtiles, int n_whole, uint32_t sA, uint32_t sB,
                                              PipeBarriers* bars, uint32_t rank, RingPos& p) {
  using TR = ModeTraits<MODE, CG>;
  volatile int* abort_flag = &bars->abort_flag;
  int4 tile; int n_tile, half;
  decode_item<TR::kGateUp>(a, item, n_mtiles, n_whole, tile, n_tile, half);
  const int width = half < 0 ? a.bn : 128;
  const int b_row = (a.b_rows_per_expert ? tile.x * a.b_rows_per_expert : 0) +
                    n_tile * (TR::kGateUp ? a.bn / 2 : a.bn) + (half > 0 ? 128 : 0);
  const int a_row = tile.y + (int)rank * kBM;
  constexpr int kCols = TR::kTernary ? 128 : 64;           // elements in the 128 bytes of a stage's row
  int kb, ke;
  item_k_range<TR::kGateUp>(a, item, kb, ke);
  for (int ks = kb; ks < ke; ++ks) {
    if (!mbar_wait(smem_u32(&bars->empty[p.stage]), p.phase ^ 1, abort_flag)) return false;
    uint32_t bar = smem_u32(&bars->full[p.stage]);
    if (CG == 1 || rank == 0) mbar_expect_tx(bar, CG * kStageA + (TR::kUnpack ? 0 : width * 128));
    if (CG == 2) bar = map_to_rank(bar, 0);
    auto load = [&](uint32_t dst, const CUtensorMap& tm, int row) {
      if (CG == 2) tma_load_2d_pair(dst, &tm, ks * kCols, row, bar);
      else tma_load_2d(dst, &tm, ks * kCols, row, bar);
    };
    load(sA + p.stage * kStageA, tm_a, a_row);
    if (!TR::kUnpack) load_weight_rows<MODE, CG>(tm_b0, tm_b1, a, sB + p.stage * TR::kStageB, 128, b_row, width, rank, load);
    p.next(S);
  }
  return true;
}

// After its last item the token producer walks the ring once more: the commits of the last S steps have arrived at this CTA's
// `empty` barriers before it may leave.  Nobody else waits for them (the epilogue waits for another commit, and arrivals of two
// commits have no order), and in a pair they come from the other CTA, whose closing cluster barrier orders its threads'
// accesses but not asynchronous arrivals.
template <int S>
__device__ __forceinline__ bool await_last_commits(PipeBarriers* bars, RingPos p) {
  for (int i = 0; i < S; ++i) {
    if (!mbar_wait(smem_u32(&bars->empty[p.stage]), p.phase ^ 1, &bars->abort_flag)) return false;
    p.next(S);
  }
  return true;
}

// weight codes (a pair: either CTA the codes of its half of the weight rows, on its own barrier)
template <int MODE, int kStagesP, int kStageP, int CG>
__device__ __forceinline__ bool load_codes(const CUtensorMap& tm_b0, const CUtensorMap& tm_b1, const UmmaArgs& a, int item, int n_mtiles, int n_whole,
                                           uint32_t sP, PipeBarriers* bars, uint32_t rank, RingPos& p) {
  using TR = ModeTraits<MODE, CG>;
  volatile int* abort_flag = &bars->abort_flag;
  constexpr int kRB = TR::kCodeRowBytes;
  int4 tile; int n_tile, half;
  decode_item<TR::kGateUp>(a, item, n_mtiles, n_whole, tile, n_tile, half);
  const int width = half < 0 ? a.bn : 128;
  const int b_row = tile.x * a.b_rows_per_expert + n_tile * (TR::kGateUp ? a.bn / 2 : a.bn) + (half > 0 ? 128 : 0);
  int kb, ke;
  item_k_range<TR::kGateUp>(a, item, kb, ke);
  for (int ks = kb; ks < ke; ++ks) {
    if (!mbar_wait(smem_u32(&bars->empty_p[p.stage]), p.phase ^ 1, abort_flag)) return false;
    const uint32_t bar = smem_u32(&bars->full_p[p.stage]);
    mbar_expect_tx(bar, width / CG * kRB);
    load_weight_rows<MODE, CG>(tm_b0, tm_b1, a, sP + p.stage * kStageP, kRB, b_row, width, rank,
                               [&](uint32_t dst, const CUtensorMap& tm, int row) { tma_load_2d(dst, &tm, ks * kRB, row, bar); });
    p.next(kStagesP);
  }
  return true;
}

// A whole warp walks the steps (in a pair the first CTA's, for both) and one elected lane issues.  Warp-uniform control flow is
// what keeps descriptors and barrier addresses in uniform registers, where tcgen05.mma takes its operands: with one lane in a
// loop of its own a step of four MMAs took the issuing thread 830 to 870 cycles beside busy unpackers and epilogue warps, and
// the tensor pipe, which needs 512, waited for it.
template <int MODE, int S, int CG>
__device__ __forceinline__ bool issue_mmas(const UmmaArgs& a, int item, int n_whole, int local, uint32_t tmem_base, uint32_t sA,
                                           uint32_t sB, PipeBarriers* bars, RingPos& p) {
  using TR = ModeTraits<MODE, CG>;
  volatile int* abort_flag = &bars->abort_flag;
  constexpr uint32_t kM = kBM * CG;
  const uint32_t idesc_whole = TR::kTernary ? make_idesc(2, 1, 0, kM, (uint32_t)a.bn)     // s32 += s8 * u8
                                            : make_idesc(1, 1, 1, kM, (uint32_t)a.bn);    // f32 += bf16 * bf16
  const uint32_t idesc_half = TR::kTernary ? make_idesc(2, 1, 0, kM, 128u) : make_idesc(1, 1, 1, kM, 128u);
  const int buf = local & 1;
  const uint32_t use = (uint32_t)(local >> 1);
  if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->tmem_empty[buf]), (use & 1) ^ 1, abort_flag))) return false;
  tc_fence_after();
  const uint32_t d_tmem = tmem_base + buf * 256;
  const uint32_t idesc = (!TR::kGateUp && item >= n_whole) ? idesc_half : idesc_whole;
  int kb, ke;
  item_k_range<TR::kGateUp>(a, item, kb, ke);
  uint32_t acc = 0;
  for (int ks = kb; ks < ke; ++ks) {
    if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->full[p.stage]), p.phase, abort_flag))) return false;
    tc_fence_after();
    const uint64_t da = smem_desc_sw128(sA + p.stage * kStageA);
    const uint64_t db = smem_desc_sw128(sB + p.stage * TR::kStageB);
    if (elect_one()) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (TR::kTernary) mma_i8<CG>(d_tmem, da + 2 * j, db + 2 * j, idesc, j > 0 ? 1u : acc);
        else mma_f16<CG>(d_tmem, da + 2 * j, db + 2 * j, idesc, j > 0 ? 1u : acc);
      }
      mma_commit<CG>(smem_u32(&bars->empty[p.stage]));
    }
    __syncwarp();
    acc = 1;
    p.next(S);
  }
  if (elect_one()) mma_commit<CG>(smem_u32(&bars->tmem_full[buf]));
  __syncwarp();
  return true;
}

// 2-bit -> int8 for the ternary experts; int8 / 4-bit -> bf16 for an RTN-coded shared expert.  group 0 (warps 4-7)
// expands the even pipeline steps, group 1 (warps 8-11) the odd ones.  p, q: positions in the rings of stages and codes
// (a pair: either CTA its half of the rows; the MMA issuer, in the first CTA, is told by both)
template <int MODE, int S, int kStagesP, int kStageP, int CG>
__device__ __forceinline__ bool expand_codes(const UmmaArgs& a, int item, int n_whole, int group, uint8_t* genB,
                                             const uint8_t* genP, PipeBarriers* bars, RingPos& p, RingPos& q, uint32_t& step) {
  using TR = ModeTraits<MODE, CG>;
  volatile int* abort_flag = &bars->abort_flag;
  const int tid = (threadIdx.x - 128) & 127, lane = threadIdx.x & 31;
  if constexpr (!TR::kUnpack) {                    // bf16 weights among items with codes: only the announcements
    int kb, ke;
    item_k_range<TR::kGateUp>(a, item, kb, ke);
    for (int ks = kb; ks < ke; ++ks, ++step, p.next(S)) {
      if ((step & 1u) != (uint32_t)group) continue;
      if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->empty[p.stage]), p.phase ^ 1, abort_flag))) return false;
      if (lane == 0) mbar_arrive(smem_u32(&bars->full[p.stage]));
    }
    return true;
  }
  // chunks of 16 code bytes, spread over 128 threads
  const int n_chunks = ((!TR::kGateUp && item >= n_whole) ? 128 : a.bn) / CG * (TR::kCodeRowBytes / 16);
  int kb, ke;
  item_k_range<TR::kGateUp>(a, item, kb, ke);
  for (int ks = kb; ks < ke; ++ks, ++step) {
    if ((step & 1u) == (uint32_t)group) {
      // In this order: once the MMA has left the operand stage, the step kStages back is done, so the code stage's last
      // use (kStagesP >= kStages steps back) has completed its phase.  Asked for first, full_p could still be in the phase
      // before that one, which its parity does not tell from the one wanted: with three code stages (INT8) a stage's
      // steps fall to the two groups in turn, and this group has not waited for the other's.
      static_assert(kStagesP >= S, "a code stage must not come round before its operand stage");
      const bool ok = mbar_wait(smem_u32(&bars->empty[p.stage]), p.phase ^ 1, abort_flag) &&
                      mbar_wait(smem_u32(&bars->full_p[q.stage]), q.phase, abort_flag);
      if (!__all_sync(0xffffffffu, ok)) return false;
      const uint8_t* src = genP + q.stage * kStageP;
      uint8_t* dst = genB + p.stage * TR::kStageB;
      // batches of four chunks per thread, all loads of a batch ahead of its conversions
      for (int c0 = tid; c0 < n_chunks; c0 += 128 * 4) {
        uint4 wv[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int c = c0 + b * 128;
          if (c < n_chunks) wv[b] = *reinterpret_cast<const uint4*>(src + c * 16);
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int c = c0 + b * 128;
          if (c >= n_chunks) break;
          const uint32_t pw[4] = {wv[b].x, wv[b].y, wv[b].z, wv[b].w};
          if (TR::kRtnBits == 8) {
            // 16 int8 codes -> two 16-byte pieces of 8 bf16 each
            const int r = c >> 2, quarter = c & 3;
            uint8_t* row = dst + (r >> 3) * 1024 + (r & 7) * 128;
            uint32_t e[8];
#pragma unroll
            for (int j = 0; j < 4; ++j) s8x4_to_bf16x2(pw[j], e[2 * j], e[2 * j + 1]);
            *reinterpret_cast<uint4*>(row + (((quarter * 2) ^ (r & 7)) << 4)) = make_uint4(e[0], e[1], e[2], e[3]);
            *reinterpret_cast<uint4*>(row + (((quarter * 2 + 1) ^ (r & 7)) << 4)) = make_uint4(e[4], e[5], e[6], e[7]);
          } else {
            const int r = c >> 1, half = c & 1;
            uint8_t* row = dst + (r >> 3) * 1024 + (r & 7) * 128;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              uint4 o;
              if (TR::kRtnBits == 4) {
                // 8 four-bit codes -> one 16-byte piece of 8 bf16
                uint32_t e[4];
                u4x8_to_bf16x2(pw[j], e);
                o = make_uint4(e[0], e[1], e[2], e[3]);
              } else {
                o.x = pw[j] & 0x03030303u;
                o.y = (pw[j] >> 2) & 0x03030303u;
                o.z = (pw[j] >> 4) & 0x03030303u;
                o.w = (pw[j] >> 6) & 0x03030303u;
              }
              *reinterpret_cast<uint4*>(row + (((half * 4 + j) ^ (r & 7)) << 4)) = o;
            }
          }
        }
      }
      fence_proxy_async_smem();                // generic-proxy writes -> visible to the MMA
      __syncwarp();
      if (lane == 0) {
        if (CG == 2) mbar_arrive_cluster(map_to_rank(smem_u32(&bars->full[p.stage]), 0));
        else mbar_arrive(smem_u32(&bars->full[p.stage]));
        mbar_arrive(smem_u32(&bars->empty_p[q.stage]));
      }
    }
    p.next(S);
    q.next(kStagesP);
  }
  return true;
}

// kFirst, kWarps: the epilogue warps of the CTA
template <int MODE, int CG, int kFirst, int kWarps>
__device__ __forceinline__ bool write_out(const UmmaArgs& a, int item, int n_mtiles, int n_whole, int local, uint32_t tmem_base,
                                          uint8_t* genE, PipeBarriers* bars, uint32_t rank) {
  using TR = ModeTraits<MODE, CG>;
  volatile int* abort_flag = &bars->abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int q = warp & 3;                          // TMEM lane quarter this warp may read
  constexpr int kParts = kWarps / 4;                // warps per lane quarter
  const int part = (warp - kFirst) >> 2;            // which part of the tile's columns
  const int r_in_tile = q * 32 + lane;
  int4 tile; int n_tile, half;
  decode_item<TR::kGateUp>(a, item, n_mtiles, n_whole, tile, n_tile, half);
  if (CG == 2) {                                   // this CTA's 128 rows of the pair's tile
    tile.y += (int)rank * kBM;
    tile.z = min(tile.z - (int)rank * kBM, kBM);
  }
  int kb_, ke_;
  const int split = item_k_range<TR::kGateUp>(a, item, kb_, ke_);
  const int buf = local & 1;
  const uint32_t use = (uint32_t)(local >> 1);
  const bool row_ok = r_in_tile < tile.z;
  const int64_t row = int64_t(tile.y) + r_in_tile;
  const uint32_t t_row = tmem_base + (uint32_t(q * 32) << 16) + buf * 256;
  float c0 = 0.f, c1 = 0.f;
  int rs = 0;
  if (TR::kTernary && row_ok) {
    const float beta = fmaxf(a.beta[row], kEpsScale);
    rs = a.rowsum[row];
    c0 = dequant_scale(a.alpha0[tile.x], beta);
    if (TR::kGateUp) c1 = dequant_scale(a.alpha1[tile.x], beta);
  }
  const bool ok = mbar_wait(smem_u32(&bars->tmem_full[buf]), use & 1, abort_flag);
  if (!__all_sync(0xffffffffu, ok)) return false;
  tc_fence_after();
  if (TR::kGateUp) {
    const int col0 = n_tile * 128;
    const bool row_fast = __fmul_rn(c0, c1) > 1e-12f;
    const uint32_t acc_bias = 0x4B400000u - (uint32_t)rs;
    const uint64_t c0x2 = f32x2(c0, c0), c1x2 = f32x2(c1, c1);
    float hmax = 0.0f;                           // max |h| (before the bf16 rounding, which is monotonic)
    constexpr int kCols = TR::kEpiCols, kPitch = TR::kEpiPitch;
    constexpr int kLanesPerRow = kCols * 2 / 16, kRowsPerStore = 32 / kLanesPerRow;
    uint8_t* stg = genE + (warp - kFirst) * 32 * kPitch;
#pragma unroll 1
    for (int cr = part * (128 / kParts); cr < (part + 1) * (128 / kParts); cr += kCols) {
#pragma unroll 1
      for (int c = cr; c < cr + kCols; c += 16) {
        uint32_t rg[16], ru[16];
        tmem_ld_32x32b_x16(t_row + c, rg);
        tmem_ld_32x32b_x16(t_row + 128 + c, ru);
        tmem_wait_ld();
        if (row_ok) {
          float hv[16];
          if (TR::kTernary) {
            float t_max = row_fast ? 0.0f : INFINITY;
            uint32_t key = 0xFFFFFFFFu;
#pragma unroll
            for (int j = 0; j < 16; j += 2) {
              float t;
              glu_h2_fast_biased(rg[j], rg[j + 1], ru[j], ru[j + 1], acc_bias, c0x2, c1x2, hv[j], hv[j + 1], t);
              t_max = fmaxf(t_max, t);
              key = min(key, min(glu_midpoint_key(hv[j]), glu_midpoint_key(hv[j + 1])));
            }
            const bool all = !(t_max <= kGluMaxT);
            if (key <= kGluMidpointKeys || all) {
              // Mostly one element.  Looked at four at a time where one CTA works on a tile, which leaves such a pass sooner (gate/up of
              // 256 x 512, top-4, 1941 tokens: 17.7 us one by one, 16.9), one by one in a pair (896 x 4864, 4096 tokens: 69 us, 77 by fours).
              constexpr int kAtATime = CG == 1 ? 4 : 1;
#pragma unroll
              for (int j0 = 0; j0 < 16; j0 += kAtATime) {
                uint32_t key_here = glu_midpoint_key(hv[j0]);
#pragma unroll
                for (int j = j0 + 1; j < j0 + kAtATime; ++j) key_here = min(key_here, glu_midpoint_key(hv[j]));
                if (key_here <= kGluMidpointKeys || all) {
#pragma unroll
                  for (int j = j0; j < j0 + kAtATime; ++j)
                    if (kAtATime == 1 || glu_midpoint_key(hv[j]) <= kGluMidpointKeys || all)
                      hv[j] = glu_h_rare((int)rg[j] - rs, (int)ru[j] - rs, c0, c1);
                }
              }
            }
#pragma unroll
            for (int j = 0; j < 16; j += 2) hmax = fmaxf(fmaxf(hmax, fabsf(hv[j])), fabsf(hv[j + 1]));
          } else if (TR::kRtn || a.alpha0 != nullptr) {
            // RTN-coded shared expert (codes expanded here, or beforehand): row scales of the
            // gate and up matrices = scales of this tile's output columns
            const float4* sgp = reinterpret_cast<const float4*>(a.alpha0 + col0 + c);
            const float4* sup = reinterpret_cast<const float4*>(a.alpha1 + col0 + c);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              const float4 sg = __ldg(sgp + v), su = __ldg(sup + v);
              const float sgv[4] = {sg.x, sg.y, sg.z, sg.w}, suv[4] = {su.x, su.y, su.z, su.w};
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const float g = __uint_as_float(rg[4 * v + u]) * sgv[u];
                hv[4 * v + u] = __uint_as_float(ru[4 * v + u]) * suv[u] * silu_fast(g);
              }
            }
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const float g = __uint_as_float(rg[j]);
              hv[j] = __uint_as_float(ru[j]) * silu_fast(g);
            }
          }
          uint32_t packed[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) packed[j] = pack_bf16x2(hv[2 * j], hv[2 * j + 1]);
          if (TR::kTernary) {
            // the thread's 16 bf16 values are one 32-byte sector of its row: one store
            st_global_v8(reinterpret_cast<uint16_t*>(a.out) + row * a.n_out + col0 + c, packed[0], packed[1], packed[2],
                         packed[3], packed[4], packed[5], packed[6], packed[7]);
          } else {
            uint4* sdst = reinterpret_cast<uint4*>(stg + lane * kPitch + (c - cr) * 2);
            sdst[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
            sdst[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
          }
          if (TR::kTernary && a.tap0) {
            int4* t0 = reinterpret_cast<int4*>(a.tap0 + row * a.n_out + col0 + c);
            int4* t1 = reinterpret_cast<int4*>(a.tap1 + row * a.n_out + col0 + c);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              t0[v] = make_int4((int)rg[4 * v] - rs, (int)rg[4 * v + 1] - rs, (int)rg[4 * v + 2] - rs, (int)rg[4 * v + 3] - rs);
              t1[v] = make_int4((int)ru[4 * v] - rs, (int)ru[4 * v + 1] - rs, (int)ru[4 * v + 2] - rs, (int)ru[4 * v + 3] - rs);
            }
          }
        }
      }
      if (!TR::kTernary) {
        __syncwarp();
        // the warp's 32 rows x kCols columns leave as whole row segments (kCols * 2 bytes each)
#pragma unroll
        for (int r0 = 0; r0 < 32; r0 += kRowsPerStore) {
          const int r = r0 + lane / kLanesPerRow, piece = lane % kLanesPerRow;
          if (q * 32 + r < tile.z) {
            const uint4 v = *reinterpret_cast<const uint4*>(stg + r * kPitch + piece * 16);
            uint16_t* orow = reinterpret_cast<uint16_t*>(a.out) + (int64_t(tile.y) + q * 32 + r) * a.n_out + col0 + cr;
            reinterpret_cast<uint4*>(orow)[piece] = v;
          }
        }
        __syncwarp();
      }
    }
    // bits of non-negative floats order like unsigned integers; bf16_rn(max) = max(bf16_rn)
    if (TR::kTernary && row_ok && a.beta_out_bits) {
      const uint32_t hb = f32_to_bf16_bits(hmax) << 16;
      if (hb) atomicMax(a.beta_out_bits + row, hb);
    }
  } else {
    const uint32_t acc_bias = 0x4B400000u - (uint32_t)rs;   // see glu_h2_fast_biased
    const int width = half < 0 ? a.bn : 128;
    const int col0 = n_tile * a.bn + (half > 0 ? 128 : 0);
    const bool combine = !TR::kTernary && a.comb_out != nullptr;
    float cw[MOTE_MAX_TOPK];
    const float* cy[MOTE_MAX_TOPK];
    if (combine && row_ok) {
#pragma unroll
      for (int j = 0; j < MOTE_MAX_TOPK; ++j)
        if (j < a.comb_k) {
          cw[j] = a.comb_w[row * a.comb_k + j];
          cy[j] = a.comb_y + int64_t(a.comb_perm[row * a.comb_k + j]) * a.n_out + col0;
        }
    }
#pragma unroll 1
    for (int c = part * 16; c < width; c += kParts * 16) {
      uint32_t ra[16];
      tmem_ld_32x32b_x16(t_row + c, ra);
      tmem_wait_ld();
      if (row_ok) {
        float o[16];
#pragma unroll
        for (int v = 0; v < 16; ++v)
          o[v] = TR::kTernary ? __fmul_rn(__fsub_rn(__uint_as_float(ra[v] + acc_bias), kMagic), c0)   // fl32(acc - rs) * c0
                              : __uint_as_float(ra[v]);
        if (TR::kRtn || (!TR::kTernary && a.alpha0 != nullptr)) {
          const float4* sp = reinterpret_cast<const float4*>(a.alpha0 + col0 + c);
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const float4 sc = __ldg(sp + v);
            o[4 * v] *= sc.x; o[4 * v + 1] *= sc.y; o[4 * v + 2] *= sc.z; o[4 * v + 3] *= sc.w;
          }
        }
        if (a.out) {
          float* dst = reinterpret_cast<float*>(a.out) + split * a.split_stride + row * a.n_out + col0 + c;
#pragma unroll
          for (int v = 0; v < 2; ++v)
            st_global_v8(dst + 8 * v, __float_as_uint(o[8 * v]), __float_as_uint(o[8 * v + 1]), __float_as_uint(o[8 * v + 2]),
                         __float_as_uint(o[8 * v + 3]), __float_as_uint(o[8 * v + 4]), __float_as_uint(o[8 * v + 5]),
                         __float_as_uint(o[8 * v + 6]), __float_as_uint(o[8 * v + 7]));
        }
        if (TR::kTernary && a.tap0) {
          int4* t0 = reinterpret_cast<int4*>(a.tap0 + row * a.n_out + col0 + c);
#pragma unroll
          for (int v = 0; v < 4; ++v)
            t0[v] = make_int4((int)ra[4 * v] - rs, (int)ra[4 * v + 1] - rs, (int)ra[4 * v + 2] - rs, (int)ra[4 * v + 3] - rs);
        }
        if (combine) {
          // fp32, slots in ascending j, then the residual, one bf16 rounding
#pragma unroll
          for (int j = 0; j < MOTE_MAX_TOPK; ++j)
            if (j < a.comb_k) {
#pragma unroll
              for (int v = 0; v < 2; ++v) {
                uint32_t yv[8];
                ld_global_v8(cy[j] + c + 8 * v, yv);
#pragma unroll
                for (int u = 0; u < 8; ++u) o[8 * v + u] = fmaf(cw[j], __uint_as_float(yv[u]), o[8 * v + u]);
              }
            }
          if (a.comb_res) {
            uint32_t rw[8];
            if (a.comb_wide) {
              ld_global_v8(a.comb_res + row * a.n_out + col0 + c, rw);
            } else {
              const uint4* rp = reinterpret_cast<const uint4*>(a.comb_res + row * a.n_out + col0 + c);
              const uint4 r0 = rp[0], r1 = rp[1];
              rw[0] = r0.x; rw[1] = r0.y; rw[2] = r0.z; rw[3] = r0.w; rw[4] = r1.x; rw[5] = r1.y; rw[6] = r1.z; rw[7] = r1.w;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) { o[2 * u] += bf16_lo(rw[u]); o[2 * u + 1] += bf16_hi(rw[u]); }
          }
          uint32_t pk[8];
#pragma unroll
          for (int v = 0; v < 8; ++v) pk[v] = f32_to_bf16_bits(o[2 * v]) | (f32_to_bf16_bits(o[2 * v + 1]) << 16);
          if (a.comb_wide) {
            st_global_v8(a.comb_out + row * a.n_out + col0 + c, pk[0], pk[1], pk[2], pk[3], pk[4], pk[5], pk[6], pk[7]);
          } else {
            uint4* od = reinterpret_cast<uint4*>(a.comb_out + row * a.n_out + col0 + c);
            od[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            od[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncwarp();
  if (lane == 0) {
    if (CG == 2) mbar_arrive_cluster(map_to_rank(smem_u32(&bars->tmem_empty[buf]), 0));
    else mbar_arrive(smem_u32(&bars->tmem_empty[buf]));
  }
  return true;
}

// ------------------------------------------------------------------------------------------------
// The CTA's walk over its items: all of mode MODE, or (pair of GEMMs) routed items of mode MODE and shared items of
// mode SMODE.  A pair takes the longer items first: gate/up the shared ones (bf16 rows are eight times as long as 2-bit
// ones), down the routed ones (the shared ones are cut along K).
template <int MODE, int SMODE, int CG>
__device__ __forceinline__ void umma_cta(const CUtensorMap& tm_a, const CUtensorMap& tm_b0, const CUtensorMap& tm_b1, const UmmaArgs& a,
                                         const CUtensorMap& ts_a, const CUtensorMap& ts_b0, const CUtensorMap& ts_b1, const UmmaArgs& as) {
  using TR = PairTraits<MODE, SMODE, CG>;
  constexpr bool kPair = SMODE >= 0;
  constexpr int kS = kPair ? SMODE : MODE;
  constexpr int S = TR::kStages, kStagesP = TR::kStagesP, kStageP = TR::kStageP;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t sA = smem_base;
  const uint32_t sB = sA + S * kStageA;
  const uint32_t sP = sB + S * TR::kStageB;
  uint8_t* genB = smem_gen + S * kStageA;
  uint8_t* genP = genB + S * TR::kStageB;
  uint8_t* genE = genP + (TR::kUnpack ? kStagesP * kStageP : 0);
  PipeBarriers* bars = reinterpret_cast<PipeBarriers*>(genE + TR::kEpiStage);
  volatile int* abort_flag = &bars->abort_flag;

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t rank = CG == 2 ? cluster_ctarank() : 0;
  const int worker = blockIdx.x / CG, workers = gridDim.x / CG;      // CTAs, or pairs of them

  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      // the operands have landed, and four unpacking warps per CTA have announced their part
      mbar_init(smem_u32(&bars->full[s]), 1 + (TR::kUnpack ? 4 * CG : 0));
      mbar_init(smem_u32(&bars->empty[s]), 1);
      mbar_init(smem_u32(&bars->full_p[s]), 1);
      mbar_init(smem_u32(&bars->empty_p[s]), 4);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&bars->tmem_full[b]), 1);
      mbar_init(smem_u32(&bars->tmem_empty[b]), TR::kEpiWarps * CG);
    }
    bars->abort_flag = 0;
    fence_barrier_init();
    prefetch_tensormap(&tm_a);
    prefetch_tensormap(&tm_b0);
    prefetch_tensormap(&tm_b1);
    if (kPair) {
      prefetch_tensormap(&ts_a);
      prefetch_tensormap(&ts_b0);
      prefetch_tensormap(&ts_b1);
    }
  }
  if (warp == 2) {
    tmem_alloc<CG>(smem_u32(&bars->tmem_base), kTmemCols);
    tmem_relinquish<CG>();
  }
  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();             // the other CTA's barriers are initialised
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, bars->tmem_base, 0);
  pdl_wait();                              // set-up above overlaps the tail of the kernel before this one
  const int n_mtiles = __shfl_sync(0xffffffffu, a.tiles[0].x, 0);
  const ItemPlan plan = plan_items<TR::kGateUp>(a, n_mtiles, workers);
  const int n_whole = plan.n_whole;
  int n_mt_s = 0, n_shared = 0;
  if (kPair) {
    n_mt_s = __shfl_sync(0xffffffffu, as.tiles[0].x, 0);
    n_shared = n_mt_s * as.n_ntiles * (TR::kGateUp ? 1 : as.k_splits);
  }
  const int n_items = plan.n_items + n_shared;
  // item -> its number among the items of its kind
  auto is_shared = [&](int item) { return kPair && (TR::kGateUp ? item < n_shared : item >= plan.n_items); };
  auto shared_no = [&](int item) { return TR::kGateUp ? item : item - plan.n_items; };
  auto routed_no = [&](int item) { return TR::kGateUp && kPair ? item - n_shared : item; };

  if (warp == 0) {
    // ---------------------------------------------------------------- token-operand producer
    if (lane == 0) {
      RingPos p;
      bool ok = true;
      for (int item = worker; ok && item < n_items; item += workers)
        ok = is_shared(item)
            ? load_operands<kS, S, CG>(ts_a, ts_b0, ts_b1, as, shared_no(item), n_mt_s, n_shared, sA, sB, bars, rank, p)
            : load_operands<MODE, S, CG>(tm_a, tm_b0, tm_b1, a, routed_no(item), n_mtiles, n_whole, sA, sB, bars, rank, p);
      if (ok) (void)await_last_commits<S>(bars, p);
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- packed-weight producer
    if (TR::kUnpack && lane == 0) {
      RingPos p;
      for (int item = worker; item < n_items; item += workers) {
        bool ok = true;
        if (!is_shared(item)) ok = load_codes<MODE, kStagesP, kStageP, CG>(tm_b0, tm_b1, a, routed_no(item), n_mtiles, n_whole, sP, bars, rank, p);
        else if (ModeTraits<kS>::kUnpack) ok = load_codes<kS, kStagesP, kStageP, CG>(ts_b0, ts_b1, as, shared_no(item), n_mt_s, n_shared, sP, bars, rank, p);
        if (!ok) break;
      }
    }
  } else if (warp == 2) {
    // ---------------------------------------------------------------- MMA issuer
    if (rank == 0) {
      RingPos p;
      int local = 0;
      for (int item = worker; item < n_items; item += workers, ++local) {
        const bool ok = is_shared(item)
            ? issue_mmas<kS, S, CG>(as, shared_no(item), n_shared, local, tmem_base, sA, sB, bars, p)
            : issue_mmas<MODE, S, CG>(a, routed_no(item), n_whole, local, tmem_base, sA, sB, bars, p);
        if (!ok) break;
      }
    }
  } else if (TR::kUnpack && warp >= 4 && warp < 12) {
    // ---------------------------------------------------------------- code unpackers
    if (TR::kUnpack) {
      const int group = (warp - 4) >> 2;
      RingPos p, q;
      uint32_t step = 0;
      for (int item = worker; item < n_items; item += workers) {
        const bool ok = is_shared(item)
            ? expand_codes<kS, S, kStagesP, kStageP, CG>(as, shared_no(item), n_shared, group, genB, genP, bars, p, q, step)
            : expand_codes<MODE, S, kStagesP, kStageP, CG>(a, routed_no(item), n_whole, group, genB, genP, bars, p, q, step);
        if (!ok) break;
      }
    }
  } else if (warp >= TR::kEpiFirst) {
    // ---------------------------------------------------------------- epilogue
    int local = 0;
    for (int item = worker; item < n_items; item += workers, ++local) {
      const bool ok = is_shared(item) ? write_out<kS, CG, TR::kEpiFirst, TR::kEpiWarps>(as, shared_no(item), n_mt_s, n_shared, local, tmem_base, genE, bars, rank)
                                      : write_out<MODE, CG, TR::kEpiFirst, TR::kEpiWarps>(a, routed_no(item), n_mtiles, n_whole, local, tmem_base, genE, bars, rank);
      if (!ok) break;
    }
  }

  // ------------------------------------------------------------------ teardown
  drain_after_abort(abort_flag);
  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();             // neither CTA's shared memory and TMEM go while the other still works with them
  if (warp == 2) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc<CG>(tmem_base, kTmemCols);
  }
  if (threadIdx.x == 0) report_abort(abort_flag, a.status);
  if (CG == 2) cluster_sync();
}

template <int MODE, int CG>
__global__ void __launch_bounds__(ModeTraits<MODE, CG>::kThreads, 1)
umma_gemm_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b0,
                 const __grid_constant__ CUtensorMap tm_b1, const UmmaArgs a) {
  umma_cta<MODE, -1, CG>(tm_a, tm_b0, tm_b1, a, tm_a, tm_b0, tm_b1, a);
}
template <int MODE, int SMODE>
__global__ void __launch_bounds__(ModeTraits<MODE>::kThreads, 1)
umma_pair_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b0,
                 const __grid_constant__ CUtensorMap tm_b1, const UmmaArgs a, const __grid_constant__ CUtensorMap ts_a,
                 const __grid_constant__ CUtensorMap ts_b0, const __grid_constant__ CUtensorMap ts_b1, const UmmaArgs as) {
  umma_cta<MODE, SMODE, 1>(tm_a, tm_b0, tm_b1, a, ts_a, ts_b0, ts_b1, as);
}

// One CTA that runs the GEMM kernels' bounded wait to its limit: an mbarrier nothing ever arrives
// at, no copy and no MMA in flight.  The wait gives up after limit_ns, the CTA takes the same
// teardown as the GEMM (drain, status word) and returns normally; the context stays usable.
__global__ void bounded_wait_selftest_kernel(uint32_t* status, uint64_t limit_ns) {
  __shared__ uint64_t bar;
  __shared__ int abort_word;
  volatile int* abort_flag = &abort_word;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_word = 0;
    fence_barrier_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) (void)mbar_wait(smem_u32(&bar), 0, abort_flag, limit_ns);
  __syncthreads();
  drain_after_abort(abort_flag);
  __syncthreads();
  if (threadIdx.x == 0) report_abort(abort_flag, status);
}

mote_status_t launch_bounded_wait_selftest(uint32_t* status, uint64_t limit_ns, cudaStream_t stream) {
  bounded_wait_selftest_kernel<<<1, 32, 0, stream>>>(status, limit_ns);
  MOTE_LAUNCH_OK();
  return MOTE_OK;
}

// ------------------------------------------------------------------------------------------------
// Host side: tensor maps and launches
// ------------------------------------------------------------------------------------------------
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

// 2-D row-major tensor [rows, cols] of elem_bytes-wide elements, box [box_rows, box_cols].
static bool make_map_2d(CUtensorMap* m, const void* base, CUtensorMapDataType dt, int elem_bytes, uint64_t rows,
                        uint64_t cols, uint32_t box_rows, uint32_t box_cols, CUtensorMapSwizzle sw) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * (uint64_t)elem_bytes};
  cuuint32_t box[2] = {box_cols, box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(m, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Width of a down-projection tile: the largest multiple of 32 up to 256 that divides N (N is a
// multiple of 128).  Wider tiles reuse the token operand for more MMA work per byte fetched.
static int pick_bn(int N) {
  for (int bn = 256; bn > 128; bn -= 32)
    if (N % bn == 0) return bn;
  return 128;
}

template <int MODE, int CG = 1>
static mote_status_t launch_umma(const CUtensorMap& ta, const CUtensorMap& tb0, const CUtensorMap& tb1,
                                 const UmmaArgs& a, int max_items, cudaStream_t stream, bool pdl) {
  using TR = ModeTraits<MODE, CG>;
  static PerDeviceOnce attr_once;                  // one per MODE and CG (this function is a template)
  MOTE_CUDA_OK(set_max_dynamic_smem(attr_once, umma_gemm_kernel<MODE, CG>, (int)TR::kSmem));
  const int grid = CG * std::max(1, std::min(device_sm_count() / CG, max_items));
  MOTE_CUDA_OK(launch_ex(umma_gemm_kernel<MODE, CG>, dim3(grid), dim3(TR::kThreads), TR::kSmem, stream, pdl, CG, ta, tb0, tb1, a));
  ++g_launch_count;
  g_gemm_tile[(TR::kTernary ? 0 : 2) + (TR::kGateUp ? 0 : 1)] = (kBM * CG) << 16 | a.bn;
  MOTE_LAUNCH_OK();
  return MOTE_OK;
}

// Rows of the (first) weight map's box; load_weight_rows fetches one or two of them.
static uint32_t weight_box_rows(int bn, bool gateup, int cg) {
  if (cg == 1 || gateup) return std::min(bn, 128);
  return bn == 256 ? 64 : bn / 2;
}

// Tensor maps and arguments of one GEMM.
struct GemmSetup {
  CUtensorMap ta, tb0, tb1;
  UmmaArgs a{};
};

// cg: CTAs per tile (row tiles of 128 * cg rows)
static bool setup_ternary(GemmSetup& u, const TernaryGemmArgs& g, bool gateup, const int4* tiles, int max_mtiles,
                          const int32_t* rowsum, uint32_t* beta_out_bits, uint32_t* status, int cg) {
  int bn = gateup ? 256 : pick_bn(g.N);
  // a down projection with few row tiles: the narrowest tiles (at least 64 wide) that are no more than the SMs (the
  // weights are the traffic here, and they are read once either way)
  if (!gateup) {
    const int workers = device_sm_count() / cg;
    for (int n = 64; n < bn; n += 32)
      if (g.N % n == 0 && max_mtiles * (g.N / n) <= workers) bn = n;
  }
  // second weight map: the up matrix (gate/up), or the rows beyond 128 of a down tile of one CTA
  const uint32_t rows0 = weight_box_rows(bn, gateup, cg);
  if (!make_map_2d(&u.ta, g.qa, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)g.P, (uint64_t)g.K, 128, 128,
                   CU_TENSOR_MAP_SWIZZLE_128B) ||
      !make_map_2d(&u.tb0, g.w0, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)g.E * g.N, (uint64_t)g.K / 4,
                   rows0, 32, CU_TENSOR_MAP_SWIZZLE_NONE) ||
      !make_map_2d(&u.tb1, gateup ? g.w1 : g.w0, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)g.E * g.N,
                   (uint64_t)g.K / 4, (gateup || bn <= 128) ? 128 : bn - 128, 32, CU_TENSOR_MAP_SWIZZLE_NONE))
    return false;
  UmmaArgs& a = u.a;
  a.tiles = tiles;
  a.n_ntiles = gateup ? g.N / 128 : g.N / bn;
  a.k_steps = g.K / 128;
  a.k_splits = 1;
  a.bn = bn;
  a.split_tail = (!gateup && bn == 256) ? 1 : 0;
  a.n_out = g.N;
  a.b_rows_per_expert = g.N;
  a.beta = g.beta; a.rowsum = rowsum; a.alpha0 = g.alpha0; a.alpha1 = g.alpha1;
  a.out = gateup ? g.h_bf16 : static_cast<void*>(g.y);
  a.tap0 = g.acc0_tap; a.tap1 = g.acc1_tap;
  a.beta_out_bits = gateup ? beta_out_bits : nullptr;
  a.status = status;
  return true;
}

mote_status_t launch_ternary_umma(const TernaryGemmArgs& g, bool gateup, const int4* tiles, int max_mtiles,
                                  const int32_t* rowsum, uint32_t* beta_out_bits, uint32_t* status,
                                  cudaStream_t stream, bool pdl, int cg) {
  if (g.P == 0) return MOTE_OK;
  GemmSetup u;
  if (!setup_ternary(u, g, gateup, tiles, max_mtiles, rowsum, beta_out_bits, status, cg)) return MOTE_ERR_CUDA;
  const int max_items = max_mtiles * u.a.n_ntiles;
  if (cg == 2)
    return gateup && g.K <= kShortK ? launch_umma<MODE_T_GATEUP_SHORT, 2>(u.ta, u.tb0, u.tb1, u.a, max_items, stream, pdl)
           : gateup ? launch_umma<MODE_T_GATEUP, 2>(u.ta, u.tb0, u.tb1, u.a, max_items, stream, pdl)
                  : launch_umma<MODE_T_DOWN, 2>(u.ta, u.tb0, u.tb1, u.a, max_items, stream, pdl);
  return gateup ? launch_umma<MODE_T_GATEUP>(u.ta, u.tb0, u.tb1, u.a, max_items, stream, pdl)
                : launch_umma<MODE_T_DOWN>(u.ta, u.tb0, u.tb1, u.a, max_items, stream, pdl);
}

// K splits of the shared down projection: with few row tiles its T x N output has too few tiles to
// occupy the SMs (one row tile of c3: 6 tiles for 27 MB of weights), so each tile's K range is cut
// into up to 16 items whose partial sums the caller adds.  At most 4096 partial rows in all.
int shared_down_k_splits(int64_t T, int N, int K) {
  const int sms = device_sm_count();
  const int64_t n_tiles = ((T + 127) / 128) * (N / pick_bn(N));
  if (n_tiles * 2 > sms) return 1;
  int64_t splits = std::min<int64_t>(16, sms / n_tiles);
  splits = std::min<int64_t>(splits, (K / 64) / 4);
  splits = std::min<int64_t>(splits, kMaxPartialRows / T);
  return (int)std::max<int64_t>(splits, 1);
}

// ------------------------------------------------------------------------------------------------
// One CTA per tile of 128 rows or a pair per tile of 256?  Per pipeline step a pair needs half the weight bytes, half of the
// expansion and half of the weight operand's reads from shared memory in each SM, but its row tiles are twice as long, which
// rounds an expert's rows up to 256, and half as many workers end in a longer last round.  So both are put as pipeline steps (a
// step of the routed gate/up GEMM on single CTAs, 0.42 us, is the unit; the other rates are measured in that unit) times rounds.
// us of the two GEMMs of the routed experts (gate/up + down), single CTAs / pairs, uniform routing: 2048 x 11008, 16 experts, top-2:
// 131 / 178 (768 tokens), 132 / 182 (960), 230 / 183 (1536), 290 / 256 (2048); 4 experts, top-1: 88 / 74 (768), 102 / 102 (1152);
// 896 x 4864, 4 experts: 48 / 48 (1024), 86 / 84 (2304), 122 / 109 (4096); 512 x 2048, 16 experts: 54 / 59 (4096); 384 x 9216,
// 2 experts, top-1: 94 / 85 (4000).  Of the shared ones: 2048 x 11008: 125 / 142 (1152: K splits fill one round of single CTAs),
// 174 / 163 (1536); 256 x 512: 33 / 35 (8192).
// The rule errs towards single CTAs where an expert's rows lie below 256, of which half a tile per expert is too much (it forgoes
// the pairs at 16 experts, 1536 tokens, and at 4 experts, 768 tokens), and once the other way (256 x 512, 8192 tokens: 32 / 34).
// It puts a routed down projection at pick_bn's width, although few row tiles are launched narrower (setup_ternary), and the
// two GEMMs of a step share a table of tiles, so they choose alike.
// ------------------------------------------------------------------------------------------------
static double gemm_steps(double row_tiles, int n_tiles, double steps, int workers, bool halves, double per_step, double least) {
  const double rounds = row_tiles * n_tiles / workers, whole = std::floor(rounds + 1e-9), tail = rounds - whole;
  const double last = tail <= 1e-6 ? 0.0 : halves && tail <= 0.5 ? 0.6 : 1.0;
  return (whole + last) * std::max(steps * per_step, least);      // least: a tile's epilogue, where K is short
}
int routed_ctas_per_tile(int64_t P, int E, int d, int f) {
  double cost[2];
  for (int cg = 1; cg <= 2; ++cg) {
    const int workers = device_sm_count() / cg, bn = pick_bn(d);
    const double row_tiles = double(P) / (128 * cg) + 0.5 * std::min<int64_t>(E, P);     // the router's choice is not known here
    const double steps = gemm_steps(row_tiles, f / 128, d / 128, workers, false, cg == 1 ? 1.0 : 0.72, cg == 1 ? 14 : 12) +
                         gemm_steps(row_tiles, d / bn, f / 128, workers, bn == 256, cg == 1 ? 0.9 : 0.75, 0);
    cost[cg - 1] = steps + (cg == 1 ? 0 : 8);                       // clusters start later
  }
  return cost[1] < cost[0] ? 2 : 1;
}
int shared_ctas_per_tile(int64_t T, int d, int f, int k_splits) {
  double cost[2];
  for (int cg = 1; cg <= 2; ++cg) {
    const int workers = device_sm_count() / cg, bn = pick_bn(d);
    const double row_tiles = double((T + 128 * cg - 1) / (128 * cg));
    const double steps = gemm_steps(row_tiles, f / 128, d / 64, workers, false, cg == 1 ? 0.93 : 0.85, 0) +
                         gemm_steps(row_tiles, d / bn * k_splits, f / 64.0 / k_splits, workers, bn == 256 && k_splits == 1,
                                    cg == 1 ? 1.1 : 1.03, 0);
    cost[cg - 1] = steps + (cg == 1 ? 0 : 8);
  }
  return cost[1] < cost[0] ? 2 : 1;
}

static bool setup_shared(GemmSetup& u, const void* act, const SharedMat& w0, const SharedMat& w1, int bits, bool gateup,
                         int64_t T, int K, int N, void* out, const int4* tiles, uint32_t* status, const CombineArgs* comb,
                         int k_splits, int cg) {
  const int bn = gateup ? 256 : pick_bn(N);
  const uint32_t rows0 = weight_box_rows(bn, gateup, cg);
  const uint32_t rows1 = (gateup || bn <= 128) ? 128 : bn - 128;
  if (!make_map_2d(&u.ta, act, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)T, (uint64_t)K, 128, 64,
                   CU_TENSOR_MAP_SWIZZLE_128B))
    return false;
  const void* wb1 = gateup ? w1.w : w0.w;
  if (bits == 16) {
    if (!make_map_2d(&u.tb0, w0.w, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)N, (uint64_t)K, rows0, 64,
                     CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_2d(&u.tb1, wb1, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)N, (uint64_t)K, rows1, 64,
                     CU_TENSOR_MAP_SWIZZLE_128B))
      return false;
  } else {
    // code rows as bytes: K (int8) or K/2 (4-bit) per row, 64 reduction elements per pipeline stage
    const uint64_t row_bytes = bits == 8 ? (uint64_t)K : (uint64_t)K / 2;
    const uint32_t box = bits == 8 ? 64 : 32;
    if (!make_map_2d(&u.tb0, w0.w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)N, row_bytes, rows0, box,
                     CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !make_map_2d(&u.tb1, wb1, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, (uint64_t)N, row_bytes, rows1, box,
                     CU_TENSOR_MAP_SWIZZLE_NONE))
      return false;
  }
  UmmaArgs& a = u.a;
  a.tiles = tiles;
  a.n_ntiles = gateup ? N / 128 : N / bn;
  a.k_steps = K / 64;
  a.k_splits = std::max(k_splits, 1);
  a.split_stride = T * N;
  a.bn = bn;
  a.split_tail = (!gateup && bn == 256 && a.k_splits == 1) ? 1 : 0;
  a.n_out = N;
  a.b_rows_per_expert = 0;
  a.out = out;
  a.status = status;
  a.alpha0 = w0.scale; a.alpha1 = w1.scale;     // row scales of an RTN-coded shared expert, else null
  if (comb && !gateup) {
    a.comb_y = comb->y; a.comb_w = comb->w; a.comb_perm = comb->perm;
    a.comb_res = static_cast<const uint16_t*>(comb->residual); a.comb_out = static_cast<uint16_t*>(comb->out);
    a.comb_k = comb->k;
    a.comb_wide = ((reinterpret_cast<uintptr_t>(comb->out) | reinterpret_cast<uintptr_t>(comb->residual)) & 31u) == 0;
  }
  return true;
}

mote_status_t launch_shared_umma(const void* act, const SharedMat& w0, const SharedMat& w1, int bits, bool gateup,
                                 int64_t T, int K, int N, void* out, const int4* tiles, int max_mtiles,
                                 uint32_t* status, const CombineArgs* comb, cudaStream_t stream, bool pdl,
                                 int k_splits, int cg) {
  if (T == 0) return MOTE_OK;
  if (k_splits > 1 && (gateup || comb || !out)) return MOTE_ERR_SHAPE;
  if (cg == 2 && bits != 16) return MOTE_ERR_SHAPE;
  GemmSetup u;
  if (!setup_shared(u, act, w0, w1, bits, gateup, T, K, N, out, tiles, status, comb, k_splits, cg)) return MOTE_ERR_CUDA;
  const UmmaArgs& a = u.a;
  const int max_items = max_mtiles * a.n_ntiles * a.k_splits;
  if (cg == 2)
    return gateup ? launch_umma<MODE_B_GATEUP, 2>(u.ta, u.tb0, u.tb1, a, max_items, stream, pdl)
                  : launch_umma<MODE_B_DOWN, 2>(u.ta, u.tb0, u.tb1, a, max_items, stream, pdl);
  if (bits == 8)
    return gateup ? launch_umma<MODE_Q8_GATEUP>(u.ta, u.tb0, u.tb1, a, max_items, stream, pdl)
                  : launch_umma<MODE_Q8_DOWN>(u.ta, u.tb0, u.tb1, a, max_items, stream, pdl);
  if (bits == 4)
    return gateup ? launch_umma<MODE_Q4_GATEUP>(u.ta, u.tb0, u.tb1, a, max_items, stream, pdl)
                  : launch_umma<MODE_Q4_DOWN>(u.ta, u.tb0, u.tb1, a, max_items, stream, pdl);
  return gateup ? launch_umma<MODE_B_GATEUP>(u.ta, u.tb0, u.tb1, a, max_items, stream, pdl)
                : launch_umma<MODE_B_DOWN>(u.ta, u.tb0, u.tb1, a, max_items, stream, pdl);
}

template <int MODE, int SMODE>
static mote_status_t launch_pair(const GemmSetup& r, const GemmSetup& sh, int max_items, cudaStream_t stream, bool pdl) {
  constexpr size_t smem = PairTraits<MODE, SMODE, 1>::kSmem;
  constexpr int kThreads = PairTraits<MODE, SMODE, 1>::kThreads;
  static PerDeviceOnce attr_once;                  // one per pair
  MOTE_CUDA_OK(set_max_dynamic_smem(attr_once, umma_pair_kernel<MODE, SMODE>, (int)smem));
  const int grid = std::max(1, std::min(device_sm_count(), max_items));
  MOTE_CUDA_OK(launch_ex(umma_pair_kernel<MODE, SMODE>, dim3(grid), dim3(kThreads), smem, stream, pdl, 1, r.ta, r.tb0, r.tb1, r.a,
                         sh.ta, sh.tb0, sh.tb1, sh.a));
  ++g_launch_count;
  MOTE_LAUNCH_OK();
  return MOTE_OK;
}

mote_status_t launch_umma_pair(const TernaryGemmArgs& g, bool gateup, const int4* tiles_routed, int max_mtiles_routed,
                               const int32_t* rowsum, uint32_t* beta_out_bits, const void* act, const SharedMat& w0,
                               const SharedMat& w1, int bits, int64_t T, void* out, const int4* tiles_shared,
                               int max_mtiles_shared, uint32_t* status, cudaStream_t stream, bool pdl, int k_splits) {
  if (g.P == 0) return MOTE_OK;
  GemmSetup r, sh;
  if (!setup_ternary(r, g, gateup, tiles_routed, max_mtiles_routed, rowsum, beta_out_bits, status, 1) ||
      !setup_shared(sh, act, w0, w1, bits, gateup, T, g.K, g.N, out, tiles_shared, status, nullptr, k_splits, 1))
    return MOTE_ERR_CUDA;
  const int max_items = max_mtiles_routed * r.a.n_ntiles + max_mtiles_shared * sh.a.n_ntiles * sh.a.k_splits;
  if (bits == 8)
    return gateup ? launch_pair<MODE_T_GATEUP, MODE_Q8_GATEUP>(r, sh, max_items, stream, pdl)
                  : launch_pair<MODE_T_DOWN, MODE_Q8_DOWN>(r, sh, max_items, stream, pdl);
  if (bits == 4)
    return gateup ? launch_pair<MODE_T_GATEUP, MODE_Q4_GATEUP>(r, sh, max_items, stream, pdl)
                  : launch_pair<MODE_T_DOWN, MODE_Q4_DOWN>(r, sh, max_items, stream, pdl);
  return gateup ? launch_pair<MODE_T_GATEUP, MODE_B_GATEUP>(r, sh, max_items, stream, pdl)
                : launch_pair<MODE_T_DOWN, MODE_B_DOWN>(r, sh, max_items, stream, pdl);
}

}  // namespace mote
