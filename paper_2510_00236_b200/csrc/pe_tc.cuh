// Tensor-core kernel for the sequence-level per-example statistics (Section 2.3; Eq. (2)).
//
// Work unit: a CTA PAIR (a cluster of two thread blocks on two SMs) owns a 256 x NT tile of the
// [d_out, d_in] output (NT = 128, 192 or 256) and a contiguous slice of the batch.  For every example of
// the slice the tile of G_b = dY_b^T X_b is formed by pair-wide tcgen05 MMAs (cta_group::2,
// M = 256: each block supplies 128 rows of dY_b^T and half of the NT rows of X_b^T from its own
// shared memory and receives its 128 accumulator rows in its own tensor memory), read back by the
// epilogue warps, passed through phi and added to register-resident running sums (sum_b phi(G_b)
// and, when asked for, sum_b G_b).  The per-example tile never leaves the SM.  Pairing cuts the
// operand bytes each SM pulls from L2 per flop; an SM sustains about 70 B/clk from L2, a lone
// 128 x 128 tile would need 128 B/clk at full tensor rate, a 256 x 128 pair 96, a 256 x 192 pair 75, a
// 256 x 256 pair 64.
//
//   MEAN_REGS, NT = 128: two running sums per thread (64 + 64 registers)         -- both outputs
//   MEAN_REGS, NT = 192: two running sums per thread (96 + 96 registers; the control
//                        warps shrink to 40 registers so that the epilogue warps can take 232) -- both outputs
//   MEAN_REGS_SIGN, NT = 128: the same plus sum_b sign(G_b), counted in 16-bit halves
//                        of 32 more registers                                      -- mean, square and sign in one pass
//   MEAN_HYBRID_SIGN, NT = 192: mean, square and sign on the wider tile: sum_b G_b^2 (96 registers), the sign
//                        counts (48) and a third of sum_b G_b (32) in registers, the other two thirds of
//                        sum_b G_b in the 128 tensor-memory columns the two accumulators leave free
//   MEAN_TMEM, NT = 256: sum_b phi(G_b) in 128 registers per thread, sum_b G_b in
//                        tensor memory beside ONE per-example accumulator       -- both outputs
//   MEAN_NONE, NT = 256: one running sum per thread (128 registers)               -- only sum_b phi(G_b) wanted
//   MEAN_NORMS, NT = 256: no running sums; every example's sum of squares over the
//                        tile is reduced and added to out_norms[b]                 -- per-example squared norms
//   PHI = 0,   NT = 256: no per-example reset (accumulate in tensor memory)        -- plain contraction over all rows
// Further template arguments: RAGGED (packed batches with per-example token ranges), OPT (the parameter
// update applied by the block that completes a tile's sums), F8 (e4m3 operands for the plain contraction), CHUNKED (several
// accumulators per example), PERSIST (several tiles per pair), PARTS (several contractions in one launch).
//
// Warp roles per block (12 warps): 0 = TMA producer of the dY boxes, 2 = TMEM allocator, then TMA
// producer of the X boxes, 1 = MMA issuer (leader block only), 3 idle, 4..11 = epilogue (warp w reads
// TMEM lanes 32*(w%4)..+31, column half (w-4)/4).  The control warps run warp-uniform code in which
// every lane waits and one elected lane issues: TMA, MMA and commit instructions take their operands
// from uniform registers, and the same loops written for "lane 0 only" spent about 140 cycles per MMA,
// 115 per TMA load and 550 per barrier probe behind queued MMAs, which bound every shape and needed two
// issuers on alternate examples with half the operand ring each.  One issuer on the whole ring instead:
// 128 x 512 tokens x 1024^2, both outputs 152 -> 127 us, three statistics 183 -> 134; 64 x 256 x 512 x 2048
// 41.3 -> 36.3 us (cuBLAS' plain GEMM of the shape: 35.8).
// The 512 TMEM columns hold 512/NT accumulators, so the MMAs of later examples overlap the epilogue of
// earlier ones.  (MEAN_TMEM has one accumulator: while the epilogue drains it the producers keep filling
// the ring, and the issuer then works the backlog off at full tensor rate, which absorbs the pause as long
// as the operand supply, not the tensor pipe, is what bounds the example.)
//
// PERSIST: layers of more tiles than pairs.  A pair per two SMs takes every (gridDim.x / 2)-th unit: the tensor work of a tile starts
// while the one before is written out (two accumulators ahead; the write-out goes from registers to memory, past the ring), and
// prologue and teardown are paid once.  The tiles of the last, partial wave are contracted in slices of the batch, as many
// as leave every pair one, and added to outputs zeroed beforehand, in no fixed order (more than two slices: the low bits may differ between
// runs).  Bound by the operand supply as
// before.  8 x 256 x 1024 x 32104, both outputs 231 -> 174 us, sign 165 -> 121;
// 64 x 256 x 512 x 32768 565 -> 527 (of which the slices 40), sign 477 -> 420; 16 x 1024 x 2048 x 8192, sign 460 -> 405, but
// sequences of 256 tokens and more gain nothing by the walk alone (64 x 256 x 512 x 16384, three statistics, 321 -> 328 us).
//
// Barriers.  full[s] lives in the leader block: its producer posts the byte count of BOTH blocks'
// loads, and the follower's TMA loads credit their bytes to it through the cluster window.
// empty[s] and acc_full[a] exist in both blocks and are signalled in both by one multicast commit.
// acc_empty[a] lives in the leader and collects the arrivals of both blocks' epilogue warps.
//
// Operand orientation: A = dY_b viewed as M = d_out x K = T and B = X_b viewed as N = d_in x K = T.
// In global memory the contraction index (the token) is the slow one, so both operands are
// "MN-major".  A TMA box is 128 bytes of features (64 bf16) x BK tokens; with the 128-byte swizzle that is
// exactly the canonical MN-major layout of the MMA: 8-token x 64-feature atoms of 1 KiB, the next
// 8 tokens 1 KiB further (stride byte offset), the next 64 features one box further (leading byte
// offset).  (X at NT = 192: 64 bytes of features per box row and the 64-byte swizzle, 512-byte atoms.)
#pragma once
#include "pe_optim.cuh"
#include "pe_sm100.cuh"

namespace pe {

constexpr int TC_TILE_M = 128;    // d_out rows per block (the pair covers 256)
constexpr int TC_PAIR_M = 2 * TC_TILE_M;
constexpr int TC_TMEM_COLS = 512;
constexpr int TC_THREADS = 384;
constexpr int TC_REGS_CONTROL = 64;     // setmaxnreg of warps 0..3
constexpr int TC_REGS_EPILOGUE = 216;   // setmaxnreg of warps 4..11  (4*32*64 + 8*32*216 = 63488 <= 384*168)
constexpr int TC_REGS_AT_LAUNCH = 168;  // registers per thread of a 384-thread block at one block per SM (65536 / 384, in eights)
constexpr int TC_BAR_BYTES = 512;
// operand ring; leaves room for barriers and alignment slack.  The 256 x 192 tile's four 56 KiB stages take 224 KiB.
__host__ __device__ constexpr int tc_smem_budget(int nt) { return (nt == 192 ? 224 : 200) * 1024; }

// Operand element type of the MMA.  bf16 (kind::f16, 16 tokens per instruction) for the per-example
// statistics; tf32 (kind::tf32, fp32 storage, 8 tokens per instruction) for the per-token statistic,
// whose squared operands need more than bf16's 8 significant bits.  NT = d_in columns per pair tile.
// Default tokens per pipeline stage: 128 for the 256 x 128 tile, 64 for the 256 x 256 tile, 32 for
// tf32.  (The statistics of sequences of at most 32 tokens have a kernel of their own, pe_short.cuh.)
__host__ __device__ constexpr int tc_default_bk(bool tf32, int nt) { return tf32 ? 32 : (nt == 256 ? 64 : 128); }
constexpr int TC_CHUNK_TOKENS = 512;    // CHUNKED: tokens per accumulator
// F8: 8-bit operands (kind::f8f6f4, e4m3, 32 tokens per instruction): the scaled squares of the two-pass
// per-token statistic's fp8 form.
template <bool TF32, int NT, int BK_ = tc_default_bk(TF32, NT), bool F8 = false>
struct TcOperand {
  static_assert(!(TF32 && F8), "one operand type");
  static constexpr int ELEM_BYTES = TF32 ? 4 : (F8 ? 1 : 2);
  static constexpr int BOX_FEATS = 128 / ELEM_BYTES;            // features per 128-byte swizzle row: 64 | 32 | 128
  // tokens per pipeline stage (one TMA box is BK tokens tall)
  static constexpr int BK = BK_;
  static constexpr int MMA_K = 32 / ELEM_BYTES;                 // tokens per MMA instruction: 16 | 8 | 32
  static constexpr int BOX_BYTES = 128 * BK;                    // one box: BK tokens x 128 bytes
  static constexpr int A_BOXES = TC_TILE_M / BOX_FEATS;         // this block's 128 rows of dY^T
  static constexpr int B_FEATS = NT / 2;                        // this block's half of the tile's d_in columns
  // NT = 192: 96 columns of X per block are one and a half 128-byte rows.  X is then loaded in
  // 64-byte rows (32 features per box, TMA SWIZZLE_64B) and described to the MMA with the 64-byte
  // swizzle (descriptor layout 4: 8-token x 32-feature atoms of 512 bytes); dY keeps 128-byte rows.
  static constexpr bool B_NARROW = (B_FEATS % BOX_FEATS) != 0;
  static_assert(!B_NARROW || !TF32, "64-byte rows are only set up for 16-bit operands");
  static constexpr int B_ROW_BYTES = B_NARROW ? 64 : 128;
  static constexpr int B_BOX_FEATS = B_ROW_BYTES / ELEM_BYTES;  // 64 | 32
  static constexpr int B_BOX_BYTES = B_ROW_BYTES * BK;
  static constexpr int B_BOXES = B_FEATS / B_BOX_FEATS;         // 1 | 2 | 3
  static constexpr int A_BYTES = A_BOXES * BOX_BYTES;           // 32 KiB (BK = 128) | 16 KiB
  static constexpr int B_BYTES = B_BOXES * B_BOX_BYTES;         // 16 KiB | 24 KiB (NT = 192)
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;         // per block: 48 KiB | 56 KiB | 32 KiB
  static constexpr int STAGES = tc_smem_budget(NT) / STAGE_BYTES;   // 4 | 4 | 6
  static constexpr int K_STEP_BYTES = MMA_K * 128;              // smem advance per MMA: 2048 | 1024
  static constexpr int B_K_STEP_BYTES = MMA_K * B_ROW_BYTES;
  static constexpr int ACC_BUFS = TC_TMEM_COLS / NT;            // 4 | 2 | 2 accumulators in tensor memory
  // MN-major swizzle atoms: bf16 = 8 tokens x 128 B with 16-byte chunks (descriptor layout 2, TMA
  // SWIZZLE_128B); tf32 = 4 tokens x 128 B with 32-byte chunks (layout 1, TMA SWIZZLE_128B_ATOM_32B).
  static constexpr uint32_t DESC_LAYOUT = TF32 ? 1u : 2u;
  static constexpr uint32_t SBO_BYTES = TF32 ? 512u : 1024u;   // next swizzle atom along the tokens
  static constexpr uint32_t B_DESC_LAYOUT = B_NARROW ? 4u : DESC_LAYOUT;
  static constexpr uint32_t B_SBO_BYTES = B_NARROW ? 512u : SBO_BYTES;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + TC_BAR_BYTES + 1024;   // + alignment slack
  // Register split between the four control warps and the eight epilogue warps (setmaxnreg).  The pool
  // is what the block was launched with, 384 threads x 168 registers, NOT the SM's whole register file: an
  // increase that the decreases of the control warps do not cover never returns.  Two running sums of
  // 96 floats each need the larger epilogue share.
  static constexpr int REGS_CONTROL = (NT == 192) ? 40 : TC_REGS_CONTROL;
  static constexpr int REGS_EPILOGUE = (NT == 192) ? 232 : TC_REGS_EPILOGUE;
};

// error codes latched in the device status word (which wait gave up)
enum : int { TC_WAIT_EMPTY = 1, TC_WAIT_FULL = 2, TC_WAIT_ACC_EMPTY = 3, TC_WAIT_ACC_FULL = 4 };

struct TcParams {
  int B, T, d_in, d_out;
  int pairs_m, tiles_n, band;   // tile grid: 256-row pair rows x NT-column tiles; pair rows per band of the tile order
  int nsplit;          // batch slices (gridDim.z); > 1 => outputs pre-zeroed, partials added atomically
  int whole_tiles;     // PERSIST: tiles that one pair contracts over the whole batch; each of the others goes to
  int tail_split;      // this many pairs, by slices of the batch, whose sums are added to (zeroed) outputs
  int slice_examples;  // 0, or the examples of such a slice (the last one may have fewer): where slices are short, 64-bit divisions would show
  int sum_run;         // short_stats_kernel, the square alone: examples summed by themselves, a power of two
  int part_chunks;     // PARTS: chunks of rows per part, slices of the square's, the mean's and the sign's chunks
  int part_slices[3];
  unsigned int part_dy, part_x;   // PARTS: the copies of dY and of X that each product takes
  const uint8_t* odd_rows;        // PARTS: [part_chunks * T] examples whose square (1) or sign (2) the copies do not carry, formed from
  const uint16_t* rows_dy;        // the operands themselves, [.., d_out] and [.., d_in]
  const uint16_t* rows_x;
  int per_example;     // 1: reset the accumulator for every example and apply phi (statistics)
                       // 0: one accumulation over the whole slice (plain contraction, phi = identity)
  int half_operands;   // 16-bit operands are IEEE half instead of bf16 (the staged per-token statistic)
  int accumulate;      // add the results to what the outputs hold (no zeroing kernel runs before this one)
  int wait_at_start;   // the kernel before this one in the stream is not the one that zeroes the outputs: wait for it before anything else
  int scalar_out;      // d_in % 4 != 0: the outputs' rows are no 16-byte multiples, so the warps write them themselves
  float* out_mean;     // may be NULL; written through tmap_mean
  float* out_stat;     // may be NULL; written through tmap_stat
  float* out_sign;     // MEAN_REGS_SIGN only: sum_b sign(G_b), written through tmap_sign
  float* out_norms;    // MEAN_NORMS only: [B], zero on entry; every tile adds its share of ||G_b||_F^2
  const int* seq_offsets;   // RAGGED only: [B + 1] token-row offsets; example b owns rows offsets[b] .. offsets[b+1]-1
  int by_tokens;            // RAGGED only: the batch is sliced by tokens instead of by examples
  const float* sq_norms;    // PHI == 3 only: [B] per-example squared norms the clipping coefficient is taken from
  const float* scale_x;     // PHI == 4 only: [B, d_in] and [B, d_out] factors of example b's columns and rows of G_b
  const float* scale_y;
  float clip_norm;          // PHI == 3 only: C of c_b = min(1, C / sqrt(N_b))
  unsigned int* dev_status;
};

// PARTS: chunk c of the launch is chunk c % n of product c / n: the operands as they are | the upper half of dY's squares by that of X's, lower
// by upper, upper by lower, lower by lower | the signs.  part_dy, part_x: the copy that a product takes, four bits each.  Where that
// chunk is in the operand.
__device__ __forceinline__ int tc_part_chunk(const TcParams& p, int c, bool of_dy) {
  const int product = c / p.part_chunks;
  return (int)(((of_dy ? p.part_dy : p.part_x) >> (4 * product)) & 15u) * p.part_chunks + c - product * p.part_chunks;
}

// PERSIST: unit u of the launch, a tile and the examples it is contracted over.
struct TcUnit {
  int tile, b_begin, b_end;
  bool whole;
};
__device__ __forceinline__ int tc_units(const TcParams& p) { return p.whole_tiles + (p.pairs_m * p.tiles_n - p.whole_tiles) * p.tail_split; }
__device__ __forceinline__ TcUnit tc_unit(const TcParams& p, int u) {
  if (u < p.whole_tiles) return {u, 0, p.B, true};
  const int rest = p.pairs_m * p.tiles_n - p.whole_tiles, v = u - p.whole_tiles, slice = v / rest;
  if (p.slice_examples) return {p.whole_tiles + v - slice * rest, slice * p.slice_examples, min(p.B, (slice + 1) * p.slice_examples), false};
  return {p.whole_tiles + v - slice * rest, (int)((long long)p.B * slice / p.tail_split), (int)((long long)p.B * (slice + 1) / p.tail_split), p.tail_split == 1};
}

// Where an example's tokens are and how many pipeline stages they take.  Fixed-length batches: the
// operand maps are 3-D (d, T, B), an example is the coordinate `seq` of the last dimension and its
// stages start at token 0.  Packed (ragged) batches: the maps are (d, rows, 1), the example starts at
// row `row0`; its whole 16-token groups (`main` tokens) come from there in `nk_main` stages, and its
// last `len % 16` tokens come, zero-padded to 16, from a side buffer that a pre-pass fills (a map
// (d, 16, B)): one more stage with one MMA step.  An empty sequence is such a tail stage of zeros, so
// that every example owns at least one stage and one accumulator.
struct SeqGeom {
  int row0, main, nk_main, nk;
};
template <bool RAGGED>
__device__ __forceinline__ SeqGeom seq_geom(const TcParams& p, int b, int bk) {
  SeqGeom g;
  if constexpr (RAGGED) {
    const int r0 = __ldg(p.seq_offsets + b), r1 = __ldg(p.seq_offsets + b + 1);
    const int len = r1 > r0 ? r1 - r0 : 0;
    g.row0 = r0;
    g.main = len & ~15;
    g.nk_main = (g.main + bk - 1) / bk;
    g.nk = g.nk_main + (((len & 15) != 0 || len == 0) ? 1 : 0);
  } else {
    g.row0 = 0;
    g.main = p.T;
    g.nk_main = g.nk = (p.T + bk - 1) / bk;
  }
  return g;
}

// Slices of a packed batch: equal shares of tokens (plus 64 per example for its hand-offs), not of examples, whose lengths
// differ: first example of the slice that starts at `target`, the smallest b with offsets[b] + 64 b >= target.  A warp
// searches 32 ways at a time (two rounds up to 1024 examples).
__device__ __forceinline__ long long ragged_key(const int* offsets, int b) { return (long long)__ldg(offsets + b) + 64ll * b; }
__device__ __forceinline__ int ragged_slice_begin(const int* offsets, int B, int slice, int nsplit, int lane) {
  if (slice <= 0) return 0;
  if (slice >= nsplit) return B;
  const long long first = ragged_key(offsets, 0), target = first + (ragged_key(offsets, B) - first) * slice / nsplit;
  int lo = 0, hi = B;
  while (lo < hi) {
    const int step = (hi - lo + 31) / 32, idx = lo + lane * step;
    const unsigned below = __ballot_sync(0xffffffffu, idx < hi && ragged_key(offsets, idx) < target);
    if (below == 0u) break;
    const int last = lo + (__popc(below) - 1) * step;
    lo = last + 1;
    hi = min(hi, last + step);
  }
  return lo < B ? lo : B;
}

// Tile order.  Pairs that run at the same time should share operand panels in L2, so consecutive
// pair indices sweep the d_in tiles inside a band of p.band pair rows before moving to the next band:
// the ~74 resident pairs then touch about band*256 columns of dY and 74/band*NT columns of X per
// example instead of all of dY.  Returns this block's 128-row tile of d_out and NT-column tile of d_in.
__device__ __forceinline__ void tc_tile_of_pair(const TcParams& p, int pair_id, uint32_t rank, int& tile_m, int& tile_n) {
  const int per_band = p.band * p.tiles_n;
  const int band = pair_id / per_band, r = pair_id - band * per_band;
  const int rows = min(p.band, p.pairs_m - band * p.band);      // pair rows in this (possibly last, shorter) band
  tile_n = r / rows;
  tile_m = 2 * (band * p.band + (r - tile_n * rows)) + (int)rank;
}

// (sign(g) + 1) / 2, i.e. 0, 0.5 or 1, with sign(+-0) = 0, in two instructions: g is scaled by 2^64 (exact, or to
// infinity; the callers do it two columns at a time), then 2^127 * g + 0.5 is rounded and saturated to [0, 1].  The
// smallest nonzero |g|, the denormal 2^-149, arrives as 2^42, so every nonzero g saturates and zero alone gives 0.5.
// Summed over nb examples this is (sum_b sign(G_b) + nb) / 2, exact in fp32 (multiples of 0.5 below 2^23).
constexpr float SIGN_PRESCALE = 18446744073709551616.f;     // 2^64
__device__ __forceinline__ float sign_half_of_scaled(float g_scaled) {
  float u;
  asm("fma.rn.sat.f32 %0, %1, 0f7F000000, 0f3F000000;" : "=f"(u) : "f"(g_scaled));
  return u;
}
__device__ __forceinline__ float sign_half(float g) { return sign_half_of_scaled(g * SIGN_PRESCALE); }
// The same for two columns: {u(lo), u(hi)} packed for the two-wide fp32 instructions.
__device__ __forceinline__ uint64_t sign_half2(uint64_t g2) {
  float a0, a1;
  sm100::f32x2_unpack(sm100::f32x2_mul(g2, sm100::f32x2_pack(SIGN_PRESCALE, SIGN_PRESCALE)), a0, a1);
  return sm100::f32x2_pack(sign_half_of_scaled(a0), sign_half_of_scaled(a1));
}
// Two columns' sign(g) + 1 in {0, 1, 2} as the low and high 16 bits of one word: 2 u + 1.5 * 2^23 has the integer in
// the low bits of its pattern, and one byte permute packs the two low halves.
__device__ __forceinline__ uint32_t sign_plus_one_packed(uint64_t g2) {
  float t0, t1;
  sm100::f32x2_unpack(sm100::f32x2_fma(sign_half2(g2), sm100::f32x2_pack(2.f, 2.f), sm100::f32x2_pack(12582912.f, 12582912.f)), t0, t1);
  return __byte_perm(__float_as_uint(t0), __float_as_uint(t1), 0x5410);
}

template <int PHI>
__device__ __forceinline__ float phi_apply(float g) {
  if (PHI == 1) return g * g;
  if (PHI == 2) {
    // sign(g) with sign(+-0) = 0: (g != 0) as 1.0f / 0.0f, then g's sign bit copied onto it (-0.0f adds nothing)
    const float nz = (g != 0.f) ? 1.f : 0.f;
    return __uint_as_float(__float_as_uint(nz) | (__float_as_uint(g) & 0x80000000u));
  }
  return g;
}

// Zeroes the outputs of a split-batch launch.  The statistics kernel that follows is launched as a
// programmatic dependent: its launch overlaps the zeroing, its blocks start as the zeroing blocks leave their SMs (no SM has room for one of
// each), and it only waits for the whole of it in its very last step, behind griddepcontrol.wait.  It is a programmatic dependent itself, and lets its successor
// start only when everything before it has completed, on which the successor relies (early: at once, for a successor that waits for this one
// before anything else).  a, b, c: n floats each, 16-byte aligned; b and c may be NULL.  counters: the tile counters of a fused update
// (n_counters words; may be NULL).
__global__ void __launch_bounds__(256) zero_outputs_kernel(float4* __restrict__ a, float4* __restrict__ b, float4* __restrict__ c,
                                                           long long n, unsigned int* __restrict__ counters, int n_counters, int early) {
  if (early) sm100::griddep_launch_dependents();
  sm100::griddep_wait();
  if (!early) sm100::griddep_launch_dependents();
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  const long long stride = (long long)gridDim.x * blockDim.x;
  if (counters)
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n_counters; k += stride) counters[k] = 0u;
  const long long n4 = n >> 2;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n4; k += stride) {
    a[k] = z;
    if (b) b[k] = z;
    if (c) c[k] = z;
  }
  const long long k = (n4 << 2) + threadIdx.x;             // the last n % 4
  if (blockIdx.x == 0 && k < n) {
    reinterpret_cast<float*>(a)[k] = 0.f;
    if (b) reinterpret_cast<float*>(b)[k] = 0.f;
    if (c) reinterpret_cast<float*>(c)[k] = 0.f;
  }
}

// Zeroes the tiles from the p.whole_tiles-th on (256 rows x nt columns each) of up to three outputs, for the launch whose last
// tiles are split over the batch; a warp takes a row of a tile.  At most half a wave of tiles (29 MB for both outputs).  A block to every SM, so
// that the contraction starts where one has left: as ordinary launches of blocks without a share of their own the same within 0.5 % (8 x 256 x 1024 x 32104,
// both outputs, 160 us, 64 x 256 x 512 x 32768 459, 16 x 1024 x 2048 x 8192, sign, 355).
__global__ void __launch_bounds__(256) zero_tail_tiles_kernel(TcParams p, int nt) {
  sm100::griddep_wait();
  sm100::griddep_launch_dependents();
  const int rest = p.pairs_m * p.tiles_n - p.whole_tiles, lane = threadIdx.x & 31;
  for (int k = blockIdx.x * 8 + (threadIdx.x >> 5); k < rest * TC_PAIR_M; k += gridDim.x * 8) {
    int tile_m, tile_n;
    tc_tile_of_pair(p, p.whole_tiles + k / TC_PAIR_M, 0, tile_m, tile_n);
    const int row = tile_m * TC_TILE_M + k % TC_PAIR_M, end = min(p.d_in, (tile_n + 1) * nt);
    if (row >= p.d_out) continue;
    for (int col = tile_n * nt + lane; col < end; col += 32) {
      const long long at = (long long)row * p.d_in + col;
      if (p.out_mean) p.out_mean[at] = 0.f;
      if (p.out_stat) p.out_stat[at] = 0.f;
      if (p.out_sign) p.out_sign[at] = 0.f;
    }
  }
}

// where sum_b G_b is kept in per-example mode; MEAN_REGS_SIGN = MEAN_REGS with phi = square plus the sign statistic
// MEAN_NORMS keeps no [d_out, d_in] sums at all: it reduces each G_b tile to its sum of squares
enum : int { MEAN_NONE = 0, MEAN_REGS = 1, MEAN_TMEM = 2, MEAN_REGS_SIGN = 3, MEAN_NORMS = 4, MEAN_HYBRID_SIGN = 5 };
constexpr int TC_SIGN_COUNT_MAX = 32767;   // examples per block in MEAN_REGS_SIGN mode: 2 * count must fit 16 bits

// gridDim = (2 * pairs_m * tiles_n, 1, nsplit); blockIdx.x = 2 * (pair index in the tile order) + rank in pair.
// The fused parameter update of one epilogue warp's 32-row x (PANELS * 32)-column piece of the tile.  The piece
// is walked as float4 groups, a warp instruction covering 128 float4 in row-major order (global accesses of a
// warp are whole 16-byte groups of one or two rows), whereas the running sums live one ROW per lane: the sums
// therefore come either from the warp's staged panels in shared memory (the 128-byte-swizzled 32 x 32 panels the
// write-out also hands to TMA; chunk k of row r sits at chunk position k ^ (r & 7)) or, when the batch was
// split and this block added the last partial sum, from the outputs in global memory (read past L1).  Eight
// float4 per array and lane are in flight at a time (about 100 KiB per SM): the step is a latency-bound tail
// during which the block's tensor cores idle, so what counts is the number of memory round trips.
template <int OPT, int PANELS>
__device__ __forceinline__ void fused_update_piece(const FusedOpt& o, const TcParams& p, int row0, int col0, int lane,
                                                   const uint8_t* stat_panels, const uint8_t* mean_panels) {
  constexpr int C4 = PANELS * 8;             // float4 groups per row of the piece
  constexpr int ITERS = C4;                  // 32 rows x C4 groups / 32 lanes
  constexpr int BATCH = 8;
  static_assert(ITERS % BATCH == 0, "whole batches");
  const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
  for (int it0 = 0; it0 < ITERS; it0 += BATCH) {
    float4 th[BATCH], mm[BATCH], vv[BATCH], s1[BATCH], s2[BATCH];
#pragma unroll
    for (int i = 0; i < BATCH; ++i) {
      const int k = (it0 + i) * 32 + lane;
      const int r = k / C4, c4 = k - r * C4;
      const int row = row0 + r, col = col0 + 4 * c4;
      const bool in = row < p.d_out && col < p.d_in;           // d_in is a multiple of 8: a group is all in or all out
      const long long idx = (long long)row * p.d_in + col;
      th[i] = in ? *reinterpret_cast<const float4*>(o.theta + idx) : zero4;
      mm[i] = in ? *reinterpret_cast<const float4*>(o.m + idx) : zero4;
      vv[i] = (OPT == OPT_ADAM && in) ? *reinterpret_cast<const float4*>(o.v + idx) : zero4;
      float4 st, mn = zero4;
      if (stat_panels) {
        const int off = (c4 >> 3) * 4096 + r * 128 + (((c4 & 7) ^ (r & 7)) << 4);
        st = *reinterpret_cast<const float4*>(stat_panels + off);
        if (OPT == OPT_ADAM) mn = *reinterpret_cast<const float4*>(mean_panels + off);
      } else {
        st = in ? __ldcg(reinterpret_cast<const float4*>(p.out_stat + idx)) : zero4;
        if (OPT == OPT_ADAM) mn = in ? __ldcg(reinterpret_cast<const float4*>(p.out_mean + idx)) : zero4;
      }
      s1[i] = (OPT == OPT_ADAM) ? mn : st;
      s2[i] = st;
    }
#pragma unroll
    for (int i = 0; i < BATCH; ++i) {
      const int k = (it0 + i) * 32 + lane;
      const int r = k / C4, c4 = k - r * C4;
      const int row = row0 + r, col = col0 + 4 * c4;
      if (row < p.d_out && col < p.d_in) {
        const long long idx = (long long)row * p.d_in + col;
        if constexpr (OPT == OPT_ADAM) {
          adam_one_rt(o.variant, th[i].x, mm[i].x, vv[i].x, s1[i].x, s2[i].x, o.adam);
          adam_one_rt(o.variant, th[i].y, mm[i].y, vv[i].y, s1[i].y, s2[i].y, o.adam);
          adam_one_rt(o.variant, th[i].z, mm[i].z, vv[i].z, s1[i].z, s2[i].z, o.adam);
          adam_one_rt(o.variant, th[i].w, mm[i].w, vv[i].w, s1[i].w, s2[i].w, o.adam);
          *reinterpret_cast<float4*>(o.v + idx) = vv[i];
        } else {
          sign_one(th[i].x, mm[i].x, s1[i].x, o.sign);
          sign_one(th[i].y, mm[i].y, s1[i].y, o.sign);
          sign_one(th[i].z, mm[i].z, s1[i].z, o.sign);
          sign_one(th[i].w, mm[i].w, s1[i].w, o.sign);
        }
        *reinterpret_cast<float4*>(o.theta + idx) = th[i];
        *reinterpret_cast<float4*>(o.m + idx) = mm[i];
        if (o.theta_lp) {
          const __nv_bfloat162 lo = __floats2bfloat162_rn(th[i].x, th[i].y), hi = __floats2bfloat162_rn(th[i].z, th[i].w);
          uint2 pk;
          pk.x = *reinterpret_cast<const unsigned int*>(&lo);
          pk.y = *reinterpret_cast<const unsigned int*>(&hi);
          *reinterpret_cast<uint2*>(o.theta_lp + idx) = pk;
        }
      }
    }
  }
}

// RAGGED: packed batch with per-example token ranges (tmap_x / tmap_dy are then (d, rows, 1), tmap_x_tail /
// tmap_dy_tail (d, 16, B) over the zero-padded last partial token groups); otherwise the tail maps are unused.
// PHI: 0 identity, 1 square, 2 sign, 3 the clipping scale c_b * g with c_b = min(1, C / sqrt(N_b)), 4 the factors
// scale_y[b, o] * scale_x[b, i] * g[o, i] (powers of two: the staged per-token statistic, whose examples are chunks of rows).
// CHUNKED: an example's tokens are contracted TC_CHUNK_TOKENS at a time, each run into an accumulator of its own, and the
// runs are added in registers (round to nearest).  The tensor core truncates when it adds to an accumulator, which shrinks a sum of
// n instructions by about n * 2^-25: 6e-6 (G_b) and 1.2e-5 (G_b^2) at 6000 tokens, against 5e-7 and 1e-6 with runs of 512, what
// fp32 FMAs in order give too.  64 more registers per epilogue thread, hence the 256 x 128 tile.
// OPT: the parameter update applied by the block that completes a tile's sums (OPT_ADAM needs both running
// sums, OPT_SIGN the sign statistic alone); `o` is ignored when OPT == OPT_NONE.
template <int PHI, bool TF32, int NT, int MEAN, int BKT = tc_default_bk(TF32, NT), bool RAGGED = false, int OPT = OPT_NONE, bool F8 = false, bool CHUNKED = false, bool PERSIST = false, bool PARTS = false>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TC_THREADS, 1)
tc_stats_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_dy,
                const __grid_constant__ CUtensorMap tmap_mean, const __grid_constant__ CUtensorMap tmap_stat,
                const __grid_constant__ CUtensorMap tmap_sign, const __grid_constant__ CUtensorMap tmap_x_tail,
                const __grid_constant__ CUtensorMap tmap_dy_tail, TcParams p, FusedOpt o) {
  using namespace sm100;
  using Op = TcOperand<TF32, NT, BKT, F8>;
  static_assert(!F8 || (PHI == 0 && NT == 256 && !RAGGED), "8-bit operands: the plain contraction of the per-token statistic");
  constexpr bool HYBRID = (MEAN == MEAN_HYBRID_SIGN);
  constexpr bool TRIPLE = (MEAN == MEAN_REGS_SIGN) || HYBRID;
  static_assert((MEAN != MEAN_REGS && MEAN != MEAN_REGS_SIGN) || NT == 128 || (NT == 192 && MEAN == MEAN_REGS), "two running sums only fit the registers up to NT = 192");
  static_assert(NT != 192 || MEAN == MEAN_REGS || HYBRID, "the 256 x 192 tile exists for both running sums");
  static_assert(!HYBRID || (NT == 192 && !RAGGED && OPT == OPT_NONE), "the hybrid mean fills the tensor-memory columns two 192-column accumulators leave free");
  static_assert(!TRIPLE || PHI == 1, "the three-statistic mode is mean + square + sign");
  constexpr bool NORMS = (MEAN == MEAN_NORMS);
  static_assert(!NORMS || (PHI == 1 && NT == 256), "per-example norms: squares on the 256 x 256 tile");
  static_assert(MEAN != MEAN_TMEM || (NT == 256 && PHI != 0), "the tensor-memory mean sits beside one 256-column accumulator");
  static_assert(!RAGGED || (!TF32 && MEAN != MEAN_TMEM), "packed batches: 16-bit operands, several accumulators");
  static_assert((PHI != 3 && PHI != 4) || MEAN == MEAN_NONE, "the clipped sum and the scaled contraction are statistic-only passes");
  static_assert(!CHUNKED || (MEAN == MEAN_REGS && NT == 128 && !RAGGED && OPT == OPT_NONE), "runs of an example: the two-sum kernel on the 256 x 128 tile");
  static_assert(!PARTS || (PHI == 0 && !TF32 && !F8 && !RAGGED && !PERSIST && OPT == OPT_NONE), "the statistics of one-token examples are plain contractions");
  static_assert(!PERSIST || (!RAGGED && OPT == OPT_NONE && MEAN != MEAN_TMEM && PHI != 0), "several tiles per pair: fixed-length batches");
  constexpr int CHUNK_STAGES = CHUNKED ? TC_CHUNK_TOKENS / BKT : 1;
  constexpr int REGS_CONTROL = CHUNKED || TRIPLE ? 40 : Op::REGS_CONTROL, REGS_EPILOGUE = CHUNKED || TRIPLE ? 232 : Op::REGS_EPILOGUE;
  static_assert(128 * REGS_CONTROL + 256 * REGS_EPILOGUE <= TC_THREADS * TC_REGS_AT_LAUNCH, "setmaxnreg: the epilogue's increase must fit what the control warps give up");
  static_assert(OPT != OPT_ADAM || (MEAN == MEAN_REGS && PHI == 1), "the Adam family consumes sum_b G_b and sum_b G_b^2");
  static_assert(OPT != OPT_SIGN || (MEAN == MEAN_NONE && PHI == 2), "MicroSignSGD consumes sum_b sign(G_b)");
  constexpr int STAGES = Op::STAGES, BK = Op::BK;
  constexpr int BOX_BYTES = Op::BOX_BYTES, A_BYTES = Op::A_BYTES, STAGE_BYTES = Op::STAGE_BYTES;
  constexpr int ACC_BUFS = (MEAN == MEAN_TMEM) ? 1 : Op::ACC_BUFS;
  constexpr int MEAN_COL0 = 256;                    // first tensor-memory column of the MEAN_TMEM running sum
  constexpr int COLS = NT / 2;                      // accumulator columns per epilogue thread
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t bar_base = smem_base + STAGES * STAGE_BYTES;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };
  auto acc_full_bar = [&](int a) { return bar_base + 8u * (2 * STAGES + a); };
  auto acc_empty_bar = [&](int a) { return bar_base + 8u * (2 * STAGES + ACC_BUFS + a); };
  static_assert(8 * (2 * STAGES + 2 * ACC_BUFS) + 16 <= TC_BAR_BYTES, "barrier area too small");
  uint8_t* tail = smem_gen + STAGES * STAGE_BYTES + 8 * (2 * STAGES + 2 * ACC_BUFS);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(tail);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 8);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;      // the warp's number, uniform to the compiler too
  const uint32_t rank = cluster_ctarank();          // 0 = leader of the pair
  int b_begin = (int)(((long long)p.B * blockIdx.z) / p.nsplit);
  int b_end = (int)(((long long)p.B * (blockIdx.z + 1)) / p.nsplit);
  if constexpr (RAGGED) {
    if (p.by_tokens) {
      b_begin = ragged_slice_begin(p.seq_offsets, p.B, blockIdx.z, p.nsplit, lane);
      b_end = max(b_begin, ragged_slice_begin(p.seq_offsets, p.B, blockIdx.z + 1, p.nsplit, lane));
    }
  }
  int which = 0;                                    // PARTS: 0 the square, 1 the mean, 2 the sign
  if constexpr (PARTS) {
    int z = blockIdx.z;
    if (z >= p.part_slices[0]) { z -= p.part_slices[0]; which = 1; }
    if (which == 1 && z >= p.part_slices[1]) { z -= p.part_slices[1]; which = 2; }
    const int first = which == 0 ? p.part_chunks : which == 1 ? 0 : 5 * p.part_chunks;
    const long long count = which == 0 ? 4ll * p.part_chunks : p.part_chunks;
    b_begin = first + (int)(count * z / p.part_slices[which]);
    b_end = first + (int)(count * (z + 1) / p.part_slices[which]);
  }
  int nb = b_end - b_begin;
  const int n_units = PERSIST ? tc_units(p) : 1;      // PERSIST: this pair takes every (gridDim.x / 2)-th of them

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int a = 0; a < ACC_BUFS; ++a) { mbar_init(acc_full_bar(a), 1); mbar_init(acc_empty_bar(a), 16); }
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 2) { tmem_alloc_pair(smem_u32(const_cast<uint32_t*>(tmem_slot)), TC_TMEM_COLS); tmem_relinquish_pair(); }
  tc_fence_before();
  cluster_sync_all();          // barriers of both blocks initialised before any remote arrival
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // The next kernel of the stream may be launched from here on (it finds no room before blocks of this one leave).  With an unsplit
  // batch this kernel is itself a programmatic dependent of whatever precedes it: everything above overlapped that
  // kernel's end, and nothing below may start before it has completed.  (With a split batch its predecessor is the kernel
  // that zeroes the outputs, which lets this one start when everything older has completed, and only the write-out waits for it.)
  // A packed batch's predecessor is the kernel that fills the side buffer (and zeroes the outputs), to the same effect: the
  // producers wait for it before the first load from there.
  griddep_launch_dependents();
  if (!RAGGED && p.wait_at_start) griddep_wait();

  // Register budget: the epilogue warpgroups hold 128 floats of running sums plus a 32-register TMEM
  // read per thread; the producer / MMA warpgroup needs little.  Each setmaxnreg sits inside the
  // branch of the role it applies to.
  if (warp < 4) {
    setmaxnreg_dec<REGS_CONTROL>();
    const bool strict = wait_cycle_limit() < WAIT_CYCLE_LIMIT_STRICT;
    if (warp == 0 || warp == 2) {
      // ---------------------------------------------------------- TMA producers (both blocks)
      // Warp 0 loads this block's rows of dY^T (and, in the leader, posts the stage's byte count);
      // warp 2 loads this block's half of the X^T rows.  Both wait for the same "stage empty" phase.
      const bool is_a = (warp == 0);
      const CUtensorMap* tmap = is_a ? &tmap_dy : &tmap_x;
      const CUtensorMap* tmap_tail = is_a ? &tmap_dy_tail : &tmap_x_tail;
      const int n_boxes = is_a ? Op::A_BOXES : Op::B_BOXES;
      const int box_feats = is_a ? Op::BOX_FEATS : Op::B_BOX_FEATS;
      const int box_bytes = is_a ? BOX_BYTES : Op::B_BOX_BYTES;
      if (elect_one()) {
        prefetch_tensormap(tmap);
        if constexpr (RAGGED) prefetch_tensormap(tmap_tail);
      }
      int s = 0;
      uint32_t ph = 1;
      bool ok = true;
      bool side_ready = false;        // RAGGED: the side buffer is complete
      int unit = blockIdx.x >> 1;
      do {
        int tile_m, tile_n;
        if (PERSIST) {
          const TcUnit t = tc_unit(p, unit);
          b_begin = t.b_begin; b_end = t.b_end; nb = b_end - b_begin;
          tc_tile_of_pair(p, t.tile, rank, tile_m, tile_n);
        } else {
          tc_tile_of_pair(p, unit, rank, tile_m, tile_n);
        }
        const int c0 = is_a ? tile_m * TC_TILE_M : tile_n * NT + (int)rank * Op::B_FEATS;   // first feature of this warp's boxes
        for (int e = 0; e < nb && ok; ++e) {
          const SeqGeom g = seq_geom<RAGGED>(p, b_begin + e, BK);
          for (int kc = 0; kc < g.nk; ++kc) {
            if (!mbar_wait_warp(empty_bar(s), ph, abort_flag, p.dev_status, TC_WAIT_EMPTY, strict)) { ok = false; break; }
            if (elect_one()) {
              const bool tail = RAGGED && kc >= g.nk_main;       // the zero-padded last partial group, from the side buffer (boxes 16 tokens tall)
              if (is_a && rank == 0) mbar_arrive_expect_tx(full_bar(s), tail ? 2 * STAGE_BYTES / (BK / 16) : 2 * STAGE_BYTES);     // both blocks' bytes
              const uint32_t leader_full = map_to_cta(full_bar(s), 0);
              const uint32_t dst = smem_base + s * STAGE_BYTES + (is_a ? 0 : A_BYTES);
              if (tail && !side_ready) griddep_wait();
              const CUtensorMap* tm = tail ? tmap_tail : tmap;
              const int c1 = tail ? 0 : g.row0 + kc * BK;
              const int c2 = PARTS ? tc_part_chunk(p, b_begin + e, is_a) : RAGGED ? (tail ? b_begin + e : 0) : b_begin + e;
              for (int b = 0; b < n_boxes; ++b) tma_load_3d_pair(dst + b * box_bytes, tm, leader_full, c0 + b * box_feats, c1, c2);
            }
            __syncwarp();
            if (RAGGED && kc >= g.nk_main) side_ready = true;
            if (++s == STAGES) { s = 0; ph ^= 1u; }
          }
        }
      } while (PERSIST && ok && (unit += gridDim.x >> 1) < n_units);
    } else if (rank == 0 && warp == 1) {
      // ---------------------------------------------------------- MMA issuer (leader block)
      // Example e goes to accumulator e % ACC_BUFS.  A plain contraction (per_example == 0)
      // alternates the same way but resets each accumulator only once, and the epilogue adds them up.
      // operand format code 0 is IEEE half under kind::f16 and e4m3 under kind::f8f6f4
      const uint32_t idesc = (F8 || (!TF32 && p.half_operands)) ? make_idesc_half_mn_major(TC_PAIR_M, NT) : make_idesc_mn_major(TC_PAIR_M, NT, TF32);
      int s = 0;
      uint32_t ph = 0;
      int run = 0;                    // accumulators filled so far (CHUNKED: several per example)
      bool ok = true;
      int unit = blockIdx.x >> 1;
      do {
        if (PERSIST) {
          const TcUnit t = tc_unit(p, unit);
          b_begin = t.b_begin; b_end = t.b_end; nb = b_end - b_begin;
        }
        for (int e = 0; e < nb && ok; ++e) {
          const SeqGeom sg = seq_geom<RAGGED>(p, b_begin + e, BK);
          int buf = (PERSIST ? run : e) % ACC_BUFS;
          if (p.per_example && !CHUNKED) {
            if (!mbar_wait_warp(acc_empty_bar(buf), ((uint32_t)((PERSIST ? run : e) / ACC_BUFS) & 1u) ^ 1u, abort_flag, p.dev_status, TC_WAIT_ACC_EMPTY, strict)) { ok = false; break; }
            tc_fence_after();
            if (PERSIST) ++run;
          }
          const bool last_of_acc = p.per_example || e + ACC_BUFS >= nb;
          for (int kc = 0; kc < sg.nk; ++kc) {
            const int kin = CHUNKED ? kc % CHUNK_STAGES : kc;           // stage within its accumulator
            const bool acc_done = kc == sg.nk - 1 || (CHUNKED && kin == CHUNK_STAGES - 1);
            if (CHUNKED && kin == 0) {
              buf = run % ACC_BUFS;
              if (!mbar_wait_warp(acc_empty_bar(buf), ((uint32_t)(run / ACC_BUFS) & 1u) ^ 1u, abort_flag, p.dev_status, TC_WAIT_ACC_EMPTY, strict)) { ok = false; break; }
              tc_fence_after();
              ++run;
            }
            const uint32_t d_tmem = tmem_base + (uint32_t)(buf * NT);
            if (!mbar_wait_warp(full_bar(s), ph, abort_flag, p.dev_status, TC_WAIT_FULL, strict)) { ok = false; break; }
            tc_fence_after();
            if (elect_one()) {
              const uint32_t a_src = smem_base + s * STAGE_BYTES;
              const uint32_t b_src = a_src + A_BYTES;
              // tokens of this example in this stage: the rest of its whole 16-token groups, or the padded tail group
              const int t_left = (RAGGED && kc >= sg.nk_main) ? 16 : sg.main - kc * BK;
              uint32_t accumulate = (kin > 0 || (!p.per_example && e >= ACC_BUFS)) ? 1u : 0u;
#pragma unroll
              for (int k = 0; k < BK / Op::MMA_K; ++k) {
                // rows past T are zero-filled by TMA; whole MMA steps past T are skipped
                if (k * Op::MMA_K < t_left) {
                  const uint64_t ad = make_smem_desc(a_src + k * Op::K_STEP_BYTES, BOX_BYTES, Op::SBO_BYTES, Op::DESC_LAYOUT);
                  const uint64_t bd = make_smem_desc(b_src + k * Op::B_K_STEP_BYTES, Op::B_BOX_BYTES, Op::B_SBO_BYTES, Op::B_DESC_LAYOUT);
                  umma_ss_pair<TF32 ? 1 : (F8 ? 2 : 0)>(d_tmem, ad, bd, idesc, accumulate);
                  accumulate = 1;
                }
              }
              umma_commit_pair(empty_bar(s));                // stage reusable in both blocks once these MMAs retire
              if (last_of_acc && acc_done) umma_commit_pair(acc_full_bar(buf));   // accumulator complete, both blocks
            }
            __syncwarp();
            if (++s == STAGES) { s = 0; ph ^= 1u; }
          }
        }
      } while (PERSIST && ok && (unit += gridDim.x >> 1) < n_units);
    }
  } else {
    // ------------------------------------------------------------ epilogue (both blocks)
    setmaxnreg_inc<REGS_EPILOGUE>();
    const int q = warp & 3;                 // TMEM lane quadrant this warp may access
    const int h = (warp - 4) >> 2;          // column half of the tile
    constexpr bool KEEP_MEAN = MEAN == MEAN_REGS || MEAN == MEAN_REGS_SIGN || PHI == 0;     // running sum of G_b in registers
    constexpr int N_STAT = (PHI != 0 && !NORMS) ? COLS : 1;
    // HYBRID: of a thread's 96 columns the first 64 have their running sum of G_b in tensor memory (columns
    // HYB_COL0 + 64 h ..), the last 32 in registers
    constexpr int HYB_TMEM_COLS = 64, HYB_COL0 = 2 * 192;
    constexpr int N_MEAN = KEEP_MEAN ? COLS : (HYBRID ? COLS - HYB_TMEM_COLS : 1);
    float acc_stat[N_STAT], acc_mean[N_MEAN];
    // TRIPLE: sum_b (sign(G_b) + 1) of two neighbouring columns in one register, as unsigned 16-bit
    // halves (each at most 2 nb <= 65534, so a plain 32-bit add never carries from one half into the
    // other); sum_b sign = count - nb.  The third statistic costs 32 registers instead of 64.
    constexpr int N_CNT = TRIPLE ? COLS / 2 : 1;
    uint32_t acc_cnt[N_CNT];
#pragma unroll
    for (int j = 0; j < N_CNT; ++j) acc_cnt[j] = 0u;
#pragma unroll
    for (int j = 0; j < N_STAT; ++j) acc_stat[j] = 0.f;
#pragma unroll
    for (int j = 0; j < N_MEAN; ++j) acc_mean[j] = 0.f;
    bool ok = true;
    // What of the unit stays in registers during the loop over its examples was measured (8 x 256 x 1024 x 32104, both outputs, 186 us with
    // the tile found before the loop, 196 to 207 otherwise; three statistics 1 %, one statistic 2 % the other way round).
    constexpr bool TILE_FIRST = PHI == 4 || (!TRIPLE && !(PERSIST && MEAN == MEAN_NONE));
    int unit = blockIdx.x >> 1, a0 = 0;    // PERSIST: accumulators of the units before this one
    do {        // (the body keeps the function's indentation)
    int tile_m, tile_n;
    bool whole = true;
    if (PERSIST) {
      const TcUnit t = tc_unit(p, unit);
      b_begin = t.b_begin; b_end = t.b_end; nb = b_end - b_begin;
      if constexpr (TILE_FIRST) {
        whole = t.whole;
        tc_tile_of_pair(p, t.tile, rank, tile_m, tile_n);
      }
    } else if constexpr (TILE_FIRST) {
      tc_tile_of_pair(p, unit, rank, tile_m, tile_n);
    }
    // per-example mode: one accumulator per example, in order; plain mode: each accumulator once
    const int n_runs = CHUNKED ? (p.T + TC_CHUNK_TOKENS - 1) / TC_CHUNK_TOKENS : 1;      // accumulators per example
    const int n_acc = p.per_example ? nb * n_runs : min(nb, ACC_BUFS);
    constexpr int N_RUN = CHUNKED ? COLS : 1;
    float acc_run[N_RUN];           // CHUNKED: the sum of the example's runs so far
#pragma unroll
    for (int j = 0; j < N_RUN; ++j) acc_run[j] = 0.f;
    // PARTS: this unit's share of the marked examples, looked up while the first operands are on their way
    int odd_begin = 0, odd_end = 0;
    bool any_odd = false;
    if constexpr (PARTS) {
      if (which != 1) {
        const int z = (int)blockIdx.z - (which == 2 ? p.part_slices[0] + p.part_slices[1] : 0), groups = p.part_chunks * p.T / 16;
        odd_begin = (int)((long long)groups * z / p.part_slices[which]) * 16;
        odd_end = (int)((long long)groups * (z + 1) / p.part_slices[which]) * 16;
        uint32_t seen = 0u;
        for (int r = odd_begin + 16 * lane; r < odd_end; r += 512) {
          const uint4 v = *reinterpret_cast<const uint4*>(p.odd_rows + r);
          seen |= v.x | v.y | v.z | v.w;
        }
        any_odd = __any_sync(0xffffffffu, (seen & (which == 0 ? 0x01010101u : 0x02020202u)) != 0u);
      }
    }
    const uint32_t lane_base = tmem_base + ((uint32_t)(q * 32) << 16);
    float norm_kept = 0.f;          // NORMS
    for (int a = 0; a < n_acc; ++a) {
      const int buf = (a0 + a) % ACC_BUFS;
      const uint32_t acc_ph = (uint32_t)((a0 + a) / ACC_BUFS) & 1u;
      // PHI == 3: this example's clipping coefficient c_b = min(1, C / sqrt(N_b)); the load is issued before
      // the wait for the accumulator, which hides its latency.  N_b = 0 (a zero gradient) gives 1.
      uint64_t coef2 = 0;
      if constexpr (PHI == 3) {
        const float nb2 = __ldg(p.sq_norms + b_begin + a);
        const float nrm = sqrtf(nb2);
        const float c = nrm > p.clip_norm ? p.clip_norm / nrm : 1.f;
        coef2 = f32x2_pack(c, c);
      }
      // PHI == 4: this row's factor; the columns' are loaded beside each tensor-memory read
      if constexpr (PHI == 4) {
        const int row = tile_m * TC_TILE_M + q * 32 + lane;
        const float c = row < p.d_out ? __ldg(p.scale_y + (long long)(b_begin + a) * p.d_out + row) : 0.f;
        coef2 = f32x2_pack(c, c);
      }
      // every lane polls, but the warp acts on one answer: the tensor-memory loads below are warp-wide
      // instructions, so no lane may leave the loop alone when its own wait is the one that gives up
      if (!mbar_wait_warp(acc_full_bar(buf), acc_ph, abort_flag, p.dev_status, TC_WAIT_ACC_FULL)) { ok = false; break; }
      tc_fence_after();
      const uint32_t taddr = lane_base + (uint32_t)(buf * NT + h * COLS);
      if constexpr (MEAN == MEAN_TMEM) {
        // sum_b G_b lives in tensor-memory columns MEAN_COL0.. of the same lanes: read it with G_b,
        // add, write it back (the first example just writes G_b).
        const uint32_t maddr = lane_base + (uint32_t)(MEAN_COL0 + h * COLS);
#pragma unroll
        for (int c = 0; c < COLS / 16; ++c) {
          uint32_t r[16], m[16];
          if (a == 0) tmem_ld_32x32b_x16_wait(taddr + c * 16, r);
          else tmem_ld_32x32b_x16_pair_wait(taddr + c * 16, r, maddr + c * 16, m);
          if (c == COLS / 16 - 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(map_to_cta(acc_empty_bar(buf), 0));   // G_b read: the issuer may start the next example
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float g = __uint_as_float(r[j]);
            acc_stat[c * 16 + j] += (PHI == 2) ? sign_half(g) : phi_apply<PHI>(g);
            if (a != 0) r[j] = __float_as_uint(g + __uint_as_float(m[j]));
          }
          tmem_st_32x32b_x16(maddr + c * 16, r);
        }
        tmem_st_wait();
      } else if constexpr (HYBRID) {
        const uint32_t maddr = lane_base + (uint32_t)(HYB_COL0 + h * HYB_TMEM_COLS);
#pragma unroll
        for (int c = 0; c < COLS / 16; ++c) {
          constexpr int LAST = COLS / 16 - 1;
          const bool in_tmem = c * 16 < HYB_TMEM_COLS;           // compile-time after unrolling
          uint32_t r[16], m[16];
          if (in_tmem && a != 0) tmem_ld_32x32b_x16_pair_wait(taddr + c * 16, r, maddr + c * 16, m);
          else tmem_ld_32x32b_x16_wait(taddr + c * 16, r);
          if (c == LAST) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(map_to_cta(acc_empty_bar(buf), 0));   // G_b read: the issuer may start its next example
          }
#pragma unroll
          for (int j = 0; j < 16; j += 2) {
            const uint64_t g2 = f32x2_pack(__uint_as_float(r[j]), __uint_as_float(r[j + 1]));
            const uint64_t s2 = f32x2_fma(g2, g2, f32x2_pack(acc_stat[c * 16 + j], acc_stat[c * 16 + j + 1]));
            f32x2_unpack(s2, acc_stat[c * 16 + j], acc_stat[c * 16 + j + 1]);
            acc_cnt[(c * 16 + j) >> 1] += sign_plus_one_packed(g2);
            if (in_tmem) {
              if (a != 0) {
                const uint64_t m2 = f32x2_add(f32x2_pack(__uint_as_float(m[j]), __uint_as_float(m[j + 1])), g2);
                float lo, hi;
                f32x2_unpack(m2, lo, hi);
                r[j] = __float_as_uint(lo);
                r[j + 1] = __float_as_uint(hi);
              }
            } else {
              const int k = c * 16 + j - HYB_TMEM_COLS;
              const uint64_t m2 = f32x2_add(f32x2_pack(acc_mean[k], acc_mean[k + 1]), g2);
              f32x2_unpack(m2, acc_mean[k], acc_mean[k + 1]);
            }
          }
          if (in_tmem) tmem_st_32x32b_x16(maddr + c * 16, r);      // the first example just writes G_b
        }
        tmem_st_wait();
      } else if constexpr (NORMS) {
        // this thread's share of ||G_b||_F^2 (its row, its 128 columns; rows and columns outside the
        // matrix are exact zeros), then the warp's, then one atomic per warp and example
        // All reads at once and the accumulator released behind them, before the arithmetic.
        constexpr int READS = COLS / 32;
        uint32_t r[READS][32];
#pragma unroll
        for (int c = 0; c < READS; ++c) tmem_ld_issue(taddr + c * 32, r[c]);
#pragma unroll
        for (int c = 0; c < READS; ++c) tmem_ld_wait_for(r[c]);
        tc_fence_before();
        __syncwarp();
        mbar_arrive_cluster_if(lane == 0, map_to_cta(acc_empty_bar(buf), 0));
        uint64_t part[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) part[i] = f32x2_pack(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < READS; ++c)
#pragma unroll
          for (int j = 0; j < 32; j += 2) {
            const uint64_t g2 = f32x2_pack(__uint_as_float(r[c][j]), __uint_as_float(r[c][j + 1]));
            part[(j / 2) % 4] = f32x2_fma(g2, g2, part[(j / 2) % 4]);
          }
        float s0, s1;
        f32x2_unpack(f32x2_add(f32x2_add(part[0], part[1]), f32x2_add(part[2], part[3])), s0, s1);
        float s = s0 + s1;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        // lane l keeps the sum of the unit's example 32 k + l: one coalesced add per 32 examples.  An add per example and warp met the other tiles' at one
        // address of L2, 2048 of them per example on 128 tiles: 128 x 64 x 2048 x 4096 254 -> 109 us, 50 x 120 x 1400 x 2000 80 -> 40, 64 x 128 x 512 x 2048 20 -> 16.
        if (lane == (a & 31)) norm_kept = s;
        if ((a & 31) == 31 || a == n_acc - 1) {
          const int first = a & ~31;
          if (first + lane <= a) atomicAdd(p.out_norms + b_begin + first + lane, norm_kept);
        }
      } else {
        // CH columns per tensor-memory read: 32, or 16 where the running sums leave few registers (NT = 192; the three
        // statistics on the 256 x 128 tile, whose 160 registers of sums leave room for two reads of 16 in flight, not 32)
        constexpr int CH = (NT == 192 || TRIPLE || CHUNKED) ? 16 : 32;
        constexpr int NCH = COLS / CH;                // reads per example
        // phi and the running sums for one read of CH columns (chunk c of this thread's COLS columns)
        float4 col_scale[PHI == 4 ? CH / 4 : 1];
        auto fold = [&](const uint32_t (&r)[CH], int c) {
          if constexpr (PHI == 2) {
            // the running sum holds sum_b (sign(G_b) + 1) / 2 until the write-out turns it into sum_b sign(G_b)
#pragma unroll
            for (int j = 0; j < CH; j += 2) {
              const uint64_t g2 = f32x2_pack(__uint_as_float(r[j]), __uint_as_float(r[j + 1]));
              if (KEEP_MEAN) {
                const uint64_t m2 = f32x2_add(f32x2_pack(acc_mean[c * CH + j], acc_mean[c * CH + j + 1]), g2);
                f32x2_unpack(m2, acc_mean[c * CH + j], acc_mean[c * CH + j + 1]);
              }
              const uint64_t s2 = f32x2_add(f32x2_pack(acc_stat[c * CH + j], acc_stat[c * CH + j + 1]), sign_half2(g2));
              f32x2_unpack(s2, acc_stat[c * CH + j], acc_stat[c * CH + j + 1]);
            }
          } else {
            // two columns per instruction: packed fp32 add for sum_b G_b, packed fma for sum_b G_b^2
#pragma unroll
            for (int j = 0; j < CH; j += 2) {
              const uint64_t g2 = f32x2_pack(__uint_as_float(r[j]), __uint_as_float(r[j + 1]));
              if (KEEP_MEAN) {
                const uint64_t m2 = f32x2_add(f32x2_pack(acc_mean[c * CH + j], acc_mean[c * CH + j + 1]), g2);
                f32x2_unpack(m2, acc_mean[c * CH + j], acc_mean[c * CH + j + 1]);
              }
              if constexpr (PHI == 4) {
                const float4 f = col_scale[j >> 2];
                const uint64_t f2 = (j & 2) ? f32x2_pack(f.z, f.w) : f32x2_pack(f.x, f.y);
                const uint64_t s2 = f32x2_fma(f32x2_mul(g2, f2), coef2, f32x2_pack(acc_stat[c * CH + j], acc_stat[c * CH + j + 1]));
                f32x2_unpack(s2, acc_stat[c * CH + j], acc_stat[c * CH + j + 1]);
              }
              if (PHI == 1 || PHI == 3) {
                const uint64_t s2 = f32x2_fma(g2, PHI == 1 ? g2 : coef2, f32x2_pack(acc_stat[c * CH + j], acc_stat[c * CH + j + 1]));
                f32x2_unpack(s2, acc_stat[c * CH + j], acc_stat[c * CH + j + 1]);
              }
              if (TRIPLE) {
                acc_cnt[(c * CH + j) >> 1] += sign_plus_one_packed(g2);
              }
            }
          }
        };
        auto release_acc = [&]() {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(map_to_cta(acc_empty_bar(buf), 0));   // buffer(s) free for the issuer's next example(s)
        };
        // Where the registers allow two reads in flight (running sums of at most 128 floats beside two 32-column
        // reads; the three statistics' 160 registers beside two 16-column reads), the reads are software-pipelined:
        // read k+1 is issued before the arithmetic on read k, so only the first read of a unit exposes the
        // tensor-memory latency.  That latency, paid twice per example, was a third of the two-sum epilogue's time
        // per example of 32 tokens (the three-statistic epilogue, bound by its instruction
        // count, gained 2-3 %).
        constexpr bool PIPELINED = (CH == 32 && PHI != 3 && PHI != 4) || (TRIPLE && NT == 128);
        if constexpr (PIPELINED) {
          uint32_t ra[CH], rb[CH];
          tmem_ld_issue(taddr, ra);
#pragma unroll
          for (int k = 0; k < NCH; ++k) {
            if (k & 1) tmem_ld_wait_for(rb); else tmem_ld_wait_for(ra);
            if (k + 1 < NCH) {
              const uint32_t next = taddr + (uint32_t)((k + 1) * CH);
              if (k & 1) tmem_ld_issue(next, ra); else tmem_ld_issue(next, rb);
            } else {
              release_acc();
            }
            if (k & 1) fold(rb, k); else fold(ra, k);
          }
        } else {
#pragma unroll
          for (int c = 0; c < NCH; ++c) {
            uint32_t r[CH];
            if constexpr (PHI == 4) {
              const int col = tile_n * NT + h * COLS + c * CH;
#pragma unroll
              for (int j = 0; j < CH / 4; ++j)
                col_scale[j] = col + 4 * j < p.d_in ? __ldg(reinterpret_cast<const float4*>(p.scale_x + (long long)(b_begin + a) * p.d_in + col) + j)
                                                    : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            if constexpr (CH == 32) tmem_ld_32x32b_x32_wait(taddr + c * CH, r);
            else tmem_ld_32x32b_x16_wait(taddr + c * CH, r);
            if (c == NCH - 1) release_acc();
            if constexpr (CHUNKED) {
              const bool last_run = a % n_runs == n_runs - 1;
#pragma unroll
              for (int j = 0; j < CH; j += 2) {
                float lo, hi;
                f32x2_unpack(f32x2_add(f32x2_pack(acc_run[c * CH + j], acc_run[c * CH + j + 1]), f32x2_pack(__uint_as_float(r[j]), __uint_as_float(r[j + 1]))), lo, hi);
                r[j] = __float_as_uint(lo); r[j + 1] = __float_as_uint(hi);
                acc_run[c * CH + j] = last_run ? 0.f : lo;
                acc_run[c * CH + j + 1] = last_run ? 0.f : hi;
              }
              if (last_run) fold(r, c);
            } else {
              fold(r, c);
            }
          }
        }
      }
    }
    // Final write-out.  By now every MMA of this block has completed (the last accumulator was
    // committed after them), so the operand ring is free: each warp stages its 32-row x COLS-column
    // piece of an output there, 32 columns (one 128-byte-swizzled 4 KiB panel) at a time, and one lane
    // hands the panels to TMA, which stores them (or, with a split batch, adds them) and drops
    // whatever lies outside the matrix.  The tensor-memory loads are warp-wide instructions: the
    // condition around them is made uniform over the warp.
    ok = __all_sync(0xffffffffu, ok);
    if constexpr (!TILE_FIRST) {
      const TcUnit t = PERSIST ? tc_unit(p, unit) : TcUnit{unit, 0, 0, true};
      whole = t.whole;
      tc_tile_of_pair(p, t.tile, rank, tile_m, tile_n);
    }
    if constexpr (PARTS) {
      // The marked examples, in fp32 as G_b: a row per lane, the columns' entries of X handed round two at a time.  Bound by the exchanges (square)
      // and by the instructions of a comparison per entry (sign).  Every example marked for both and every piece holding a zero product,
      // three statistics: 1024 x 1024^2 1075 us (ordinary examples 29; 288 with the kernel that forms every G_b for all), 512 x 4096^2 3364 (159;
      // 2058).  Both rows have to span more than 2^33 for that (or hold an infinity or NaN).
      if (ok && any_odd) {
        const int row = tile_m * TC_TILE_M + q * 32 + lane, col0 = tile_n * NT + h * COLS;
        // +-1 or 0 as bf16
        auto sgn = [](uint32_t bits) { return (bits & 0x7fffu) != 0u && (bits & 0x7fffu) <= 0x7f80u ? 0x3f80u | (bits & 0x8000u) : 0u; };
        auto lowest = [](uint32_t bits) { return (bits & 0x7fffu) != 0u ? (int)(bits & 0x7fffu) : 0x7fff; };
        for (int r0 = odd_begin; r0 < odd_end; r0 += 32) {
          unsigned int todo = __ballot_sync(0xffffffffu, r0 + lane < odd_end && (p.odd_rows[r0 + lane] & (which == 0 ? 1 : 2)) != 0);
          for (; todo != 0u; todo &= todo - 1u) {
            const long long b = r0 + __ffs((int)todo) - 1;
            const uint32_t yb = row < p.d_out ? p.rows_dy[b * p.d_out + row] : 0u;
            const float y = __uint_as_float(yb << 16);
            const uint16_t* const xb = p.rows_x + b * p.d_in;
            uint32_t mine[COLS / 64];
            int low = 0x7fff;
#pragma unroll
            for (int c = 0; c < COLS / 64; ++c) {
              const int col = col0 + 64 * c + 2 * lane;
              const uint32_t x0 = col < p.d_in ? xb[col] : 0u, x1 = col + 1 < p.d_in ? xb[col + 1] : 0u;
              mine[c] = x0 | x1 << 16;
              low = min(low, min(lowest(x0), lowest(x1)));
            }
            if (which == 0) {
#pragma unroll
              for (int c = 0; c < COLS / 64; ++c) {
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                  const uint32_t x2 = __shfl_sync(0xffffffffu, mine[c], j);
                  const int k = 64 * c + 2 * j;
                  const uint64_t g2 = f32x2_mul(f32x2_pack(__uint_as_float(x2 << 16), __uint_as_float(x2 & 0xffff0000u)), f32x2_pack(y, y));
                  f32x2_unpack(f32x2_fma(g2, g2, f32x2_pack(acc_mean[k], acc_mean[k + 1])), acc_mean[k], acc_mean[k + 1]);
                }
              }
            } else {
              // counted by the signs of its factors: taken back where the product is zero, if one of this piece may be
              const int ex = __reduce_min_sync(0xffffffffu, low) >> 7, ey = __reduce_min_sync(0xffffffffu, lowest(yb)) >> 7;
              if ((ex > 0 ? ex : -6) + (ey > 0 ? ey : -6) >= 254 - 149) continue;
              const float sy = __uint_as_float(sgn(yb) << 16);
#pragma unroll
              for (int c = 0; c < COLS / 64; ++c) {
                const uint32_t signs = sgn(mine[c] & 0xffffu) | sgn(mine[c] >> 16) << 16;
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                  const uint32_t x2 = __shfl_sync(0xffffffffu, mine[c], j), s2 = __shfl_sync(0xffffffffu, signs, j);
                  const int k = 64 * c + 2 * j;
                  if (__uint_as_float(x2 << 16) * y == 0.f) acc_mean[k] -= __uint_as_float(s2 << 16) * sy;
                  if (__uint_as_float(x2 & 0xffff0000u) * y == 0.f) acc_mean[k + 1] -= __uint_as_float(s2 & 0xffff0000u) * sy;
                }
              }
            }
          }
        }
      }
    }
    if constexpr (PHI == 2) {
      // sum_b (sign(G_b) + 1) / 2  ->  sum_b sign(G_b)
      const float nbf = (float)nb;
#pragma unroll
      for (int j = 0; j < N_STAT; ++j) acc_stat[j] = fmaf(2.f, acc_stat[j], -nbf);
    }
    if constexpr (PERSIST && NORMS) {
      a0 += n_acc;                  // (nothing to write out)
    } else if constexpr (PERSIST) {
      // Several tiles per pair: straight from the registers, since the operand ring already fills for the next tile.  Lanes
      // exchange their rows' values first, so that four of them store 128 bytes side by side (stores of 32 bytes to 32 rows: 8 x 256
      // x 1024 x 32104, both outputs, 201 us against 179).  Slices of a tile add 128 bytes of a row per instruction (16-byte adds, 32
      // bytes to a lane, were 2 % of a call of 235 us slower).
      const int row0 = tile_m * TC_TILE_M + q * 32, col0 = tile_n * NT + h * COLS;
      if (!whole) griddep_wait();                                   // the kernel that zeroes this tile
      auto put = [&](float* out, int c, float (&v)[32]) {           // 32 columns from the c-th on
        if (whole) {
          const int row = row0 + (lane & ~3), col = col0 + c + 8 * (lane & 3);
          quad_transpose(v, lane);
          if (ok && col < p.d_in) {                                 // d_in is a multiple of 8: a group is all in or all out
            float* const dst = out + (long long)row * p.d_in + col;
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (row + j < p.d_out) st_global_v8(dst + (long long)j * p.d_in, &v[8 * j]);
          }
        } else {
          const int col = col0 + c + lane;
          warp_transpose(v, lane);
          if (ok && col < p.d_in) {
            float* const dst = out + (long long)row0 * p.d_in + col;
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (row0 + j < p.d_out) atomicAdd(dst + (long long)j * p.d_in, v[j]);
          }
        }
      };
      if (p.out_stat) {
#pragma unroll
        for (int c = 0; c < COLS; c += 32) {
          float v[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = acc_stat[c + j];
          put(p.out_stat, c, v);
        }
      }
      if (p.out_mean && (KEEP_MEAN || HYBRID)) {
#pragma unroll
        for (int c = 0; c < COLS; c += 32) {
          float v[32];
          if (HYBRID && c < HYB_TMEM_COLS) {
            uint32_t m[32];
            tmem_ld_32x32b_x32_wait(lane_base + (uint32_t)(HYB_COL0 + h * HYB_TMEM_COLS) + c, m);
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(m[j]);
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = acc_mean[HYBRID ? (c - HYB_TMEM_COLS + j) & 31 : (KEEP_MEAN ? c + j : 0)];
          }
          put(p.out_mean, c, v);
        }
      }
      if constexpr (TRIPLE) {
        const float nbf = (float)nb;
#pragma unroll
        for (int c = 0; c < COLS; c += 32) {
          float v[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = (float)((acc_cnt[(c + j) >> 1] >> (16 * (j & 1))) & 0xFFFFu) - nbf;
          if (p.out_sign) put(p.out_sign, c, v);
        }
#pragma unroll
        for (int j = 0; j < N_CNT; ++j) acc_cnt[j] = 0u;
      }
#pragma unroll
      for (int j = 0; j < N_STAT; ++j) acc_stat[j] = 0.f;
#pragma unroll
      for (int j = 0; j < N_MEAN; ++j) acc_mean[j] = 0.f;
      a0 += n_acc;
    } else {
    constexpr int PANELS = COLS / 32;
    // each epilogue warp stages in its own eighth of the operand ring: 6 panels of 4 KiB (7 at NT = 192)
    constexpr int WARP_PANELS = (STAGES * STAGE_BYTES / 8) / 4096;
    static_assert(WARP_PANELS >= PANELS, "an epilogue warp stages one output at a time");
    static_assert(OPT != OPT_ADAM || WARP_PANELS >= 2 * PANELS, "the fused Adam update reads both staged sums");
    const uint32_t stage_base = smem_base + (uint32_t)(warp - 4) * (uint32_t)(WARP_PANELS * 4096);
    const int row0 = tile_m * TC_TILE_M + q * 32;
    const int col0 = tile_n * NT + h * COLS;
    // fused update on the unsplit schedule: the sums are staged even when the caller does not want them written
    const bool stage_for_update = OPT != OPT_NONE && p.nsplit == 1;
    if (ok && n_acc > 0) {
      auto put_panel = [&](uint32_t panel_addr, const float* v) {      // v: this lane's 32 consecutive columns
        uint8_t* dst = smem_gen + (panel_addr - smem_base) + lane * 128;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          *reinterpret_cast<float4*>(dst + ((k ^ (lane & 7)) << 4)) = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
      };
      auto send = [&](const CUtensorMap* tm, float* out, uint32_t first_panel) {
        if (p.scalar_out) {
          if (p.nsplit > 1 && !p.accumulate) griddep_wait();
          __syncwarp();
          for (int c = 0; c < PANELS; ++c) {
            const int col = col0 + c * 32 + lane;
            const uint8_t* src = smem_gen + (first_panel + c * 4096 - smem_base) + (lane & 3) * 4;
            for (int r = 0; r < 32 && row0 + r < p.d_out; ++r) {
              const float v = *reinterpret_cast<const float*>(src + r * 128 + (((lane >> 2) ^ (r & 7)) << 4));
              if (col < p.d_in) {
                float* const at = out + (size_t)(row0 + r) * p.d_in + col;
                if (p.nsplit == 1 && !p.accumulate) *at = v;
                else atomicAdd(at, v);
              }
            }
          }
          __syncwarp();           // the panels may be refilled for the next output
          return;
        }
        fence_async_smem();
        __syncwarp();
        if (row0 < p.d_out && elect_one()) {
          if (p.nsplit > 1 && !p.accumulate) griddep_wait();       // the kernel that zeroes the outputs may still be running
          for (int c = 0; c < PANELS; ++c) {
            if (col0 + c * 32 < p.d_in) {
              if (p.nsplit == 1 && !p.accumulate) tma_store_2d<false>(tm, first_panel + c * 4096, col0 + c * 32, row0);
              else tma_store_2d<true>(tm, first_panel + c * 4096, col0 + c * 32, row0);
            }
          }
          bulk_commit_group();
        }
      };
      if constexpr (PARTS) {
#pragma unroll
        for (int c = 0; c < PANELS; ++c) put_panel(stage_base + c * 4096, &acc_mean[c * 32]);
        send(which == 0 ? &tmap_stat : which == 1 ? &tmap_mean : &tmap_sign, which == 0 ? p.out_stat : which == 1 ? p.out_mean : p.out_sign, stage_base);
      }
      // sum_b phi(G_b), or the plain contraction when PHI == 0
      if (!PARTS && (p.out_stat || stage_for_update)) {
#pragma unroll
        for (int c = 0; c < PANELS; ++c) put_panel(stage_base + c * 4096, (PHI != 0) ? &acc_stat[c * 32] : &acc_mean[c * 32]);
        if (p.out_stat) send(&tmap_stat, p.out_stat, stage_base);
      }
      // sum_b G_b
      if (!PARTS && (p.out_mean || (stage_for_update && OPT == OPT_ADAM)) && (KEEP_MEAN || MEAN == MEAN_TMEM || HYBRID)) {
        uint32_t first = stage_base + PANELS * 4096;          // MEAN_REGS / PHI == 0: second half of the warp's 16 KiB
        if constexpr (HYBRID) {
          // two panels from tensor memory, the third from registers; staged behind the statistic's three panels
          const uint32_t maddr = lane_base + (uint32_t)(HYB_COL0 + h * HYB_TMEM_COLS);
#pragma unroll
          for (int c = 0; c < HYB_TMEM_COLS / 32; ++c) {
            uint32_t m[32];
            tmem_ld_32x32b_x32_wait(maddr + c * 32, m);
            put_panel(first + c * 4096, reinterpret_cast<const float*>(m));
          }
          put_panel(first + (HYB_TMEM_COLS / 32) * 4096, &acc_mean[0]);
        } else if constexpr (MEAN == MEAN_TMEM) {
          // the panels are needed again: wait until TMA has read the first output out of them
          if (elect_one()) bulk_wait_read_all();
          __syncwarp();
          first = stage_base;
          const uint32_t maddr = lane_base + (uint32_t)(MEAN_COL0 + h * COLS);
#pragma unroll
          for (int c = 0; c < PANELS; ++c) {
            uint32_t m[32];
            tmem_ld_32x32b_x32_wait(maddr + c * 32, m);
            put_panel(first + c * 4096, reinterpret_cast<const float*>(m));
          }
        } else if constexpr (KEEP_MEAN) {
          if constexpr (PANELS * 2 > WARP_PANELS) {           // PHI == 0 at NT = 256: one output only ever
            if (elect_one()) bulk_wait_read_all();
            __syncwarp();
            first = stage_base;
          }
#pragma unroll
          for (int c = 0; c < PANELS; ++c) put_panel(first + c * 4096, &acc_mean[c * 32]);
        }
        if (p.out_mean) send(&tmap_mean, p.out_mean, first);
      }
      if constexpr (TRIPLE) {
        // sum_b sign(G_b): the warp's staging area is in use, so wait until TMA has read it
        if (p.out_sign) {
          if (elect_one()) bulk_wait_read_all();
          __syncwarp();
          const float nbf = (float)nb;
#pragma unroll
          for (int c = 0; c < PANELS; ++c) {
            float v[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = (float)((acc_cnt[(c * 32 + j) >> 1] >> (16 * (j & 1))) & 0xFFFFu) - nbf;
            put_panel(stage_base + c * 4096, v);
          }
          send(&tmap_sign, p.out_sign, stage_base);
        }
      }
      if (elect_one()) bulk_wait_read_all();       // shared memory must outlive TMA's reads
    }
    __syncwarp();
    if constexpr (OPT != OPT_NONE) {
      // The parameter update, by the block that holds (unsplit batch) or has just completed (split batch)
      // the tile's sums over the whole batch.  Split batch: every block adds its partial tile to the
      // outputs, waits until those adds have been performed, and takes a ticket from the tile's counter;
      // the block that draws the last ticket reads the finished sums back and applies the update.  A block
      // that gave up on a wait marks the counter so that nobody updates the parameters from incomplete sums.
      bool apply = ok && n_acc > 0;
      if (p.nsplit > 1) {
        if (elect_one()) { bulk_wait_all(); __threadfence(); }
        __syncwarp();
        named_bar_sync(1, 256);                   // the eight epilogue warps; executed by all of them whatever `ok` says
        volatile int* last_flag = reinterpret_cast<volatile int*>(tail + 12);
        if (warp == 4 && lane == 0) {
          griddep_wait();                         // the counters are zeroed by the kernel that zeroes the outputs
          const unsigned int inc = 1u + (*abort_flag ? 0x10000u : 0u);
          const unsigned int now = atomicAdd(o.tile_counters + blockIdx.x, inc) + inc;
          int last = 0;
          if ((now & 0xffffu) == (unsigned int)p.nsplit) {
            last = (now >> 16) ? 0 : 1;
            atomicExch(o.tile_counters + blockIdx.x, 0u);
          }
          *last_flag = last;
        }
        named_bar_sync(1, 256);
        apply = (*last_flag != 0);
        if (apply) __threadfence();
      }
      if (apply) {
        const bool from_smem = p.nsplit == 1;
        const uint8_t* stat_panels = from_smem ? smem_gen + (stage_base - smem_base) : nullptr;
        fused_update_piece<OPT, PANELS>(o, p, row0, col0, lane, stat_panels, stat_panels ? stat_panels + PANELS * 4096 : nullptr);
      }
      __syncwarp();
    }
    }
    } while (PERSIST && ok && (unit += gridDim.x >> 1) < n_units);
  }

  // ---------------------------------------------------------------- teardown
  // Sequences of whole 16-token groups need nothing of the side buffer, and with an unsplit batch nothing above has waited for the kernel
  // that fills it.  This one may not complete before it does: the next call may fill the same workspace.
  if constexpr (RAGGED) griddep_wait();
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // A wait gave up.  Loads this block issued may still be landing in its shared memory: give them
    // time (bounded) before the block exits and its shared memory is handed to another block.
    const long long t0 = clock64();
    while (clock64() - t0 < (1ll << 22)) __nanosleep(1000);
  }
  // Neither block may leave while its peer can still arrive on its barriers or read its shared memory.
  __syncwarp();
  cluster_sync_all();
  if (warp == 2) { tc_fence_after(); tmem_dealloc_pair(tmem_base, TC_TMEM_COLS); }
}

}  // namespace pe
