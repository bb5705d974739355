// Tensor-core kernel for the statistics of short sequences (T <= 32): sum_b G_b, sum_b G_b^2 and sum_b sign(G_b), G_b = dY_b^T X_b, those
// that are wanted.  Work unit as in tc_stats_kernel: a CTA pair, a 256 x 128 tile of [d_out, d_in], a slice of the batch; a pair per two SMs
// walks over the tiles.  An example is one or two MMAs, so neither the tensor pipe nor memory is the bound but the epilogue: its fp32
// instructions on 32 768 entries of G_b per SM and unit of two examples (packed: 512 cycles for two sums, 768 for the sign, 1472 for all three;
// half- and full-rate instructions share the issue, so integer ones are not free beside them), and the barriers between the roles.  Hence:
//  - Two examples to a stage, an accumulator unit and a hand-off, folded side by side.
//  - One barrier pair per stage.  go: the operands' bytes and the 16 arrivals of the epilogue warps that free the accumulator unit (on the barrier of
//    the stage that will be contracted into it), so that the issuer waits once per unit; done: one commit, which the epilogue and the producers
//    wait for.  Separate barriers for stages and accumulators cost the issuer 680 of 901 cycles per unit.
//  - The epilogue asks for the next unit's barrier a read ahead, without blocking, and issues that unit's first reads, by a predicate, before its
//    last arithmetic; it arrives by a predicated instruction (a branch around it costs about 80 cycles).  Releasing and looking ahead took 300 cycles a unit.
//  - Results leave through a panel of shared memory of their own (TMA stores, or adds for a slice of the batch), so that the operand ring is
//    filled for the next tile meanwhile.  Adds from registers, lanes transposed, took 7 us per tile and two sums.
// 1024 x 32 tokens x 1024^2: both outputs 135 -> 110 us (clock cycles a unit: 901 -> 750), sign 166 -> 155, three statistics
// 275 -> 244; 128 x 32 x 4096^2: 219 -> 196, 304 -> 270, 472 -> 429; 512 x 2 x 1024^2: 72 -> 58, 92 -> 81, 142 -> 127.  The
// square alone gains where tiles or tokens are few (512 x 8 x 4096 x 2048 407 -> 368, 64 x 32 x 4096^2 105 -> 99, 40 drawn layers 14 %, geometric mean); large layers of 32 tokens are
// equal or up to 4 % slower than on the 256 x 256 tile, at a quarter of its rounding error (800 x 32 x 1024 x 4096 279 -> 287 us, 4.2e-7 -> 7.9e-8).
// (before: stages and accumulators of tc_stats_kernel with two examples each).  What is left above the arithmetic is the two units' round trip
// from release to the next unit's reads, about 780 cycles at T = 32.  Measured and dropped: signs counted from the sign bits by byte
// permutes and 16-bit adds with zeros looked for by three-way minima (three statistics 244 -> 228 us where G_b holds no zeros, but every zero
// is a second pass over the unit: 2-token sequences 127 -> 197); a lag of half a unit between a scheduler's two epilogue warps (no change).
#pragma once
#include "pe_tc.cuh"

namespace pe {

constexpr int SHORT_NT = 128;                       // d_in columns per pair tile
constexpr int SHORT_T = 32;                         // tokens of a stage, and the longest sequence
constexpr int SHORT_G = 2;                          // examples per stage and unit of work
constexpr int SHORT_A_BOX = SHORT_G * SHORT_T * 128;              // 64 rows of dY^T: 8 KiB, two of them per block
constexpr int SHORT_B_BOX = SHORT_G * SHORT_T * 128;              // 64 columns of X: 8 KiB
constexpr int SHORT_STAGE = 2 * SHORT_A_BOX + SHORT_B_BOX;        // 24 KiB
constexpr int SHORT_STAGES = 8;
constexpr int SHORT_RUN_MIN = 16, SHORT_RUN_MAX = 256;      // examples summed by themselves where the square alone is wanted: powers of two
constexpr int SHORT_UNITS = TC_TMEM_COLS / (SHORT_G * SHORT_NT);  // accumulator units in tensor memory: 2
constexpr int SHORT_PANEL = 4096;                   // per epilogue warp: 32 x 32 results on their way out
constexpr int SHORT_RING = SHORT_STAGES * SHORT_STAGE + 8 * SHORT_PANEL;
constexpr int SHORT_SMEM_BYTES = SHORT_RING + TC_BAR_BYTES + 1024;
static_assert(SHORT_SMEM_BYTES <= 227 * 1024, "shared memory of a block");
constexpr int SHORT_REGS_CONTROL = 40, SHORT_REGS_EPILOGUE = 232;
static_assert(128 * SHORT_REGS_CONTROL + 256 * SHORT_REGS_EPILOGUE <= TC_THREADS * TC_REGS_AT_LAUNCH, "setmaxnreg: the epilogue's increase must fit what the control warps give up");
enum : int { SHORT_WAIT_DONE = 21, SHORT_WAIT_GO = 22, SHORT_WAIT_ACC = 23 };

// The same for the sum over two examples, sign + sign + 2 in {0 .. 4}: the saturated halves are added before the integer is
// extracted (1.5 * 2^22 has steps of 0.5).
__device__ __forceinline__ uint32_t signs_plus_two_packed(uint64_t g2, uint64_t h2) {
  float t0, t1;
  sm100::f32x2_unpack(sm100::f32x2_add(sm100::f32x2_add(sign_half2(g2), sm100::f32x2_pack(6291456.f, 6291456.f)), sign_half2(h2)), t0, t1);
  return __byte_perm(__float_as_uint(t0), __float_as_uint(t1), 0x5410);
}

template <bool MEAN, bool SQUARE, bool SIGN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TC_THREADS, 1)
short_stats_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_dy, const __grid_constant__ CUtensorMap tmap_mean,
                   const __grid_constant__ CUtensorMap tmap_square, const __grid_constant__ CUtensorMap tmap_sign, TcParams p) {
  using namespace sm100;
  constexpr int COLS = SHORT_NT / 2;                // accumulator columns per epilogue thread
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t bar_base = smem_base + SHORT_RING;
  auto go_bar = [&](int s) { return bar_base + 8u * s; };
  auto done_bar = [&](int s) { return bar_base + 8u * (SHORT_STAGES + s); };
  uint8_t* tail = smem_gen + SHORT_RING + 16 * SHORT_STAGES;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(tail);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 8);
  static_assert(16 * SHORT_STAGES + 16 <= TC_BAR_BYTES, "barrier area too small");

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();          // 0 = leader of the pair
  const int n_units = tc_units(p), step = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < SHORT_STAGES; ++s) { mbar_init(go_bar(s), 1 + 16); mbar_init(done_bar(s), 1); }
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 2) { tmem_alloc_pair(smem_u32(const_cast<uint32_t*>(tmem_slot)), TC_TMEM_COLS); tmem_relinquish_pair(); }
  tc_fence_before();
  cluster_sync_all();          // barriers of both blocks initialised before any remote arrival
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  griddep_launch_dependents();            // as in tc_stats_kernel
  if (p.wait_at_start) griddep_wait();

  if (warp < 4) {
    setmaxnreg_dec<SHORT_REGS_CONTROL>();
    const bool strict = wait_cycle_limit() < WAIT_CYCLE_LIMIT_STRICT;
    if (warp == 0 || warp == 2) {
      // ---------------------------------------------------------- TMA producers (both blocks)
      const bool is_a = (warp == 0);
      const CUtensorMap* tmap = is_a ? &tmap_dy : &tmap_x;
      if (elect_one()) prefetch_tensormap(tmap);
      int s = 0;
      uint32_t ph = 1;
      bool ok = true;
      for (int u = blockIdx.x >> 1; ok && u < n_units; u += step) {
        const TcUnit t = tc_unit(p, u);
        int tile_m, tile_n;
        tc_tile_of_pair(p, t.tile, rank, tile_m, tile_n);
        const int c0 = is_a ? tile_m * TC_TILE_M : tile_n * SHORT_NT + (int)rank * (SHORT_NT / 2);
        for (int b = t.b_begin; b < t.b_end; b += SHORT_G) {
          if (!mbar_wait_warp(done_bar(s), ph, abort_flag, p.dev_status, SHORT_WAIT_DONE, strict)) { ok = false; break; }
          if (elect_one()) {
            if (is_a && rank == 0) mbar_arrive_expect_tx(go_bar(s), 2 * SHORT_STAGE);       // both blocks' bytes
            const uint32_t leader_go = map_to_cta(go_bar(s), 0);
            const uint32_t dst = smem_base + s * SHORT_STAGE;
            // (the box is SHORT_G examples deep; past the batch's end it reads zeros)
            if (is_a) {
              tma_load_3d_pair(dst, tmap, leader_go, c0, 0, b);
              tma_load_3d_pair(dst + SHORT_A_BOX, tmap, leader_go, c0 + 64, 0, b);
            } else {
              tma_load_3d_pair(dst + 2 * SHORT_A_BOX, tmap, leader_go, c0, 0, b);
            }
          }
          __syncwarp();
          if (++s == SHORT_STAGES) { s = 0; ph ^= 1u; }
        }
      }
    } else if (rank == 0 && warp == 1) {
      // ---------------------------------------------------------- MMA issuer (leader block)
      const uint32_t idesc = make_idesc_mn_major(TC_PAIR_M, SHORT_NT, false);
      const bool two_steps = p.T > 16;
      int s = 0, buf = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int u = blockIdx.x >> 1; ok && u < n_units; u += step) {
        const TcUnit t = tc_unit(p, u);
        for (int b = t.b_begin; b < t.b_end; b += SHORT_G) {
          if (!mbar_wait_warp(go_bar(s), ph, abort_flag, p.dev_status, SHORT_WAIT_GO, strict)) { ok = false; break; }
          tc_fence_after();
          if (elect_one()) {
            const uint32_t a_src = smem_base + s * SHORT_STAGE, d = tmem_base + (uint32_t)(buf * SHORT_G * SHORT_NT);
            const uint64_t ad = make_smem_desc(a_src, SHORT_A_BOX, 1024u, 2u), bd = make_smem_desc(a_src + 2 * SHORT_A_BOX, SHORT_B_BOX, 1024u, 2u);
#pragma unroll
            for (int j = 0; j < SHORT_G; ++j) {
              const uint64_t at = (uint64_t)(j * SHORT_T * 128 >> 4);
              umma_ss_pair<0>(d + (uint32_t)(j * SHORT_NT), ad + at, bd + at, idesc, 0u);
              if (two_steps) umma_ss_pair<0>(d + (uint32_t)(j * SHORT_NT), ad + at + (2048 >> 4), bd + at + (2048 >> 4), idesc, 1u);
            }
            umma_commit_pair(done_bar(s));
          }
          __syncwarp();
          buf ^= 1;
          if (++s == SHORT_STAGES) { s = 0; ph ^= 1u; }
        }
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue (both blocks)
    setmaxnreg_inc<SHORT_REGS_EPILOGUE>();
    const int q = warp & 3, h = (warp - 4) >> 2;     // tensor-memory lane quadrant, column half of the tile
    constexpr int W = MEAN && SQUARE && SIGN ? 8 : 16;             // columns per read of each example
    constexpr int STEPS = COLS / W;
    static_assert(STEPS % 2 == 0, "two buffers in turn");
    // Three sums: sum_b (sign(G_b) + 1) of two neighbouring columns in one word, as in tc_stats_kernel; otherwise sum_b (sign(G_b) + 1) / 2 in fp32.
    constexpr bool COUNT = SIGN && SQUARE;
    float acc_mean[MEAN ? COLS : 1], acc_stat[SQUARE || SIGN ? COLS : 1];
    uint32_t acc_cnt[COUNT ? COLS / 2 : 1];
    // The square alone: sum_run examples at a time in sums of their own.  This tile leaves more of the batch to a pair than the 256 x 256 tile of
    // tc_stats_kernel does, and plain sums would round more often than there.  Each run costs about 260 cycles at its end: 1024 x 32 x 4096^2
    // 1495 us in runs of 16 (error 1.2e-7), 1472 of 64 (8e-8).
    constexpr bool RUNS = SQUARE && !MEAN && !SIGN;
    float acc_run[RUNS ? COLS : 1];
    auto clear = [&]() {
#pragma unroll
      for (int j = 0; j < COLS; ++j) {
        if (MEAN) acc_mean[j] = 0.f;
        if (SQUARE || SIGN) acc_stat[j] = 0.f;
        if (RUNS) acc_run[j] = 0.f;
        if (COUNT && j % 2 == 0) acc_cnt[j / 2] = 0u;
      }
    };
    clear();
    const uint32_t lane_base = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * COLS);
    const uint32_t leader_go = map_to_cta(go_bar(0), 0);
#pragma unroll
    for (int k = 0; k < SHORT_UNITS; ++k) mbar_arrive_cluster_if(lane == 0, leader_go + 8u * k);          // both accumulator units are free
    int s = 0, buf = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int u = blockIdx.x >> 1; ok && u < n_units; u += step) {
      const TcUnit t = tc_unit(p, u);
      int tile_m, tile_n;
      tc_tile_of_pair(p, t.tile, rank, tile_m, tile_n);
      const int row0 = tile_m * TC_TILE_M + q * 32, col0 = tile_n * SHORT_NT + h * COLS;
      uint32_t g[2][W], f[2][W];              // the two examples' entries, two reads in turn
      bool read_ahead = false;
      for (int b = t.b_begin; b < t.b_end; b += SHORT_G) {
        const bool pair_of = b + 1 < t.b_end;
        const uint32_t taddr = lane_base + (uint32_t)(buf * SHORT_G * SHORT_NT);
        int next_s = s + 1, free_s = s + SHORT_UNITS;
        uint32_t next_ph = ph;
        if (next_s == SHORT_STAGES) { next_s = 0; next_ph ^= 1u; }
        if (free_s >= SHORT_STAGES) free_s -= SHORT_STAGES;
        auto fold = [&](int k) {
#pragma unroll
          for (int j = 0; j < W; j += 2) {
            const int c = k * W + j;
            const uint64_t g2 = f32x2_pack(__uint_as_float(g[k & 1][j]), __uint_as_float(g[k & 1][j + 1]));
            const uint64_t f2 = f32x2_pack(__uint_as_float(f[k & 1][j]), __uint_as_float(f[k & 1][j + 1]));
            if constexpr (MEAN) f32x2_unpack(f32x2_add(f32x2_add(f32x2_pack(acc_mean[c], acc_mean[c + 1]), g2), f2), acc_mean[c], acc_mean[c + 1]);
            if constexpr (SQUARE) {
              float& s0 = RUNS ? acc_run[RUNS ? c : 0] : acc_stat[c];
              float& s1 = RUNS ? acc_run[RUNS ? c + 1 : 0] : acc_stat[c + 1];
              f32x2_unpack(f32x2_fma(f2, f2, f32x2_fma(g2, g2, f32x2_pack(s0, s1))), s0, s1);
            }
            if constexpr (COUNT) acc_cnt[c / 2] += signs_plus_two_packed(g2, f2);
            if constexpr (SIGN && !COUNT)
              f32x2_unpack(f32x2_add(f32x2_add(f32x2_pack(acc_stat[c], acc_stat[c + 1]), sign_half2(g2)), sign_half2(f2)), acc_stat[c], acc_stat[c + 1]);
          }
        };
        // Reads that are in flight cross no join of branches that defines their registers: what the compiler might move there would be read before it
        // has arrived.
        if (!read_ahead) {
          if (!mbar_wait_warp(done_bar(s), ph, abort_flag, p.dev_status, SHORT_WAIT_ACC)) { ok = false; break; }
          tc_fence_after();
          tmem_ld_issue(taddr, g[0]);
          tmem_ld_issue(taddr + SHORT_NT, f[0]);
          tmem_ld_wait_for(g[0], f[0]);
        }
        bool next_done = false;
#pragma unroll
        for (int k = 0; k < STEPS; ++k) {
          if (k > 0) tmem_ld_wait_for(g[k & 1], f[k & 1]);
          if (k + 1 < STEPS) {
            tmem_ld_issue(taddr + (k + 1) * W, g[(k + 1) & 1]);
            tmem_ld_issue(taddr + SHORT_NT + (k + 1) * W, f[(k + 1) & 1]);
            // whether the next unit is there already is asked a step before the answer is needed
            if (k + 2 == STEPS && b + SHORT_G < t.b_end) next_done = mbar_test_wait(done_bar(next_s), next_ph);
          }
          if (!pair_of) {
#pragma unroll
            for (int j = 0; j < W; ++j) f[k & 1][j] = 0u;
          }
          if (k + 1 < STEPS) {
            fold(k);
          }
        }
        tc_fence_before();
        __syncwarp();
        mbar_arrive_cluster_if(lane == 0, leader_go + 8u * free_s);        // this accumulator unit may be filled again
        read_ahead = __all_sync(0xffffffffu, next_done);
        if (read_ahead) tc_fence_after();
        const uint32_t ahead = lane_base + (uint32_t)((buf ^ 1) * SHORT_G * SHORT_NT);
        tmem_ld_issue_if(read_ahead, ahead, g[0]);
        tmem_ld_issue_if(read_ahead, ahead + SHORT_NT, f[0]);
        fold(STEPS - 1);
        tmem_ld_wait_for(g[0], f[0]);
        if constexpr (RUNS) {
          if (((b - t.b_begin + SHORT_G) & (p.sum_run - 1)) == 0 || b + SHORT_G >= t.b_end) {
#pragma unroll
            for (int j = 0; j < COLS; j += 2) {
              f32x2_unpack(f32x2_add(f32x2_pack(acc_stat[j], acc_stat[j + 1]), f32x2_pack(acc_run[j], acc_run[j + 1])), acc_stat[j], acc_stat[j + 1]);
              acc_run[j] = acc_run[j + 1] = 0.f;
            }
          }
        }
        buf ^= 1;
        if (++s == SHORT_STAGES) { s = 0; ph ^= 1u; }
      }
      ok = __all_sync(0xffffffffu, ok);
      // Write-out, while the next tile's first units are contracted: 32 columns at a time through the warp's own panel of shared memory, which TMA
      // stores or, for a slice of the batch, adds to the output, dropping what lies outside the matrix.
      const bool add = !t.whole || p.accumulate;
      if (!t.whole && !p.accumulate) griddep_wait();                 // the kernel that zeroes the outputs
      const uint32_t panel = smem_base + SHORT_STAGES * SHORT_STAGE + (uint32_t)(warp - 4) * SHORT_PANEL;
      uint8_t* const panel_gen = smem_gen + (panel - smem_base);
      auto put = [&](const CUtensorMap* tm, float* out, int c, const float (&v)[32]) {            // 32 columns from the c-th on
        if (!ok || row0 >= p.d_out || col0 + c >= p.d_in) return;
        if (elect_one()) bulk_wait_read_all();                       // the panel's last use
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 8; ++k)
          *reinterpret_cast<float4*>(panel_gen + lane * 128 + ((k ^ (lane & 7)) << 4)) = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
        if (p.scalar_out) {                                          // rows that are no 16-byte multiples
          __syncwarp();
          const int col = col0 + c + lane;
          for (int r = 0; r < 32 && row0 + r < p.d_out; ++r) {
            const float x = *reinterpret_cast<const float*>(panel_gen + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + (lane & 3) * 4);
            float* const at = out + (long long)(row0 + r) * p.d_in + col;
            if (col < p.d_in) {
              if (add) atomicAdd(at, x);
              else *at = x;
            }
          }
          return;
        }
        fence_async_smem();
        __syncwarp();
        if (elect_one()) {
          if (add) tma_store_2d<true>(tm, panel, col0 + c, row0);
          else tma_store_2d<false>(tm, panel, col0 + c, row0);
          bulk_commit_group();
        }
        __syncwarp();
      };
#pragma unroll
      for (int c = 0; c < COLS; c += 32) {
        float v[32];
        if constexpr (SQUARE) {
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = acc_stat[c + j];
          if (p.out_stat) put(&tmap_square, p.out_stat, c, v);
        }
        if constexpr (MEAN) {
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = acc_mean[c + j];
          put(&tmap_mean, p.out_mean, c, v);
        }
        if constexpr (SIGN) {
          const float nbf = (float)((t.b_end - t.b_begin + SHORT_G - 1) / SHORT_G * SHORT_G);      // (an example missing from the last unit is one of zeros)
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            if constexpr (COUNT) v[j] = (float)((acc_cnt[(c + j) / 2] >> (16 * (j & 1))) & 0xFFFFu) - nbf;
            else v[j] = fmaf(2.f, acc_stat[c + j], -nbf);
          }
          put(&tmap_sign, p.out_sign, c, v);
        }
      }
      clear();
    }
    if (elect_one()) bulk_wait_read_all();           // shared memory must outlive TMA's reads
    __syncwarp();
  }

  // ---------------------------------------------------------------- teardown, as in tc_stats_kernel
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    const long long t0 = clock64();
    while (clock64() - t0 < (1ll << 22)) __nanosleep(1000);
  }
  __syncwarp();
  cluster_sync_all();
  if (warp == 2) { tc_fence_after(); tmem_dealloc_pair(tmem_base, TC_TMEM_COLS); }
}

}  // namespace pe
