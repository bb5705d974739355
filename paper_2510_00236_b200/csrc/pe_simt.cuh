// SIMT (CUDA-core) kernels for the per-example statistics: the fp32-input path and the path for
// shapes the tensor-core kernel does not take.  A thread block owns a (16 TM) x (16 TN) tile of the
// [d_out, d_in] output and walks over the examples of its slice of the batch; the per-example
// gradient tile lives in registers and never reaches global memory.
//
// Bound: fp32 FMA (148 SMs x 128 lanes, 72 TFLOP/s) on layers that fill the chip, the latency of one load
// and one reduction on those that do not.  Each thread forms TM x TN entries (two columns per packed FMA) from
// 128-bit shared-memory reads; the next chunk of tokens is loaded into registers while the current one is
// contracted, across example boundaries, and the two chunk buffers need one barrier per chunk.  The batch is
// split over the blocks of a cluster, whose partial sums meet in shared memory: nothing is zeroed first, no
// atomics, and the result does not depend on timing (more slices than a cluster holds fall back to atomics).
// Measured, both outputs, against a 64 x 64 tile of 4 x 4 entries, one buffer and scalar reads: 32 x 128 x 256 x 1024 157.8 -> 65 us, 8 x 16 x 64 x 64
// 18.7 -> 11.4 us per call; 8 x 256 x 1024 x 16384 1438 us, 48 TFLOP/s (packed FMAs from shared memory alone, in a loop: 61; of the difference a
// seventh are the warps that wait at the chunks' barrier).  Not faster: 8 x 8 entries (one block per SM, 38 TFLOP/s), scalar FMAs (42), packed FMAs
// over diagonals of 2 x 2 entries, which need no doubled operands (3 to 6 % slower), clusters of 16, 16-token chunks of the largest tile.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "pe_optim.cuh"
#include "pe_sm100.cuh"

namespace pe {

constexpr int SIMT_MAX_CLUSTER = 8;     // batch slices whose partial sums meet in shared memory

enum : int { MODE_STATS = 0, MODE_TOKEN = 1, MODE_NORMS = 2 };

// Tile shapes.  TM x TN entries per thread; KT tokens per chunk.  The large tile has the most FMAs per shared-memory
// read, the small ones spread a small layer over the chip.
template <int TM_, int TN_, int KT_, int THREADS_ = 256>
struct SimtTile {
  static constexpr int TM = TM_, TN = TN_, KT = KT_, THREADS = THREADS_;
  static constexpr int TY = THREADS / 16;                        // TY x 16 threads
  static constexpr int BLOCKS = TM * TN == 4 ? 3 : 512 / THREADS;       // an SM holds at least (32 x 32: 86 to 92 registers, and two blocks, if left alone)
  static constexpr int ROWS = TY * TM, COLS = 16 * TN;
  static constexpr int CHUNK = KT * (ROWS + COLS);               // floats of one chunk: dY part, then X part
  static constexpr int YV = KT * ROWS / 4 / THREADS, XV = KT * COLS / 4 / THREADS;   // 4-column groups per thread
  static_assert(YV * 4 * THREADS == KT * ROWS && XV * 4 * THREADS == KT * COLS, "whole groups per thread");
  // the largest tile keeps its running sums in shared memory (64 registers of sums beside 32 of G_b would leave one block per SM)
  static constexpr bool SUMS_IN_SMEM = TM * TN > 16;
  // the chunk buffers; the sums' exchange at the end lies behind them where the sums live there, on top of them otherwise
  static constexpr int smem_floats(int sums) {
    return SUMS_IN_SMEM ? 2 * CHUNK + sums * ROWS * COLS : (2 * CHUNK > sums * ROWS * COLS ? 2 * CHUNK : sums * ROWS * COLS);
  }
};
using SimtTile84 = SimtTile<8, 4, 32>;
// Half of the largest tile in blocks of half the threads, four to an SM: the same FMAs per read in twice as many pieces, which spread layers of a
// few hundred rows and columns more evenly.  10 x 200 x 800 x 400, both outputs, 78 -> 64 us, 64 x 32 x 500 x 300 43 -> 35, 8 x 256 x 1024 x 2048 255 -> 208,
// and per token 230 -> 187.  Shorter chunks beside running sums, whose shared memory would leave room for three blocks.
template <int MODE>
using SimtTileHalf = SimtTile<8, 4, MODE == MODE_TOKEN ? 32 : 16, 128>;
using SimtTile44 = SimtTile<4, 4, 16>;
using SimtTile22 = SimtTile<2, 2, 32>;
using SimtTile11 = SimtTile<1, 1, 64>;

// What a packed batch or a clipped sum adds to the plain call; all NULL / 0 otherwise.
struct SimtExtra {
  const int* seq_offsets;     // [B + 1]: example b owns token rows offsets[b] .. offsets[b+1]-1 of X [rows, d_in], dY [rows, d_out]
  long long total_rows;       // rows of the packed tensors (reads are kept inside)
  const float* sq_norms;      // phi == 3: [B] squared norms N_b;  coef_b = min(1, clip_norm / sqrt(N_b))
  float clip_norm;
};

// phi: 0 identity, 1 square, 2 sign, 3 the clipping scale coef * g
__device__ __forceinline__ float apply_phi(float g, int phi, float coef) {
  if (phi == 1) return g * g;
  if (phi == 2) return (g > 0.f ? 1.f : 0.f) - (g < 0.f ? 1.f : 0.f);
  if (phi == 3) return coef * g;
  return g;
}

// Four elements from p on, `left` of which are inside the row, as they are loaded.  whole: all four, as one aligned load.  Widened only when they are
// written to shared memory, so that a chunk's loads are in flight together: norms
// of 17 x 136 x 63 x 928 42.9 -> 24.7 us, of 33 x 245 x 98 x 434 77.8 -> 49.2.
__device__ __forceinline__ float4 load_group(const float* p, int left, bool whole) {
  if (whole) return __ldg(reinterpret_cast<const float4*>(p));
  float v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) v[j] = j < left ? __ldg(p + j) : 0.f;
  return make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ uint4 load_group(const __nv_bfloat16* p, int left, bool whole) {
  if (whole) {
    const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
    return make_uint4(u.x, u.y, 0u, 0u);
  }
  uint32_t w[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) w[j] = j < left ? (uint32_t)__ldg(reinterpret_cast<const unsigned short*>(p) + j) : 0u;
  return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ float4 widen_group(float4 v, bool) { return v; }
__device__ __forceinline__ float4 widen_group(uint4 v, bool whole) {
  if (whole) return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xFFFF0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xFFFF0000u));
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.y << 16), __uint_as_float(v.z << 16), __uint_as_float(v.w << 16));
}

// A thread's N operands of one token: N = 1, 2 or 4 consecutive floats, 8 as two groups of four, 4 * SIDE floats apart (SIDE: threads on this
// side of the tile).
template <int N, int SIDE>
__device__ __forceinline__ void lds_vec(const float* p, float (&v)[N]) {
  if constexpr (N == 1) {
    v[0] = *p;
  } else if constexpr (N == 2) {
    const float2 t = *reinterpret_cast<const float2*>(p);
    v[0] = t.x; v[1] = t.y;
  } else {
#pragma unroll
    for (int h = 0; h < N / 4; ++h) {
      const float4 t = *reinterpret_cast<const float4*>(p + 4 * SIDE * h);
      v[4 * h] = t.x; v[4 * h + 1] = t.y; v[4 * h + 2] = t.z; v[4 * h + 3] = t.w;
    }
  }
}
// Tile row (column) of entry j of a thread's N: the layout lds_vec reads.
template <int N, int SIDE>
__device__ __forceinline__ int micro_index(int thread, int j) { return N <= 4 ? thread * N + j : thread * 4 + (j & 3) + 4 * SIDE * (j >> 2); }

// MODE_STATS: out_mean = sum_b G_b, out_stat = sum_b phi(G_b)         (Section 2.3, Eq. (2))
// MODE_TOKEN: out_stat = sum_{b,t} dY^2 X^2; operands are squared as they are staged and the
//             accumulator is never reset between examples             (Section 2.3, per-token form)
// MODE_NORMS: out_stat is a [B] array, zero on entry; every tile adds its share of ||G_b||_F^2 to
//             out_stat[b] (Section 2.3, per-example squared norms); no [d_out, d_in] output
// gridDim = (ceil(d_in/COLS) * ceil(d_out/ROWS), 1, slices) in clusters of (1, 1, cluster), cluster a power of two that divides
// slices; slice z handles examples [z*B/slices, (z+1)*B/slices), or that share of the B*T rows (MODE_TOKEN).  With more
// slices than one cluster the outputs must be zero on entry and the clusters' sums are added atomically; with
// accumulate != 0 the results are added to whatever the outputs hold.  opt.kind != 0 (one cluster only): the block that
// ends up with an entry's sums also applies the parameter update (phi must then be square for the Adam family,
// sign for MicroSignSGD); out_mean / out_stat may then be NULL.
// ldx, ldy: elements from one token's row of X, dY to the next.
// SUMS: running sums per entry: 2 = sum_b phi(G_b) and sum_b G_b, 1 = the former alone (or the contraction of MODE_TOKEN).
template <typename TIn, int MODE, class Tile, int SUMS>
__global__ void __launch_bounds__(Tile::THREADS, Tile::BLOCKS)
simt_stats_kernel(const TIn* __restrict__ X, const TIn* __restrict__ dY, int B, int T, int d_in, int d_out,
                  int phi, float* __restrict__ out_mean, float* __restrict__ out_stat, int accumulate, int cluster, int ldx, int ldy, int vec_x, int vec_y,
                  SimtExtra ex, FusedOpt opt) {
  constexpr int TM = Tile::TM, TN = Tile::TN, KT = Tile::KT, ROWS = Tile::ROWS, COLS = Tile::COLS;
  constexpr bool IN_SMEM = Tile::SUMS_IN_SMEM && MODE == MODE_STATS;
  extern __shared__ __align__(16) float simt_smem[];
  // a warp is 4 x 8 threads of the TY x 16: four distinct operands of dY and eight of X per shared-memory read
  const int tx = (threadIdx.x & 7) | ((threadIdx.x >> 2) & 8), ty = ((threadIdx.x >> 3) & 3) | ((threadIdx.x >> 6) << 2);
  const int tiles_in = (d_in + COLS - 1) / COLS;
  const int i0 = (int)(blockIdx.x % tiles_in) * COLS, o0 = (int)(blockIdx.x / tiles_in) * ROWS;
  const int slices = gridDim.z;

  // g: this thread's entries of G_b.  Running sums ([0] = the statistic, [1] = sum_b G_b) in registers, or, IN_SMEM, in a
  // thread-private arrangement of shared memory (one float4 per thread, the block's threads side by side: no bank conflicts).
  float g[TM][TN];
  float sum[IN_SMEM ? 1 : SUMS][TM][TN];
  float* const smem_sums = simt_smem + 2 * Tile::CHUNK;
  auto slot = [&](int s, int r, int c4) { return reinterpret_cast<float4*>(smem_sums) + ((s * TM + r) * (TN / 4) + c4) * Tile::THREADS + threadIdx.x; };
#pragma unroll
  for (int r = 0; r < TM; ++r) {
#pragma unroll
    for (int c = 0; c < TN; ++c) g[r][c] = 0.f;
#pragma unroll
    for (int s = 0; s < SUMS; ++s) {
      if constexpr (IN_SMEM) {
#pragma unroll
        for (int c4 = 0; c4 < TN / 4; ++c4) *slot(s, r, c4) = make_float4(0.f, 0.f, 0.f, 0.f);
      } else {
#pragma unroll
        for (int c = 0; c < TN; ++c) sum[s][r][c] = 0.f;
      }
    }
  }

  // The walk: example b, tokens t .. t+KT-1 of it.  MODE_TOKEN: the slice's rows, in "examples" of 2^20 rows.
  constexpr int TOKEN_RUN = 1 << 20;
  int b = 0, b_end = 0, t = 0, Tb = 0;
  long long row0 = 0, slice_row0 = 0, slice_rows = 0;
  auto open_example = [&]() {
    if (MODE == MODE_TOKEN) {
      row0 = slice_row0 + (long long)b * TOKEN_RUN;
      const long long rest = slice_rows - (long long)b * TOKEN_RUN;
      Tb = rest < TOKEN_RUN ? (int)rest : TOKEN_RUN;
      return;
    }
    row0 = (long long)b * T;
    Tb = T;
    if (ex.seq_offsets) {            // packed batch: this example's own token range, clamped to the tensor
      const long long r0 = ex.seq_offsets[b], r1 = ex.seq_offsets[b + 1];
      row0 = r0 < 0 ? 0 : r0;
      const long long end = r1 > ex.total_rows ? ex.total_rows : r1;
      Tb = end > row0 ? (int)(end - row0) : 0;
    }
  };
  if (MODE == MODE_TOKEN) {
    const long long rows = (long long)B * T;
    slice_row0 = rows * blockIdx.z / slices;
    slice_rows = rows * (blockIdx.z + 1) / slices - slice_row0;
    b_end = (int)((slice_rows + TOKEN_RUN - 1) / TOKEN_RUN);
  } else {
    b = (int)(((long long)B * blockIdx.z) / slices);
    b_end = (int)(((long long)B * (blockIdx.z + 1)) / slices);
  }
  if (b < b_end) open_example();

  // A thread's groups of a chunk lie in one column, Y_STEP and X_STEP tokens apart, so that a chunk's addresses take one multiplication per
  // operand: spelled out per group, their 64-bit multiplications were a fifth of the FMA pipe's work.
  constexpr int Y_STEP = 4 * Tile::THREADS / ROWS, X_STEP = 4 * Tile::THREADS / COLS;
  static_assert(Y_STEP * ROWS == 4 * Tile::THREADS && X_STEP * COLS == 4 * Tile::THREADS, "whole rows of groups per round");
  const int y_tok = threadIdx.x / (ROWS / 4), x_tok = threadIdx.x / (COLS / 4);
  const int y_col = o0 + 4 * (threadIdx.x % (ROWS / 4)), x_col = i0 + 4 * (threadIdx.x % (COLS / 4));
  const bool y_whole = vec_y != 0 && y_col + 3 < d_out, x_whole = vec_x != 0 && x_col + 3 < d_in;
  using Group = std::conditional_t<sizeof(TIn) == 2, uint4, float4>;
  Group sy[Tile::YV], sx[Tile::XV];
  auto load_chunk = [&]() {            // zero past the example's end and past the matrix edge
    const TIn* yp = dY + (row0 + t + y_tok) * (long long)ldy + y_col;
    const TIn* xp = X + (row0 + t + x_tok) * (long long)ldx + x_col;
    const int y_left = y_col < d_out ? Tb - t - y_tok : 0, x_left = x_col < d_in ? Tb - t - x_tok : 0;
#pragma unroll
    for (int k = 0; k < Tile::YV; ++k) {
      sy[k] = Group{};
      if (k * Y_STEP < y_left) sy[k] = load_group(yp, d_out - y_col, y_whole);
      yp += (size_t)Y_STEP * ldy;
    }
#pragma unroll
    for (int k = 0; k < Tile::XV; ++k) {
      sx[k] = Group{};
      if (k * X_STEP < x_left) sx[k] = load_group(xp, d_in - x_col, x_whole);
      xp += (size_t)X_STEP * ldx;
    }
  };
  auto put = [&](float* at, float4 v) {
    *reinterpret_cast<float4*>(at) = MODE == MODE_TOKEN ? make_float4(v.x * v.x, v.y * v.y, v.z * v.z, v.w * v.w) : v;
  };
  // end of example eb: phi and the running sums
  auto fold = [&](int eb) {
    if constexpr (MODE == MODE_NORMS) {
      float s = 0.f;            // entries outside the matrix are exact zeros (their operands were zero-filled)
#pragma unroll
      for (int r = 0; r < TM; ++r)
#pragma unroll
        for (int c = 0; c < TN; ++c) s = fmaf(g[r][c], g[r][c], s);
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
      if ((threadIdx.x & 31) == 0) atomicAdd(out_stat + eb, s);
    } else if constexpr (MODE == MODE_STATS) {
      float coef = 1.f;
      if (phi == 3) {
        const float nrm = sqrtf(ex.sq_norms[eb]);
        coef = nrm > ex.clip_norm ? ex.clip_norm / nrm : 1.f;
      }
#pragma unroll
      for (int r = 0; r < TM; ++r) {
        if constexpr (IN_SMEM) {
#pragma unroll
          for (int c4 = 0; c4 < TN / 4; ++c4) {
            float v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = g[r][4 * c4 + j];
            float4 s = *slot(0, r, c4);
            s.x += apply_phi(v[0], phi, coef); s.y += apply_phi(v[1], phi, coef);
            s.z += apply_phi(v[2], phi, coef); s.w += apply_phi(v[3], phi, coef);
            *slot(0, r, c4) = s;
            if constexpr (SUMS == 2) {
              float4 m = *slot(1, r, c4);
              m.x += v[0]; m.y += v[1]; m.z += v[2]; m.w += v[3];
              *slot(1, r, c4) = m;
            }
          }
        } else {
#pragma unroll
          for (int c = 0; c < TN; ++c) {
            const float v = g[r][c];
            sum[0][r][c] += apply_phi(v, phi, coef);
            if constexpr (SUMS == 2) sum[1][r][c] += v;
          }
        }
      }
    }
    if constexpr (MODE != MODE_TOKEN) {
#pragma unroll
      for (int r = 0; r < TM; ++r)
#pragma unroll
        for (int c = 0; c < TN; ++c) g[r][c] = 0.f;
    }
  };

  bool more = b < b_end;
  if (more) load_chunk();
  for (int buf = 0; more; buf ^= 1) {
    const int left = Tb - t, cur_b = b;            // tokens of this example from this chunk on
    float* const y = simt_smem + buf * Tile::CHUNK;
    float* const x = y + KT * ROWS;
#pragma unroll
    for (int k = 0; k < Tile::YV; ++k) put(y + 4 * (threadIdx.x + k * Tile::THREADS), widen_group(sy[k], y_whole));
#pragma unroll
    for (int k = 0; k < Tile::XV; ++k) put(x + 4 * (threadIdx.x + k * Tile::THREADS), widen_group(sx[k], x_whole));
    __syncthreads();           // a buffer is written again two chunks later, behind the barrier that follows its last reads
    // the next chunk's loads are in flight during this one's arithmetic
    t += KT;
    const bool ends = t >= Tb;
    if (ends) {
      t = 0;
      if (++b < b_end) open_example();
    }
    more = b < b_end;
    if (more) load_chunk();
    // tokens past the example's end are zero: whole groups of 8 of them are skipped.  (A whole chunk without a loop: the reads of one group overlap the
    // FMAs of the one before; 3 to 5 %.)
    auto tokens = [&](auto count, int k0) {
#pragma unroll
      for (int kk = 0; kk < decltype(count)::value; ++kk) {
        float yv[TM], xv[TN];
        lds_vec<TM, Tile::TY>(y + (k0 + kk) * ROWS + (TM < 4 ? TM : 4) * ty, yv);
        lds_vec<TN, 16>(x + (k0 + kk) * COLS + (TN < 4 ? TN : 4) * tx, xv);
#pragma unroll
        for (int r = 0; r < TM; ++r) {
          if constexpr (TN >= 2) {
            const uint64_t y2 = sm100::f32x2_pack(yv[r], yv[r]);
#pragma unroll
            for (int c = 0; c < TN; c += 2) {
              const uint64_t a = sm100::f32x2_fma(y2, sm100::f32x2_pack(xv[c], xv[c + 1]), sm100::f32x2_pack(g[r][c], g[r][c + 1]));
              sm100::f32x2_unpack(a, g[r][c], g[r][c + 1]);
            }
          } else {
            g[r][0] = fmaf(yv[r], xv[0], g[r][0]);
          }
        }
      }
    };
    if (left >= KT) {
      tokens(std::integral_constant<int, KT>{}, 0);
    } else {
#pragma unroll 1
      for (int k0 = 0; k0 < left; k0 += 8) tokens(std::integral_constant<int, 8>{}, k0);
    }
    if (ends) fold(cur_b);
  }

  if constexpr (MODE != MODE_NORMS) {       // MODE_NORMS has no [d_out, d_in] output
    // Every block lays its partial sums out in its shared memory as [sum][row][column]; each block of the cluster
    // then adds up its share of the rows over all of them, in slice order, and writes the result.
    float* const xch = IN_SMEM ? smem_sums : simt_smem;
    if constexpr (IN_SMEM) {
      // the thread-private slots are overwritten by their own rearrangement: one sum at a time, through registers
#pragma unroll
      for (int s = 0; s < SUMS; ++s) {
        float4 v[TM][TN / 4];
#pragma unroll
        for (int r = 0; r < TM; ++r)
#pragma unroll
          for (int c4 = 0; c4 < TN / 4; ++c4) v[r][c4] = *slot(s, r, c4);
        __syncthreads();
#pragma unroll
        for (int r = 0; r < TM; ++r)
#pragma unroll
          for (int c4 = 0; c4 < TN / 4; ++c4)
            *reinterpret_cast<float4*>(xch + (s * ROWS + micro_index<TM, Tile::TY>(ty, r)) * COLS + micro_index<TN, 16>(tx, 4 * c4)) = v[r][c4];
      }
    } else {
      __syncthreads();         // the chunk buffers are idle from here on
#pragma unroll
      for (int s = 0; s < SUMS; ++s)
#pragma unroll
        for (int r = 0; r < TM; ++r)
#pragma unroll
          for (int c = 0; c < TN; ++c)
            xch[(s * ROWS + micro_index<TM, Tile::TY>(ty, r)) * COLS + micro_index<TN, 16>(tx, c)] = MODE == MODE_TOKEN ? g[r][c] : sum[s][r][c];
    }
    if (cluster > 1) sm100::cluster_sync_all();
    else __syncthreads();
    const int rank = cluster > 1 ? (int)sm100::cluster_ctarank() : 0;
    const bool add = slices > cluster || accumulate;
    const uint32_t local = sm100::smem_u32(xch);
    const int share = ROWS / cluster;         // rows this block finishes
    for (int e = threadIdx.x; e < share * COLS; e += Tile::THREADS) {
      const int r = rank * share + e / COLS, c = e % COLS;
      const int o = o0 + r, i = i0 + c;
      if (o >= d_out || i >= d_in) continue;
      float v[SUMS];
#pragma unroll
      for (int s = 0; s < SUMS; ++s) {
        const int at = (s * ROWS + r) * COLS + c;
        if (cluster == 1) {
          v[s] = xch[at];
        } else {
          float q[SIMT_MAX_CLUSTER];
#pragma unroll
          for (int k = 0; k < SIMT_MAX_CLUSTER; ++k) q[k] = k < cluster ? sm100::ld_shared_cluster(sm100::map_to_cta(local + 4u * (uint32_t)at, (uint32_t)k)) : 0.f;
          float a = q[0];
#pragma unroll
          for (int k = 1; k < SIMT_MAX_CLUSTER; ++k) a += q[k];
          v[s] = a;
        }
      }
      const size_t at = (size_t)o * d_in + i;
      if (!add) {
        if (out_stat) out_stat[at] = v[0];
        if (SUMS == 2 && out_mean) out_mean[at] = v[SUMS - 1];
        // the parameter update of Algorithm 1 / Section 3.1, applied where the sums over the whole batch are
        if (MODE == MODE_STATS && SUMS == 2 && opt.kind == OPT_ADAM) fused_update_one<OPT_ADAM>(opt, (long long)at, v[SUMS - 1], v[0]);
        if (MODE == MODE_STATS && SUMS == 1 && opt.kind == OPT_SIGN) fused_update_one<OPT_SIGN>(opt, (long long)at, v[0], 0.f);
      } else {
        if (out_stat) atomicAdd(out_stat + at, v[0]);
        if (SUMS == 2 && out_mean) atomicAdd(out_mean + at, v[SUMS - 1]);
      }
    }
    if (cluster > 1) sm100::cluster_sync_all();          // shared memory must outlive the peers' reads
  }
}

}  // namespace pe
