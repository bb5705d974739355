// C-ABI entry points of libpestats: argument validation, path selection, tensor-map creation and
// kernel launches.  Everything that computes runs in the CUDA kernels included below.
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <cmath>
#include <functional>
#include <mutex>
#include <vector>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "../../include/pestats.h"
#include "pe_layout.cuh"
#include "pe_optim.cuh"
#include "pe_stage.cuh"
#include "pe_short.cuh"
#include "pe_simt.cuh"
#include "pe_tc.cuh"
#include "pe_tok.cuh"

namespace pe {

__device__ unsigned int g_dev_status = 0;   // first device-side wait that gave up (0 = none)

static std::atomic<int> g_path{PE_PATH_AUTO};
static std::atomic<int> g_last_path{PE_PATH_AUTO};
static std::atomic<long long> g_launches{0};
static std::atomic<int> g_fused_mode{PE_FUSED_AUTO};
// Both outputs of a layer whose d_in fills neither 192- nor 128-column tiles well: from this sequence length on the running sum
// of G_b may live in tensor memory beside a 256-column accumulator.
constexpr int TC_MEAN_TMEM_MIN_T = 4096;
constexpr int TC_WIDE_MAX_PAD_PERCENT = 13;
constexpr int PHI_UNSCALE = 4;      // internal phi of the staged per-token statistic: a chunk's scales undone
constexpr int PHI_CLIP_SCALE = 3;   // internal phi of the clipped sum: c_b * G_b (not part of pe_phi_t)
constexpr int TC_BAND = 8;          // pair rows per band of the tile order (8 x 256 rows of d_out)

constexpr int MAX_DEVICES = 64;
struct DeviceInfo {
  std::atomic<int> state{0};     // 0 unknown, 1 ready, -1 failed
  int cc_major = 0, sm_count = 0;
  unsigned int* status_ptr = nullptr;
  bool tc_attr_set[64] = {};
  bool tok_attr_set = false;
};
static DeviceInfo g_dev[MAX_DEVICES];
static std::mutex g_dev_mutex;      // guards the lazily filled per-device state (first calls from several host threads)

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static std::atomic<EncodeTiledFn> g_encode{nullptr};

static pe_status_t device_info(DeviceInfo** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) { cudaGetLastError(); return PE_ERR_CUDA; }
  DeviceInfo& d = g_dev[dev];
  if (d.state.load(std::memory_order_acquire) == 0) {
    std::lock_guard<std::mutex> lock(g_dev_mutex);
    if (d.state.load(std::memory_order_relaxed) != 0) { *out = &d; return d.cc_major == 10 ? PE_OK : PE_ERR_ARCH; }
    int major = 0, sms = 0;
    void* sp = nullptr;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      cudaGetLastError();
      return PE_ERR_CUDA;
    }
    d.cc_major = major;
    d.sm_count = sms;
    if (major == 10) {
      if (cudaGetSymbolAddress(&sp, g_dev_status) != cudaSuccess) { cudaGetLastError(); return PE_ERR_CUDA; }
      d.status_ptr = static_cast<unsigned int*>(sp);
    }
    d.state.store(1, std::memory_order_release);
  }
  *out = &d;
  return d.cc_major == 10 ? PE_OK : PE_ERR_ARCH;
}

static EncodeTiledFn encode_fn() {
  EncodeTiledFn f = g_encode.load();
  if (f) return f;
  void* sym = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess || !sym) {
    cudaGetLastError();
    return nullptr;
  }
  f = reinterpret_cast<EncodeTiledFn>(sym);
  g_encode.store(f);
  return f;
}

static bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

static pe_status_t check_launch() {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return PE_ERR_CUDA;
  g_launches.fetch_add(1);
  return PE_OK;
}

// [B, T, d] row-major (bf16, or fp32 read as tf32) viewed as a 3-D tensor (d, T, B); one box = 128
// bytes of features x one pipeline stage of tokens of one example, 128-byte swizzled (16-byte chunks for bf16, 32-byte
// chunks for fp32: the MN-major tf32 MMA accepts no other layout).  rows64: 64 bytes of features per box row with
// the 64-byte swizzle (X of the 256 x 192 tile).  Tokens past T and features past d read as zero.
// pitch: elements from one token's row to the next (a multiple of 8 for bf16), 0 = d.
static pe_status_t make_operand_map(CUtensorMap* m, const void* base, int B, int T, int d, bool f32, int box_feats, int box_tokens,
                                    bool rows64 = false, int box_examples = 1, int pitch = 0) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return PE_ERR_CUDA;
  const cuuint64_t es = f32 ? 4ull : 2ull;
  cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)T, (cuuint64_t)B};
  const cuuint64_t row = (cuuint64_t)(pitch ? pitch : d) * es;
  cuuint64_t strides[2] = {row, (cuuint64_t)T * row};
  cuuint32_t box[3] = {(cuuint32_t)box_feats, (cuuint32_t)box_tokens, (cuuint32_t)box_examples};
  cuuint32_t estr[3] = {1u, 1u, 1u};
  CUresult r = enc(m, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE,
                   f32 ? CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B : (rows64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B),
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? PE_OK : PE_ERR_CUDA;
}

// The tensor-core per-token statistic rounds each squared operand to 11 significant bits (tf32 in the
// one-kernel form, column-scaled IEEE half in the two-pass form): relative error at most 2^-11 per
// factor, so at most ~1e-3 on any entry, all terms being non-negative.  Tiny problems
// gain nothing from the tensor cores and take the SIMT kernel (fp32 squares).
constexpr long long TOKEN_TC_MIN_ROWS = 256;

// [d_out, d_in] fp32 output viewed as a 2-D tensor (d_in, d_out); one box = 32 columns (128 bytes,
// 128-byte swizzled) x 32 rows, the piece one epilogue warp stages at a time.
static pe_status_t make_output_map(CUtensorMap* m, float* base, int d_in, int d_out) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return PE_ERR_CUDA;
  cuuint64_t dims[2] = {(cuuint64_t)d_in, (cuuint64_t)d_out};
  cuuint64_t strides[1] = {(cuuint64_t)d_in * 4ull};
  cuuint32_t box[2] = {32u, 32u};
  cuuint32_t estr[2] = {1u, 1u};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? PE_OK : PE_ERR_CUDA;
}

static bool tc_shape_ok(int B, int T, int d_in, int d_out);
static bool token_tc_ok(int B, int T, int d_in, int d_out) {
  return tc_shape_ok(B, T, d_in, d_out) && (long long)B * T >= TOKEN_TC_MIN_ROWS;
}

static bool tc_shape_ok(int B, int T, int d_in, int d_out) {
  if (B < 1 || T < 1) return false;
  if ((d_in % 8) || (d_out % 8)) return false;                        // 16-byte row pitch for TMA
  if ((long long)T * (d_in > d_out ? d_in : d_out) * 4ll >= (1ll << 40)) return false;   // TMA stride limit (fp32 staging included)
  return true;
}

// What a unit of work (one tile, one slice of the batch) costs a CTA pair on a given kernel, in microseconds, for choosing the tile
// and the number of slices.  Fitted to sweeps of both over layers from 512 x 512 to 1024 x 32104 with T = 1 to 1000.
struct UnitCost {
  int nt;                     // d_in columns per tile
  double token_lo, token_hi;  // per token of an example, with few pairs running and with all of them (operand supply from L2)
  double example;             // added per example
  double example_min;         // at least this much per example (what the epilogue takes)
  double fixed;               // per unit: prologue, first stage, write-out, teardown
};
constexpr double NORMS_UNIT = 0.15;                 // per tile and slice of the batch that a pair takes in turn
constexpr double FUSED_UPDATE_FIXED = 20.0;       // the parameter update of a 256 x 192 tile inside the statistics kernel
constexpr double SPLIT_FIXED = 2.0;               // adding to the outputs instead of storing, per unit
constexpr double ZERO_BYTES_PER_US = 6.4e6;       // zeroing the outputs of a split launch
constexpr UnitCost COST_STAT = {256, 0.51 / 128, 0.68 / 128, 0.0, 0.34, 8.5};            // one statistic (square, clipping) on 256 x 256
constexpr UnitCost COST_SIGN = {256, 0.51 / 128, 0.68 / 128, 0.0, 0.66, 8.5};
constexpr UnitCost COST_NORMS = {256, 0.51 / 128, 0.68 / 128, 0.0, 0.30, 7.0};
constexpr UnitCost COST_PLAIN = {256, 0.51 / 128, 0.68 / 128, 0.0, 0.0, 8.5};
constexpr UnitCost COST_TOKEN = {TOK_NT, 0.42 / TOK_BK, 0.45 / TOK_BK, 0.0, 0.0, 8.5};     // an "example" is one 32-row stage
// The per-token statistic's chunks dealt out over the pairs: two tiles instead of one to write out per pair, and rows that are read at
// different times for the tiles that share them.  64 x 256 x 512 x 2048 (16 tiles) 68.9 -> 63.0 us; 128 x 512 x 512 x 1024 (8 tiles, whose nine slices leave
// two pairs idle) 117 -> 119, which stays in slices.
constexpr double TOK_EVEN_FIXED = 4.0;
// ... and rows of operands that L2 does not hold (126 MB together, or a quarter of that for one beside the other's stream) are then read from HBM once for
// every tile, at about 4 TB/s: 60000 rows x 2048 x 2304 (72 tiles) 906 us whole and 1123 dealt out, 512 x 4608 (36) 447 and 531, 256 x 6656 (26) 379 in
// slices and 339 dealt out; 16384 x 1792 x 2560 (70) 238 and 276, 1280 x 2560 (50) 190 and 180.
constexpr double TOK_L2_BYTES = 126e6, TOK_DEALT_BYTES_PER_US = 4.0e6;
constexpr UnitCost COST_PLAIN_FP8 = {256, 0.28 / 128, 0.40 / 128, 0.0, 0.0, 8.5};
constexpr UnitCost COST_BOTH_192 = {192, 0.375 / 128, 0.55 / 128, 0.02, 0.35, 10.0};     // two sums
constexpr UnitCost COST_BOTH_128 = {128, 0.35 / 128, 0.44 / 128, 0.12, 0.20, 8.3};
constexpr UnitCost COST_ALL_192 = {192, 0.375 / 128, 0.60 / 128, 0.05, 0.95, 11.0};      // three statistics
constexpr UnitCost COST_ALL_128 = {128, 0.35 / 128, 0.44 / 128, 0.16, 0.55, 9.5};

// One pair per two SMs that walks over the tiles (PERSIST) instead of a pair per tile.  It saves the prologue and the teardown, and
// tensor work of the next tile overlaps the write-out.  What is lost: pairs that run faster cannot take more tiles (64 x 256 x 512 x 16384,
// three statistics: 321 -> 328 us).  Slices of the last wave stay one to a pair: 40 x 200 x 640 x 8000 (54 tiles left), both outputs, 104 us
// unsplit, 125 to 135 in 2 to 5 slices.
constexpr double PERSIST_SAVES = 3.5;             // per unit after a pair's first
constexpr double PERSIST_DRIFT = 1.025;
constexpr double TAIL_SPLIT_OUTPUT = 3.5;         // per output of a unit whose sums are added: exchange over the lanes, atomic adds

struct LaunchCost {
  double us;
  int tail_split;             // 0: a pair per tile; otherwise one pair per two SMs, the tiles of the last wave in this many slices
};
// Time of a launch of `tiles` tiles in ns slices of the batch: waves of `slots` pairs, the last one with fewer pairs.
static LaunchCost launch_cost(const UnitCost& c, long long tiles, int B, double T, int slots, int ns, int outputs, double out_bytes, bool may_persist) {
  auto unit = [&](long long examples, double busy) {
    const double ex = T * (c.token_lo + (c.token_hi - c.token_lo) * busy) + c.example;
    return examples * (ex > c.example_min ? ex : c.example_min);
  };
  const long long units = tiles * ns, full = units / slots, rest = units % slots, per = ((long long)B + ns - 1) / ns;
  const double fixed = c.fixed + (ns > 1 ? SPLIT_FIXED : 0.0), last = (double)rest / slots;
  LaunchCost best = {full * (unit(per, 1.0) + fixed) + (rest ? unit(per, last) + fixed : 0.0) + (ns > 1 ? out_bytes / ZERO_BYTES_PER_US : 0.0), 0};
  if (!may_persist || ns > 1 || tiles <= slots) return best;
  const double whole = full * (unit(per, 1.0) * PERSIST_DRIFT + c.fixed - PERSIST_SAVES) + PERSIST_SAVES;
  const double plain = whole + (rest ? unit(per, last) + c.fixed - PERSIST_SAVES : 0.0);
  if (plain < best.us) best = {plain, 1};
  // the last wave's tiles in slices, as many as leave one unit to a pair
  const int k = rest ? (int)std::min<long long>(slots / rest, B) : 1;
  if (k > 1) {
    const double split = whole + unit(((long long)B + k - 1) / k, last * k) + c.fixed - PERSIST_SAVES + outputs * TAIL_SPLIT_OUTPUT;
    if (split < best.us) best = {split, k};
  }
  return best;
}
struct TilePlan {
  int choice, ns;             // index into the candidates, batch slices
  int tail_split;             // as in LaunchCost
};
// The cheapest of the candidate kernels and slice counts.
static TilePlan plan_tiles(const UnitCost* cand, int n_cand, int B, double T, int d_in, int d_out, int slots, int max_split, int outputs,
                           bool may_persist = false) {
  TilePlan best = {0, 1, 0};
  double best_cost = 1e300;
  const long long pairs_m = ((long long)d_out + TC_PAIR_M - 1) / TC_PAIR_M;
  const double out_bytes = 4.0 * outputs * d_in * d_out;
  for (int k = 0; k < n_cand; ++k) {
    const long long tiles = pairs_m * ((d_in + cand[k].nt - 1) / cand[k].nt);
    for (int ns = 1; ns <= max_split && ns <= B && (ns == 1 || tiles * (ns - 1) < 16ll * slots); ++ns) {
      const LaunchCost cost = launch_cost(cand[k], tiles, B, T, slots, ns, outputs, out_bytes, may_persist);
      if (cost.us < best_cost * 0.995) { best_cost = cost.us; best = {k, ns, cost.tail_split}; }
    }
  }
  return best;
}

// Pair rows per band of the tile order (tc_tile_of_pair).  Thread blocks start in the order of their index, `slots`
// CTA pairs at a time, the batch slices one after the other; such a wave streams, for every example of its slice, the dY
// panels of the pair rows and the X panels of the column tiles it touches, and between two waves the batch has passed
// through L2.  So the bytes a launch reads from HBM follow the sum over waves of (pair rows x 256 + column tiles x nt):
// measured on the 8192 x 2048 layer with 256 sequences of 1024 tokens in five slices, 18.5 GB with bands of 8 pair rows, which the
// waves cut unevenly there, against 13.0 GB with bands of 1 (the model gives 2.54 and 1.88 times the operands' size).
// The candidates are walked on the host; the previous default is kept unless another band saves more than 3 %.
static int choose_band(int pairs_m, int tiles_n, int nt, int nsplit, int slots) {
  const int fallback = pairs_m < TC_BAND ? pairs_m : TC_BAND;
  const long long total = (long long)pairs_m * tiles_n;
  if (slots < 1 || pairs_m <= 1 || total * nsplit <= slots) return fallback;       // one wave: the order does not matter
  struct Key { int pairs_m, tiles_n, nt, nsplit, slots, band; };
  thread_local Key cache[16] = {};
  thread_local int cache_next = 0;
  for (const Key& k : cache)
    if (k.band > 0 && k.pairs_m == pairs_m && k.tiles_n == tiles_n && k.nt == nt && k.nsplit == nsplit && k.slots == slots) return k.band;
  // units walked per candidate: the whole launch, or its first 16 Ki thread-block pairs (over 200 waves; the pattern repeats)
  const long long units = total * nsplit < (1ll << 14) ? total * nsplit : (1ll << 14);
  thread_local std::vector<int> row_seen, col_seen;
  row_seen.assign((size_t)pairs_m, -1);
  col_seen.assign((size_t)tiles_n, -1);
  static const int candidates[] = {TC_BAND, 1, 2, 3, 4, 6, 12, 16};
  double best_cost = 0.0, fallback_cost = 0.0;
  int best = fallback;
  for (int band : candidates) {
    if (band > pairs_m) band = pairs_m;
    std::fill(row_seen.begin(), row_seen.end(), -1);
    std::fill(col_seen.begin(), col_seen.end(), -1);
    const long long per_band = (long long)band * tiles_n;
    double cost = 0.0;
    for (long long u = 0; u < units; ++u) {
      const int wave = (int)(u / slots);
      const long long pair_id = u % total;
      const int b = (int)(pair_id / per_band);
      const int r = (int)(pair_id - (long long)b * per_band);
      const int rows = band < pairs_m - b * band ? band : pairs_m - b * band;
      const int tile_n = r / rows, pair_row = b * band + (r - tile_n * rows);
      if (row_seen[pair_row] != wave) { row_seen[pair_row] = wave; cost += TC_PAIR_M; }
      if (col_seen[tile_n] != wave) { col_seen[tile_n] = wave; cost += nt; }
    }
    if (band == fallback) fallback_cost = cost;
    if (best_cost == 0.0 || cost < best_cost) { best_cost = cost; best = band; }
  }
  if (fallback_cost > 0.0 && best_cost > 0.97 * fallback_cost) best = fallback;
  cache[cache_next] = Key{pairs_m, tiles_n, nt, nsplit, slots, best};
  cache_next = (cache_next + 1) % 16;
  return best;
}

static pe_status_t zero_outputs(float* a, float* b, size_t bytes, cudaStream_t st) {
  if (a && cudaMemsetAsync(a, 0, bytes, st) != cudaSuccess) { cudaGetLastError(); return PE_ERR_CUDA; }
  if (b && cudaMemsetAsync(b, 0, bytes, st) != cudaSuccess) { cudaGetLastError(); return PE_ERR_CUDA; }
  return PE_OK;
}

// Launches `kernel` as a programmatic dependent of the kernel before it in the stream (every kernel launched this way waits for
// that one to complete before it touches what others may have written: griddep_wait).
template <typename Kernel, typename... Args>
static pe_status_t launch_dependent(Kernel kernel, dim3 grid, int threads, int smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = (size_t)smem; cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr; cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, kernel, args...) != cudaSuccess) { cudaGetLastError(); return PE_ERR_CUDA; }
  return check_launch();
}
// Zeroes up to three [d_out, d_in] outputs with a kernel that lets its successor start when everything older has completed: the successor's
// blocks follow on each SM as the zeroing block leaves it.  A programmatic dependent itself: against ordinary launches 1024 x 32 x 1024^2, both outputs,
// 113 -> 110, 64 x 32 x 256 x 4096 18.6 -> 16.2 us (25 layers with MicroAdam 1597 -> 1576, which is within the runs' spread).  early: the successor starts at once and has to wait for it before anything else (what came
// before may still be running), worth it where there is little to zero: the norms of 64 x 256 x 512 x 2048 36.1 -> 32.6 us.
// Shared memory that these kernels do not use, so that an SM takes one block: as dependents they would else crowd the SMs that become free first, and
// zero 8 MB from there (64 x 256 x 512 x 2048, three statistics, calls one after the other, 47.2 us against 43.4; 45.2 as ordinary launches).
constexpr int ZERO_SMEM = 120 * 1024;
template <typename Kernel>
static pe_status_t one_block_per_sm(DeviceInfo* di, int slot, Kernel kernel) {
  std::lock_guard<std::mutex> lock(g_dev_mutex);
  if (!di->tc_attr_set[slot]) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ZERO_SMEM) != cudaSuccess) { cudaGetLastError(); return PE_ERR_CUDA; }
    di->tc_attr_set[slot] = true;
  }
  return PE_OK;
}
static pe_status_t zero_for_split(DeviceInfo* di, float* a, float* b, size_t n, cudaStream_t st, float* c = nullptr,
                                  unsigned int* counters = nullptr, int n_counters = 0, bool early = false) {
  float* first = a ? a : b;
  float* second = a ? b : nullptr;
  if (!first) return PE_OK;
  long long blocks = ((long long)(n / 4) + 255) / 256;
  if (blocks > di->sm_count) blocks = di->sm_count;   // few blocks: the dependent kernel needs the SMs
  const dim3 grid((int)(blocks < 1 ? 1 : blocks));
  float4 *const o1 = reinterpret_cast<float4*>(first), *const o2 = reinterpret_cast<float4*>(second), *const o3 = reinterpret_cast<float4*>(c);
  if (!early) {
    const pe_status_t rc = one_block_per_sm(di, 5, zero_outputs_kernel);
    if (rc != PE_OK) return rc;
  }
  return launch_dependent(zero_outputs_kernel, grid, 256, early ? 0 : ZERO_SMEM, st, o1, o2, o3, (long long)n, counters, n_counters, early ? 1 : 0);
}

// mxt, myt: the maps of the zero-padded tail groups of a packed batch (RAGGED); any valid map otherwise.
template <int PHI, bool TF32, int NT, int MEAN, int BKT = tc_default_bk(TF32, NT), bool RAGGED = false, int OPT = OPT_NONE, bool F8 = false, bool CHUNKED = false, bool PERSIST = false, bool PARTS = false>
static pe_status_t launch_tc_inst(DeviceInfo* di, int slot, const CUtensorMap& mx, const CUtensorMap& my, const CUtensorMap& mm,
                                  const CUtensorMap& ms, const CUtensorMap& msgn, const TcParams& p, dim3 grid, cudaStream_t st,
                                  const CUtensorMap* mxt = nullptr, const CUtensorMap* myt = nullptr, const FusedOpt* opt = nullptr) {
  constexpr int smem = TcOperand<TF32, NT, BKT, F8>::SMEM_BYTES;
  {
    std::lock_guard<std::mutex> lock(g_dev_mutex);
    if (!di->tc_attr_set[slot]) {
      if (cudaFuncSetAttribute(tc_stats_kernel<PHI, TF32, NT, MEAN, BKT, RAGGED, OPT, F8, CHUNKED, PERSIST, PARTS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) {
        cudaGetLastError();
        return PE_ERR_CUDA;
      }
      di->tc_attr_set[slot] = true;
    }
  }
  return launch_dependent(tc_stats_kernel<PHI, TF32, NT, MEAN, BKT, RAGGED, OPT, F8, CHUNKED, PERSIST, PARTS>, grid, TC_THREADS, smem, st, mx, my, mm, ms, msgn,
                            mxt ? *mxt : mx, myt ? *myt : my, p, opt ? *opt : FusedOpt{});
}

// The same with one tile per pair, or (persist) one pair per two SMs that walks over the tiles.
template <int PHI, int NT, int MEAN, int BKT = tc_default_bk(false, NT), bool CHUNKED = false>
static pe_status_t launch_tc_tiles(DeviceInfo* di, int slot, bool persist, const CUtensorMap& mx, const CUtensorMap& my, const CUtensorMap& mm,
                                   const CUtensorMap& ms, const CUtensorMap& msgn, const TcParams& p, dim3 grid, cudaStream_t st) {
  if (!persist) return launch_tc_inst<PHI, false, NT, MEAN, BKT, false, OPT_NONE, false, CHUNKED>(di, slot, mx, my, mm, ms, msgn, p, grid, st);
  grid.x = 2 * (di->sm_count / 2);
  return launch_tc_inst<PHI, false, NT, MEAN, BKT, false, OPT_NONE, false, CHUNKED, true>(di, 32 + slot, mx, my, mm, ms, msgn, p, grid, st);
}

// What makes the operands of a launch (a layout kernel): called with the outputs to zero by the way.
using LayoutStep = std::function<pe_status_t(const LayoutZero&)>;
static bool any_output(const LayoutZero& z) { return z.out[0] || z.out[1] || z.out[2]; }

// Statistics of short sequences (T <= SHORT_T).  out_mean, out_square, out_sign: those wanted; out_mean and out_sign with or without
// out_square, out_square with or without out_mean.
// Whole tiles per pair or slices of the batch: by time, fitted to sweeps of both over layers from 512 x 512 to 4096 x 4096 (both outputs, 2000 x 3 x 512^2, 8
// tiles in 1, 8, 9, 10 and 18 slices: 366, 56, 52, 86 and 56 us; 300 x 16 x 2048^2, 128 tiles: 120 whole, 122 with the last wave's in four slices, three
// statistics 258 and 246).
struct ShortCost {
  double example, fixed, add;      // us per example of a tile, per tile, more for a tile whose sums are added
};
static ShortCost short_cost(bool mean, bool square, bool sign) {
  if (mean && square && sign) return {0.45, 2.2, 3.2};
  if (mean && sign) return {0.345, 1.5, 2.3};
  if (mean) return {0.19, 1.5, 2.3};
  return sign ? ShortCost{0.28, 1.0, 1.5} : ShortCost{0.155, 1.0, 1.5};
}
// Rounding error of the sums, as variances up to a factor: p examples at a time in order, in runs of r summed by themselves, and `parts` such sums added
// in order.  Terms of either sign (G_b): p + parts; terms of one sign (G_b^2): r^2 + p^2 / r + B parts, or p^2 + B parts without runs.  (1395 x 5 x
// 1696 x 1336, square alone, p = 1395: errors of 5.2e-7, 1.32e-7, 9.5e-8 and 7.3e-8 without runs and in runs of 16, 32 and 64.)
static double mean_rounding(double p, double parts) { return p + parts; }
static double square_rounding(int B, double p, double r, double parts) { return (r < p ? r * r + p * p / r : p * p) + B * parts; }
// The sums' lengths are bounded by those of the plan that a pair per tile and slice would have, at these costs (one, two sums, three), so that a
// plan that takes fewer slices for the time's sake does not lose precision: 2021 x 24 x 2336 x 1728, mean and square, whole tiles 716 us with errors of 6.6e-7
// and 5.3e-7, in five slices 733 us, 3.7e-7 and 1.5e-7; 1545 x 4 x 1624 x 2296, three statistics, 1157 and 1184.  It decides on 1 to 3 % of the layers from
// 256 x 256 to 4096 x 4096.
constexpr UnitCost SUMS_OF_ONE = COST_STAT;
constexpr UnitCost SUMS_OF_TWO = {128, 0.05 / 32, 0.10 / 32, 0.0, 0.245, 8.3};
constexpr UnitCost SUMS_OF_THREE = {128, 0.05 / 32, 0.10 / 32, 0.0, 0.54, 9.5};
struct ShortPlan {
  int whole, split;                // tiles that a pair takes over the whole batch; slices of the batch for each of the others
  int run;                         // the square alone: examples that are summed by themselves, a power of two
};
// Every pair takes whole tiles in turn; the tiles of a last partial wave, or all of them where that is cheaper, go to several
// pairs each, by slices of the batch.  Three statistics: a unit, whole tile or slice, has no more examples than its 16-bit counts of signs hold.
static ShortPlan plan_short(bool mean, bool square, bool sign, int B, int T, int d_in, int d_out, int slots, bool accumulate, bool may_persist) {
  const ShortCost c = short_cost(mean, square, sign);
  const bool counts = mean && square && sign, runs = square && !mean;
  const long long tiles = (((long long)d_in + SHORT_NT - 1) / SHORT_NT) * (((long long)d_out + TC_PAIR_M - 1) / TC_PAIR_M);
  ShortPlan plan = {0, 1, SHORT_RUN_MIN};
  double most_mean = 1e300, most_square = 1e300;
  if (mean || square) {
    const UnitCost& cost = counts ? SUMS_OF_THREE : mean ? SUMS_OF_TWO : SUMS_OF_ONE;
    const int outputs = (mean ? 1 : 0) + (square ? 1 : 0) + (sign ? 1 : 0);
    int ns = plan_tiles(&cost, 1, B, T, d_in, d_out, slots, std::max(16, slots), outputs, may_persist && !(counts && B > TC_SIGN_COUNT_MAX)).ns;
    if (counts && (B + ns - 1) / ns > TC_SIGN_COUNT_MAX) ns = (B + TC_SIGN_COUNT_MAX - 1) / TC_SIGN_COUNT_MAX;
    const double p = (B + ns - 1) / ns, parts = ns > 1 ? ns : 0;
    if (mean) most_mean = mean_rounding(p, parts);
    if (square) most_square = square_rounding(B, p, p, parts);
    plan.split = ns;               // (where nothing below is good enough)
  }
  auto run_of = [&](double p, double parts) {        // the longest runs that round within 2 % as little as any
    double least = 1e300;
    for (int r = SHORT_RUN_MIN; r <= SHORT_RUN_MAX; r *= 2) least = std::min(least, square_rounding(B, p, r, parts));
    int r = SHORT_RUN_MAX;
    while (r > SHORT_RUN_MIN && square_rounding(B, p, r, parts) > 1.02 * least) r /= 2;
    return r;
  };
  auto good = [&](double p, double parts) {
    return (!counts || p <= TC_SIGN_COUNT_MAX) && (!mean || mean_rounding(p, parts) <= most_mean) &&
           (!square || square_rounding(B, p, runs ? run_of(p, parts) : p, parts) <= most_square);
  };
  double best = 1e300;
  for (int pass = 0; pass < 2; ++pass) {
    const long long w = pass == 0 ? 0 : tiles - tiles % slots, rest = tiles - w;
    if (pass == 1 && (w == 0 || rest == 0 || !good(B, 0))) break;
    for (int k = 1; k <= B && k <= 4 * slots && (k == 1 || rest * (k - 1) < 16ll * slots); ++k) {
      const double per = (double)((B + k - 1) / k);
      const bool add = k > 1 || accumulate;
      const double us = (double)(w / slots) * (B * c.example + c.fixed) +
                        (double)((rest * k + slots - 1) / slots) * (per * c.example + c.fixed + (add ? c.add : 0.0)) + (add && !accumulate ? 2.0 : 0.0);
      if (us < best * 0.995 && good(per, k > 1 ? k : 0)) { best = us; plan.whole = (int)(k == 1 ? tiles : w); plan.split = k; }
    }
  }
  if (runs) plan.run = plan.whole > 0 ? run_of(B, 0) : run_of((B + plan.split - 1) / plan.split, plan.split > 1 ? plan.split : 0);
  return plan;
}
static pe_status_t launch_short(DeviceInfo* di, const void* X, const void* dY, int B, int T, int d_in, int d_out, float* out_mean, float* out_square,
                                float* out_sign, cudaStream_t st, bool accumulate, int pitch_x, int pitch_y, const LayoutStep& before) {
  CUtensorMap mx, my;
  pe_status_t rc = make_operand_map(&mx, X, B, T, d_in, false, 64, SHORT_T, false, SHORT_G, pitch_x);
  if (rc == PE_OK) rc = make_operand_map(&my, dY, B, T, d_out, false, 64, SHORT_T, false, SHORT_G, pitch_y);
  if (rc != PE_OK) return rc;
  const int tiles_n = (d_in + SHORT_NT - 1) / SHORT_NT, pairs_m = (d_out + TC_PAIR_M - 1) / TC_PAIR_M;
  if ((long long)tiles_n * pairs_m > (1ll << 29)) return PE_ERR_DIM;
  const long long tiles = (long long)tiles_n * pairs_m;
  const int slots = di->sm_count / 2 > 0 ? di->sm_count / 2 : 1;
  const ShortPlan plan = plan_short(out_mean, out_square, out_sign, B, T, d_in, d_out, slots, accumulate,
                                    !accumulate && d_in % 8 == 0 && aligned(out_mean, 32) && aligned(out_square, 32) && aligned(out_sign, 32));
  const int whole = plan.whole, split = plan.split;
  TcParams p{};
  p.B = B; p.T = T; p.d_in = d_in; p.d_out = d_out; p.accumulate = accumulate ? 1 : 0;
  p.pairs_m = pairs_m; p.tiles_n = tiles_n; p.band = choose_band(pairs_m, tiles_n, SHORT_NT, whole == 0 ? split : 1, slots);
  p.whole_tiles = whole; p.tail_split = split; p.sum_run = plan.run;
  p.scalar_out = d_in % 4 != 0 ? 1 : 0;
  CUtensorMap mm = mx, msq = mx, msgn = mx;           // an output that is not wanted gets a map that is never used
  if (!p.scalar_out) {
    if (out_mean) rc = make_output_map(&mm, out_mean, d_in, d_out);
    if (rc == PE_OK && out_square) rc = make_output_map(&msq, out_square, d_in, d_out);
    if (rc == PE_OK && out_sign) rc = make_output_map(&msgn, out_sign, d_in, d_out);
    if (rc != PE_OK) return rc;
  }
  p.out_mean = out_mean; p.out_stat = out_square; p.out_sign = out_sign; p.dev_status = di->status_ptr;
  const bool to_zero = split > 1 && !accumulate;
  const bool zero_tail = to_zero && whole > 0;           // the sliced tiles alone, behind a layout kernel too: 49 x 2 x 1120 x 5035 134 -> 45 us
  p.wait_at_start = !to_zero || (before && !zero_tail) ? 1 : 0;
  if (before) {
    LayoutZero zero = {{nullptr, nullptr, nullptr}, (long long)d_in * d_out};
    if (to_zero && !zero_tail) { zero.out[0] = out_mean; zero.out[1] = out_square; zero.out[2] = out_sign; }
    if ((rc = before(zero)) != PE_OK) return rc;
  }
  if (zero_tail) {
    rc = one_block_per_sm(di, 24, zero_tail_tiles_kernel);
    if (rc == PE_OK) rc = launch_dependent(zero_tail_tiles_kernel, dim3(di->sm_count), 256, ZERO_SMEM, st, p, SHORT_NT);
  } else if (to_zero && !before) {
    float* const outs[3] = {out_mean, out_square, out_sign};
    float* list[3] = {nullptr, nullptr, nullptr};
    int n = 0;
    for (float* o : outs)
      if (o) list[n++] = o;
    rc = zero_for_split(di, list[0], list[1], (size_t)d_in * d_out, st, list[2]);
  }
  if (rc != PE_OK) return rc;
  const long long units = whole + (tiles - whole) * split;
  const dim3 grid((unsigned)(2 * std::min<long long>(slots, units)));
  auto run = [&](auto kernel, int slot) {
    {
      std::lock_guard<std::mutex> lock(g_dev_mutex);
      if (!di->tc_attr_set[slot]) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SHORT_SMEM_BYTES) != cudaSuccess) { cudaGetLastError(); return PE_ERR_CUDA; }
        di->tc_attr_set[slot] = true;
      }
    }
    return launch_dependent(kernel, grid, TC_THREADS, SHORT_SMEM_BYTES, st, mx, my, mm, msq, msgn, p);
  };
  if (out_sign && out_mean && out_square) return run(short_stats_kernel<true, true, true>, 8);
  if (out_sign && out_mean) return run(short_stats_kernel<true, false, true>, 9);
  if (out_sign) return run(short_stats_kernel<false, false, true>, 27);
  if (out_mean) return run(short_stats_kernel<true, true, false>, 40);
  return run(short_stats_kernel<false, true, false>, 41);
}

// Tensor-core launch.  per_example = 0 runs the plain contraction over all B*T rows (its result goes
// to whichever of out_mean / out_stat is not NULL).  With per_example = 1 and both outputs wanted the
// pair tile is 256 x 128 (two running sums per thread); with only out_stat it is 256 x 256.
static pe_status_t launch_tc(DeviceInfo* di, const void* X, const void* dY, int B, int T, int d_in, int d_out, int phi,
                             int per_example, float* out_mean, float* out_stat, cudaStream_t st, bool half_ops = false,
                             float* out_sign = nullptr, bool accumulate = false, const float* sq_norms = nullptr, float clip_norm = 0.f,
                             int pitch_x = 0, int pitch_y = 0, bool chunked = false, const float* scale_x = nullptr,
                             const float* scale_y = nullptr, const LayoutStep& before = nullptr) {
  const bool triple = out_sign != nullptr;       // mean + square + sign in one pass (phi = square, all three outputs given)
  const bool both = per_example && ((out_mean && out_stat) || chunked);
  const bool runs = chunked && T > TC_CHUNK_TOKENS;     // several accumulators per example
  const int forced = g_path.load();
  if (per_example && T <= SHORT_T && forced != PE_PATH_TENSOR_WIDE && (phi == PE_PHI_SQUARE || phi == PE_PHI_SIGN))
    return launch_short(di, X, dY, B, T, d_in, d_out, out_mean, phi == PE_PHI_SQUARE ? out_stat : nullptr, phi == PE_PHI_SIGN ? out_stat : out_sign, st,
                        accumulate, pitch_x, pitch_y, before);
  const int slots = di->sm_count / 2 > 0 ? di->sm_count / 2 : 1, max_split = std::max(16, slots);
  // Tile and batch slices by estimated time.  Both outputs: 256 x 192 or 256 x 128 (22 % more operand traffic per flop, but
  // less padding and more even waves on some layers: 64 x 256 x 512 x 32768 528 us against 497).
  UnitCost cand[2];
  int n_cand = 0;
  bool cand_wide[2] = {false, false};
  if (both) {
    if (forced != PE_PATH_TENSOR_NARROW && !runs) { cand_wide[n_cand] = true; cand[n_cand++] = triple ? COST_ALL_192 : COST_BOTH_192; }
    if (forced != PE_PATH_TENSOR_WIDE || n_cand == 0) cand[n_cand++] = triple ? COST_ALL_128 : COST_BOTH_128;
  } else {
    cand[n_cand++] = !per_example ? COST_PLAIN : phi == PE_PHI_SIGN ? COST_SIGN : COST_STAT;
  }
  // Several tiles per pair: rows of whole 32-byte sectors (others, written in parts of sectors, 12 x 100 x 900 x 20001, three statistics: 160 us
  // against 252), and 16-bit counts of examples.
  const bool may_persist = per_example && !accumulate && d_in % 8 == 0 && aligned(out_mean, 32) && aligned(out_stat, 32) && aligned(out_sign, 32) &&
                           !(triple && B > TC_SIGN_COUNT_MAX);
  const TilePlan plan = plan_tiles(cand, n_cand, B, T, d_in, d_out, slots, max_split, (out_mean ? 1 : 0) + (out_stat ? 1 : 0) + (out_sign ? 1 : 0), may_persist);
  const long long pad192 = (long long)((d_in + 191) / 192) * 192, pad128 = (long long)((d_in + 127) / 128) * 128;
  const bool mean_tmem = both && !triple && !runs && forced != PE_PATH_TENSOR_NARROW && forced != PE_PATH_TENSOR_WIDE && T >= TC_MEAN_TMEM_MIN_T &&
                         pad192 * 100 > pad128 * (100 + TC_WIDE_MAX_PAD_PERCENT);
  const bool wide = both && !mean_tmem && cand_wide[plan.choice];
  const bool mean_regs = both && !mean_tmem;
  const int nt = mean_regs ? (wide ? 192 : 128) : 256;
  const int box_feats = TcOperand<false, 256>::BOX_FEATS;
  const int box_tokens = tc_default_bk(false, nt);
  CUtensorMap mx, my;
  pe_status_t rc = wide ? make_operand_map(&mx, X, B, T, d_in, false, TcOperand<false, 192>::B_BOX_FEATS, box_tokens, true, 1, pitch_x)
                        : make_operand_map(&mx, X, B, T, d_in, false, box_feats, box_tokens, false, 1, pitch_x);
  if (rc != PE_OK) return rc;
  rc = make_operand_map(&my, dY, B, T, d_out, false, box_feats, box_tokens, false, 1, pitch_y);
  if (rc != PE_OK) return rc;
  // an output that is not wanted gets the other one's map and is never used; rows that are no 16-byte multiples cannot be
  // described by a map at all and are written without one (scalar_out)
  const bool scalar_out = d_in % 4 != 0;
  CUtensorMap mm = mx, ms = mx, msgn = mx;
  if (!scalar_out) {
    rc = make_output_map(&mm, out_mean ? out_mean : out_stat, d_in, d_out);
    if (rc == PE_OK) rc = make_output_map(&ms, out_stat ? out_stat : out_mean, d_in, d_out);
    if (rc == PE_OK && triple) rc = make_output_map(&msgn, out_sign, d_in, d_out);
    if (rc != PE_OK) return rc;
  }
  const int tiles_n = (d_in + nt - 1) / nt, pairs_m = (d_out + TC_PAIR_M - 1) / TC_PAIR_M;
  if ((long long)tiles_n * pairs_m > (1ll << 29)) return PE_ERR_DIM;
  int ns = mean_tmem ? plan_tiles(&COST_STAT, 1, B, T, d_in, d_out, slots, max_split, 2).ns : plan.ns;
  if (triple && (B + ns - 1) / ns > TC_SIGN_COUNT_MAX) ns = (B + TC_SIGN_COUNT_MAX - 1) / TC_SIGN_COUNT_MAX;   // 16-bit sign counters
  const bool to_zero = ns > 1 && !accumulate;
  if (before) {
    LayoutZero zero = {{nullptr, nullptr, nullptr}, (long long)d_in * d_out};
    if (to_zero) { zero.out[0] = out_mean; zero.out[1] = out_stat; zero.out[2] = out_sign; }
    rc = before(zero);
  } else if (to_zero) {
    rc = zero_for_split(di, out_mean, out_stat, (size_t)d_in * d_out, st, out_sign);
  }
  if (rc != PE_OK) return rc;
  TcParams p{};
  p.B = B; p.T = T; p.d_in = d_in; p.d_out = d_out; p.nsplit = ns; p.per_example = per_example; p.half_operands = half_ops ? 1 : 0;
  p.accumulate = accumulate ? 1 : 0; p.scalar_out = scalar_out ? 1 : 0; p.wait_at_start = !to_zero || before ? 1 : 0;
  p.pairs_m = pairs_m; p.tiles_n = tiles_n; p.band = choose_band(pairs_m, tiles_n, nt, ns, di->sm_count / 2);
  p.out_mean = out_mean; p.out_stat = out_stat; p.out_sign = out_sign; p.out_norms = nullptr; p.dev_status = di->status_ptr;
  p.seq_offsets = nullptr; p.sq_norms = sq_norms; p.clip_norm = clip_norm; p.scale_x = scale_x; p.scale_y = scale_y;
  dim3 grid(2 * pairs_m * tiles_n, 1, ns);
  const bool persist = plan.tail_split > 0 && ns == 1 && !mean_tmem;
  if (persist) {
    const int tiles = pairs_m * tiles_n;
    p.tail_split = plan.tail_split;
    p.whole_tiles = plan.tail_split > 1 ? tiles - tiles % slots : tiles;
    if (plan.tail_split > 1) {
      p.wait_at_start = 0;
      rc = one_block_per_sm(di, 24, zero_tail_tiles_kernel);
      if (rc == PE_OK) rc = launch_dependent(zero_tail_tiles_kernel, dim3(di->sm_count), 256, ZERO_SMEM, st, p, nt);
      if (rc != PE_OK) return rc;
    }
  }
  if (phi == PHI_UNSCALE) return launch_tc_tiles<4, 256, MEAN_NONE>(di, 30, persist, mx, my, mm, ms, msgn, p, grid, st);
  if (phi == PHI_CLIP_SCALE) return launch_tc_tiles<3, 256, MEAN_NONE>(di, 14, persist, mx, my, mm, ms, msgn, p, grid, st);
  if (runs) {
    if (phi == PE_PHI_SQUARE) return launch_tc_tiles<1, 128, MEAN_REGS, 128, true>(di, 28, persist, mx, my, mm, ms, msgn, p, grid, st);
    return launch_tc_tiles<2, 128, MEAN_REGS, 128, true>(di, 29, persist, mx, my, mm, ms, msgn, p, grid, st);
  }
  if (triple && wide) return launch_tc_tiles<1, 192, MEAN_HYBRID_SIGN>(di, 26, persist, mx, my, mm, ms, msgn, p, grid, st);
  if (triple) return launch_tc_tiles<1, 128, MEAN_REGS_SIGN>(di, 10, persist, mx, my, mm, ms, msgn, p, grid, st);
  if (!per_example) return launch_tc_inst<0, false, 256, MEAN_NONE>(di, 4, mx, my, mm, ms, msgn, p, grid, st);
  if (wide) {
    if (phi == PE_PHI_SQUARE) return launch_tc_tiles<1, 192, MEAN_REGS>(di, 12, persist, mx, my, mm, ms, msgn, p, grid, st);
    return launch_tc_tiles<2, 192, MEAN_REGS>(di, 13, persist, mx, my, mm, ms, msgn, p, grid, st);
  }
  if (mean_regs) {
    if (phi == PE_PHI_SQUARE) return launch_tc_tiles<1, 128, MEAN_REGS>(di, 0, persist, mx, my, mm, ms, msgn, p, grid, st);
    return launch_tc_tiles<2, 128, MEAN_REGS>(di, 1, persist, mx, my, mm, ms, msgn, p, grid, st);
  }
  if (both) {
    if (phi == PE_PHI_SQUARE) return launch_tc_inst<1, false, 256, MEAN_TMEM>(di, 6, mx, my, mm, ms, msgn, p, grid, st);
    return launch_tc_inst<2, false, 256, MEAN_TMEM>(di, 7, mx, my, mm, ms, msgn, p, grid, st);
  }
  if (phi == PE_PHI_SQUARE) return launch_tc_tiles<1, 256, MEAN_NONE>(di, 2, persist, mx, my, mm, ms, msgn, p, grid, st);
  return launch_tc_tiles<2, 256, MEAN_NONE>(di, 3, persist, mx, my, mm, ms, msgn, p, grid, st);
}

// Example norms: examples > 0: one pair per two SMs that takes every slots-th of the tiles' slices of so many examples, since nothing is
// written out at the end of a tile: no pair is idle in a last wave.  16 x 512 x 2048 x 4096 (128 tiles) 95 -> 88 us, 32 x 512 x 1024 x 4096 97 -> 92.
// 0: a pair per tile and slice.
struct NormsPlan {
  int slices, examples;
  int order_slices;              // slices that the tile order is chosen for: a walk's one like the other, so that another B takes no new search
};
static NormsPlan plan_norms(int B, int T, int d_in, int d_out, int slots) {
  const long long tiles = (((long long)d_in + 255) / 256) * (((long long)d_out + TC_PAIR_M - 1) / TC_PAIR_M);
  NormsPlan plan = {plan_tiles(&COST_NORMS, 1, B, T, d_in, d_out, slots, std::max(16, slots), 0).ns, 0, 0};
  double best = launch_cost(COST_NORMS, tiles, B, T, slots, plan.slices, 0, 0.0, false).us - (plan.slices > 1 ? SPLIT_FIXED : 0.0);
  // (beyond 64 examples the cost of a unit is less than one per cent, and more slices only even the waves out)
  for (int examples = 1; examples <= B && examples <= 64; ++examples) {
    const long long slices = ((long long)B + examples - 1) / examples, rounds = (tiles * slices + slots - 1) / slots;
    if (tiles * slices >= (1ll << 30)) continue;
    if (tiles * slices < slots) break;
    const double us = rounds * (examples * std::max(T * COST_NORMS.token_hi, COST_NORMS.example_min) + NORMS_UNIT) + COST_NORMS.fixed;
    if (us < best * 0.99) { best = us; plan.slices = (int)slices; plan.examples = examples; }
  }
  plan.order_slices = plan.examples == 0 ? plan.slices : 1;
  return plan;
}

// Per-example squared norms on the tensor cores: the statistic-only 256 x 256 schedule, but every
// example's tile is reduced to one number and added to norms[b] (zeroed by the caller of this function).
static pe_status_t launch_tc_norms(DeviceInfo* di, const void* X, const void* dY, int B, int T, int d_in, int d_out, float* norms,
                                   cudaStream_t st) {
  CUtensorMap mx, my;
  const int box_feats = TcOperand<false, 256>::BOX_FEATS, box_tokens = tc_default_bk(false, 256);
  pe_status_t rc = make_operand_map(&mx, X, B, T, d_in, false, box_feats, box_tokens);
  if (rc != PE_OK) return rc;
  rc = make_operand_map(&my, dY, B, T, d_out, false, box_feats, box_tokens);
  if (rc != PE_OK) return rc;
  const int tiles_n = (d_in + 255) / 256, pairs_m = (d_out + TC_PAIR_M - 1) / TC_PAIR_M;
  if ((long long)tiles_n * pairs_m > (1ll << 29)) return PE_ERR_DIM;
  const int slots = di->sm_count / 2 > 0 ? di->sm_count / 2 : 1;
  const NormsPlan plan = plan_norms(B, T, d_in, d_out, slots);
  const int ns = plan.slices;
  const bool walk = plan.examples > 0;
  TcParams p{};
  p.B = B; p.T = T; p.d_in = d_in; p.d_out = d_out; p.nsplit = walk ? 1 : ns; p.per_example = 1; p.half_operands = 0;
  p.accumulate = 1;       // no matrix is written
  p.whole_tiles = 0; p.tail_split = ns; p.slice_examples = plan.examples;
  // norms[b] = 0 (by a kernel that overlaps the launch of this one, 16-byte alignment allowing)
  p.wait_at_start = 1;
  rc = aligned(norms, 16) ? zero_for_split(di, norms, nullptr, (size_t)B, st, nullptr, nullptr, 0, true)
                          : zero_outputs(norms, nullptr, (size_t)B * sizeof(float), st);
  if (rc != PE_OK) return rc;
  p.pairs_m = pairs_m; p.tiles_n = tiles_n; p.band = choose_band(pairs_m, tiles_n, 256, plan.order_slices, di->sm_count / 2);
  p.out_mean = nullptr; p.out_stat = nullptr; p.out_sign = nullptr; p.out_norms = norms; p.dev_status = di->status_ptr;
  p.seq_offsets = nullptr; p.sq_norms = nullptr; p.clip_norm = 0.f;
  // the three output maps are never used by this variant: any valid map will do
  if (walk)
    return launch_tc_inst<1, false, 256, MEAN_NORMS, 64, false, OPT_NONE, false, false, true>(di, 32 + 11, mx, my, mx, mx, mx, p, dim3(2 * slots), st);
  return launch_tc_inst<1, false, 256, MEAN_NORMS>(di, 11, mx, my, mx, mx, mx, p, dim3(2 * pairs_m * tiles_n, 1, ns), st);
}

// Tile and batch slices of a SIMT launch: the cheapest by an estimate in microseconds, fitted to sweeps of all tiles and slice
// counts over layers from 48 x 48 to 1100 x 1100 (the choice 5 % above the sweep's best, geometric mean).  A chunk of
// tokens costs its FMAs times the blocks that share the SM, but for a block alone at least that and a latency.
constexpr int SIMT_MAX_D_OUT = 65535 * 128;
struct SimtPlan {
  int tile, slices, cluster;      // tile: index into the five shapes
};
static SimtPlan plan_simt(int sm_count, int mode, bool two_sums, bool exact, int B, int T, int d_in, int d_out) {
  constexpr int HALF = 4;
  static constexpr int rows[5] = {SimtTile84::ROWS, SimtTile44::ROWS, SimtTile22::ROWS, SimtTile11::ROWS, SimtTileHalf<MODE_STATS>::ROWS};
  static constexpr int cols[5] = {SimtTile84::COLS, SimtTile44::COLS, SimtTile22::COLS, SimtTile11::COLS, SimtTileHalf<MODE_STATS>::COLS};
  const int kt[5] = {SimtTile84::KT, SimtTile44::KT, SimtTile22::KT, SimtTile11::KT, mode == MODE_TOKEN ? SimtTileHalf<MODE_TOKEN>::KT : SimtTileHalf<MODE_STATS>::KT};
  static constexpr int per_sm[5] = {2, 2, 3, 4, 4};                           // blocks an SM holds
  static constexpr double chunk_us[5] = {1.95, 0.60, 0.85, 0.80, 0.46};       // a full chunk's FMAs, one block
  static constexpr double latency_us[5] = {0.25, 0.35, 0.45, 0.50, 0.0};
  static constexpr double fold_us[5] = {0.35, 0.10, 0.05, 0.05, 0.0};         // phi and the sums at the end of an example
  const bool by_rows = mode == MODE_TOKEN;                            // what the slices divide: rows or examples
  const long long units = by_rows ? (long long)B * T : B;
  const int loose = (d_in % 4 != 0) + (d_out % 4 != 0);
  // roundings that a sum over the batch goes through: a slice's own examples, the slices of a cluster, the clusters
  auto chain = [&](long long s) { const long long c = std::min<long long>(s, SIMT_MAX_CLUSTER); return (units + s - 1) / s + c + (s + c - 1) / c; };
  SimtPlan best = {0, 1, 1};
  double best_cost = 1e300;
  int other_slices = 1;
  int least = 1;             // slices: sums of all rows are not to grow longer, and with them their rounding error, for the last tile's sake
  for (int k = 0; k < 5; ++k) {
    if (k == HALF) {
      other_slices = best.slices;
      if (by_rows) least = best.slices;
    }
    const long long tiles = (long long)((d_in + cols[k] - 1) / cols[k]) * ((d_out + rows[k] - 1) / rows[k]);
    for (int s = least; s <= 32 && s <= units; s *= 2) {
      const long long blocks = tiles * s, slots = (long long)per_sm[k] * sm_count;
      const long long per = (units + s - 1) / s;
      const double tokens = (double)(by_rows ? per : (long long)T), whole = std::floor(tokens / kt[k]);
      const double rest = (double)(((long long)(tokens - whole * kt[k]) + 7) / 8 * 8) / kt[k];
      double cost;
      if (k == HALF) {
        // whole rounds of blocks, then those that are left: blocks that share an SM take turns, one alone is as long as 1.27
        const double chunk = by_rows ? 2 * chunk_us[k] : chunk_us[k], edge = 0.195 + 0.075 * loose, fold = by_rows ? 0.0 : two_sums ? 0.294 : 0.05;
        auto round = [&](double together) {
          const double share = std::max(together, 1.27);
          return (by_rows ? 1.0 : (double)per) * (((whole + rest) * chunk + fold) * share + (whole + (rest > 0.0 ? 1.0 : 0.0)) * edge) + 4.7;
        };
        const long long most = (blocks + sm_count - 1) / sm_count, left = most % per_sm[k];
        cost = (double)(most / per_sm[k]) * round(per_sm[k]) + (left ? round((double)left) : 0.0) + 1.86 + (s > 1 ? 1.475 : 0.0) + (s > SIMT_MAX_CLUSTER ? 5.0 : 0.0);
        cost *= 0.88;          // (both estimates are high; chosen only where it is the faster one: at 70 layers never more than 2 % behind)
      } else {
        double sharing = (double)std::min<long long>(per_sm[k], (blocks + sm_count - 1) / sm_count);
        if (k == 0 && s >= SIMT_MAX_CLUSTER && blocks <= sm_count) sharing = 1.5;      // clusters of eight are placed densely
        auto chunk = [&](double f) { return std::max(sharing * chunk_us[k] * f, latency_us[k] + chunk_us[k] * f); };
        double walk = whole * chunk(1.0) + (rest > 0.0 ? chunk(rest) : 0.0);
        if (!by_rows) walk = per * (walk + fold_us[k] * sharing);
        const double waves = (double)((blocks + slots - 1) / slots);
        cost = waves * (walk + 2.0) + 1.5 + 0.12 * s + (s > SIMT_MAX_CLUSTER ? 3.0 : 0.0);
      }
      if (cost < best_cost) { best_cost = cost; best = {k, s, s < SIMT_MAX_CLUSTER ? s : SIMT_MAX_CLUSTER}; }
    }
  }
  // Nor are sums over the examples, but for those of signs alone, which are exact: the last tile in more slices, or in as many as the best of the other tiles has (60 x 24 x 900 x 300, both sums: error of
  // the mean 1.23e-7 at 53 us in 4 slices, 1.16e-7 at 56 in 16, 1.16e-7 at 79 on the 128 x 64 tile in 32).
  if (best.tile == HALF && mode == MODE_STATS && !exact) {
    int s = best.slices;
    while (chain(s) > chain(other_slices) && s < 32 && 2ll * s <= units) s *= 2;
    if (chain(s) > chain(other_slices)) s = other_slices;
    best = {HALF, s, s < SIMT_MAX_CLUSTER ? s : SIMT_MAX_CLUSTER};
  }
  if (mode == MODE_NORMS) best.cluster = 1;      // nothing is exchanged
  return best;
}

template <typename TIn, int MODE, class Tile, int SUMS>
static pe_status_t launch_simt_inst(const SimtPlan& plan, const TIn* X, const TIn* dY, int B, int T, int d_in, int d_out, int phi,
                                    float* out_mean, float* out_stat, cudaStream_t st, bool accumulate, int ldx, int ldy, const SimtExtra& ex,
                                    const FusedOpt& opt) {
  auto kernel = simt_stats_kernel<TIn, MODE, Tile, SUMS>;
  constexpr int smem = (MODE == MODE_STATS ? Tile::smem_floats(SUMS) : (2 * Tile::CHUNK > Tile::ROWS * Tile::COLS ? 2 * Tile::CHUNK : Tile::ROWS * Tile::COLS)) * 4;
  if constexpr (smem > 48 * 1024) {
    int dev = 0;
    static std::atomic<bool> attr_set[MAX_DEVICES];
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) { cudaGetLastError(); return PE_ERR_CUDA; }
    if (!attr_set[dev].load(std::memory_order_acquire)) {       // (concurrent first calls set the same value)
      if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) { cudaGetLastError(); return PE_ERR_CUDA; }
      attr_set[dev].store(true, std::memory_order_release);
    }
  }
  // a group of four columns is one load when every row of the operand starts on such a boundary
  const size_t group = 4 * sizeof(TIn);
  const int vec_x = ldx % 4 == 0 && aligned(X, group) ? 1 : 0, vec_y = ldy % 4 == 0 && aligned(dY, group) ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  const long long tiles = (long long)((d_in + Tile::COLS - 1) / Tile::COLS) * ((d_out + Tile::ROWS - 1) / Tile::ROWS);
  if (d_out > SIMT_MAX_D_OUT || tiles >= (1ll << 31)) return PE_ERR_DIM;
  cfg.gridDim = dim3((unsigned)tiles, 1, plan.slices);
  cfg.blockDim = dim3(Tile::THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 1; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = plan.cluster;
  cfg.attrs = &attr; cfg.numAttrs = plan.cluster > 1 ? 1 : 0;
  if (cudaLaunchKernelEx(&cfg, kernel, X, dY, B, T, d_in, d_out, phi, out_mean, out_stat, accumulate ? 1 : 0, plan.cluster, ldx, ldy, vec_x, vec_y, ex, opt) != cudaSuccess) {
    cudaGetLastError();
    return PE_ERR_CUDA;
  }
  return check_launch();
}

template <typename TIn, int MODE>
static pe_status_t launch_simt(DeviceInfo* di, const TIn* X, const TIn* dY, int B, int T, int d_in, int d_out, int phi,
                               float* out_mean, float* out_stat, cudaStream_t st, bool accumulate = false, SimtExtra ex = SimtExtra{},
                               const FusedOpt* opt = nullptr, int pitch_x = 0, int pitch_y = 0) {
  const int ldx = pitch_x ? pitch_x : d_in, ldy = pitch_y ? pitch_y : d_out;
  const bool two_sums = out_mean || (opt && opt->kind == OPT_ADAM);
  SimtPlan plan = plan_simt(di->sm_count, MODE, two_sums, phi == PE_PHI_SIGN && !two_sums, B, T, d_in, d_out);
  if (opt && plan.slices > SIMT_MAX_CLUSTER) plan.slices = SIMT_MAX_CLUSTER;      // a fused update needs the whole batch in one cluster
  if (MODE != MODE_NORMS && plan.slices > plan.cluster && !accumulate) {
    pe_status_t rc = zero_outputs(out_mean, out_stat, (size_t)d_in * d_out * sizeof(float), st);
    if (rc != PE_OK) return rc;
  }
  const FusedOpt o = opt ? *opt : FusedOpt{};
  auto run = [&](auto tile) {
    using Tile = decltype(tile);
    if constexpr (MODE == MODE_STATS) {
      if (two_sums)
        return launch_simt_inst<TIn, MODE, Tile, 2>(plan, X, dY, B, T, d_in, d_out, phi, out_mean, out_stat, st, accumulate, ldx, ldy, ex, o);
    }
    return launch_simt_inst<TIn, MODE, Tile, 1>(plan, X, dY, B, T, d_in, d_out, phi, out_mean, out_stat, st, accumulate, ldx, ldy, ex, o);
  };
  switch (plan.tile) {
    case 0: return run(SimtTile84{});
    case 1: return run(SimtTile44{});
    case 2: return run(SimtTile22{});
    case 4: return run(SimtTileHalf<MODE>{});
    default: return run(SimtTile11{});
  }
}

static int grid_for(long long work_items, int sm_count) {
  long long blocks = (work_items + OPT_THREADS - 1) / OPT_THREADS;
  long long cap = (long long)sm_count * 8;
  if (blocks < 1) blocks = 1;
  return (int)(blocks < cap ? blocks : cap);
}

// The update kernels.  skip_if_set: NULL, or the device status word that makes the step leave the parameters alone.
static pe_status_t launch_microadam(DeviceInfo* di, int variant, float* theta, __nv_bfloat16* lp, float* m, float* v, const float* sum_g,
                                    const float* sum_g2, long long n, const AdamParams& p, const unsigned int* skip_if_set, cudaStream_t st) {
  const dim3 grid(grid_for(n / 4 + 4, di->sm_count));
  switch (variant) {
    case ADAM_ORIGINAL: return launch_dependent(microadam_kernel<ADAM_ORIGINAL>, grid, OPT_THREADS, 0, st, theta, lp, m, v, sum_g, sum_g2, n, p, skip_if_set);
    case ADAM_MICRO: return launch_dependent(microadam_kernel<ADAM_MICRO>, grid, OPT_THREADS, 0, st, theta, lp, m, v, sum_g, sum_g2, n, p, skip_if_set);
    case ADAM_MICRO_VAR: return launch_dependent(microadam_kernel<ADAM_MICRO_VAR>, grid, OPT_THREADS, 0, st, theta, lp, m, v, sum_g, sum_g2, n, p, skip_if_set);
    default: return launch_dependent(microadam_kernel<ADAM_MICRO_MSQ>, grid, OPT_THREADS, 0, st, theta, lp, m, v, sum_g, sum_g2, n, p, skip_if_set);
  }
}
static pe_status_t launch_microsignsgd(DeviceInfo* di, float* theta, __nv_bfloat16* lp, float* m, const float* sum_sign, long long n,
                                       const SignParams& p, const unsigned int* skip_if_set, cudaStream_t st) {
  return launch_dependent(microsignsgd_kernel, dim3(grid_for(n / 4 + 4, di->sm_count)), OPT_THREADS, 0, st, theta, lp, m, sum_sign, n, p, skip_if_set);
}

// Side buffer of a packed batch: the zero-padded last partial 16-token group of every sequence, X's [B, 16, d_in]
// then dY's [B, 16, d_out] (bf16), each part 256-byte aligned.
struct RaggedLayout {
  size_t x_bytes, y_bytes;
  size_t total() const { return x_bytes + y_bytes; }
};
static RaggedLayout ragged_layout(int B, int d_in, int d_out) {
  RaggedLayout l;
  l.x_bytes = ((size_t)B * 16 * (size_t)d_in * 2 + 255) / 256 * 256;
  l.y_bytes = ((size_t)B * 16 * (size_t)d_out * 2 + 255) / 256 * 256;
  return l;
}

// Tensor-core launch for a packed batch.  norms != NULL: per-example squared norms (zeroed by the caller);
// otherwise the statistics of pe_linear_stats.  phi = identity (or only out_mean wanted) runs the per-example
// kernel with the identity, whose running sum is sum_b G_b.
static pe_status_t launch_tc_ragged(DeviceInfo* di, const void* X, const void* dY, const int* offsets, int B, long long rows, int d_in,
                                    int d_out, int phi, float* out_mean, float* out_stat, float* norms, void* ws, cudaStream_t st) {
  const RaggedLayout l = ragged_layout(B, d_in, d_out);
  uint16_t* xt = static_cast<uint16_t*>(ws);
  uint16_t* yt = reinterpret_cast<uint16_t*>(static_cast<char*>(ws) + l.x_bytes);
  const TailTensor tx = {static_cast<const uint16_t*>(X), xt, d_in}, ty = {static_cast<const uint16_t*>(dY), yt, d_out};
  pe_status_t rc = PE_OK;
  const bool both = !norms && out_mean && out_stat && phi != PE_PHI_IDENTITY;
  const bool plain = !norms && (phi == PE_PHI_IDENTITY || !out_stat);      // only sum_b G_b
  const int nt = both ? 192 : 256;
  const int box_tokens = tc_default_bk(false, nt);
  const int rows_i = (int)(rows > 0 ? rows : 1);
  CUtensorMap mx, my, mxt, myt;
  const int bf = TcOperand<false, 256>::BOX_FEATS;
  if (both) {
    rc = make_operand_map(&mx, X, 1, rows_i, d_in, false, TcOperand<false, 192>::B_BOX_FEATS, box_tokens, true);
    if (rc == PE_OK) rc = make_operand_map(&mxt, xt, B, 16, d_in, false, TcOperand<false, 192>::B_BOX_FEATS, 16, true);
  } else {
    rc = make_operand_map(&mx, X, 1, rows_i, d_in, false, bf, box_tokens);
    if (rc == PE_OK) rc = make_operand_map(&mxt, xt, B, 16, d_in, false, bf, 16);
  }
  if (rc == PE_OK) rc = make_operand_map(&my, dY, 1, rows_i, d_out, false, bf, box_tokens);
  if (rc == PE_OK) rc = make_operand_map(&myt, yt, B, 16, d_out, false, bf, 16);
  if (rc != PE_OK) return rc;
  float* first = plain ? (out_mean ? out_mean : out_stat) : out_stat;
  CUtensorMap mm = mx, ms = mx;       // never used by the norms variant
  if (!norms) {
    rc = make_output_map(&ms, first, d_in, d_out);
    if (rc == PE_OK) rc = make_output_map(&mm, both ? out_mean : first, d_in, d_out);
    if (rc != PE_OK) return rc;
  }
  const int tiles_n = (d_in + nt - 1) / nt, pairs_m = (d_out + TC_PAIR_M - 1) / TC_PAIR_M;
  if ((long long)tiles_n * pairs_m > (1ll << 29)) return PE_ERR_DIM;
  const long long t_avg = rows / B > 0 ? rows / B : 1;
  const int slots = di->sm_count / 2 > 0 ? di->sm_count / 2 : 1;
  const UnitCost& unit = norms ? COST_NORMS : both ? COST_BOTH_192 : plain ? COST_STAT : phi == PE_PHI_SIGN ? COST_SIGN : COST_STAT;
  const int ns = plan_tiles(&unit, 1, B, (double)t_avg, d_in, d_out, slots, std::max(16, slots), norms ? 0 : both ? 2 : 1).ns;
  // the pre-pass: the partial 16-token groups to the side buffer, and the outputs of a split batch to zero
  const bool zero = ns > 1 && !norms;
  const int chunks = (int)std::min<long long>(8, std::max<long long>(1, 8ll * di->sm_count / (2ll * B)));
  rc = launch_dependent(pack_tails_kernel, dim3((unsigned)B, 2, (unsigned)chunks), STAGE_THREADS, 0, st, tx, ty, offsets, rows, zero ? first : (float*)nullptr,
                        zero && both ? out_mean : (float*)nullptr, (long long)d_in * d_out);
  if (rc != PE_OK) return rc;
  TcParams p{};
  p.B = B; p.T = 0; p.d_in = d_in; p.d_out = d_out; p.nsplit = ns; p.per_example = 1; p.half_operands = 0;
  p.accumulate = norms ? 1 : 0;
  p.pairs_m = pairs_m; p.tiles_n = tiles_n; p.band = choose_band(pairs_m, tiles_n, nt, ns, di->sm_count / 2);
  p.out_mean = both ? out_mean : nullptr; p.out_stat = norms ? nullptr : first; p.out_sign = nullptr; p.out_norms = norms;
  p.by_tokens = ns > 1 && (phi != PE_PHI_SIGN || B <= TC_SIGN_COUNT_MAX) ? 1 : 0;
  p.seq_offsets = offsets; p.sq_norms = nullptr; p.clip_norm = 0.f; p.dev_status = di->status_ptr;
  const dim3 grid(2 * pairs_m * tiles_n, 1, ns);
  if (norms) return launch_tc_inst<1, false, 256, MEAN_NORMS, 64, true>(di, 15, mx, my, mm, ms, ms, p, grid, st, &mxt, &myt);
  if (plain) {
    rc = launch_tc_inst<0, false, 256, MEAN_NONE, 64, true>(di, 20, mx, my, mm, ms, ms, p, grid, st, &mxt, &myt);
    if (rc == PE_OK && out_mean && out_stat &&
        cudaMemcpyAsync(out_stat, out_mean, (size_t)d_in * d_out * sizeof(float), cudaMemcpyDeviceToDevice, st) != cudaSuccess) {
      cudaGetLastError();
      return PE_ERR_CUDA;
    }
    return rc;
  }
  if (both) {
    if (phi == PE_PHI_SQUARE) return launch_tc_inst<1, false, 192, MEAN_REGS, 128, true>(di, 16, mx, my, mm, ms, ms, p, grid, st, &mxt, &myt);
    return launch_tc_inst<2, false, 192, MEAN_REGS, 128, true>(di, 17, mx, my, mm, ms, ms, p, grid, st, &mxt, &myt);
  }
  if (phi == PE_PHI_SQUARE) return launch_tc_inst<1, false, 256, MEAN_NONE, 64, true>(di, 18, mx, my, mm, ms, ms, p, grid, st, &mxt, &myt);
  return launch_tc_inst<2, false, 256, MEAN_NONE, 64, true>(di, 19, mx, my, mm, ms, ms, p, grid, st, &mxt, &myt);
}

static pe_status_t validate_stats(const void* X, const void* dY, int B, int T, int d_in, int d_out, const float* o1,
                                  const float* o2, bool need_both_null_check, size_t in_align) {
  if (B < 0 || T < 0 || d_in < 1 || d_out < 1) return PE_ERR_DIM;
  if ((!X || !dY) && B > 0 && T > 0) return PE_ERR_NULL;      // empty inputs may be NULL
  if (need_both_null_check && !o1 && !o2) return PE_ERR_NULL;
  if ((long long)B * T * (long long)(d_in > d_out ? d_in : d_out) >= (1ll << 40)) return PE_ERR_DIM;
  if ((long long)d_in * d_out >= (1ll << 40)) return PE_ERR_DIM;
  if (!aligned(X, in_align) || !aligned(dY, in_align)) return PE_ERR_ALIGN;
  if ((o1 && !aligned(o1, 16)) || (o2 && !aligned(o2, 16))) return PE_ERR_ALIGN;
  return PE_OK;
}

// A plain contraction over all B*T rows does not care where one sequence ends: short sequences are
// regrouped into full two-stage "examples" when the rows divide evenly (fewer, fuller pipeline stages).
static void regroup_rows(int& B, int& T) {
  constexpr int REGROUP = 2 * TcOperand<false, 256>::BK;
  const long long rows = (long long)B * T;
  if (T < REGROUP && rows % REGROUP == 0) { B = (int)(rows / REGROUP); T = REGROUP; }
}

// pe_linear_stats on the tensor cores.
static pe_status_t tc_linear_stats(DeviceInfo* di, const void* X, const void* dY, int B, int T, int d_in, int d_out, int phi, float* out_mean,
                                   float* out_stat, bool accumulate, cudaStream_t st, const LayoutStep& before = nullptr) {
  g_last_path.store(PE_PATH_TENSOR);
  auto plain = [&](float* out, const LayoutStep& first = nullptr) {
    return launch_tc(di, X, dY, B, T, d_in, d_out, phi, 0, out, nullptr, st, false, nullptr, accumulate, nullptr, 0.f, 0, 0, false, nullptr, nullptr, first);
  };
  if (phi == PE_PHI_IDENTITY || !out_stat) {
    // phi = identity, or only sum_b G_b wanted: the plain contraction over all B*T rows, where B and T only enter
    // through B*T: regroup short sequences into full two-stage "examples" when the rows divide evenly.
    regroup_rows(B, T);
    pe_status_t rc = plain(out_mean ? out_mean : out_stat, before);
    if (rc != PE_OK || !out_mean || !out_stat) return rc;
    if (accumulate) return plain(out_stat);          // a copy would overwrite: contract once more into the second
    if (cudaMemcpyAsync(out_stat, out_mean, (size_t)d_in * d_out * sizeof(float), cudaMemcpyDeviceToDevice, st) != cudaSuccess) {
      cudaGetLastError();
      return PE_ERR_CUDA;
    }
    return PE_OK;
  }
  return launch_tc(di, X, dY, B, T, d_in, d_out, phi, 1, out_mean, out_stat, st, false, nullptr, accumulate, nullptr, 0.f, 0, 0, false, nullptr, nullptr,
                   before);
}

// The same for layers that the SIMT kernel would otherwise serve, from copies whose rows are pitch_x, pitch_y elements
// apart (multiples of 8; 0: back to back), held to that kernel's accuracy: at most TC_CHUNK_TOKENS tokens per accumulator, and sum_b G_b
// from the examples' sums rather than from one accumulation over all rows.  out_sign != NULL: the three statistics of
// pe_linear_stats_all (phi = square).
static pe_status_t tc_linear_stats_pitched(DeviceInfo* di, const void* X, const void* dY, int B, int T, int d_in, int d_out, int phi,
                                           float* out_mean, float* out_stat, float* out_sign, bool accumulate, int pitch_x, int pitch_y,
                                           cudaStream_t st, const LayoutStep& before) {
  g_last_path.store(PE_PATH_TENSOR);
  auto run = [&](int f, float* mean, float* stat, float* sign, const LayoutStep& first = nullptr) {
    return launch_tc(di, X, dY, B, T, d_in, d_out, f, 1, mean, stat, st, false, sign, accumulate, nullptr, 0.f, pitch_x, pitch_y, true, nullptr, nullptr,
                     first);
  };
  if (phi == PE_PHI_IDENTITY) {
    pe_status_t rc = run(PE_PHI_SQUARE, out_mean ? out_mean : out_stat, nullptr, nullptr, before);
    if (rc != PE_OK || !out_mean || !out_stat) return rc;
    if (accumulate) return run(PE_PHI_SQUARE, out_stat, nullptr, nullptr);
    if (cudaMemcpyAsync(out_stat, out_mean, (size_t)d_in * d_out * sizeof(float), cudaMemcpyDeviceToDevice, st) != cudaSuccess) {
      cudaGetLastError();
      return PE_ERR_CUDA;
    }
    return PE_OK;
  }
  if (out_sign && T > TC_CHUNK_TOKENS) {
    pe_status_t rc = run(PE_PHI_SQUARE, out_mean, out_stat, nullptr, before);
    return rc == PE_OK ? run(PE_PHI_SIGN, nullptr, out_sign, nullptr) : rc;
  }
  return run(phi, out_mean, out_stat, out_sign, before);
}

template <typename TIn>
static pe_status_t linear_stats_impl(const TIn* X, const TIn* dY, int B, int T, int d_in, int d_out, pe_phi_t phi,
                                     float* out_mean, float* out_stat, cudaStream_t st, bool allow_tc, bool accumulate = false) {
  pe_status_t rc = validate_stats(X, dY, B, T, d_in, d_out, out_mean, out_stat, true, allow_tc ? 16 : 4);
  if (rc != PE_OK) return rc;
  if (phi != PE_PHI_IDENTITY && phi != PE_PHI_SQUARE && phi != PE_PHI_SIGN) return PE_ERR_PHI;
  DeviceInfo* di = nullptr;
  rc = device_info(&di);
  if (rc != PE_OK) return rc;
  if (B == 0 || T == 0) return accumulate ? PE_OK : zero_outputs(out_mean, out_stat, (size_t)d_in * d_out * sizeof(float), st);
  const int forced = g_path.load();
  const bool tc_ok = allow_tc && tc_shape_ok(B, T, d_in, d_out);
  if (forced >= PE_PATH_TENSOR && !tc_ok) return PE_ERR_UNSUPPORTED_SHAPE;
  if (tc_ok && forced != PE_PATH_SIMT) {
    if constexpr (sizeof(TIn) == 2) return tc_linear_stats(di, X, dY, B, T, d_in, d_out, phi, out_mean, out_stat, accumulate, st);
  }
  g_last_path.store(PE_PATH_SIMT);
  return launch_simt<TIn, MODE_STATS>(di, X, dY, B, T, d_in, d_out, (int)phi, out_mean, out_stat, st, accumulate);
}

static size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Constants of one Adam-family step (Algorithm 1): the scales that turn the sums into averages, the
// bias corrections of step t, and the factor 1 / (1 - 1/B) of Eq. (6).
static AdamParams make_adam_params(int B, float grad_scale, float lr, float beta1, float beta2, float eps, int eps_inside_sqrt,
                                   float weight_decay, int step) {
  AdamParams p;
  p.mu_scale = (float)((double)grad_scale / (double)B);
  p.nu_scale = (float)((double)grad_scale * (double)grad_scale / (double)B);
  p.beta1 = beta1; p.beta2 = beta2;
  p.inv_c1 = (float)(1.0 / (1.0 - std::pow((double)beta1, (double)step)));
  p.inv_c2 = (float)(1.0 / (1.0 - std::pow((double)beta2, (double)step)));
  p.eps = eps; p.lr = lr; p.wd = weight_decay; p.eps_inside = eps_inside_sqrt ? 1 : 0;
  p.inv_B = (float)(1.0 / (double)B);
  p.bessel = B > 1 ? (float)(1.0 / (1.0 - 1.0 / (double)B)) : 1.f;
  return p;
}

// Words of tile counters a fused statistics + update launch may need: one per thread block of the widest grid
// (256 x 128 tiles), i.e. two per pair tile.
static size_t fused_counter_words(int d_in, int d_out) {
  return 2 * (size_t)((d_out + TC_PAIR_M - 1) / TC_PAIR_M) * (size_t)((d_in + 127) / 128);
}

// Statistics and parameter update in one tensor-core launch.  kind = OPT_ADAM: sum_b G_b and sum_b G_b^2 (256 x 192 or
// 256 x 128 tile, both sums in registers) feed Algorithm 1; kind = OPT_SIGN: sum_b sign(G_b) (256 x 256 tile) feeds
// MicroSignSGD.  out_a = out_mean (Adam only), out_b = the statistic; they may be NULL when the schedule does not
// split the batch, which is forced when they (or the counters) are missing.
static pe_status_t launch_tc_fused(DeviceInfo* di, const void* X, const void* dY, int B, int T, int d_in, int d_out, int kind,
                                   float* out_a, float* out_b, FusedOpt opt, unsigned int* counters, size_t counter_words,
                                   cudaStream_t st) {
  const bool adam = kind == OPT_ADAM;
  const int forced = g_path.load();
  const int slots = di->sm_count / 2 > 0 ? di->sm_count / 2 : 1;
  // the batch is only split if somebody can complete a tile: outputs to add to and a counter per block
  const bool can_split = out_b && (!adam || out_a) && counters && counter_words >= fused_counter_words(d_in, d_out);
  UnitCost cand[2];
  int n_cand = 0;
  if (adam && forced != PE_PATH_TENSOR_NARROW) cand[n_cand++] = COST_BOTH_192;
  if (adam && (forced != PE_PATH_TENSOR_WIDE || n_cand == 0)) cand[n_cand++] = COST_BOTH_128;
  if (!adam) cand[n_cand++] = COST_SIGN;
  for (int k = 0; k < n_cand; ++k) cand[k].fixed += FUSED_UPDATE_FIXED * cand[k].nt / 192.0;
  const TilePlan plan = plan_tiles(cand, n_cand, B, T, d_in, d_out, slots, can_split ? std::max(16, slots) : 1, adam ? 2 : 1);
  const bool wide = adam && cand[plan.choice].nt == 192;
  const int nt = adam ? (wide ? 192 : 128) : 256;
  const int box_feats = TcOperand<false, 256>::BOX_FEATS, box_tokens = tc_default_bk(false, nt);
  CUtensorMap mx, my, mm, ms;
  pe_status_t rc = wide ? make_operand_map(&mx, X, B, T, d_in, false, TcOperand<false, 192>::B_BOX_FEATS, box_tokens, true)
                        : make_operand_map(&mx, X, B, T, d_in, false, box_feats, box_tokens);
  if (rc == PE_OK) rc = make_operand_map(&my, dY, B, T, d_out, false, box_feats, box_tokens);
  // an output that is not wanted gets a map over the parameters and is never written through it
  if (rc == PE_OK) rc = make_output_map(&mm, out_a ? out_a : opt.theta, d_in, d_out);
  if (rc == PE_OK) rc = make_output_map(&ms, out_b ? out_b : opt.theta, d_in, d_out);
  if (rc != PE_OK) return rc;
  const int tiles_n = (d_in + nt - 1) / nt, pairs_m = (d_out + TC_PAIR_M - 1) / TC_PAIR_M;
  if ((long long)tiles_n * pairs_m > (1ll << 29)) return PE_ERR_DIM;
  const int ns = plan.ns;
  const size_t blocks = 2 * (size_t)tiles_n * pairs_m;
  if (ns > 1) {
    rc = zero_for_split(di, adam ? out_a : nullptr, out_b, (size_t)d_in * d_out, st, nullptr, counters, (int)blocks);
    if (rc != PE_OK) return rc;
  }
  TcParams p{};
  p.B = B; p.T = T; p.d_in = d_in; p.d_out = d_out; p.nsplit = ns; p.per_example = 1; p.half_operands = 0; p.accumulate = 0;
  p.wait_at_start = ns == 1 ? 1 : 0;
  p.pairs_m = pairs_m; p.tiles_n = tiles_n; p.band = choose_band(pairs_m, tiles_n, nt, ns, di->sm_count / 2);
  p.out_mean = adam ? out_a : nullptr; p.out_stat = out_b; p.out_sign = nullptr; p.out_norms = nullptr; p.dev_status = di->status_ptr;
  p.seq_offsets = nullptr; p.sq_norms = nullptr; p.clip_norm = 0.f;
  opt.kind = kind;
  opt.tile_counters = counters;
  const dim3 grid((unsigned)blocks, 1, ns);
  if (!adam) return launch_tc_inst<2, false, 256, MEAN_NONE, 64, false, OPT_SIGN>(di, 23, mx, my, mm, ms, ms, p, grid, st, nullptr, nullptr, &opt);
  if (wide) return launch_tc_inst<1, false, 192, MEAN_REGS, 128, false, OPT_ADAM>(di, 21, mx, my, mm, ms, ms, p, grid, st, nullptr, nullptr, &opt);
  return launch_tc_inst<1, false, 128, MEAN_REGS, 128, false, OPT_ADAM>(di, 22, mx, my, mm, ms, ms, p, grid, st, nullptr, nullptr, &opt);
}

// Per-token statistic: `units` chunks of rows for each tile.  ns: slices of the rows, a pair per tile and slice; deal_tiles > 0: instead, the chunks of
// every deal_tiles tiles (the last ones may be fewer) dealt out evenly over deal_pairs pairs, pairs in all.
struct TokPlan {
  int ns, deal_tiles, deal_pairs, pairs;
};
static TokPlan plan_tok(int units, int d_in, int d_out, int slots) {
  const long long tiles = (((long long)d_in + TOK_NT - 1) / TOK_NT) * (((long long)d_out + TC_PAIR_M - 1) / TC_PAIR_M);
  const double out_bytes = 4.0 * d_in * d_out;
  TokPlan plan = {plan_tiles(&COST_TOKEN, 1, units, TOK_BK, d_in, d_out, slots, std::max(32, slots), 1).ns, 0, 0, 0};
  if (tiles >= slots || tiles * units < slots || units < 2) return plan;
  const double in_slices = launch_cost(COST_TOKEN, tiles, units, TOK_BK, slots, plan.ns, 1, out_bytes, false).us;
  // Evenly over all pairs, which gives a tile three parts and more, added in no fixed order.  A call whose tiles would be whole or in two slices repeats bit for bit
  // (two parts on zero, whatever their order), and keeps to that: groups of k tiles on k + 1 pairs, which give every tile two parts.
  const long long k = plan.ns > 2 ? tiles : (slots - 1) / (slots - tiles), pairs = plan.ns > 2 ? slots : k + 1;
  const double load = std::ceil((double)units * k / pairs);
  // Tiles that share rows read them at different times, and so from HBM, unless what they share stays in L2.
  const double rows = (double)units * TOK_BK, x_bytes = 2.0 * rows * d_in, y_bytes = 2.0 * rows * d_out, tile_bytes = 2.0 * rows * 256;
  const bool all_stay = x_bytes + y_bytes <= TOK_L2_BYTES;
  const double traffic = (all_stay || x_bytes <= TOK_L2_BYTES / 4 ? x_bytes : tiles * tile_bytes) + (all_stay || y_bytes <= TOK_L2_BYTES / 4 ? y_bytes : tiles * tile_bytes);
  const double dealt = std::max(load * TOK_BK * COST_TOKEN.token_hi, traffic / TOK_DEALT_BYTES_PER_US) + COST_TOKEN.fixed + SPLIT_FIXED + out_bytes / ZERO_BYTES_PER_US +
                       TOK_EVEN_FIXED;
  if (dealt < in_slices) {
    plan.deal_tiles = (int)k; plan.deal_pairs = (int)pairs;
    plan.pairs = (int)(plan.ns > 2 ? slots : tiles + (tiles + k - 1) / k);
  }
  return plan;
}


// Fused per-token statistic: squares, rounds to tf32 and contracts inside one kernel.
static pe_status_t launch_tok(DeviceInfo* di, const void* X, const void* dY, long long rows, int d_in, int d_out, float* out,
                              cudaStream_t st) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return PE_ERR_CUDA;
  CUtensorMap mx, my, mo;
  auto operand_map = [&](CUtensorMap* m, const void* base, int d) {
    cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)d * 2ull};
    cuuint32_t box[2] = {64u, (cuuint32_t)TOK_BK};
    cuuint32_t estr[2] = {1u, 1u};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  };
  if (!operand_map(&mx, X, d_in) || !operand_map(&my, dY, d_out)) return PE_ERR_CUDA;
  pe_status_t rc = make_output_map(&mo, out, d_in, d_out);
  if (rc != PE_OK) return rc;
  const int tiles_n = (d_in + TOK_NT - 1) / TOK_NT, pairs_m = (d_out + TC_PAIR_M - 1) / TC_PAIR_M;
  if ((long long)tiles_n * pairs_m > (1ll << 29)) return PE_ERR_DIM;
  const long long n_chunks = (rows + TOK_BK - 1) / TOK_BK;
  const int units = n_chunks > (1 << 30) ? (1 << 30) : (int)n_chunks;
  const int slots = di->sm_count / 2 > 0 ? di->sm_count / 2 : 1;
  const TokPlan plan = plan_tok(units, d_in, d_out, slots);
  const int ns = plan.ns;
  const bool even = plan.deal_tiles > 0;
  if (ns > 1 || even) {
    rc = zero_for_split(di, out, nullptr, (size_t)d_in * d_out, st);
    if (rc != PE_OK) return rc;
  }
  {
    std::lock_guard<std::mutex> lock(g_dev_mutex);
    if (!di->tok_attr_set) {
      if (cudaFuncSetAttribute(tok_sqstats_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TOK_SMEM_BYTES) != cudaSuccess) {
        cudaGetLastError();
        return PE_ERR_CUDA;
      }
      di->tok_attr_set = true;
    }
  }
  TokParams p;
  p.rows = rows; p.d_in = d_in; p.d_out = d_out; p.pairs_m = pairs_m; p.tiles_n = tiles_n;
  p.band = choose_band(pairs_m, tiles_n, TOK_NT, even ? 1 : ns, di->sm_count / 2); p.nsplit = even ? 1 : ns;
  p.deal_tiles = plan.deal_tiles; p.deal_pairs = plan.deal_pairs; p.dev_status = di->status_ptr;
  return launch_dependent(tok_sqstats_kernel, even ? dim3(2 * plan.pairs) : dim3(2 * pairs_m * tiles_n, 1, ns), TOK_THREADS, TOK_SMEM_BYTES, st, mx, my, mo, p);
}

}  // namespace pe

using namespace pe;

extern "C" {

pe_status_t pe_linear_stats(const void* X, const void* dY, int B, int T, int d_in, int d_out, pe_phi_t phi,
                            float* out_mean, float* out_stat, pe_stream_t stream) {
  return linear_stats_impl<__nv_bfloat16>(static_cast<const __nv_bfloat16*>(X), static_cast<const __nv_bfloat16*>(dY), B, T,
                                          d_in, d_out, phi, out_mean, out_stat, reinterpret_cast<cudaStream_t>(stream), true);
}

pe_status_t pe_example_sqnorms(const void* X, const void* dY, int B, int T, int d_in, int d_out, float* out_norms,
                               pe_stream_t stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (!out_norms && B > 0) return PE_ERR_NULL;
  pe_status_t rc = validate_stats(X, dY, B, T, d_in, d_out, nullptr, nullptr, false, 16);
  if (rc != PE_OK) return rc;
  if (out_norms && !aligned(out_norms, 4)) return PE_ERR_ALIGN;
  DeviceInfo* di = nullptr;
  rc = device_info(&di);
  if (rc != PE_OK) return rc;
  if (B == 0) return PE_OK;
  if (T == 0) return zero_outputs(out_norms, nullptr, (size_t)B * sizeof(float), st);
  const int forced = g_path.load();
  const bool tc_ok = tc_shape_ok(B, T, d_in, d_out);
  if (forced >= PE_PATH_TENSOR && !tc_ok) return PE_ERR_UNSUPPORTED_SHAPE;
  if (tc_ok && forced != PE_PATH_SIMT) {
    g_last_path.store(PE_PATH_TENSOR);
    return launch_tc_norms(di, X, dY, B, T, d_in, d_out, out_norms, st);
  }
  g_last_path.store(PE_PATH_SIMT);
  rc = zero_outputs(out_norms, nullptr, (size_t)B * sizeof(float), st);
  if (rc != PE_OK) return rc;
  // every block handles whole examples of its slice and adds to out_norms[b]: "accumulate" keeps launch_simt from zeroing
  return launch_simt<__nv_bfloat16, MODE_NORMS>(di, static_cast<const __nv_bfloat16*>(X), static_cast<const __nv_bfloat16*>(dY), B, T,
                                                d_in, d_out, 1, nullptr, out_norms, st, true);
}

pe_status_t pe_linear_stats_accumulate(const void* X, const void* dY, int B, int T, int d_in, int d_out, pe_phi_t phi,
                                       float* out_mean, float* out_stat, pe_stream_t stream) {
  return linear_stats_impl<__nv_bfloat16>(static_cast<const __nv_bfloat16*>(X), static_cast<const __nv_bfloat16*>(dY), B, T,
                                          d_in, d_out, phi, out_mean, out_stat, reinterpret_cast<cudaStream_t>(stream), true, true);
}

pe_status_t pe_linear_stats_all(const void* X, const void* dY, int B, int T, int d_in, int d_out, float* out_mean,
                                float* out_square, float* out_sign, pe_stream_t stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (!out_mean || !out_square || !out_sign) return PE_ERR_NULL;
  pe_status_t rc = validate_stats(X, dY, B, T, d_in, d_out, out_mean, out_square, true, 16);
  if (rc != PE_OK) return rc;
  if (!aligned(out_sign, 16)) return PE_ERR_ALIGN;
  DeviceInfo* di = nullptr;
  rc = device_info(&di);
  if (rc != PE_OK) return rc;
  const int forced = g_path.load();
  // One pass when the tensor-core kernel takes the shape; otherwise the two calls this one stands for.
  if (B > 0 && T > 0 && forced != PE_PATH_SIMT && tc_shape_ok(B, T, d_in, d_out)) {
    g_last_path.store(PE_PATH_TENSOR);
    return launch_tc(di, X, dY, B, T, d_in, d_out, PE_PHI_SQUARE, 1, out_mean, out_square, st, false, out_sign);
  }
  const __nv_bfloat16* Xb = static_cast<const __nv_bfloat16*>(X);
  const __nv_bfloat16* Yb = static_cast<const __nv_bfloat16*>(dY);
  rc = linear_stats_impl<__nv_bfloat16>(Xb, Yb, B, T, d_in, d_out, PE_PHI_SQUARE, out_mean, out_square, st, true);
  if (rc != PE_OK) return rc;
  return linear_stats_impl<__nv_bfloat16>(Xb, Yb, B, T, d_in, d_out, PE_PHI_SIGN, nullptr, out_sign, st, true);
}

// Copies of the operands at 16-byte row pitches: X's, then dY's, each 256-byte aligned; a tensor whose width is a multiple of 8
// needs none.
struct PaddedLayout {
  int pitch_x, pitch_y;
  size_t x_bytes, y_bytes;
};
static PaddedLayout padded_layout(int B, int T, int d_in, int d_out, bool always) {
  PaddedLayout l;
  l.pitch_x = (d_in + 7) & ~7;
  l.pitch_y = (d_out + 7) & ~7;
  l.x_bytes = (always || d_in % 8) ? align_up((size_t)B * T * l.pitch_x * 2, 256) : 0;
  l.y_bytes = (always || d_out % 8) ? align_up((size_t)B * T * l.pitch_y * 2, 256) : 0;
  return l;
}
// Widths that are no multiples of 8: from this many multiply-adds on, copying the operands to a padded pitch and
// contracting them on the tensor cores beats the SIMT kernel.  Two launches against one, at least 15 us of host and device time per call.
// SIMT / padded, us: 8 x 64 x 129 x 257 (2^24) 10.4 / 16.4, 8 x 64 x 257 x 255 (2^25) 12.4 / 16.3, 8 x 128 x 129 x 257 (2^25) 14.5 / 15.2,
// 8 x 64 x 257 x 511 (2^26) 18.6 / 16.5, 32 x 8 x 513 x 511 (2^26) 26.5 / 23.7, 8 x 256 x 129 x 257 (2^26) 22.7 / 15.3, 2 x 2048 x 129 x 255 (2^27)
// 61.6 / 20.7.  (One width below 16, where the SIMT tile is mostly empty, would gain earlier: 64 x 256 x 1024 x 1 (2^24) 94 / 17.)
constexpr long long PAD_MIN_MACS = 1ll << 26;
static bool padding_pays(int B, int T, int d_in, int d_out) {
  return B > 0 && T > 0 && (d_in % 8 || d_out % 8) && tc_shape_ok(B, T, (d_in + 7) & ~7, (d_out + 7) & ~7) &&
         (double)B * T * d_in * d_out >= (double)PAD_MIN_MACS && (long long)B * T < (1ll << 31);
}

// Examples of one token: the statistics that are wanted, and where their copies of the operands are among those that are made (the mean
// needs the operands as they are, the square the two halves of their squares, the sign their signs).
struct OneTokenWant {
  bool mean, square, sign;
  int first_half() const { return mean ? 1 : 0; }
  int first_sign() const { return first_half() + (square ? 2 : 0); }
  int copies() const { return first_sign() + (sign ? 1 : 0); }
};
static OneTokenWant one_token_want(int phi, bool mean, bool stat, bool sign) {
  if (phi == PE_PHI_IDENTITY) return {mean || stat, false, false};
  if (phi == PE_PHI_SIGN) return {mean, false, stat};
  return {mean, stat, sign};
}

// The copies of each operand, in n chunks of `chunk` rows.  A chunk is what one accumulator takes, and the
// accumulators are added in registers; the square's error against fp64, 2-norm, at 1024 x 1024^2: 1.4e-6 with 512 rows, 3.0e-7 with
// 128, 1.7e-7 with 64, and 2.4e-7 with the kernel that forms every G_b.  64 rows cost 10 % there.
constexpr int ONE_TOKEN_CHUNK = 64;
struct OneTokenLayout {
  int chunk, n, pitch_x, pitch_y;
  size_t x_bytes, y_bytes, odd_bytes;     // odd: a byte per row (the marks of one_token_operands_kernel)
  size_t total() const { return x_bytes + y_bytes + odd_bytes; }
};
static OneTokenLayout one_token_layout(int B, int d_in, int d_out, const OneTokenWant& want) {
  OneTokenLayout l;
  l.n = (B + ONE_TOKEN_CHUNK - 1) / ONE_TOKEN_CHUNK;
  l.chunk = ((B + l.n - 1) / l.n + 15) / 16 * 16;
  l.pitch_x = (d_in + 7) & ~7;
  l.pitch_y = (d_out + 7) & ~7;
  l.x_bytes = align_up((size_t)want.copies() * l.n * l.chunk * l.pitch_x * 2, 256);
  l.y_bytes = align_up((size_t)want.copies() * l.n * l.chunk * l.pitch_y * 2, 256);
  l.odd_bytes = want.square || want.sign ? align_up((size_t)l.n * l.chunk, 256) : 0;
  return l;
}
// From this many entries of all G_b on, the two launches (16 us at least, and 8 us more of host time) beat the kernel that forms every
// G_b and is bound by reading them: mean and square, three statistics, sign alone, us: 128 x 1024^2 26.8, 49.6, 31.0 -> 16.7, 17.8,
// 15.7 (64 x 1024^2 18.7, 31.0, 20.7 stays); 1024 x 1024^2 133, 313, 162 -> 23, 28, 16; 512 x 4096^2 781, 2145, 1112 -> 123, 157, 48.
constexpr double ONE_TOKEN_MIN_MACS = 1.2e8;
static bool one_token_pays(int B, int T, int d_in, int d_out) {
  return T == 1 && B > 0 && B <= (1 << 24) && tc_shape_ok(B, T, (d_in + 7) & ~7, (d_out + 7) & ~7) && (double)B * d_in * d_out >= ONE_TOKEN_MIN_MACS;
}
// Slices of each product's chunks: units of at most `len` chunks of a tile, by the estimated time of the launch: the units shared out
// over the pairs, at least the longest.
static void one_token_slices(const OneTokenLayout& l, const bool (&want)[3], long long tiles, int slots, double out_bytes, int (&slices)[3]) {
  const double per_chunk = l.chunk * (COST_PLAIN.token_lo + COST_PLAIN.token_hi) * 0.5;
  const int counts[3] = {4 * l.n, l.n, l.n};
  double best = 1e300;
  for (int parts = 1; parts <= 4 * l.n && parts <= 128; ++parts) {
    const int len = (4 * l.n + parts - 1) / parts;
    double work = 0.0, longest = 0.0;
    int s[3];
    bool split = false;
    for (int k = 0; k < 3; ++k) {
      s[k] = want[k] ? (counts[k] + len - 1) / len : 0;
      if (s[k] > 1) split = true;
    }
    for (int k = 0; k < 3; ++k) {
      if (!s[k]) continue;
      const double unit = (double)((counts[k] + s[k] - 1) / s[k]) * per_chunk + COST_PLAIN.fixed + (split ? SPLIT_FIXED : 0.0);
      work += unit * s[k] * tiles;
      longest = std::max(longest, unit);
    }
    const double units = (double)tiles * (s[0] + s[1] + s[2]);
    const double us = std::max(longest, work / units * std::ceil(units / slots)) + (split ? out_bytes / ZERO_BYTES_PER_US : 0.0);
    if (us < best * 0.995) {
      best = us;
      for (int k = 0; k < 3; ++k) slices[k] = s[k];
    }
  }
}
static pe_status_t one_token_stats(DeviceInfo* di, const void* X, const void* dY, int B, int d_in, int d_out, float* out_mean, float* out_square,
                                   float* out_sign, bool accumulate, void* workspace, cudaStream_t st) {
  const OneTokenWant want = {out_mean != nullptr, out_square != nullptr, out_sign != nullptr};
  const OneTokenLayout l = one_token_layout(B, d_in, d_out, want);
  uint8_t* const odd = static_cast<uint8_t*>(workspace) + l.x_bytes + l.y_bytes;
  const OneTokenTensor tx = {static_cast<const uint16_t*>(X), static_cast<uint16_t*>(workspace), d_in, l.pitch_x};
  const OneTokenTensor ty = {static_cast<const uint16_t*>(dY), reinterpret_cast<uint16_t*>(static_cast<char*>(workspace) + l.x_bytes), d_out, l.pitch_y};
  const int tiles_n = (d_in + 255) / 256, pairs_m = (d_out + TC_PAIR_M - 1) / TC_PAIR_M;
  if ((long long)tiles_n * pairs_m > (1ll << 29)) return PE_ERR_DIM;
  const int slots = di->sm_count / 2 > 0 ? di->sm_count / 2 : 1;
  float* const outs[3] = {out_square, out_mean, out_sign};
  TcParams p{};
  one_token_slices(l, {want.square, want.mean, want.sign}, (long long)tiles_n * pairs_m, slots, 4.0 * (want.mean + want.square + want.sign) * d_in * d_out,
                   p.part_slices);
  const bool split = p.part_slices[0] > 1 || p.part_slices[1] > 1 || p.part_slices[2] > 1;
  LayoutZero zero = {{nullptr, nullptr, nullptr}, (long long)d_in * d_out};
  if (split && !accumulate)
    for (int k = 0; k < 3; ++k) zero.out[k] = outs[k];
  const int rows = l.n * l.chunk, zero_blocks = split && !accumulate ? 2 * di->sm_count : 0;
  pe_status_t rc = launch_dependent(one_token_operands_kernel, dim3(rows + zero_blocks), LAYOUT_THREADS, 0, st, tx, ty, odd, B, l.chunk, l.n, want.mean ? 0 : -1,
                                    want.square ? want.first_half() : -1, want.sign ? want.first_sign() : -1, zero);
  if (rc != PE_OK) return rc;
  CUtensorMap mx, my;
  constexpr int box_feats = TcOperand<false, 256>::BOX_FEATS, box_tokens = TcOperand<false, 256>::BK;
  rc = make_operand_map(&mx, tx.dst, want.copies() * l.n, l.chunk, d_in, false, box_feats, box_tokens, false, 1, l.pitch_x);
  if (rc == PE_OK) rc = make_operand_map(&my, ty.dst, want.copies() * l.n, l.chunk, d_out, false, box_feats, box_tokens, false, 1, l.pitch_y);
  if (rc != PE_OK) return rc;
  const bool scalar_out = d_in % 4 != 0;
  CUtensorMap mo[3] = {mx, mx, mx};
  for (int k = 0; k < 3 && !scalar_out; ++k) {
    if (!outs[k]) continue;
    rc = make_output_map(&mo[k], outs[k], d_in, d_out);
    if (rc != PE_OK) return rc;
  }
  p.B = 6 * l.n; p.T = l.chunk; p.d_in = d_in; p.d_out = d_out; p.nsplit = split ? 2 : 1; p.per_example = 1;
  p.accumulate = accumulate ? 1 : 0; p.scalar_out = scalar_out ? 1 : 0; p.wait_at_start = 1; p.part_chunks = l.n;
  // the copies that products 0 to 5 take (tc_part_chunk), four bits each: mean | upper and lower halves of dY by those of X | sign
  const unsigned int half = want.first_half(), sign = want.first_sign();
  p.part_dy = half * 0x11110u + 0x10100u + (sign << 20);
  p.part_x = half * 0x11110u + 0x11000u + (sign << 20);
  p.odd_rows = odd; p.rows_dy = static_cast<const uint16_t*>(dY); p.rows_x = static_cast<const uint16_t*>(X);
  p.pairs_m = pairs_m; p.tiles_n = tiles_n;
  const int units = p.part_slices[0] + p.part_slices[1] + p.part_slices[2];
  p.band = choose_band(pairs_m, tiles_n, 256, units, slots);
  p.out_stat = out_square; p.out_mean = out_mean; p.out_sign = out_sign; p.dev_status = di->status_ptr;
  return launch_tc_inst<0, false, 256, MEAN_NONE, tc_default_bk(false, 256), false, OPT_NONE, false, false, false, true>(
      di, 31, mx, my, mo[1], mo[0], mo[2], p, dim3(2 * pairs_m * tiles_n, 1, units), st);
}

static size_t padded_workspace_bytes(int B, int T, int d_in, int d_out, const OneTokenWant& want) {
  if (B < 1 || T < 1 || d_in < 1 || d_out < 1 || g_path.load() != PE_PATH_AUTO) return 0;
  if (one_token_pays(B, T, d_in, d_out)) {
    // the mean alone of widths that TMA can address is a contraction of the operands as they are
    if (!want.square && !want.sign && (!want.mean || (d_in % 8 == 0 && d_out % 8 == 0))) return 0;
    return one_token_layout(B, d_in, d_out, want).total();
  }
  if (!padding_pays(B, T, d_in, d_out)) return 0;
  const PaddedLayout l = padded_layout(B, T, d_in, d_out, false);
  return l.x_bytes + l.y_bytes;
}

size_t pe_linear_stats_padded_workspace_bytes(int B, int T, int d_in, int d_out) {
  return padded_workspace_bytes(B, T, d_in, d_out, {true, true, true});
}
size_t pe_linear_stats_padded_workspace_bytes_for(int B, int T, int d_in, int d_out, pe_phi_t phi, int want_mean, int want_stat, int want_sign) {
  return padded_workspace_bytes(B, T, d_in, d_out, one_token_want(phi, want_mean != 0, want_stat != 0, want_sign != 0));
}

pe_status_t pe_linear_stats_padded(const void* X, const void* dY, int B, int T, int d_in, int d_out, pe_phi_t phi, int accumulate,
                                   float* out_mean, float* out_stat, float* out_sign, void* workspace, size_t workspace_bytes,
                                   pe_stream_t stream) {
  const size_t need = pe_linear_stats_padded_workspace_bytes_for(B, T, d_in, d_out, phi, out_mean != nullptr, out_stat != nullptr, out_sign != nullptr);
  if (out_sign && (accumulate || phi != PE_PHI_SQUARE)) return PE_ERR_PHI;
  if (need == 0) {
    if (out_sign) return pe_linear_stats_all(X, dY, B, T, d_in, d_out, out_mean, out_stat, out_sign, stream);
    return accumulate ? pe_linear_stats_accumulate(X, dY, B, T, d_in, d_out, phi, out_mean, out_stat, stream)
                      : pe_linear_stats(X, dY, B, T, d_in, d_out, phi, out_mean, out_stat, stream);
  }
  if (out_sign && (!out_mean || !out_stat)) return PE_ERR_NULL;
  pe_status_t rc = validate_stats(X, dY, B, T, d_in, d_out, out_mean, out_stat, true, 16);
  if (rc != PE_OK) return rc;
  if (phi != PE_PHI_IDENTITY && phi != PE_PHI_SQUARE && phi != PE_PHI_SIGN) return PE_ERR_PHI;
  if (out_sign && !aligned(out_sign, 16)) return PE_ERR_ALIGN;
  if (!workspace || workspace_bytes < need) return PE_ERR_WORKSPACE;
  if (!aligned(workspace, 256)) return PE_ERR_ALIGN;
  DeviceInfo* di = nullptr;
  rc = device_info(&di);
  if (rc != PE_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const long long rows = (long long)B * T;
  if (one_token_pays(B, T, d_in, d_out)) {
    g_last_path.store(PE_PATH_TENSOR);
    if (phi == PE_PHI_SQUARE) return one_token_stats(di, X, dY, B, d_in, d_out, out_mean, out_stat, out_sign, accumulate != 0, workspace, st);
    if (phi == PE_PHI_SIGN) return one_token_stats(di, X, dY, B, d_in, d_out, out_mean, nullptr, out_stat, accumulate != 0, workspace, st);
    rc = one_token_stats(di, X, dY, B, d_in, d_out, out_mean ? out_mean : out_stat, nullptr, nullptr, accumulate != 0, workspace, st);
    if (rc != PE_OK || !out_mean || !out_stat) return rc;
    return one_token_stats(di, X, dY, B, d_in, d_out, out_stat, nullptr, nullptr, accumulate != 0, workspace, st);
  }
  const PaddedLayout l = padded_layout(B, T, d_in, d_out, false);
  PadTensor px = {static_cast<const uint16_t*>(X), static_cast<uint16_t*>(workspace), d_in, l.pitch_x};
  PadTensor py = {static_cast<const uint16_t*>(dY), reinterpret_cast<uint16_t*>(static_cast<char*>(workspace) + l.x_bytes), d_out, l.pitch_y};
  const bool pad_x = l.x_bytes > 0, pad_y = l.y_bytes > 0;
  const long long groups = rows * ((pad_x && pad_y ? std::max(l.pitch_x, l.pitch_y) : pad_x ? l.pitch_x : l.pitch_y) / 8);
  long long blocks = (groups + 4 * LAYOUT_THREADS - 1) / (4 * LAYOUT_THREADS);
  if (blocks > 16ll * di->sm_count) blocks = 16ll * di->sm_count;
  const LayoutStep pad = [&](const LayoutZero& zero) {
    // few rows, large outputs: blocks for the zeros (34 x 10 x 793 x 1270 in two slices 29.6 -> 20.2 us)
    const int outputs = (zero.out[0] ? 1 : 0) + (zero.out[1] ? 1 : 0) + (zero.out[2] ? 1 : 0);
    const long long for_zeros = std::min<long long>(2 * di->sm_count, outputs * zero.n / (4 * 8 * LAYOUT_THREADS)), n_blocks = std::max(blocks, for_zeros);
    return launch_dependent(any_output(zero) ? pad_rows_kernel<true> : pad_rows_kernel<false>, dim3((unsigned)n_blocks, pad_x && pad_y ? 2 : 1), LAYOUT_THREADS, 0, st, pad_x ? px : py, py, rows, zero);
  };
  return tc_linear_stats_pitched(di, pad_x ? (const void*)px.dst : X, pad_y ? (const void*)py.dst : dY, B, T, d_in, d_out, phi, out_mean, out_stat, out_sign,
                         accumulate != 0, l.pitch_x, l.pitch_y, st, pad);
}

// Tile of the unfolding kernel: output positions across and down, and channels per round, so that a block's shared memory (the input
// rows) stays within its budget.  False: a receptive field too large for that.
struct UnfoldTile {
  int tile_w, tile_h, chan, cols, img_rows, row_step, kh_step, smem;
};
static bool unfold_tile(const ConvGeom& g, int sm_count, UnfoldTile* t) {
  const int kk = g.Kh * g.Kw;
  auto smem = [&](int chan, int cols) { return (long long)((chan * kk + 7) / 8 * 8) * 4 + ((long long)chan * g.Kh * cols + 8) * 2; };
  auto cols_of = [&](int w) { return (long long)(w - 1) * g.sw + (long long)(g.Kw - 1) * g.dw + 1; };
  for (int w = g.Wo < 128 ? g.Wo : 128;; w = (w + 1) / 2) {
    const long long cols = cols_of(w);
    for (int chan = g.C; chan > 0; chan = chan > 8 ? (chan - 1) / 8 * 8 : 0) {
      if ((long long)chan * kk < (1 << 14) && cols < (1 << 16) && smem(chan, (int)cols) <= UNFOLD_SMEM_BYTES) {
        // one output row: the kernel's rows alone.  (An extra column where pairs have to start at an even one, and a whole pair at the end: less than
        // the 4 bytes per feature counted above.)
        int even = ((int)cols + 2) & ~1;
        // Rows an odd number of words apart, where there is room: threads side by side gather from rows two or three apart (12 images of 64 x 76 x 76, 3 x 3: 40
        // words 93 us, 39 before pairs were loaded 85, 41 60; 32 of 3 x 56 x 56, 7 x 7, 44.5 -> 38.2).
        if (even % 4 == 0 && (long long)chan * g.Kh * (even + 2) * 2 <= UNFOLD_SMEM_BYTES) even += 2;
        *t = {w, 1, chan, even, g.Kh, g.dh, 1, chan * g.Kh * even * 2};
        // Several output rows share their input rows, as long as about four blocks are left to an SM: fewer blocks hide less of each other's
        // latency (8 images of 64 x 28 x 28, 3 x 3, one row to a block 32 us, eight 39 before the loads were batched).
        const long long w_tiles = (g.Wo + w - 1) / w;
        for (int h = 8; h > 1; h /= 2) {
          const long long rows = (long long)(h - 1) * g.sh + (long long)(g.Kh - 1) * g.dh + 1, bytes = chan * rows * even * 2;
          if (h > g.Ho || bytes > UNFOLD_SMEM_BYTES || w_tiles * ((g.Ho + h - 1) / h) * g.B < 4ll * sm_count) continue;
          *t = {w, h, chan, even, (int)rows, 1, g.dh, (int)bytes};
          break;
        }
        return true;
      }
    }
    if (w == 1) return false;
  }
}
static bool conv_geom(int B, int C, int H, int W, int F, int Kh, int Kw, int sh, int sw, int ph, int pw, int dh, int dw, ConvGeom* g) {
  if (B < 1 || C < 1 || H < 1 || W < 1 || F < 1 || Kh < 1 || Kw < 1 || sh < 1 || sw < 1 || ph < 0 || pw < 0 || dh < 1 || dw < 1) return false;
  const long long ho = ((long long)H + 2ll * ph - (long long)dh * (Kh - 1) - 1) / sh + 1, wo = ((long long)W + 2ll * pw - (long long)dw * (Kw - 1) - 1) / sw + 1;
  if ((long long)H + 2ll * ph < (long long)dh * (Kh - 1) + 1 || (long long)W + 2ll * pw < (long long)dw * (Kw - 1) + 1) return false;
  if (ho > 65535 || wo > (1 << 24) || B > 65535 || (double)C * Kh * Kw >= (double)(1 << 28) || (double)ho * wo * B >= (double)(1ll << 31)) return false;
  *g = {B, C, H, W, F, Kh, Kw, sh, sw, ph, pw, dh, dw, (int)ho, (int)wo};
  return true;
}

size_t pe_conv2d_stats_workspace_bytes(int B, int C, int H, int W, int F, int Kh, int Kw, int stride_h, int stride_w, int pad_h, int pad_w,
                                       int dil_h, int dil_w) {
  ConvGeom g;
  UnfoldTile t;
  if (!conv_geom(B, C, H, W, F, Kh, Kw, stride_h, stride_w, pad_h, pad_w, dil_h, dil_w, &g) || !unfold_tile(g, 0, &t)) return 0;
  const PaddedLayout l = padded_layout(B, g.Ho * g.Wo, C * Kh * Kw, F, true);
  return l.x_bytes + l.y_bytes;
}

pe_status_t pe_conv2d_stats(const void* x, const void* grad_out, int B, int C, int H, int W, int F, int Kh, int Kw, int stride_h, int stride_w,
                            int pad_h, int pad_w, int dil_h, int dil_w, pe_phi_t phi, float* out_mean, float* out_stat, void* workspace,
                            size_t workspace_bytes, pe_stream_t stream) {
  ConvGeom g;
  UnfoldTile t;
  if (!conv_geom(B, C, H, W, F, Kh, Kw, stride_h, stride_w, pad_h, pad_w, dil_h, dil_w, &g)) return PE_ERR_DIM;
  if (!unfold_tile(g, 0, &t)) return PE_ERR_UNSUPPORTED_SHAPE;
  if (!x || !grad_out) return PE_ERR_NULL;
  const int T = g.Ho * g.Wo, d_in = C * Kh * Kw;
  const PaddedLayout l = padded_layout(B, T, d_in, F, true);
  if (!workspace || workspace_bytes < l.x_bytes + l.y_bytes) return PE_ERR_WORKSPACE;
  if (!aligned(workspace, 256) || !aligned(x, 2) || !aligned(grad_out, 2)) return PE_ERR_ALIGN;
  uint16_t* const X = static_cast<uint16_t*>(workspace);
  uint16_t* const dY = reinterpret_cast<uint16_t*>(static_cast<char*>(workspace) + l.x_bytes);
  pe_status_t rc = validate_stats(X, dY, B, T, d_in, F, out_mean, out_stat, true, 16);
  if (rc != PE_OK) return rc;
  if (phi != PE_PHI_IDENTITY && phi != PE_PHI_SQUARE && phi != PE_PHI_SIGN) return PE_ERR_PHI;
  const int forced = g_path.load();
  const bool whole = tc_shape_ok(B, T, d_in, F);
  if (forced >= PE_PATH_TENSOR && !whole) return PE_ERR_UNSUPPORTED_SHAPE;
  DeviceInfo* di = nullptr;
  rc = device_info(&di);
  if (rc != PE_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  ConvOperands o;
  o.x = static_cast<const uint16_t*>(x); o.gy = static_cast<const uint16_t*>(grad_out); o.X = X; o.dY = dY;
  o.pitch_x = l.pitch_x; o.pitch_y = l.pitch_y;
  unfold_tile(g, di->sm_count, &t);
  o.tile_w = t.tile_w; o.tile_h = t.tile_h; o.chan = t.chan; o.cols = t.cols; o.img_rows = t.img_rows; o.row_step = t.row_step; o.kh_step = t.kh_step;
  o.pairs = W % 2 == 0 && aligned(x, 4) ? 1 : 0;
  const uint32_t per_row = (uint32_t)(o.pairs ? t.cols / 2 : t.cols);
  o.per_row_magic = (uint32_t)(((1ull << 32) + per_row - 1) / per_row); o.img_rows_magic = (uint32_t)(((1ull << 32) + t.img_rows - 1) / t.img_rows);
  o.w_tiles = (g.Wo + t.tile_w - 1) / t.tile_w; o.h_tiles = (g.Ho + t.tile_h - 1) / t.tile_h;
  o.unfold_blocks = (long long)o.w_tiles * o.h_tiles * B;
  o.t_tiles = (T + 63) / 64; o.f_tiles = (l.pitch_y + 63) / 64;
  o.vec = T % 8 == 0 && aligned(grad_out, 16) ? 1 : 0;
  const long long blocks = o.unfold_blocks + (long long)o.t_tiles * o.f_tiles * B;
  if (blocks >= (1ll << 31)) return PE_ERR_DIM;
  const LayoutStep operands = [&](const LayoutZero& zero) {
    return launch_dependent(any_output(zero) ? conv_operands_kernel<true> : conv_operands_kernel<false>, dim3((unsigned)blocks), LAYOUT_THREADS, std::max(t.smem, 64 * TRANSPOSE_PITCH * 2), st, o, g, zero);
  };
  if (forced != PE_PATH_SIMT && whole) return tc_linear_stats(di, X, dY, B, T, d_in, F, phi, out_mean, out_stat, false, st, operands);
  if (forced != PE_PATH_SIMT && padding_pays(B, T, d_in, F))
    return tc_linear_stats_pitched(di, X, dY, B, T, d_in, F, phi, out_mean, out_stat, nullptr, false, l.pitch_x, l.pitch_y, st, operands);
  if ((rc = operands(LayoutZero{})) != PE_OK) return rc;
  g_last_path.store(PE_PATH_SIMT);
  return launch_simt<__nv_bfloat16, MODE_STATS>(di, reinterpret_cast<const __nv_bfloat16*>(X), reinterpret_cast<const __nv_bfloat16*>(dY), B, T, d_in, F,
                                                (int)phi, out_mean, out_stat, st, false, SimtExtra{}, nullptr, l.pitch_x, l.pitch_y);
}

size_t pe_linear_stats_ragged_workspace_bytes(int B, int d_in, int d_out) {
  if (B < 1 || d_in < 1 || d_out < 1 || (d_in % 8) || (d_out % 8) || g_path.load() == PE_PATH_SIMT) return 0;
  return ragged_layout(B, d_in, d_out).total();
}

// Shared by pe_linear_stats_ragged and pe_example_sqnorms_ragged (norms != NULL).
static pe_status_t ragged_impl(const void* X, const void* dY, const int* seq_offsets, int B, long long total_rows, int d_in, int d_out,
                               int phi, float* out_mean, float* out_stat, float* norms, void* workspace, size_t workspace_bytes,
                               cudaStream_t st) {
  if (B < 0 || total_rows < 0 || total_rows >= (1ll << 31) || d_in < 1 || d_out < 1) return PE_ERR_DIM;
  if (B > 0 && !seq_offsets) return PE_ERR_NULL;
  if ((!X || !dY) && B > 0 && total_rows > 0) return PE_ERR_NULL;
  if (!norms && !out_mean && !out_stat) return PE_ERR_NULL;
  if (total_rows * (long long)(d_in > d_out ? d_in : d_out) >= (1ll << 40) || (long long)d_in * d_out >= (1ll << 40)) return PE_ERR_DIM;
  if (!aligned(X, 16) || !aligned(dY, 16) || !aligned(seq_offsets, 4)) return PE_ERR_ALIGN;
  if ((out_mean && !aligned(out_mean, 16)) || (out_stat && !aligned(out_stat, 16)) || (norms && !aligned(norms, 4))) return PE_ERR_ALIGN;
  if (!norms && phi != PE_PHI_IDENTITY && phi != PE_PHI_SQUARE && phi != PE_PHI_SIGN) return PE_ERR_PHI;
  DeviceInfo* di = nullptr;
  pe_status_t rc = device_info(&di);
  if (rc != PE_OK) return rc;
  if (norms) {
    if (B == 0) return PE_OK;
    if (cudaMemsetAsync(norms, 0, (size_t)B * sizeof(float), st) != cudaSuccess) { cudaGetLastError(); return PE_ERR_CUDA; }
  }
  if (B == 0 || total_rows == 0) return norms ? PE_OK : zero_outputs(out_mean, out_stat, (size_t)d_in * d_out * sizeof(float), st);
  const int forced = g_path.load();
  const bool tc_ok = (d_in % 8) == 0 && (d_out % 8) == 0;
  if (forced >= PE_PATH_TENSOR && !tc_ok) return PE_ERR_UNSUPPORTED_SHAPE;
  if (tc_ok && forced != PE_PATH_SIMT) {
    if (!workspace || workspace_bytes < ragged_layout(B, d_in, d_out).total()) return PE_ERR_WORKSPACE;
    if (!aligned(workspace, 256)) return PE_ERR_ALIGN;
    g_last_path.store(PE_PATH_TENSOR);
    return launch_tc_ragged(di, X, dY, seq_offsets, B, total_rows, d_in, d_out, phi, out_mean, out_stat, norms, workspace, st);
  }
  g_last_path.store(PE_PATH_SIMT);
  SimtExtra ex{};
  ex.seq_offsets = seq_offsets; ex.total_rows = total_rows;
  const long long t_avg = total_rows / B > 0 ? total_rows / B : 1;
  const __nv_bfloat16* Xb = static_cast<const __nv_bfloat16*>(X);
  const __nv_bfloat16* Yb = static_cast<const __nv_bfloat16*>(dY);
  if (norms) return launch_simt<__nv_bfloat16, MODE_NORMS>(di, Xb, Yb, B, (int)t_avg, d_in, d_out, 1, nullptr, norms, st, true, ex);
  return launch_simt<__nv_bfloat16, MODE_STATS>(di, Xb, Yb, B, (int)t_avg, d_in, d_out, phi, out_mean, out_stat, st, false, ex);
}

pe_status_t pe_linear_stats_ragged(const void* X, const void* dY, const int* seq_offsets, int B, long long total_rows, int d_in,
                                   int d_out, pe_phi_t phi, float* out_mean, float* out_stat, void* workspace,
                                   size_t workspace_bytes, pe_stream_t stream) {
  return ragged_impl(X, dY, seq_offsets, B, total_rows, d_in, d_out, (int)phi, out_mean, out_stat, nullptr, workspace, workspace_bytes,
                     reinterpret_cast<cudaStream_t>(stream));
}

pe_status_t pe_example_sqnorms_ragged(const void* X, const void* dY, const int* seq_offsets, int B, long long total_rows, int d_in,
                                      int d_out, float* out_norms, void* workspace, size_t workspace_bytes, pe_stream_t stream) {
  if (!out_norms && B > 0) return PE_ERR_NULL;
  return ragged_impl(X, dY, seq_offsets, B, total_rows, d_in, d_out, PE_PHI_SQUARE, nullptr, nullptr, out_norms, workspace,
                     workspace_bytes, reinterpret_cast<cudaStream_t>(stream));
}

pe_status_t pe_linear_clipped_sum(const void* X, const void* dY, int B, int T, int d_in, int d_out, float clip_norm, float* sq_norms,
                                  int norms_given, float* out_sum, pe_stream_t stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (!out_sum || (!sq_norms && B > 0)) return PE_ERR_NULL;
  if (!(clip_norm >= 0.f)) return PE_ERR_DIM;
  pe_status_t rc = validate_stats(X, dY, B, T, d_in, d_out, out_sum, nullptr, false, 16);
  if (rc != PE_OK) return rc;
  if (sq_norms && !aligned(sq_norms, 4)) return PE_ERR_ALIGN;
  DeviceInfo* di = nullptr;
  rc = device_info(&di);
  if (rc != PE_OK) return rc;
  if (B == 0 || T == 0) return zero_outputs(out_sum, nullptr, (size_t)d_in * d_out * sizeof(float), st);
  if (!norms_given) {
    rc = pe_example_sqnorms(X, dY, B, T, d_in, d_out, sq_norms, stream);
    if (rc != PE_OK) return rc;
  }
  const int forced = g_path.load();
  const bool tc_ok = tc_shape_ok(B, T, d_in, d_out);
  if (forced >= PE_PATH_TENSOR && !tc_ok) return PE_ERR_UNSUPPORTED_SHAPE;
  if (tc_ok && forced != PE_PATH_SIMT) {
    g_last_path.store(PE_PATH_TENSOR);
    return launch_tc(di, X, dY, B, T, d_in, d_out, PHI_CLIP_SCALE, 1, nullptr, out_sum, st, false, nullptr, false, sq_norms, clip_norm);
  }
  g_last_path.store(PE_PATH_SIMT);
  SimtExtra ex{};
  ex.sq_norms = sq_norms; ex.clip_norm = clip_norm;
  return launch_simt<__nv_bfloat16, MODE_STATS>(di, static_cast<const __nv_bfloat16*>(X), static_cast<const __nv_bfloat16*>(dY), B, T,
                                                d_in, d_out, PHI_CLIP_SCALE, nullptr, out_sum, st, false, ex);
}

size_t pe_linear_fused_workspace_bytes(int d_in, int d_out) {
  if (d_in < 1 || d_out < 1) return 0;
  return align_up(fused_counter_words(d_in, d_out) * sizeof(unsigned int), 256);
}

// Shared by the three fused entry points.  kind: OPT_ADAM / OPT_SIGN; out_a: sum_b G_b (Adam), out_b: the statistic.
extern "C++" template <typename TIn>
pe_status_t fused_impl(const TIn* X, const TIn* dY, int B, int T, int d_in, int d_out, int kind, float* theta, void* theta_lp,
                              float* m, float* v, float* out_a, float* out_b, FusedOpt opt, void* workspace, size_t workspace_bytes,
                              cudaStream_t st, bool allow_tc) {
  if (!theta || !m || (kind == OPT_ADAM && !v)) return PE_ERR_NULL;
  if (B < 1 || T < 1) return PE_ERR_DIM;
  pe_status_t rc = validate_stats(X, dY, B, T, d_in, d_out, out_a, out_b, false, allow_tc ? 16 : 4);
  if (rc != PE_OK) return rc;
  if (!aligned(theta, 16) || !aligned(m, 16) || (v && !aligned(v, 16)) || (theta_lp && !aligned(theta_lp, 16))) return PE_ERR_ALIGN;
  if (workspace && !aligned(workspace, 256)) return PE_ERR_ALIGN;
  DeviceInfo* di = nullptr;
  rc = device_info(&di);
  if (rc != PE_OK) return rc;
  opt.kind = kind;
  opt.theta = theta; opt.theta_lp = static_cast<__nv_bfloat16*>(theta_lp); opt.m = m; opt.v = v; opt.tile_counters = nullptr;
  const int forced = g_path.load();
  const bool tc_ok = allow_tc && tc_shape_ok(B, T, d_in, d_out);
  if (forced >= PE_PATH_TENSOR && !tc_ok) return PE_ERR_UNSUPPORTED_SHAPE;
  if (tc_ok && forced != PE_PATH_SIMT) {
    if constexpr (sizeof(TIn) == 2) {
      g_last_path.store(PE_PATH_TENSOR);
      // The update inside the statistics kernel cannot overlap the contraction: the blocks of a wave finish
      // together, so a wave's update traffic reaches memory at once while the tensor cores idle (measured: about
      // 25 us per wave, against a separate update kernel that streams at the HBM rate).  Fusing saves memory (no
      // [d_out, d_in] statistic buffers) rather than time.  PE_FUSED_AUTO
      // therefore fuses only when the caller gave no buffers for the statistics; with buffers it runs the
      // statistics kernel and the update kernel back to back.
      const int mode = g_fused_mode.load();
      const bool have_stats = out_b && (kind != OPT_ADAM || out_a);
      if (mode == PE_FUSED_NEVER && !have_stats) return PE_ERR_NULL;
      if (mode == PE_FUSED_NEVER || (mode == PE_FUSED_AUTO && have_stats)) {
        rc = launch_tc(di, X, dY, B, T, d_in, d_out, kind == OPT_ADAM ? (int)PE_PHI_SQUARE : (int)PE_PHI_SIGN, 1,
                       kind == OPT_ADAM ? out_a : nullptr, out_b, st);
        if (rc != PE_OK) return rc;
        const long long n = (long long)d_in * d_out;
        __nv_bfloat16* lp = static_cast<__nv_bfloat16*>(theta_lp);
        if (kind == OPT_ADAM) return launch_microadam(di, opt.variant, theta, lp, m, v, out_a, out_b, n, opt.adam, di->status_ptr, st);
        return launch_microsignsgd(di, theta, lp, m, out_b, n, opt.sign, di->status_ptr, st);
      }
      return launch_tc_fused(di, X, dY, B, T, d_in, d_out, kind, out_a, out_b, opt, static_cast<unsigned int*>(workspace),
                             workspace_bytes / sizeof(unsigned int), st);
    }
  }
  g_last_path.store(PE_PATH_SIMT);
  return launch_simt<TIn, MODE_STATS>(di, X, dY, B, T, d_in, d_out, kind == OPT_ADAM ? (int)PE_PHI_SQUARE : (int)PE_PHI_SIGN, out_a, out_b, st,
                                      false, SimtExtra{}, &opt);
}

static pe_status_t check_adam_args(int B, pe_adam_variant_t variant, int step) {
  if (B < 1 || step < 1) return PE_ERR_DIM;
  if ((int)variant < 0 || (int)variant > 3) return PE_ERR_PHI;
  if (((int)variant == ADAM_MICRO_VAR || (int)variant == ADAM_MICRO_MSQ) && B < 2) return PE_ERR_DIM;
  return PE_OK;
}

pe_status_t pe_linear_microadam_step(const void* X, const void* dY, int B, int T, int d_in, int d_out, float* theta, void* theta_lp,
                                     float* m, float* v, float* out_mean, float* out_stat, pe_adam_variant_t variant, float grad_scale,
                                     float lr, float beta1, float beta2, float eps, int eps_inside_sqrt, float weight_decay, int step,
                                     void* workspace, size_t workspace_bytes, pe_stream_t stream) {
  pe_status_t rc = check_adam_args(B, variant, step);
  if (rc != PE_OK) return rc;
  FusedOpt opt{};
  opt.variant = (int)variant;
  opt.adam = make_adam_params(B, grad_scale, lr, beta1, beta2, eps, eps_inside_sqrt, weight_decay, step);
  return fused_impl<__nv_bfloat16>(static_cast<const __nv_bfloat16*>(X), static_cast<const __nv_bfloat16*>(dY), B, T, d_in, d_out, OPT_ADAM,
                                   theta, theta_lp, m, v, out_mean, out_stat, opt, workspace, workspace_bytes,
                                   reinterpret_cast<cudaStream_t>(stream), true);
}

pe_status_t pe_linear_microadam_step_f32(const float* X, const float* dY, int B, int T, int d_in, int d_out, float* theta, void* theta_lp,
                                         float* m, float* v, float* out_mean, float* out_stat, pe_adam_variant_t variant,
                                         float grad_scale, float lr, float beta1, float beta2, float eps, int eps_inside_sqrt,
                                         float weight_decay, int step, pe_stream_t stream) {
  pe_status_t rc = check_adam_args(B, variant, step);
  if (rc != PE_OK) return rc;
  FusedOpt opt{};
  opt.variant = (int)variant;
  opt.adam = make_adam_params(B, grad_scale, lr, beta1, beta2, eps, eps_inside_sqrt, weight_decay, step);
  return fused_impl<float>(X, dY, B, T, d_in, d_out, OPT_ADAM, theta, theta_lp, m, v, out_mean, out_stat, opt, nullptr, 0,
                           reinterpret_cast<cudaStream_t>(stream), false);
}

pe_status_t pe_linear_microsignsgd_step(const void* X, const void* dY, int B, int T, int d_in, int d_out, float* theta, void* theta_lp,
                                        float* m, float* out_sign, float lr, float beta, float weight_decay, void* workspace,
                                        size_t workspace_bytes, pe_stream_t stream) {
  if (B < 1) return PE_ERR_DIM;
  FusedOpt opt{};
  opt.sign.inv_B = (float)(1.0 / (double)B); opt.sign.beta = beta; opt.sign.lr = lr; opt.sign.wd = weight_decay;
  return fused_impl<__nv_bfloat16>(static_cast<const __nv_bfloat16*>(X), static_cast<const __nv_bfloat16*>(dY), B, T, d_in, d_out, OPT_SIGN,
                                   theta, theta_lp, m, nullptr, nullptr, out_sign, opt, workspace, workspace_bytes,
                                   reinterpret_cast<cudaStream_t>(stream), true);
}

pe_status_t pe_linear_stats_f32(const float* X, const float* dY, int B, int T, int d_in, int d_out, pe_phi_t phi,
                                float* out_mean, float* out_stat, pe_stream_t stream) {
  return linear_stats_impl<float>(X, dY, B, T, d_in, d_out, phi, out_mean, out_stat, reinterpret_cast<cudaStream_t>(stream), false);
}

pe_status_t pe_token_sqstats(const void* X, const void* dY, int B, int T, int d_in, int d_out, float* out_stat,
                             pe_stream_t stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (!out_stat) return PE_ERR_NULL;
  pe_status_t rc = validate_stats(X, dY, B, T, d_in, d_out, out_stat, nullptr, false, 16);
  if (rc != PE_OK) return rc;
  DeviceInfo* di = nullptr;
  rc = device_info(&di);
  if (rc != PE_OK) return rc;
  if (B == 0 || T == 0) return zero_outputs(out_stat, nullptr, (size_t)d_in * d_out * sizeof(float), st);
  const int forced = g_path.load();
  const long long rows = (long long)B * T;
  const bool shape_ok = tc_shape_ok(B, T, d_in, d_out) && rows < (1ll << 31);
  if (forced >= PE_PATH_TENSOR && !shape_ok) return PE_ERR_UNSUPPORTED_SHAPE;
  if (shape_ok && rows >= TOKEN_TC_MIN_ROWS && forced != PE_PATH_SIMT) {
    g_last_path.store(PE_PATH_TENSOR);
    return launch_tok(di, X, dY, rows, d_in, d_out, out_stat, st);
  }
  g_last_path.store(PE_PATH_SIMT);
  return launch_simt<__nv_bfloat16, MODE_TOKEN>(di, static_cast<const __nv_bfloat16*>(X), static_cast<const __nv_bfloat16*>(dY), B, T,
                                                d_in, d_out, 0, nullptr, out_stat, st);
}

// Workspace of the staged per-token statistic: the column maxima of X and dY (one 32-bit word per
// column), then the scaled squares of X and of dY (IEEE half, or e4m3 in the fp8 form), each part 256-byte aligned.
// On large layers (half form) the squares are staged chunk by chunk in one pass instead: the scales of every chunk, then the
// squares, padded to whole chunks.
struct StagedLayout {
  size_t max_bytes, x_bytes, y_bytes;
  long long chunks;           // 0: two passes over the inputs
  size_t total() const { return max_bytes + x_bytes + y_bytes; }
};
// From this many input elements on.  The line is where callers begin to prefer a staged form to the one-kernel one; it is not where the
// one-pass staging begins to win, and a workspace of the two-pass form's size stays enough below it.  One kernel / one-pass / two-pass, us:
// 16 x 128 x 512 x 2048 (5e6) 19 / 23 / 35, 64 x 256 x 512 x 2048 (4e7) 69 / 68 / 88, 64 x 256 x 1024 x 4096 (8e7) 225 / 154 / 203,
// 40 x 1000 x 1024 x 1400 (9.7e7) 212 / 171 / 223, 40 x 1000 x 1024 x 1600 (1.05e8) 269 / 190 / 243, 16 x 1024 x 2048 x 8192 (1.7e8) 941 / 491 / 672,
// 128 x 512 x 512 x 1024 (1.0e8, few tiles) 141 / 151 / 196.
constexpr double STAGE_CHUNKS_MIN_ELEMS = 1e8;
static StagedLayout chunked_layout(int B, int T, int d_in, int d_out) {
  StagedLayout l;
  l.chunks = ((long long)B * T + STAGE_CHUNK - 1) / STAGE_CHUNK;
  l.max_bytes = align_up((size_t)l.chunks * ((size_t)d_in + (size_t)d_out) * sizeof(float), 256);
  l.x_bytes = align_up((size_t)l.chunks * STAGE_CHUNK * d_in * 2, 256);
  l.y_bytes = align_up((size_t)l.chunks * STAGE_CHUNK * d_out * 2, 256);
  return l;
}
static bool chunks_pay(int B, int T, int d_in, int d_out) {
  return (double)B * T * ((double)d_in + d_out) >= STAGE_CHUNKS_MIN_ELEMS && ((long long)B * T + STAGE_CHUNK - 1) / STAGE_CHUNK <= 65535;
}
static StagedLayout staged_layout(int B, int T, int d_in, int d_out, bool fp8 = false) {
  const size_t rows = (size_t)B * (size_t)T, es = fp8 ? 1 : 2;
  StagedLayout l;
  l.chunks = 0;
  l.max_bytes = align_up(((size_t)d_in + (size_t)d_out) * 4, 256);
  l.x_bytes = align_up(rows * d_in * es, 256);
  l.y_bytes = align_up(rows * d_out * es, 256);
  return l;
}
// the fp8 form stages one byte per element: TMA wants 16-byte row pitches
static bool token_fp8_ok(int B, int T, int d_in, int d_out) { return token_tc_ok(B, T, d_in, d_out) && (d_in % 16) == 0 && (d_out % 16) == 0; }

size_t pe_token_sqstats_staged_workspace_bytes(int B, int T, int d_in, int d_out) {
  if (g_path.load() == PE_PATH_SIMT || !token_tc_ok(B, T, d_in, d_out)) return 0;
  return (chunks_pay(B, T, d_in, d_out) ? chunked_layout(B, T, d_in, d_out) : staged_layout(B, T, d_in, d_out)).total();
}
size_t pe_token_sqstats_fp8_workspace_bytes(int B, int T, int d_in, int d_out) {
  if (g_path.load() == PE_PATH_SIMT || !token_tc_ok(B, T, d_in, d_out)) return 0;
  return staged_layout(B, T, d_in, d_out, token_fp8_ok(B, T, d_in, d_out)).total();
}

// Grid of the column-wise staging kernels: x covers the columns in groups of 256, y slices the rows
// so that the whole grid is a few blocks per SM.
static dim3 stage_grid(long long rows, int d, int sm_count) {
  const int gx = (d + 255) / 256;
  long long gy = ((long long)sm_count * 8 + gx - 1) / gx;
  const long long max_gy = rows / 64 > 0 ? rows / 64 : 1;
  if (gy > max_gy) gy = max_gy;
  if (gy > 65535) gy = 65535;
  if (gy < 1) gy = 1;
  return dim3((unsigned)gx, (unsigned)gy, 1);
}

// The plain contraction of e4m3 operands x8 [B, T, d_in], y8 [B, T, d_out] (one byte per element) into out.
static pe_status_t launch_tc_fp8(DeviceInfo* di, const void* x8, const void* y8, int B, int T, int d_in, int d_out, float* out,
                                 cudaStream_t st) {
  using Op = TcOperand<false, 256, 128, true>;
  EncodeTiledFn enc = encode_fn();
  if (!enc) return PE_ERR_CUDA;
  auto operand_map = [&](CUtensorMap* m, const void* base, int d) {
    cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)T, (cuuint64_t)B};
    cuuint64_t strides[2] = {(cuuint64_t)d, (cuuint64_t)T * (cuuint64_t)d};
    cuuint32_t box[3] = {(cuuint32_t)Op::BOX_FEATS, (cuuint32_t)Op::BK, 1u};
    cuuint32_t estr[3] = {1u, 1u, 1u};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  };
  CUtensorMap mx, my, mo;
  if (!operand_map(&mx, x8, d_in) || !operand_map(&my, y8, d_out)) return PE_ERR_CUDA;
  pe_status_t rc = make_output_map(&mo, out, d_in, d_out);
  if (rc != PE_OK) return rc;
  const int tiles_n = (d_in + 255) / 256, pairs_m = (d_out + TC_PAIR_M - 1) / TC_PAIR_M;
  if ((long long)tiles_n * pairs_m > (1ll << 29)) return PE_ERR_DIM;
  const int slots = di->sm_count / 2 > 0 ? di->sm_count / 2 : 1;
  const int ns = plan_tiles(&COST_PLAIN_FP8, 1, B, T, d_in, d_out, slots, std::max(16, slots), 1).ns;
  if (ns > 1) {
    rc = zero_for_split(di, out, nullptr, (size_t)d_in * d_out, st);
    if (rc != PE_OK) return rc;
  }
  TcParams p{};
  p.B = B; p.T = T; p.d_in = d_in; p.d_out = d_out; p.nsplit = ns; p.per_example = 0; p.half_operands = 0; p.accumulate = 0;
  p.wait_at_start = ns == 1 ? 1 : 0;
  p.pairs_m = pairs_m; p.tiles_n = tiles_n; p.band = choose_band(pairs_m, tiles_n, 256, ns, di->sm_count / 2);
  p.out_mean = nullptr; p.out_stat = out; p.out_sign = nullptr; p.out_norms = nullptr; p.dev_status = di->status_ptr;
  p.seq_offsets = nullptr; p.sq_norms = nullptr; p.clip_norm = 0.f;
  return launch_tc_inst<0, false, 256, MEAN_NONE, 128, false, OPT_NONE, true>(di, 25, mx, my, mo, mo, mo, p, dim3(2 * pairs_m * tiles_n, 1, ns), st);
}

// The two-pass per-token statistic on half (fp8 = false) or e4m3 (fp8 = true) squares.
static pe_status_t token_staged_impl(const void* X, const void* dY, int B, int T, int d_in, int d_out, float* out_stat, void* workspace,
                                     size_t workspace_bytes, cudaStream_t st, bool want_fp8) {
  if (!out_stat) return PE_ERR_NULL;
  pe_status_t rc = validate_stats(X, dY, B, T, d_in, d_out, out_stat, nullptr, false, 16);
  if (rc != PE_OK) return rc;
  DeviceInfo* di = nullptr;
  rc = device_info(&di);
  if (rc != PE_OK) return rc;
  if (B == 0 || T == 0) return zero_outputs(out_stat, nullptr, (size_t)d_in * d_out * sizeof(float), st);
  const int forced = g_path.load();
  const bool tc_ok = token_tc_ok(B, T, d_in, d_out);
  if (forced >= PE_PATH_TENSOR && !tc_shape_ok(B, T, d_in, d_out)) return PE_ERR_UNSUPPORTED_SHAPE;
  if (tc_ok && forced != PE_PATH_SIMT) {
    const bool fp8 = want_fp8 && token_fp8_ok(B, T, d_in, d_out);
    const long long rows = (long long)B * T;
    const StagedLayout l = staged_layout(B, T, d_in, d_out, fp8);
    if (!workspace || workspace_bytes < l.total()) return PE_ERR_WORKSPACE;
    if (!aligned(workspace, 256)) return PE_ERR_ALIGN;
    if (!fp8 && chunks_pay(B, T, d_in, d_out) && workspace_bytes >= chunked_layout(B, T, d_in, d_out).total()) {
      const StagedLayout c = chunked_layout(B, T, d_in, d_out);
      float* const scale_x = static_cast<float*>(workspace);
      float* const scale_y = scale_x + c.chunks * d_in;
      __half* const hx = reinterpret_cast<__half*>(static_cast<char*>(workspace) + c.max_bytes);
      __half* const hy = reinterpret_cast<__half*>(static_cast<char*>(workspace) + c.max_bytes + c.x_bytes);
      const ChunkTensor cx = {static_cast<const uint16_t*>(X), hx, scale_x, d_in}, cy = {static_cast<const uint16_t*>(dY), hy, scale_y, d_out};
      const int gx = (d_in + 63) / 64, gy = (d_out + 63) / 64;
      square_chunks_kernel<<<dim3((unsigned)(gx + gy), (unsigned)c.chunks), STAGE_THREADS, 0, st>>>(cx, cy, gx, rows);
      if ((rc = check_launch()) != PE_OK) return rc;
      g_last_path.store(PE_PATH_TENSOR);
      return launch_tc(di, hx, hy, (int)c.chunks, STAGE_CHUNK, d_in, d_out, PHI_UNSCALE, 1, nullptr, out_stat, st, true, nullptr, false, nullptr, 0.f, 0, 0,
                       false, scale_x, scale_y);
    }
    uint32_t* max_x = static_cast<uint32_t*>(workspace);
    uint32_t* max_y = max_x + d_in;
    void* x2 = static_cast<char*>(workspace) + l.max_bytes;
    void* y2 = static_cast<char*>(workspace) + l.max_bytes + l.x_bytes;
    const uint16_t* Xb = static_cast<const uint16_t*>(X);
    const uint16_t* Yb = static_cast<const uint16_t*>(dY);
    if (cudaMemsetAsync(max_x, 0, ((size_t)d_in + (size_t)d_out) * 4, st) != cudaSuccess) { cudaGetLastError(); return PE_ERR_CUDA; }
    // one launch per pass serves both tensors (gridDim.z picks X or dY; the grid is sized for the wider one)
    dim3 grid = stage_grid(rows, d_in > d_out ? d_in : d_out, di->sm_count);
    grid.y = (grid.y + 1) / 2;
    grid.z = 2;
    const StageTensor sx = {Xb, x2, max_x, d_in}, sy = {Yb, y2, max_y, d_out};
    column_max_kernel<<<grid, STAGE_THREADS, 0, st>>>(sx, sy, rows);
    if ((rc = check_launch()) != PE_OK) return rc;
    if (fp8) square_to_lp_kernel<true><<<grid, STAGE_THREADS, 0, st>>>(sx, sy, rows);
    else square_to_lp_kernel<false><<<grid, STAGE_THREADS, 0, st>>>(sx, sy, rows);
    if ((rc = check_launch()) != PE_OK) return rc;
    // B and T only enter through B*T: regroup the rows into two-stage "examples" when possible so
    // the batch split has many units to balance.
    const int regroup = fp8 ? 2 * TcOperand<false, 256, 128, true>::BK : 2 * TcOperand<false, 256>::BK;
    int Bp = B, Tp = T;
    if (T % regroup == 0 && rows / regroup < (1ll << 30)) { Bp = (int)(rows / regroup); Tp = regroup; }
    g_last_path.store(PE_PATH_TENSOR);
    rc = fp8 ? launch_tc_fp8(di, x2, y2, Bp, Tp, d_in, d_out, out_stat, st)
             : launch_tc(di, x2, y2, Bp, Tp, d_in, d_out, PE_PHI_IDENTITY, 0, nullptr, out_stat, st, true);
    if (rc != PE_OK) return rc;
    const int ugrid = grid_for((long long)d_in * d_out / 4 + 4, di->sm_count);
    if (fp8) unscale_kernel<true><<<ugrid, STAGE_THREADS, 0, st>>>(out_stat, d_out, d_in, max_x, max_y);
    else unscale_kernel<false><<<ugrid, STAGE_THREADS, 0, st>>>(out_stat, d_out, d_in, max_x, max_y);
    return check_launch();
  }
  g_last_path.store(PE_PATH_SIMT);
  return launch_simt<__nv_bfloat16, MODE_TOKEN>(di, static_cast<const __nv_bfloat16*>(X), static_cast<const __nv_bfloat16*>(dY), B, T,
                                                d_in, d_out, 0, nullptr, out_stat, st);
}

pe_status_t pe_token_sqstats_staged(const void* X, const void* dY, int B, int T, int d_in, int d_out, float* out_stat,
                                    void* workspace, size_t workspace_bytes, pe_stream_t stream) {
  return token_staged_impl(X, dY, B, T, d_in, d_out, out_stat, workspace, workspace_bytes, reinterpret_cast<cudaStream_t>(stream), false);
}

pe_status_t pe_token_sqstats_fp8(const void* X, const void* dY, int B, int T, int d_in, int d_out, float* out_stat,
                                 void* workspace, size_t workspace_bytes, pe_stream_t stream) {
  return token_staged_impl(X, dY, B, T, d_in, d_out, out_stat, workspace, workspace_bytes, reinterpret_cast<cudaStream_t>(stream), true);
}

// ---------------------------------------------------------------------------------------------
// Allocation-free per-token statistic.  The staging buffer is a device array inside this module's
// image.  In host code its name is only a handle for the runtime's symbol lookups, never a device
// address: the address each device gave the array is looked up once per device (with that device
// current) and cached; that looked-up pointer is what the kernels receive.
static __device__ __align__(256) unsigned char g_static_scratch[PE_STATIC_SCRATCH_BYTES];

struct StaticScratchSlot {
  std::atomic<int> ready{0};
  void* ptr = nullptr;
};
static StaticScratchSlot g_static_slot[MAX_DEVICES];

static pe_status_t static_scratch_ptr(void** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) { cudaGetLastError(); return PE_ERR_CUDA; }
  StaticScratchSlot& slot = g_static_slot[dev];
  if (!slot.ready.load(std::memory_order_acquire)) {
    void* p = nullptr;
    if (cudaGetSymbolAddress((void**)&p, g_static_scratch) != cudaSuccess || !p) { cudaGetLastError(); return PE_ERR_CUDA; }
    slot.ptr = p;                       // concurrent first calls look up the same address
    slot.ready.store(1, std::memory_order_release);
  }
  *out = slot.ptr;
  return PE_OK;
}

pe_status_t pe_token_sqstats_static(const void* X, const void* dY, int B, int T, int d_in, int d_out, float* out_stat,
                                    pe_stream_t stream) {
  if (!out_stat) return PE_ERR_NULL;
  pe_status_t rc = validate_stats(X, dY, B, T, d_in, d_out, out_stat, nullptr, false, 16);
  if (rc != PE_OK) return rc;
  // Refuse what does not fit before touching the device.
  if (pe_token_sqstats_staged_workspace_bytes(B, T, d_in, d_out) > (size_t)PE_STATIC_SCRATCH_BYTES) return PE_ERR_WORKSPACE;
  DeviceInfo* di = nullptr;
  rc = device_info(&di);
  if (rc != PE_OK) return rc;
  void* scratch = nullptr;
  rc = static_scratch_ptr(&scratch);
  if (rc != PE_OK) return rc;
  // Nothing in the array has to start at zero: the squaring pre-pass rewrites every element the
  // contraction reads.  Everything below only enqueues kernels and memsets on `stream`.
  return pe_token_sqstats_staged(X, dY, B, T, d_in, d_out, out_stat, scratch, (size_t)PE_STATIC_SCRATCH_BYTES, stream);
}

pe_status_t pe_token_sqstats_f32(const float* X, const float* dY, int B, int T, int d_in, int d_out, float* out_stat,
                                 pe_stream_t stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (!out_stat) return PE_ERR_NULL;
  pe_status_t rc = validate_stats(X, dY, B, T, d_in, d_out, out_stat, nullptr, false, 4);
  if (rc != PE_OK) return rc;
  DeviceInfo* di = nullptr;
  rc = device_info(&di);
  if (rc != PE_OK) return rc;
  if (B == 0 || T == 0) return zero_outputs(out_stat, nullptr, (size_t)d_in * d_out * sizeof(float), st);
  g_last_path.store(PE_PATH_SIMT);
  return launch_simt<float, MODE_TOKEN>(di, X, dY, B, T, d_in, d_out, 0, nullptr, out_stat, st);
}

pe_status_t microadam_family_step(float* theta, void* theta_lp, float* m, float* v, const float* sum_g, const float* sum_g2,
                                  long long n, int B, pe_adam_variant_t variant, float grad_scale, float lr, float beta1,
                                  float beta2, float eps, int eps_inside_sqrt, float weight_decay, int step,
                                  pe_stream_t stream) {
  if (!theta || !m || !v || !sum_g || !sum_g2) return PE_ERR_NULL;
  if (n < 0 || B < 1 || step < 1) return PE_ERR_DIM;
  if ((int)variant < 0 || (int)variant > 3) return PE_ERR_PHI;
  if (((int)variant == ADAM_MICRO_VAR || (int)variant == ADAM_MICRO_MSQ) && B < 2) return PE_ERR_DIM;   // a variance needs two examples
  if (!aligned(theta, 16) || !aligned(m, 16) || !aligned(v, 16) || !aligned(sum_g, 16) || !aligned(sum_g2, 16) ||
      (theta_lp && !aligned(theta_lp, 16)))
    return PE_ERR_ALIGN;
  DeviceInfo* di = nullptr;
  pe_status_t rc = device_info(&di);
  if (rc != PE_OK) return rc;
  if (n == 0) return PE_OK;
  const AdamParams p = make_adam_params(B, grad_scale, lr, beta1, beta2, eps, eps_inside_sqrt, weight_decay, step);
  return launch_microadam(di, (int)variant, theta, static_cast<__nv_bfloat16*>(theta_lp), m, v, sum_g, sum_g2, n, p, nullptr,
                          reinterpret_cast<cudaStream_t>(stream));
}

pe_status_t microadam_step(float* theta, void* theta_lp, float* m, float* v, const float* sum_g, const float* sum_g2,
                           long long n, int B, float grad_scale, float lr, float beta1, float beta2, float eps,
                           int eps_inside_sqrt, float weight_decay, int step, pe_stream_t stream) {
  return microadam_family_step(theta, theta_lp, m, v, sum_g, sum_g2, n, B, PE_ADAM_MICRO, grad_scale, lr, beta1, beta2, eps,
                               eps_inside_sqrt, weight_decay, step, stream);
}

pe_status_t microsignsgd_step(float* theta, void* theta_lp, float* m, const float* sum_sign, long long n, int B, float lr,
                              float beta, float weight_decay, pe_stream_t stream) {
  if (!theta || !m || !sum_sign) return PE_ERR_NULL;
  if (n < 0 || B < 1) return PE_ERR_DIM;
  if (!aligned(theta, 16) || !aligned(m, 16) || !aligned(sum_sign, 16) || (theta_lp && !aligned(theta_lp, 16))) return PE_ERR_ALIGN;
  DeviceInfo* di = nullptr;
  pe_status_t rc = device_info(&di);
  if (rc != PE_OK) return rc;
  if (n == 0) return PE_OK;
  SignParams p;
  p.inv_B = (float)(1.0 / (double)B); p.beta = beta; p.lr = lr; p.wd = weight_decay;
  return launch_microsignsgd(di, theta, static_cast<__nv_bfloat16*>(theta_lp), m, sum_sign, n, p, nullptr, reinterpret_cast<cudaStream_t>(stream));
}

const char* pe_status_string(pe_status_t s) {
  switch (s) {
    case PE_OK: return "PE_OK";
    case PE_ERR_NULL: return "PE_ERR_NULL";
    case PE_ERR_DIM: return "PE_ERR_DIM";
    case PE_ERR_ALIGN: return "PE_ERR_ALIGN";
    case PE_ERR_UNSUPPORTED_SHAPE: return "PE_ERR_UNSUPPORTED_SHAPE";
    case PE_ERR_PHI: return "PE_ERR_PHI";
    case PE_ERR_ARCH: return "PE_ERR_ARCH";
    case PE_ERR_CUDA: return "PE_ERR_CUDA";
    case PE_ERR_TIMEOUT: return "PE_ERR_TIMEOUT";
    case PE_ERR_WORKSPACE: return "PE_ERR_WORKSPACE";
  }
  return "PE_ERR_UNKNOWN";
}

pe_status_t pe_get_async_status(pe_stream_t stream, int* detail) {
  if (detail) *detail = 0;
  DeviceInfo* di = nullptr;
  pe_status_t rc = device_info(&di);
  if (rc != PE_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (cudaStreamSynchronize(st) != cudaSuccess) { cudaGetLastError(); return PE_ERR_CUDA; }
  unsigned int word = 0;
  if (cudaMemcpy(&word, di->status_ptr, sizeof word, cudaMemcpyDeviceToHost) != cudaSuccess) { cudaGetLastError(); return PE_ERR_CUDA; }
  if (word == 0) return PE_OK;
  if (cudaMemset(di->status_ptr, 0, sizeof word) != cudaSuccess) { cudaGetLastError(); return PE_ERR_CUDA; }
  if (detail) *detail = (int)word;
  return PE_ERR_TIMEOUT;
}

pe_status_t pe_set_wait_limit_cycles(long long cycles) {
  DeviceInfo* di = nullptr;
  pe_status_t rc = device_info(&di);
  if (rc != PE_OK) return rc;
  const long long v = cycles > 0 ? cycles : sm100::WAIT_CYCLE_LIMIT_DEFAULT;
  if (cudaMemcpyToSymbol(sm100::g_wait_cycle_limit, &v, sizeof v) != cudaSuccess) { cudaGetLastError(); return PE_ERR_CUDA; }
  return PE_OK;
}

int pe_set_fused_update(int mode) {
  if (mode < PE_FUSED_AUTO || mode > PE_FUSED_NEVER) return -1;
  return g_fused_mode.exchange(mode);
}

int pe_set_path(int path) {
  if (path < PE_PATH_AUTO || path > PE_PATH_TENSOR_WIDE) return -1;
  return g_path.exchange(path);
}
int pe_tile_order_band(int d_in, int d_out, int tile_cols, int batch_slices, int sm_count) {
  if (d_in < 1 || d_out < 1 || batch_slices < 1 || sm_count < 2) return 0;
  if (tile_cols != 128 && tile_cols != 192 && tile_cols != 256) return 0;
  const long long tiles_n = ((long long)d_in + tile_cols - 1) / tile_cols, pairs_m = ((long long)d_out + pe::TC_PAIR_M - 1) / pe::TC_PAIR_M;
  if (tiles_n * pairs_m > (1ll << 29)) return 0;
  return pe::choose_band((int)pairs_m, (int)tiles_n, tile_cols, batch_slices, sm_count / 2);
}
pe_status_t pe_plan_query(int what, int outputs, int B, int T, int d_in, int d_out, int sm_count, long long* plan) {
  if (!plan) return PE_ERR_NULL;
  if (B < 1 || T < 1 || d_in < 1 || d_out < 1 || sm_count < 2) return PE_ERR_DIM;
  const bool mean = outputs & 1, square = outputs & 2, sign = outputs & 4;
  switch (what) {
    case PE_PLAN_SHORT: {
      if (!(mean || square || sign) || T > pe::SHORT_T) return PE_ERR_DIM;
      const long long tiles = (((long long)d_in + pe::SHORT_NT - 1) / pe::SHORT_NT) * (((long long)d_out + pe::TC_PAIR_M - 1) / pe::TC_PAIR_M);
      if (tiles > (1ll << 29)) return PE_ERR_DIM;
      const pe::ShortPlan p = pe::plan_short(mean, square, sign, B, T, d_in, d_out, sm_count / 2, false, d_in % 8 == 0);
      plan[0] = p.whole; plan[1] = p.split; plan[2] = p.whole > 0 ? B : (B + p.split - 1) / p.split; plan[3] = p.run;
      return PE_OK;
    }
    case PE_PLAN_SIMT_STATS:
    case PE_PLAN_SIMT_TOKEN:
    case PE_PLAN_SIMT_NORMS: {
      if (d_out > pe::SIMT_MAX_D_OUT) return PE_ERR_DIM;
      const int mode = what == PE_PLAN_SIMT_STATS ? pe::MODE_STATS : what == PE_PLAN_SIMT_TOKEN ? pe::MODE_TOKEN : pe::MODE_NORMS;
      const pe::SimtPlan p = pe::plan_simt(sm_count, mode, mean, sign && !mean, B, T, d_in, d_out);
      plan[0] = p.tile; plan[1] = p.slices; plan[2] = p.cluster;
      return PE_OK;
    }
    case PE_PLAN_TOKEN: {
      const long long chunks = ((long long)B * T + pe::TOK_BK - 1) / pe::TOK_BK;
      const pe::TokPlan p = pe::plan_tok((int)std::min<long long>(chunks, 1 << 30), d_in, d_out, sm_count / 2);
      plan[0] = p.ns; plan[1] = p.deal_tiles; plan[2] = p.deal_pairs; plan[3] = p.pairs;
      return PE_OK;
    }
    case PE_PLAN_NORMS: {
      const pe::NormsPlan p = pe::plan_norms(B, T, d_in, d_out, sm_count / 2);
      plan[0] = p.slices; plan[1] = p.examples; plan[2] = p.order_slices;
      return PE_OK;
    }
    default: return PE_ERR_DIM;
  }
}
int pe_last_path(void) { return g_last_path.load(); }
long long pe_launch_count(void) { return g_launches.load(); }
void pe_reset_launch_count(void) { g_launches.store(0); }

}  // extern "C"
