// Layout kernels in front of the tensor-core contraction.  For operands whose rows TMA cannot address (it wants 16-byte
// row pitches): rows of a width that is no multiple of 8 copied to a padded pitch, and the operands of a convolution's
// weight gradient (Appendix B.4) unfolded straight into that form.  For the contractions that stand for the statistics of one-token
// examples: the halves of their squares and their signs.  The padding kernel is bound by HBM bandwidth, the unfolding kernel by its
// gathers from shared memory, the one-token kernel by launch latency and HBM.  The columns
// between the width and the pitch are never read (the tensor maps end at the width).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "pe_sm100.cuh"

namespace pe {

constexpr int LAYOUT_THREADS = 256;
constexpr int UNFOLD_SMEM_BYTES = 48 * 1024;

// These kernels also zero the outputs of a split batch, which saves a launch between them and the statistics kernel, and are launched as
// programmatic dependents: 8 x 64 x 257 x 511 19.6 -> 17.3 us, 16 x 100 x 333 x 2001 24.9 -> 21.6, 16 images of 16 x 56 x 56 under 3 x 3 filters
// 33.5 -> 29.4.  ZERO = false where there is nothing to zero: the loops alone cost 30 x 50 x 900 x 1501 27.1 -> 28.9 us.
struct LayoutZero {
  float* out[3];                // NULL: none; 16-byte aligned
  long long n;                  // floats per output
};
// first, step: this thread's share of the floats, in groups of four
__device__ __forceinline__ void zero_share(const LayoutZero& z, long long first, long long step) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (!z.out[k]) continue;
    for (long long i = first; i < z.n >> 2; i += step) reinterpret_cast<float4*>(z.out[k])[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (long long i = (z.n & ~3ll) + first; i < z.n; i += step) z.out[k][i] = 0.f;
  }
}

// dst[r, 0..d) = src[r, 0..d): src rows back to back, dst rows `pitch` elements apart (a multiple of 8, at least d).
// A thread writes 16-byte groups; their eight source elements start at any even byte, so it reads the two aligned 16-byte
// words around them (the second one is its neighbour's first: an L1 hit) and shifts.  gridDim.y = 1 or 2 picks the tensor.
// Bound by HBM: each element is read and written once (8 x 256 x 1024 x 32101, the whole call: 8192 -> 240 us, was SIMT).
struct PadTensor {
  const uint16_t* src;
  uint16_t* dst;
  int d, pitch;
};
template <bool ZERO>
__global__ void __launch_bounds__(LAYOUT_THREADS)
pad_rows_kernel(PadTensor ta, PadTensor tb, long long rows, LayoutZero zero) {
  sm100::griddep_launch_dependents();
  sm100::griddep_wait();
  if (ZERO) zero_share(zero, ((long long)blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x, (long long)gridDim.x * gridDim.y * blockDim.x);
  const PadTensor& t = blockIdx.y == 0 ? ta : tb;
  const int groups = t.pitch >> 3;
  const long long total = rows * groups, elems = rows * t.d;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < total; k += stride) {
    const long long r = k / groups;
    const int c = (int)(k - r * groups) * 8;
    const long long e = r * t.d + c;                     // first source element
    const long long a = e & ~7ll;                        // its aligned 16-byte word (src is 16-byte aligned)
    uint32_t o[4];
    if (a + 16 <= elems) {
      const uint4 lo = __ldg(reinterpret_cast<const uint4*>(t.src + a)), hi = __ldg(reinterpret_cast<const uint4*>(t.src + a + 8));
      uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
      const int s = (int)(e - a);                        // 0..7 elements
      if (s & 4) {
#pragma unroll
        for (int j = 0; j < 6; ++j) w[j] = w[(j + 2) & 7];
      }
      if (s & 2) {
#pragma unroll
        for (int j = 0; j < 5; ++j) w[j] = w[j + 1];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) o[j] = __funnelshift_r(w[j], w[j + 1], (s & 1) * 16);
    } else {                                             // the end of the tensor: nothing beyond it is read
      uint16_t v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = (c + j < t.d && e + j < elems) ? t.src[e + j] : (uint16_t)0;
#pragma unroll
      for (int j = 0; j < 4; ++j) o[j] = (uint32_t)v[2 * j] | ((uint32_t)v[2 * j + 1] << 16);
    }
    *reinterpret_cast<uint4*>(t.dst + r * t.pitch + c) = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

// Geometry of a 2-D convolution (the weight is [F, C, Kh, Kw]); Ho, Wo: output size.
struct ConvGeom {
  int B, C, H, W, F, Kh, Kw, sh, sw, ph, pw, dh, dw, Ho, Wo;
};

// The two operands of a convolution's weight gradient, in one launch: blocks below unfold_blocks unfold the input, the others
// transpose the cotangents.
//
// Unfolding: X[(b, oh, ow), f] = x[b, c, oh*sh - ph + kh*dh, ow*sw - pw + kw*dw] (0 outside the image), f = (c*Kh + kh)*Kw + kw: one
// row of pitch_x bf16 per output position.  A block handles tile_h x tile_w output positions: the input rows they touch go to shared
// memory once, `chan` channels at a time, two elements per load where the rows allow, and with the image's border as zeros; every 16-byte
// group of the result is gathered from there.  A thread keeps its group, whose eight offsets stay in registers, and walks over the positions.
// chan is a multiple of 8 or C, so that a round's features start on a group.
//
// Transposing: dY[b, t, f] = gy[b, f, t], [B, F, T] -> [B, T, pitch_y], through 64 x 64 tiles of shared memory; vec: rows of gy are
// 16-byte multiples and read as such.
//
// Bound by the gathers' instructions and the latency of a block's loads.  Whole calls, against a block per output row whose warps load one input row
// after the other: 32 images of 3 x 112 x 112, 7 x 7, stride 2, 64 filters (43 MB written) 46 -> 39 us; 32 of 64 x 14 x 14, 3 x 3, 128 filters
// 34 -> 20; 64 of 64 x 15 x 15, 3 x 3, stride 2, 96 filters 30 -> 21; 16 of 16 x 56 x 56, 3 x 3, 96 filters 33 -> 31.
struct ConvOperands {
  const uint16_t* x;
  const uint16_t* gy;
  uint16_t* X;
  uint16_t* dY;
  int pitch_x, pitch_y;
  int tile_w, tile_h, chan;     // unfolding: positions per block, across and down, channels per round
  int cols, img_rows;           // image columns and rows per channel in shared memory
  int row_step, kh_step;        // image rows from one of those to the next; of those from one kernel row to the next
  int pairs;                    // the image's rows are whole aligned pairs of elements
  uint32_t per_row_magic, img_rows_magic;     // ceil(2^32 / loads per row), ceil(2^32 / img_rows): exact quotients of numbers below 2^16 (not by 1)
  int w_tiles, h_tiles;         // ceil(Wo / tile_w), ceil(Ho / tile_h)
  long long unfold_blocks;      // w_tiles * h_tiles * B
  int t_tiles, f_tiles;         // transposing: ceil(T / 64), ceil(pitch_y / 64)
  int vec;
};
__device__ __forceinline__ void unfold_block(const ConvOperands& o, const ConvGeom& g, uint16_t* smem) {
  const int kk = g.Kh * g.Kw;
  const int ow0 = (int)(blockIdx.x % o.w_tiles) * o.tile_w;
  const int rest = (int)(blockIdx.x / o.w_tiles), oh0 = rest % o.h_tiles * o.tile_h, b = rest / o.h_tiles;
  const int n_ow = min(o.tile_w, g.Wo - ow0), positions = min(o.tile_h, g.Ho - oh0) * n_ow;
  const int shift = o.pairs ? (ow0 * g.sw - g.pw) & 1 : 0;           // pairs start at even columns of the image
  const int iw0 = ow0 * g.sw - g.pw - shift, ih0 = oh0 * g.sh - g.ph;
  for (int c0 = 0; c0 < g.C; c0 += o.chan) {
    const int nc = min(o.chan, g.C - c0);
    const int feats = nc * kk, groups = (feats + 7) >> 3;
    // smem: [nc][img_rows][cols], eight loads of a thread in flight (a warp per row, one after the other, spent 20 us on latency)
    const int per_row = o.pairs ? o.cols / 2 : o.cols, total = nc * o.img_rows * per_row;
    for (int base = threadIdx.x; base < total; base += 8 * LAYOUT_THREADS) {
      uint32_t v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t k = (uint32_t)(base + j * LAYOUT_THREADS);
        const uint32_t r = per_row > 1 ? __umulhi(k, o.per_row_magic) : k, ch = o.img_rows > 1 ? __umulhi(r, o.img_rows_magic) : r;
        const int ih = ih0 + (int)(r - ch * o.img_rows) * o.row_step, iw = iw0 + (int)(k - r * per_row) * (o.pairs ? 2 : 1);
        v[j] = 0u;
        if ((int)k < total && ih >= 0 && ih < g.H && iw >= 0 && iw < g.W) {
          const uint16_t* const at = o.x + (((long long)b * g.C + c0 + ch) * g.H + ih) * g.W + iw;
          v[j] = o.pairs ? __ldg(reinterpret_cast<const uint32_t*>(at)) : (uint32_t)__ldg(at);
        }
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int k = base + j * LAYOUT_THREADS;
        if (k >= total) break;
        if (o.pairs) reinterpret_cast<uint32_t*>(smem)[k] = v[j];
        else smem[k] = (uint16_t)v[j];
      }
    }
    __syncthreads();
    for (int g0 = 0; g0 < groups; g0 += LAYOUT_THREADS) {
      const int width = min(groups - g0, LAYOUT_THREADS), together = LAYOUT_THREADS / width;      // groups side by side, positions at once
      const int grp = g0 + (int)threadIdx.x % width, first = (int)threadIdx.x / width;
      if (first >= together) continue;
      // features past the last one: any element will do, those columns are never read
      int at[8];
      int ch = 8 * grp / kk, kh = (8 * grp - ch * kk) / g.Kw, kw = 8 * grp - ch * kk - kh * g.Kw;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        at[j] = 8 * grp + j < feats ? (ch * o.img_rows + kh * o.kh_step) * o.cols + kw * g.dw + shift : 0;
        if (++kw == g.Kw) {
          kw = 0;
          if (++kh == g.Kh) { kh = 0; ++ch; }
        }
      }
      uint16_t* const out = o.X + (((long long)b * g.Ho + oh0) * g.Wo + ow0) * o.pitch_x + c0 * kk + 8 * grp;
      int r = first / n_ow, w = first - r * n_ow;
#pragma unroll 2
      for (int pos = first; pos < positions; pos += together) {
        const uint16_t* const img = smem + r * g.sh * o.cols + w * g.sw;
        uint32_t v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = img[at[j]];
        *reinterpret_cast<uint4*>(out + ((long long)r * g.Wo + w) * o.pitch_x) = make_uint4(v[0] | (v[1] << 16), v[2] | (v[3] << 16), v[4] | (v[5] << 16), v[6] | (v[7] << 16));
        for (w += together; w >= n_ow; w -= n_ow) ++r;
      }
    }
    __syncthreads();
  }
}
constexpr int TRANSPOSE_PITCH = 74;       // elements: 37 words, so that the rows of a column read fall into different banks
__device__ __forceinline__ void transpose_block(const ConvOperands& o, int F, int T, uint16_t* smem) {
  const long long k0 = (long long)blockIdx.x - o.unfold_blocks;
  const int t0 = (int)(k0 % o.t_tiles) * 64;
  const int rest = (int)(k0 / o.t_tiles), f0 = rest % o.f_tiles * 64, b = rest / o.f_tiles;
  const uint16_t* const s = o.gy + (long long)b * F * T;
  if (o.vec) {
    for (int k = threadIdx.x; k < 64 * 8; k += LAYOUT_THREADS) {
      const int f = k >> 3, t = (k & 7) * 8;
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (f0 + f < F && t0 + t < T) v = __ldg(reinterpret_cast<const uint4*>(s + (long long)(f0 + f) * T + t0 + t));       // T is a multiple of 8
      uint32_t* const d = reinterpret_cast<uint32_t*>(smem + f * TRANSPOSE_PITCH + t);
      d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
    }
  } else {
    for (int k = threadIdx.x; k < 64 * 64; k += LAYOUT_THREADS) {
      const int f = k >> 6, t = k & 63;
      smem[f * TRANSPOSE_PITCH + t] = (f0 + f < F && t0 + t < T) ? __ldg(s + (long long)(f0 + f) * T + t0 + t) : (uint16_t)0;
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < 64 * 8; k += LAYOUT_THREADS) {
    const int t = k >> 3, f = (k & 7) * 8;
    if (t0 + t >= T || f0 + f >= o.pitch_y) continue;
    uint32_t v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      v[j] = (uint32_t)smem[(f + 2 * j) * TRANSPOSE_PITCH + t] | ((uint32_t)smem[(f + 2 * j + 1) * TRANSPOSE_PITCH + t] << 16);
    *reinterpret_cast<uint4*>(o.dY + ((long long)b * T + t0 + t) * o.pitch_y + f0 + f) = make_uint4(v[0], v[1], v[2], v[3]);
  }
}
template <bool ZERO>
__global__ void __launch_bounds__(LAYOUT_THREADS)
conv_operands_kernel(ConvOperands o, ConvGeom g, LayoutZero zero) {
  extern __shared__ __align__(16) uint16_t layout_smem[];
  sm100::griddep_launch_dependents();
  sm100::griddep_wait();
  if (ZERO) zero_share(zero, (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x);
  if ((long long)blockIdx.x < o.unfold_blocks) unfold_block(o, g, layout_smem);
  else transpose_block(o, g.F, g.Ho * g.Wo, layout_smem);
}

// Operands of the statistics of examples of a single token, where G_b[o,i] = dY[b,o] X[b,i] and the sums over b are contractions of
// row-wise functions of the operands: sum G_b = dY^T X, sum G_b^2 = (dY o dY)^T (X o X), sum sign(G_b) = sign(dY)^T sign(X).
// The square of a bf16 has 16 significant bits: its upper and lower half are bf16 numbers, exactly, and four products of halves make up
// the contraction without a rounding of the operands.  Each example's two rows are first scaled by 2^-s and 2^s (nothing changes in the
// product), which keeps the squares finite and their lower halves normal while the magnitudes that matter (those whose product with
// the other row's largest has a square in fp32) lie within 2^-55 .. 2^63 after it.  s is the one that does so and is nearest to that of equal
// maxima.  An example for which there is none, or that holds an infinity or a NaN, is left out of the halves and marked in `odd`, as is one with
// a product of nonzero entries that may be zero in fp32, whose sign would count: the contraction forms G_b of those, entry by entry.
//
// A copy of an operand is [n][chunk][pitch], rows past B zero.  at_mean, at_halves, at_sign: the number of the copy as it is, of the upper half
// (the lower one follows) and of the sign, -1 for one that is not wanted.  A block takes a row; blocks
// past the rows zero the outputs.  Bound by launch latency and HBM: two reads of 2 bytes and up to 8 written per element.  The whole
// call, mean and square: 1024 x 1024^2 160 -> 23 us, 512 x 4096^2 1061 -> 124, against forming every G_b.  Finding the rows' ranges costs 0 to
// 2.5 us of that.
enum : int { ONE_TOKEN_ODD_SQUARE = 1, ONE_TOKEN_ODD_SIGN = 2 };
struct OneTokenTensor {
  const uint16_t* src;
  uint16_t* dst;
  int d, pitch;
};
// Eight entries as four words.
__device__ __forceinline__ uint4 one_token_load(const uint16_t* row, int d, int g, bool vec) {
  if (vec) return __ldg(reinterpret_cast<const uint4*>(row) + g);
  uint32_t v[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = 8 * g + j < d ? (uint32_t)__ldg(row + 8 * g + j) : 0u;
  return make_uint4(v[0] | v[1] << 16, v[2] | v[3] << 16, v[4] | v[5] << 16, v[6] | v[7] << 16);
}
// Largest and smallest nonzero magnitude of what a thread sees, as bf16 patterns, two entries at a time.  low: the pattern plus 0x7fff, which
// as a signed number orders the nonzero patterns and puts zero last.
struct PairExtremes {
  uint32_t top = 0u, low = 0x7fff7fffu;
  __device__ __forceinline__ void see(uint4 v) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t m = w[j] & 0x7fff7fffu;
      top = __vmaxu2(top, m);
      low = __vmins2(low, m + 0x7fff7fffu);
    }
  }
  __device__ __forceinline__ int top_bits() const { return (int)max(top & 0xffffu, top >> 16); }
  __device__ __forceinline__ int low_bits() const { return min((int)(int16_t)(low & 0xffffu), (int)(int16_t)(low >> 16)) + 0x8001; }
};
// Exponent of a nonzero magnitude; a subnormal counts as the smallest there is.
__device__ __forceinline__ int one_token_exponent(int bits) { return bits < 0x80 ? -133 : (bits >> 7) - 127; }
struct RowExtremes {
  int top, low;
  __device__ __forceinline__ bool zero() const { return top == 0; }
  __device__ __forceinline__ bool finite() const { return top < 0x7f80; }
  __device__ __forceinline__ int top_exponent() const { return max(1, top >> 7) - 127; }
  __device__ __forceinline__ int low_exponent() const { return one_token_exponent(low); }
};
__device__ __forceinline__ void block_extremes(const PairExtremes& px, const PairExtremes& py, RowExtremes& x, RowExtremes& y) {
  __shared__ int part[4][LAYOUT_THREADS / 32];
  x = {__reduce_max_sync(0xffffffffu, px.top_bits()), __reduce_min_sync(0xffffffffu, px.low_bits())};
  y = {__reduce_max_sync(0xffffffffu, py.top_bits()), __reduce_min_sync(0xffffffffu, py.low_bits())};
  if ((threadIdx.x & 31) == 0) {
    const int warp = threadIdx.x >> 5;
    part[0][warp] = x.top; part[1][warp] = x.low; part[2][warp] = y.top; part[3][warp] = y.low;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < LAYOUT_THREADS / 32; ++k) {
    x.top = max(x.top, part[0][k]); x.low = min(x.low, part[1][k]);
    y.top = max(y.top, part[2][k]); y.low = min(y.low, part[3][k]);
  }
}
__global__ void __launch_bounds__(LAYOUT_THREADS)
one_token_operands_kernel(OneTokenTensor tx, OneTokenTensor ty, uint8_t* odd, int B, int chunk, int n, int at_mean, int at_halves, int at_sign,
                          LayoutZero zero) {
  sm100::griddep_launch_dependents();
  sm100::griddep_wait();
  const int rows = n * chunk, b = blockIdx.x;
  if (b >= rows) {
    zero_share(zero, (long long)(b - rows) * LAYOUT_THREADS + threadIdx.x, (long long)(gridDim.x - rows) * LAYOUT_THREADS);
    return;
  }
  const bool vx = tx.d % 8 == 0, vy = ty.d % 8 == 0;
  const uint16_t* const x = tx.src + (long long)b * tx.d;
  const uint16_t* const y = ty.src + (long long)b * ty.d;
  float scale_x = 0.f, scale_y = 0.f;
  bool in_halves = false;
  PairExtremes px, py;
  int flags = 0;
  if (at_halves >= 0 && b < B) {
    for (int g = threadIdx.x; g < tx.pitch / 8; g += LAYOUT_THREADS) px.see(one_token_load(x, tx.d, g, vx));
    for (int g = threadIdx.x; g < ty.pitch / 8; g += LAYOUT_THREADS) py.see(one_token_load(y, ty.d, g, vy));
    RowExtremes ex, ey;
    block_extremes(px, py, ex, ey);
    const bool finite = ex.finite() && ey.finite(), some = !ex.zero() && !ey.zero();
    if (finite && some) {
      const int top_x = ex.top_exponent(), top_y = ey.top_exponent();
      // entries below these: a product with the other row's largest under 2^-75, a square that fp32 does not have
      const int low_x = max(ex.low_exponent(), -76 - top_y), low_y = max(ey.low_exponent(), -76 - top_x);
      const int least = max(max(top_x - 62, -55 - low_y), -126), most = min(min(62 - top_y, low_x + 55), 126);
      const int s = min(max((top_x - top_y) / 2, least), most);
      in_halves = least <= most;
      scale_x = __uint_as_float((uint32_t)(127 - s) << 23);
      scale_y = __uint_as_float((uint32_t)(127 + s) << 23);
    }
    // (a row of zeros and one without infinities: G_b is zero, as the zeros in the copies make it)
    if (!in_halves && (some || !finite)) flags = ONE_TOKEN_ODD_SQUARE;
    if (at_sign >= 0 && some && ex.low_exponent() + ey.low_exponent() < -149) flags |= ONE_TOKEN_ODD_SIGN;
  }
  const bool look = at_halves < 0 && at_sign >= 0 && b < B;            // the smallest entries are found on the way
  auto write = [&](const OneTokenTensor& t, const uint16_t* row, bool vec, float scale, PairExtremes& e) {
    const long long copy = (long long)rows * t.pitch;
    uint16_t* const dst = t.dst + (long long)b * t.pitch;
    for (int g = threadIdx.x; g < t.pitch / 8; g += LAYOUT_THREADS) {
      const uint4 v = b < B ? one_token_load(row, t.d, g, vec) : make_uint4(0u, 0u, 0u, 0u);
      if (look) e.see(v);
      const uint32_t w[8] = {v.x << 16, v.x & 0xffff0000u, v.y << 16, v.y & 0xffff0000u, v.z << 16, v.z & 0xffff0000u, v.w << 16, v.w & 0xffff0000u};
      auto put = [&](int k, const uint32_t (&v)[8]) {                  // the upper halves of the words
        *reinterpret_cast<uint4*>(dst + k * copy + 8 * g) = make_uint4(__byte_perm(v[0], v[1], 0x7632), __byte_perm(v[2], v[3], 0x7632),
                                                                       __byte_perm(v[4], v[5], 0x7632), __byte_perm(v[6], v[7], 0x7632));
      };
      if (at_mean >= 0) *reinterpret_cast<uint4*>(dst + at_mean * copy + 8 * g) = v;
      if (at_halves >= 0) {
        uint32_t hi[8], lo[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float f = in_halves ? __uint_as_float(w[j]) * scale : 0.f, q = f * f;
          hi[j] = __float_as_uint(q);
          lo[j] = __float_as_uint(q - __uint_as_float(hi[j] & 0xffff0000u));      // exact
        }
        put(at_halves, hi);
        put(at_halves + 1, lo);
      }
      if (at_sign >= 0) {
        uint32_t sg[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float f = __uint_as_float(w[j]);
          sg[j] = f > 0.f ? 0x3f800000u : f < 0.f ? 0xbf800000u : 0u;
        }
        put(at_sign, sg);
      }
    }
  };
  write(tx, x, vx, scale_x, px);
  write(ty, y, vy, scale_y, py);
  // a product below 2^-149 has a factor below 2^-74
  if (look && __syncthreads_or(one_token_exponent(px.low_bits()) < -74 || one_token_exponent(py.low_bits()) < -74)) flags = ONE_TOKEN_ODD_SIGN;
  if (threadIdx.x == 0 && (at_halves >= 0 || at_sign >= 0)) odd[b] = (uint8_t)flags;
}

}  // namespace pe
