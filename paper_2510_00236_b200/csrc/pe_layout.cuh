// Layout kernels in front of the tensor-core contraction, for operands whose rows TMA cannot address (it wants 16-byte
// row pitches): rows of a width that is no multiple of 8 copied to a padded pitch, and the operands of a convolution's
// weight gradient (Appendix B.4) unfolded straight into that form.  Streaming kernels, bound by HBM bandwidth; the columns
// between the width and the pitch are never read (the tensor maps end at the width).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace pe {

constexpr int LAYOUT_THREADS = 256;
constexpr int UNFOLD_SMEM_BYTES = 48 * 1024;

// dst[r, 0..d) = src[r, 0..d): src rows back to back, dst rows `pitch` elements apart (a multiple of 8, at least d).
// A thread writes 16-byte groups; their eight source elements start at any even byte, so it reads the two aligned 16-byte
// words around them (the second one is its neighbour's first: an L1 hit) and shifts.  gridDim.y = 1 or 2 picks the tensor.
// Bound by HBM: each element is read and written once (8 x 256 x 1024 x 32101, the whole call: 8192 -> 271 us, was SIMT).
struct PadTensor {
  const uint16_t* src;
  uint16_t* dst;
  int d, pitch;
};
__global__ void __launch_bounds__(LAYOUT_THREADS)
pad_rows_kernel(PadTensor ta, PadTensor tb, long long rows) {
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

// dst[(b, oh, ow), f] = x[b, c, oh*sh - ph + kh*dh, ow*sw - pw + kw*dw] (0 outside the image), f = (c*Kh + kh)*Kw + kw: one row of
// `pitch` bf16 per output position.  A block handles one output row (a run of tile_w of its positions): the input rows it
// touches go to shared memory once, `chan` channels at a time and with the image's border as zeros, and every 16-byte
// group of the result is gathered from there through a table of the features' offsets.  chan is a multiple of 8 or C, so
// that a chunk's features start on a group.  gridDim = (ceil(Wo / tile_w), Ho, B).
// 32 images of 3 x 112 x 112, 7 x 7, stride 2, 64 filters, the whole call: 1158 -> 65 us (torch's unfold launches one kernel per
// image, in fp32, and a transpose and two conversions follow).
__global__ void __launch_bounds__(LAYOUT_THREADS)
unfold_kernel(const uint16_t* __restrict__ x, uint16_t* __restrict__ dst, ConvGeom g, int pitch, int tile_w, int chan, int cols) {
  extern __shared__ __align__(16) uint16_t unfold_smem[];
  const int kk = g.Kh * g.Kw, d = g.C * kk;
  const int chunk_feats = (chan * kk + 7) & ~7;
  int* const off = reinterpret_cast<int*>(unfold_smem);                     // [chunk_feats]: element offset of a feature at position 0
  uint16_t* const img = unfold_smem + 2 * chunk_feats;                      // [chan][Kh][cols], then one zero
  const int ow0 = blockIdx.x * tile_w, oh = blockIdx.y, b = blockIdx.z;
  const int n_ow = min(tile_w, g.Wo - ow0);
  for (int c0 = 0; c0 < g.C; c0 += chan) {
    const int nc = min(chan, g.C - c0), n_img = nc * g.Kh * cols;
    const int feats = nc * kk, groups = (feats + 7) >> 3;
    for (int k = threadIdx.x; k < n_img; k += LAYOUT_THREADS) {
      const int ch = k / (g.Kh * cols), rest = k - ch * g.Kh * cols, kh = rest / cols, w = rest - kh * cols;
      const int ih = oh * g.sh - g.ph + kh * g.dh, iw = ow0 * g.sw - g.pw + w;
      uint16_t v = 0;
      if (ih >= 0 && ih < g.H && iw >= 0 && iw < g.W) v = __ldg(x + (((long long)b * g.C + c0 + ch) * g.H + ih) * g.W + iw);
      img[k] = v;
    }
    for (int f = threadIdx.x; f < groups * 8; f += LAYOUT_THREADS) {
      const int ch = f / kk, rest = f - ch * kk, kh = rest / g.Kw, kw = rest - kh * g.Kw;
      off[f] = f < feats ? (ch * g.Kh + kh) * cols + kw * g.dw : -1;
    }
    __syncthreads();
    uint16_t* const out = dst + (((long long)b * g.Ho + oh) * g.Wo + ow0) * pitch + c0 * kk;
    for (int k = threadIdx.x; k < n_ow * groups; k += LAYOUT_THREADS) {
      const int tok = k / groups, grp = k - tok * groups;
      const int4 o0 = *reinterpret_cast<const int4*>(off + 8 * grp), o1 = *reinterpret_cast<const int4*>(off + 8 * grp + 4);
      const int o[8] = {o0.x, o0.y, o0.z, o0.w, o1.x, o1.y, o1.z, o1.w};
      uint32_t v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = o[j] >= 0 ? (uint32_t)img[o[j] + tok * g.sw] : 0u;
      *reinterpret_cast<uint4*>(out + (long long)tok * pitch + 8 * grp) =
          make_uint4(v[0] | (v[1] << 16), v[2] | (v[3] << 16), v[4] | (v[5] << 16), v[6] | (v[7] << 16));
    }
    __syncthreads();
  }
}

// dst[b, t, f] = src[b, f, t]: [B, F, T] -> [B, T, pitch], through 64 x 64 tiles of shared memory.
// gridDim = (ceil(T / 64), ceil(pitch / 64), B).
__global__ void __launch_bounds__(LAYOUT_THREADS)
transpose_rows_kernel(const uint16_t* __restrict__ src, uint16_t* __restrict__ dst, int F, int T, int pitch) {
  __shared__ uint16_t tile[64][66];            // 66: neighbouring f of one t in different banks
  const int t0 = blockIdx.x * 64, f0 = blockIdx.y * 64;
  const uint16_t* const s = src + (long long)blockIdx.z * F * T;
  for (int k = threadIdx.x; k < 64 * 64; k += LAYOUT_THREADS) {
    const int f = k >> 6, t = k & 63;
    tile[f][t] = (f0 + f < F && t0 + t < T) ? __ldg(s + (long long)(f0 + f) * T + t0 + t) : (uint16_t)0;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < 64 * 8; k += LAYOUT_THREADS) {
    const int t = k >> 3, f = (k & 7) * 8;
    if (t0 + t >= T || f0 + f >= pitch) continue;
    uint32_t o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) o[j] = (uint32_t)tile[f + 2 * j][t] | ((uint32_t)tile[f + 2 * j + 1][t] << 16);
    *reinterpret_cast<uint4*>(dst + ((long long)blockIdx.z * T + t0 + t) * pitch + f0 + f) = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

}  // namespace pe
