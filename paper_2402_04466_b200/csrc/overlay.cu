// S6: alpha-blend the thresholded tool masks as colours onto an RGBA8 copy of the source
// frame (integer arithmetic, bit-exact).  HBM-bound: 3 bytes in, 4 bytes out per pixel.
// When the frame is dense (pitch == 3*W) and 4-byte aligned the image is processed as a
// flat stream: a thread takes 4 consecutive pixels = three 32-bit loads and one 128-bit
// store, both fully coalesced.  The mask sample of a pixel, floor(x * Wm / W), is found once per
// thread with multiply-and-shift divisions whose constants the host prepares, then stepped from pixel to pixel
// by the quotient and remainder of Wm / W.  Red and blue are blended as two 16-bit halves of one register.  Six 854x480
// frames (17 MB, stage time with its event): 30.7 us with two 64-bit divisions per pixel and a loop over each pixel's own
// tools, 24.6 us without the divisions, 16.4 us with the packed blend over the tools a warp needs.
#include "tt_internal.h"

namespace tt {
namespace {

// Exact floor(n / d) for 0 <= n < 2^31 (n * e < 2^(31 + l) with l = ceil(log2 d), mul * d = 2^(31 + l) + e, 0 < e <= d).
struct FastDiv {
  uint32_t mul = 0, shift = 0;   // mul 0: d == 1
};
FastDiv fast_div(uint32_t d) {
  FastDiv f;
  if (d <= 1) return f;
  uint32_t l = 0;
  while ((1ull << l) < d) ++l;
  f.mul = (uint32_t)((1ull << (31 + l)) / d + 1);
  f.shift = l - 1;
  return f;
}
__device__ __forceinline__ uint32_t div_by(uint32_t n, FastDiv f) { return f.mul ? __umulhi(n, f.mul) >> f.shift : n; }

struct OverlayArgs {
  OverlayParams p;
  FastDiv by_w, by_h;            // source width and height
  uint32_t k_rb[TT_MAX_TOOLS];   // 102 * colour + 127 of red and blue, 16 bits each
  uint32_t k_g[TT_MAX_TOOLS];    // and of green
  int32_t step_q, step_r;        // Wm / src_w and its remainder
};

template <bool PACKED>
__device__ __forceinline__ uint32_t mask_bits(const OverlayParams& p, int n, int mx, int my) {
  const int plane = p.Hm * p.Wm;
  if (PACKED) return __ldg(p.bits + (size_t)n * plane + my * p.Wm + mx);
  uint32_t b = 0;
  for (int t = 0; t < p.T; ++t) b |= (uint32_t)(__ldg(p.masks + ((size_t)n * p.T + t) * plane + my * p.Wm + mx) != 0) << t;
  return b;
}

// Blends tool t into one pixel (red and blue in one register, 16 bits each).  (153 * c + 102 * colour + 127) / 255: the
// numerator stays below 65153, for which v / 255 = (v + 1 + v / 256) / 256 exactly, and no sum leaves its 16 bits.
__device__ __forceinline__ void blend(uint32_t& rb, uint32_t& g, uint32_t k_rb, uint32_t k_g) {
  const uint32_t v = rb * 153u + k_rb, w = g * 153u + k_g;
  rb = ((v + 0x00010001u + ((v >> 8) & 0x00FF00FFu)) >> 8) & 0x00FF00FFu;
  g = (w + 1u + (w >> 8)) >> 8;
}

// Tools ascend from 0.  The loop runs over the tools that any lane of the warp needs, so that the colours are uniform
// loads and lanes with other tools do not serialise.  The whole warp takes part.
template <int N>
__device__ __forceinline__ void blend_all(uint32_t (&rb)[N], uint32_t (&g)[N], const uint32_t (&bits)[N], const OverlayArgs& a) {
  uint32_t some = 0;
#pragma unroll
  for (int j = 0; j < N; ++j) some |= bits[j];
  some = __reduce_or_sync(0xffffffffu, some);
  while (some) {
    const int t = __ffs(some) - 1;
    some &= some - 1;
    const uint32_t k_rb = a.k_rb[t], k_g = a.k_g[t];
#pragma unroll
    for (int j = 0; j < N; ++j) {
      uint32_t x = rb[j], y = g[j];
      blend(x, y, k_rb, k_g);
      const bool m = (bits[j] >> t) & 1u;
      rb[j] = m ? x : rb[j];
      g[j] = m ? y : g[j];
    }
  }
}

__device__ __forceinline__ uint32_t rgba(uint32_t rb, uint32_t g) { return rb | (g << 8) | 0xFF000000u; }

template <bool PACKED, bool FLAT>
__global__ void __launch_bounds__(256) overlay_kernel(const __grid_constant__ OverlayArgs a) {
  const OverlayParams& p = a.p;
  pdl_wait();   // the masks are the previous kernel's output
  const int n = blockIdx.y;
  const uint8_t* __restrict__ src = p.src_tab ? p.src_tab[n] : p.src.p[n];
  const uint32_t npx = (uint32_t)p.src_w * (uint32_t)p.src_h;           // at most 2^28
  uint8_t* dst = p.dst + (size_t)n * npx * 4;
  const uint32_t i0 = (blockIdx.x * blockDim.x + threadIdx.x) * 4;      // first of 4 pixels
  int y = (int)div_by(i0, a.by_w), x = (int)i0 - y * p.src_w;
  // mask sample of (x, y) and the remainder of x * Wm / src_w, which the next pixel's sample follows from
  int mx = (int)div_by((uint32_t)(x * p.Wm), a.by_w), rem = x * p.Wm - mx * p.src_w;
  int my = (int)div_by((uint32_t)(y * p.Hm), a.by_h);
  auto next = [&]() {
    mx += a.step_q;
    rem += a.step_r;
    if (rem >= p.src_w) { rem -= p.src_w; ++mx; }
    if (++x == p.src_w) {
      x = 0; mx = 0; rem = 0; ++y;
      my = (int)div_by((uint32_t)(y * p.Hm), a.by_h);
    }
  };
  uint32_t bits[4] = {};
  // the same for all lanes of a warp (its 128 pixels all exist): both branches vote with the whole warp
  if (FLAT && (i0 & ~127u) + 128 <= npx) {
    const uint32_t* s32 = reinterpret_cast<const uint32_t*>(src) + (i0 >> 2) * 3;
    const uint32_t w0 = __ldg(s32), w1 = __ldg(s32 + 1), w2 = __ldg(s32 + 2);
    // bytes R0 G0 B0 R1 | G1 B1 R2 G2 | B2 R3 G3 B3
    uint32_t rb[4] = {w0 & 0x00FF00FFu, (w0 >> 24) | ((w1 & 0xFF00u) << 8), ((w1 >> 16) & 0xFFu) | ((w2 & 0xFFu) << 16), ((w2 >> 8) & 0xFFu) | ((w2 >> 24) << 16)};
    uint32_t g[4] = {(w0 >> 8) & 0xFFu, w1 & 0xFFu, w1 >> 24, (w2 >> 16) & 0xFFu};
    uint32_t out[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      bits[j] = mask_bits<PACKED>(p, n, mx, my);
      if (j < 3) next();
    }
    blend_all<4>(rb, g, bits, a);
#pragma unroll
    for (int j = 0; j < 4; ++j) out[j] = rgba(rb[j], g[j]);
    *reinterpret_cast<uint4*>(dst + (size_t)i0 * 4) = make_uint4(out[0], out[1], out[2], out[3]);
  } else {
    // lanes behind the last pixel stay for the vote: they have no bits set, load and store nothing
    const int live = i0 < npx ? (int)min(npx - i0, 4u) : 0;
    uint32_t rb[4] = {}, g[4] = {};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (j < live) {
        bits[j] = mask_bits<PACKED>(p, n, mx, my);
        const uint8_t* s = src + (size_t)y * p.src_pitch + 3 * x;
        rb[j] = (uint32_t)s[0] | ((uint32_t)s[2] << 16);
        g[j] = s[1];
      }
      if (j < 3) next();
    }
    blend_all<4>(rb, g, bits, a);
    uint32_t* out = reinterpret_cast<uint32_t*>(dst + (size_t)i0 * 4);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < live) out[j] = rgba(rb[j], g[j]);
  }
}

}  // namespace

cudaError_t launch_overlay(const OverlayParams& p, cudaStream_t s) {
  const long long npx = (long long)p.src_w * p.src_h;
  const long long groups = (npx + 3) / 4;
  OverlayArgs a;
  a.p = p;
  a.by_w = fast_div((uint32_t)p.src_w);
  a.by_h = fast_div((uint32_t)p.src_h);
  a.step_q = p.Wm / p.src_w;
  a.step_r = p.Wm % p.src_w;
  for (int t = 0; t < TT_MAX_TOOLS; ++t) {
    const uint32_t r = p.palette[t][0], gr = p.palette[t][1], b = p.palette[t][2];
    a.k_rb[t] = (102 * r + 127) | ((102 * b + 127) << 16);
    a.k_g[t] = 102 * gr + 127;
  }
  dim3 grid((unsigned)((groups + 255) / 256), p.K);
  bool flat = p.src_pitch == 3 * p.src_w;
  for (int n = 0; n < p.K; ++n) flat = flat && (((uintptr_t)p.src.p[n] & 3) == 0);
  flat = flat && (((uintptr_t)p.dst & 15) == 0) && ((npx * 4) % 16 == 0 || p.K == 1);
  const bool packed = p.bits != nullptr, pdl = p.pdl != 0;
  if (packed && flat) return launch_kernel(overlay_kernel<true, true>, grid, 256, 0, s, a, pdl);
  if (packed) return launch_kernel(overlay_kernel<true, false>, grid, 256, 0, s, a, pdl);
  if (flat) return launch_kernel(overlay_kernel<false, true>, grid, 256, 0, s, a, pdl);
  return launch_kernel(overlay_kernel<false, false>, grid, 256, 0, s, a, pdl);
}

}  // namespace tt
