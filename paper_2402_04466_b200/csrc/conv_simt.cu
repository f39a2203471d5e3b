// S2/S3 on plain fp32 ALUs: direct 3x3 convolution (pad 1, stride 1 or 2) with fused
// bias + ReLU, or with the fused ConvLSTM gate math.  Used by the fp32 precision path and
// for the first encoder layer of the bf16 path where the tensor-core kernel does not apply.
//
// Bound by instruction issue where there is work for every multiprocessor, by latency where there is not.  A thread holds 4 (or 8) neighbouring
// pixels x 8 output channels in registers, so that one channel's row of 3 taps costs 96 FMAs against 2 input loads and 6
// broadcast weight loads from shared memory.  The channels are taken in pairs (fma.rn.f32x2, half the instructions): a 128-bit load of weights is
// two pairs as it stands, and only the inputs have to be doubled, 6 values a row.  A warp covers 32 x 4 (16 x 16) pixels of one group of 8 channels.
// Blocks are made of WY warps along y, WO channel groups that share the input tile, and KS warps that share
// out the input channels of a tile and add their sums up in shared memory at the end: small maps have too few
// outputs to occupy the device otherwise.  KS orders the sums and follows from the layer alone; WY, WO and PX also from the batch.  Input tile
// (haloed; at stride 2 even and odd columns apart) and weights of CB channels are copied asynchronously into one of three buffers, two chunks ahead.
//
// Against one pixel x 16/32 channels per thread, 32 x 8 pixels per block and synchronous staging (stage times with
// their event): ConvLSTM of one 64x64 map with 16 channels 51 -> 15 us, of three 80x60 maps with 32 channels 135 -> 70 us.  With single FMAs those took
// 16.2 and 69.9 us (80 % of the issue slots, a quarter of them for other things than FMAs), in pairs 14.4 and 67.8.  Pairs of
// pixels instead of channels lost (94 us), with register moves for every shifted pair and with every weight twice in shared memory alike: a 128-bit load takes the
// load/store unit four cycles whether its lanes read one address or 32, so that weights are what it is busy with (6 loads for 96 FMA instructions: 75 % of it with
// the inputs').  4 x 4 pixels of 4 channels per thread halve those loads and were slower all the same (75 us).
#include <algorithm>

#include "tt_internal.h"
#include "tc_ptx.cuh"

namespace tt {
namespace {

constexpr int OC = 8;           // output channels per thread

__device__ __forceinline__ uint32_t cs_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// asynchronous copies; `ok` false writes zeros and reads nothing
__device__ __forceinline__ void copy4(uint32_t dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(ok ? 4 : 0) : "memory");
}
__device__ __forceinline__ void copy16(uint32_t dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ float sigmoid_acc(float z) { return 1.0f / (1.0f + expf(-z)); }
// on the bf16 path every contraction takes bf16 operands, like the tensor-core layers
__device__ __forceinline__ float round_bf16(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// PX: pixels per thread, in runs of 4.  4: a warp covers 32 x 4 pixels.  8 (stride 1): 16 x 16, a lane's two runs 8 columns apart.
template <int STRIDE, int WY, int WO, int KS, int PX>
struct SimtCfg {
  static_assert(PX == 4 || (PX == 8 && STRIDE == 1), "pixels per thread");
  static constexpr int WARPS = WY * WO * KS, THREADS = 32 * WARPS;
  static constexpr int TW = PX == 8 ? 16 : 32;                    // pixels of a block along x
  static constexpr int WH = PX == 8 ? 16 : 4;                     // rows of a warp
  static constexpr int TH = WH * WY;
  static constexpr int CB = STRIDE == 1 ? 8 : 4;                  // input channels per staged chunk
  static constexpr int IN_W = (TW - 1) * STRIDE + 3, IN_H = (TH - 1) * STRIDE + 3;
  static constexpr int ODD = 36;                                  // stride 2: where a row's odd columns begin (33 even ones before)
  static constexpr int PITCH = PX == 8 ? 24 : STRIDE == 1 ? 36 : 68;   // floats per staged row, a multiple of 4 that keeps the 128-bit loads free of bank conflicts
  static constexpr int IN_FLOATS = CB * IN_H * PITCH;
  static constexpr int W_FLOATS = CB * 9 * WO * OC;
  static constexpr int BUF_FLOATS = IN_FLOATS + W_FLOATS;
  static constexpr int BUFS = 3;
  static constexpr int SMEM_BYTES = BUFS * BUF_FLOATS * 4;
  static constexpr int N_POS = (IN_H * IN_W + THREADS - 1) / THREADS;   // positions of the input tile per thread
  static constexpr int W_VECS = CB * 9 * WO * (OC / 4);                 // 16-byte vectors of weights per chunk
  static_assert((KS - 1) * WY * WO * 32 * OC * PX <= BUFS * BUF_FLOATS, "the channel groups' partial sums reuse the staging buffers");
};

// the six input columns under a run of four pixels
__device__ __forceinline__ void load_row(const float* r, float (&x)[6]) {
  const float4 a = *reinterpret_cast<const float4*>(r);
  const float2 b = *reinterpret_cast<const float2*>(r + 4);
  x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y;
}

template <int STRIDE, int EPI, int WY, int WO, int KS, int PX>
__global__ void __launch_bounds__(32 * WY * WO * KS) conv3x3_simt_kernel(const __grid_constant__ ConvSimtParams p) {
  using Cfg = SimtCfg<STRIDE, WY, WO, KS, PX>;
  // Whether a row of taps is fetched while the one before it is multiplied: two or three warps to a scheduler do not hide a shared-memory load.  Only where that
  // pays for its registers (blocks, or spills of more than a word); us without / with it: not at stride 2 (a tick of six 480x360 inputs 80 / 85), not with bf16 outputs of four pixels a thread (eight 502x374
  // images to 32 channels 97 / 115; eight pixels, eight 320x240 to 96 channels 111 / 107), not in encoder layers of four channel groups to a tile (eight 320x240 images to 64 channels
  // 73.5 / 78.2; two groups 28.5 / 27.9; channels shared out by four warps 8.3 / 7.6), nor in a ConvLSTM whose channels four warps share (two 32x32 maps of 32 channels 17.9 / 18.7) or
  // with eight pixels a thread and two groups to a tile (eight 320x240 maps of 12 channels 313 / 320).  The other ConvLSTMs: eight 320x240 maps of 16 channels 486 / 449, three 80x60 of 32
  // 69.2 / 68.3.
  constexpr bool AHEAD = STRIDE == 1 && (EPI == EPI_LSTM_F32_NCHW    ? KS <= 2 && !(WO == 2 && PX == 8)
                                         : EPI == EPI_RELU_F32_NCHW ? WO < 4
                                                                    : PX == 8);
  constexpr int CB = Cfg::CB, IN_H = Cfg::IN_H, IN_W = Cfg::IN_W, PITCH = Cfg::PITCH, NT = Cfg::THREADS, TW = Cfg::TW;
  constexpr int RUNS = PX / 4, RUN_STEP = 8;         // runs of 4 pixels of a thread, and columns from one to the next
  extern __shared__ __align__(16) float smem[];
  pdl_launch_dependents();

  const int tiles_x = (p.Wo + TW - 1) / TW;
  const int tile_x = blockIdx.x % tiles_x, tile_y = blockIdx.x / tiles_x;
  const int n = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wo = warp % WO, wy = (warp / WO) % WY, ks = warp / (WO * WY);
  const int ly = wy * Cfg::WH + (PX == 8 ? lane >> 1 : lane >> 3), lx = (PX == 8 ? lane & 1 : lane & 7) * 4;
  const int xo = tile_x * TW + lx, yo = tile_y * Cfg::TH + ly;
  const int grp = blockIdx.y * WO + wo;              // group of 8 packed output channels
  const int cin = p.C0 + p.C1;
  const size_t in_plane = (size_t)p.H * p.W;
  const float* base0 = p.in0 + (size_t)p.idx0.v[n] * p.img_stride0;
  const float* base1 = p.C1 ? p.in1 + (size_t)p.idx1.v[n] * p.img_stride1 : base0;

  // the input positions this thread copies, the same for every channel: offset in a channel's plane (-1: padding) and in a staged one
  int g_off[Cfg::N_POS], s_off[Cfg::N_POS];
#pragma unroll
  for (int j = 0; j < Cfg::N_POS; ++j) {
    const int i = tid + j * NT, r = i / IN_W, col = i - r * IN_W;
    const int yi = tile_y * Cfg::TH * STRIDE - 1 + r, xi = tile_x * TW * STRIDE - 1 + col;
    g_off[j] = (yi >= 0 && yi < p.H && xi >= 0 && xi < p.W) ? yi * p.W + xi : -1;
    s_off[j] = r * PITCH + (STRIDE == 1 ? col : (col & 1) * Cfg::ODD + (col >> 1));
    if (r >= IN_H) s_off[j] = -1;
  }
  auto stage_weights = [&](int c0, float* buf) {
    const uint32_t dst = cs_smem(buf + Cfg::IN_FLOATS);
    for (int i = tid; i < Cfg::W_VECS; i += NT) {
      const int row = i / (WO * 2), v = i - row * (WO * 2);      // row = channel * 9 + tap
      const bool ok = c0 * 9 + row < cin * 9;
      copy16(dst + i * 16, p.wgt + (ok ? (size_t)(c0 * 9 + row) * p.cout_packed + (size_t)blockIdx.y * WO * OC + v * 4 : 0), ok);
    }
  };
  auto stage_input = [&](int c0, float* buf) {
    const uint32_t dst = cs_smem(buf);
#pragma unroll
    for (int c = 0; c < CB; ++c) {
      const int ci = c0 + c;
      const float* src = ci < p.C0 ? base0 + (size_t)ci * in_plane : base1 + (size_t)(ci - p.C0) * in_plane;
      if (ci >= cin) src = base0;
#pragma unroll
      for (int j = 0; j < Cfg::N_POS; ++j) {
        const bool ok = g_off[j] >= 0 && ci < cin;
        if (s_off[j] >= 0) copy4(dst + (c * IN_H * PITCH + s_off[j]) * 4, src + (ok ? g_off[j] : 0), ok);
      }
    }
  };

  stage_weights(0, smem);
  pdl_wait();   // the weights are nobody's output; from here on the previous kernel's results are read
  stage_input(0, smem);
  copies_commit();
  if (CB < cin) {
    stage_weights(CB, smem + Cfg::BUF_FLOATS);
    stage_input(CB, smem + Cfg::BUF_FLOATS);
  }
  copies_commit();

  // the old cell state is fetched now and used after the main loop
  constexpr int HB = OC / 4;
  float c_old[EPI == EPI_LSTM_F32_NCHW ? HB * PX : 1];
  const size_t out_plane = (size_t)p.Ho * p.Wo;
  const size_t pix = (size_t)yo * p.Wo + xo;
  if (EPI == EPI_LSTM_F32_NCHW && ks == 0) {
    const float* c_img = p.c_state + (size_t)p.c_idx.v[n] * p.hidden * out_plane;
#pragma unroll
    for (int jj = 0; jj < HB; ++jj)
#pragma unroll
      for (int i = 0; i < PX; ++i) {
        const int dx = (i >> 2) * RUN_STEP + (i & 3);
        c_old[jj * PX + i] = (grp * HB + jj < p.hidden && yo < p.Ho && xo + dx < p.Wo) ? c_img[(size_t)(grp * HB + jj) * out_plane + pix + dx] : 0.0f;
      }
  }

  unsigned long long acc2[OC / 2][PX];               // [pair of channels][pixel]
#pragma unroll
  for (int i = 0; i < PX * OC / 2; ++i) acc2[i / PX][i % PX] = 0ull;

  int buf = 0;
  for (int c0 = 0; c0 < cin; c0 += CB) {
    const float* cur = smem + buf * Cfg::BUF_FLOATS;
    copies_wait<1>();                                // all but the newest group: this chunk has landed
    __syncthreads();                                 // ... for every thread, and nobody reads the chunk before it any more
    if (c0 + 2 * CB < cin) {
      float* nxt = smem + (buf == 0 ? 2 : buf - 1) * Cfg::BUF_FLOATS;
      stage_weights(c0 + 2 * CB, nxt);
      stage_input(c0 + 2 * CB, nxt);
    }
    copies_commit();                                 // also where there is nothing left to copy, so that the wait above counts alike
    buf = buf == 2 ? 0 : buf + 1;
    const int c_end = min(CB, cin - c0);
    if constexpr (AHEAD) {
      const float* in_c = cur + (ks * IN_H + ly) * PITCH + lx;
      const float* w_c = cur + Cfg::IN_FLOATS + (ks * 9 * WO + wo) * OC;
      float xn[RUNS][6];
      ulonglong2 wn[3][OC / 4];
      auto fetch = [&](const float* in, const float* w) {
#pragma unroll
        for (int g = 0; g < RUNS; ++g) load_row(in + g * RUN_STEP, xn[g]);
#pragma unroll
        for (int kx = 0; kx < 3; ++kx)
#pragma unroll
          for (int o = 0; o < OC / 4; ++o) wn[kx][o] = *reinterpret_cast<const ulonglong2*>(w + kx * WO * OC + 4 * o);
      };
      if (ks < c_end) fetch(in_c, w_c);
#pragma unroll 1
      for (int c = ks; c < c_end; c += KS) {
        const bool more = c + KS < c_end;
        const float* in_next = in_c + (more ? KS * IN_H * PITCH : 0);     // behind the last channel: that one again, unused
        const float* w_next = w_c + (more ? KS * 9 * WO * OC : 0);
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
          unsigned long long x2[RUNS][6];               // each value twice
#pragma unroll
          for (int g = 0; g < RUNS; ++g)
#pragma unroll
            for (int i = 0; i < 6; ++i) {
              const float v = EPI == EPI_RELU_BF16_NHWC ? round_bf16(xn[g][i]) : xn[g][i];
              x2[g][i] = tc::pack2(v, v);
            }
          ulonglong2 w[3][OC / 4];
#pragma unroll
          for (int kx = 0; kx < 3; ++kx)
#pragma unroll
            for (int o = 0; o < OC / 4; ++o) w[kx][o] = wn[kx][o];
          if (ky < 2) fetch(in_c + (ky + 1) * PITCH, w_c + (ky + 1) * 3 * WO * OC);
          else fetch(in_next, w_next);
#pragma unroll
          for (int kx = 0; kx < 3; ++kx) {
#pragma unroll
            for (int o = 0; o < OC; o += 4) {
#pragma unroll
              for (int i = 0; i < PX; ++i) {
                const unsigned long long v = x2[i >> 2][(i & 3) + kx];
                tc::fma2(acc2[o / 2][i], v, w[kx][o >> 2].x);
                tc::fma2(acc2[o / 2 + 1][i], v, w[kx][o >> 2].y);
              }
            }
          }
        }
        in_c = in_next;
        w_c = w_next;
      }
    } else {
#pragma unroll 1
      for (int c = ks; c < c_end; c += KS) {
        const float* in_c = cur + (c * IN_H + ly * STRIDE) * PITCH + lx;
        const float* w_c = cur + Cfg::IN_FLOATS + (c * 9 * WO + wo) * OC;
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
          // x[g][i]: input column (lx + 8 g) * STRIDE + i of this row
          float x[RUNS][3 * STRIDE + 3];
#pragma unroll
          for (int g = 0; g < RUNS; ++g) {
            const float* r = in_c + ky * PITCH + g * RUN_STEP;
            if constexpr (STRIDE == 1) {
              load_row(r, x[g]);
            } else {
              const float4 e = *reinterpret_cast<const float4*>(r);
              const float4 o = *reinterpret_cast<const float4*>(r + Cfg::ODD);
              x[g][0] = e.x; x[g][2] = e.y; x[g][4] = e.z; x[g][6] = e.w; x[g][8] = r[4];
              x[g][1] = o.x; x[g][3] = o.y; x[g][5] = o.z; x[g][7] = o.w;
            }
            if (EPI == EPI_RELU_BF16_NHWC) {
#pragma unroll
              for (int i = 0; i < 3 * STRIDE + 3; ++i) x[g][i] = round_bf16(x[g][i]);
            }
          }
          unsigned long long x2[RUNS][3 * STRIDE + 3];   // each value twice
#pragma unroll
          for (int g = 0; g < RUNS; ++g)
#pragma unroll
            for (int i = 0; i < 3 * STRIDE + 3; ++i) x2[g][i] = tc::pack2(x[g][i], x[g][i]);
#pragma unroll
          for (int kx = 0; kx < 3; ++kx) {
            const ulonglong2* w = reinterpret_cast<const ulonglong2*>(w_c + (ky * 3 + kx) * WO * OC);
#pragma unroll
            for (int o = 0; o < OC; o += 4) {
              const ulonglong2 w4 = w[o >> 2];
#pragma unroll
              for (int i = 0; i < PX; ++i) {
                const unsigned long long v = x2[i >> 2][(i & 3) * STRIDE + kx];
                tc::fma2(acc2[o / 2][i], v, w4.x);
                tc::fma2(acc2[o / 2 + 1][i], v, w4.y);
              }
            }
          }
        }
      }
    }
  }

  float acc[OC][PX];                                 // [channel][pixel]
#pragma unroll
  for (int o = 0; o < OC; o += 2)
#pragma unroll
    for (int i = 0; i < PX; ++i) tc::unpack2(acc2[o / 2][i], acc[o][i], acc[o + 1][i]);

  if (KS > 1) {
    // partial sums of the other channel groups, [group - 1][tile warp][value][lane], added in a fixed order
    const int tw = warp % (WO * WY);
    __syncthreads();                                 // the last chunk has been read
    if (ks > 0) {
#pragma unroll
      for (int i = 0; i < PX * OC; ++i) smem[(((ks - 1) * WO * WY + tw) * PX * OC + i) * 32 + lane] = acc[i / PX][i % PX];
    }
    __syncthreads();
    if (ks > 0) return;
#pragma unroll
    for (int k = 0; k < KS - 1; ++k)
#pragma unroll
      for (int i = 0; i < PX * OC; ++i) acc[i / PX][i % PX] += smem[((k * WO * WY + tw) * PX * OC + i) * 32 + lane];
  }

  if (yo >= p.Ho || xo >= p.Wo) return;
  const float* bias = p.bias + grp * OC;
  // four pixels of a planar map: one 128-bit store where the row length keeps them aligned
  const bool vec = (p.Wo & 3) == 0;
  auto store4 = [&](float* dst, int n_px, const float (&v)[4]) {
    if (vec) {
      *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < n_px) dst[i] = v[i];
    }
  };
#pragma unroll
  for (int g = 0; g < RUNS; ++g) {
  const int dx = g * RUN_STEP, n_px = min(4, p.Wo - xo - dx);
  if (n_px <= 0) break;

  if (EPI == EPI_RELU_F32_NCHW) {
    float* out = reinterpret_cast<float*>(p.out) + (size_t)n * p.out_img_stride;
#pragma unroll
    for (int o = 0; o < OC; ++o) {
      if (grp * OC + o < p.cout) {
        const float b = __ldg(bias + o);
        const float v[4] = {fmaxf(acc[o][4 * g] + b, 0.0f), fmaxf(acc[o][4 * g + 1] + b, 0.0f), fmaxf(acc[o][4 * g + 2] + b, 0.0f), fmaxf(acc[o][4 * g + 3] + b, 0.0f)};
        store4(out + (size_t)(grp * OC + o) * out_plane + pix + dx, n_px, v);
      }
    }
  } else if (EPI == EPI_RELU_BF16_NHWC) {
    // channels-last with a multiple of 8 channels: this thread's 8 are one aligned 16-byte piece of each pixel
    __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(p.out) + (size_t)n * p.out_img_stride + (pix + dx) * p.cout + grp * OC;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (i < n_px) {
        uint32_t u[4];
#pragma unroll
        for (int o = 0; o < OC; o += 2) {
          const __nv_bfloat162 h = __floats2bfloat162_rn(fmaxf(acc[o][4 * g + i] + __ldg(bias + o), 0.0f), fmaxf(acc[o + 1][4 * g + i] + __ldg(bias + o + 1), 0.0f));
          u[o >> 1] = *reinterpret_cast<const uint32_t*>(&h);
        }
        *reinterpret_cast<uint4*>(out + (size_t)i * p.cout) = make_uint4(u[0], u[1], u[2], u[3]);
      }
    }
  } else {
    // Packed order inside the group: local = gate*2 + jj, hidden unit j = grp*2 + jj.
    float* c_img = p.c_state + (size_t)p.c_idx.v[n] * p.hidden * out_plane;
    float* h_img = p.h_state + (size_t)p.h_out_idx.v[n] * p.hidden * out_plane;
#pragma unroll
    for (int jj = 0; jj < HB; ++jj) {
      const int j = grp * HB + jj;
      if (j < p.hidden) {
        float c_new[4], h_new[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float gi = acc[0 * HB + jj][4 * g + i] + __ldg(bias + 0 * HB + jj);
          const float gf = acc[1 * HB + jj][4 * g + i] + __ldg(bias + 1 * HB + jj);
          const float gg = acc[2 * HB + jj][4 * g + i] + __ldg(bias + 2 * HB + jj);
          const float go = acc[3 * HB + jj][4 * g + i] + __ldg(bias + 3 * HB + jj);
          c_new[i] = sigmoid_acc(gf) * c_old[jj * PX + 4 * g + i] + sigmoid_acc(gi) * tanhf(gg);
          h_new[i] = sigmoid_acc(go) * tanhf(c_new[i]);
        }
        store4(c_img + (size_t)j * out_plane + pix + dx, n_px, c_new);
        store4(h_img + (size_t)j * out_plane + pix + dx, n_px, h_new);
      }
    }
  }
  }
}

template <int STRIDE, int EPI, int WY, int WO, int KS, int PX = 4>
cudaError_t launch_one(const ConvSimtParams& p, cudaStream_t s) {
  using Cfg = SimtCfg<STRIDE, WY, WO, KS, PX>;
  auto kern = conv3x3_simt_kernel<STRIDE, EPI, WY, WO, KS, PX>;
  const int tiles = ((p.Wo + Cfg::TW - 1) / Cfg::TW) * ((p.Ho + Cfg::TH - 1) / Cfg::TH), groups = p.cout_packed / (WO * OC);
  // As a dependent the grid starts while its predecessor still holds some multiprocessors, and the others would be filled with as many blocks
  // as fit (three ConvLSTM maps of 80x60: 90 us instead of 67).  So a block asks for enough shared memory that one more than the busiest
  // multiprocessor's even share does not fit.  An encoder layer of one block to a multiprocessor asks for no more than it takes, so that it can lie beside its
  // predecessor's blocks; a ConvLSTM of one block asks for its half all the same: its blocks ran in piles of up to four, how many depending on the registers of the layer
  // before it (one and three maps of 40x30, 64 channels behind 64: 120, 161 -> 49, 69 us; of 80x60, 64 behind 32: 55, 127 -> 38, 60).
  constexpr int SMEM_SM = 228 * 1024, SMEM_RESERVED = 1024;      // of a multiprocessor, and per block beside its own
  const long share = ((long)tiles * groups * p.K + p.sm_count - 1) / p.sm_count;
  const int smem = share == 1 && EPI != EPI_LSTM_F32_NCHW ? Cfg::SMEM_BYTES : std::max<int>(Cfg::SMEM_BYTES, (int)(SMEM_SM / (std::min<long>(share, 15) + 1)) - SMEM_RESERVED + 16);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_SM - SMEM_RESERVED);
  if (e != cudaSuccess) return e;
  return launch_kernel(kern, dim3(tiles, groups, p.K), Cfg::THREADS, smem, s, p, p.pdl != 0);
}

// How many warps share out the input channels of a tile.  Their partial sums are added up in an order that depends on this number, so
// it follows from the layer's shape for ONE stream: a stream's results must not change with the streams that share its tick, nor with
// the multiprocessors left to another workload.  `warps` is what one stream's unsplit launch would have.  Below one per
// multiprocessor four warps share a tile's channels, up to 400 two do (the line lies between the measured 256 and 540).  K = 1, 3, 8 streams, us
// with 1 / 2 / 4 warps to a tile:
//   40x30 x 128 channels from 64, stride 2 (64 warps)    25.9 25.9 26.3 / 17.4 17.4 25.8 / 12.9 18.0 28.7
//   64x64 x 64 from 32 (256)                             14.1 20.0 34.2 / 10.4 17.4 36.1 /  9.9 23.4 43.7
//   80x60 x 96 from 48 (540)                             19.9 39.5 95.8 / 18.7 45.1 103 / 19.7 52.6 124
//   80x60 x 128 from 64 (720)                            36.5 64.0 157  / 30.9 73.5 177 / 30.2 82.8 208
// Three input channels (a first layer) have little to share: two warps below the first line, else one; bf16 outputs are always one
// warp's sums.
int simt_split(const ConvSimtParams& p) {
  const long warps = (long)((p.Wo + 31) / 32) * ((p.Ho + 3) / 4) * (p.cout_packed / OC);
  if (p.epilogue == EPI_RELU_BF16_NHWC) return 1;
  if (p.C0 + p.C1 < 8) return warps < 148 ? 2 : 1;
  return warps < 148 ? 4 : warps < 400 ? 2 : 1;
}

// The block shape and the pixels per thread, which change no bit: what leaves the busiest multiprocessor least to do, in warps of 4 pixels per
// thread.  As many channel groups on one staged input tile as divide the layer's; twice the output rows where that is no more (half the weight
// copies and less halo); at stride 1 eight pixels per thread where that is less, or no more than four or more of them (fewer loads per FMA, but
// coarser).  80x60 x 128 channels from 64, 1, 2, 3, 4, 5, 8 maps, stage times with their event: four pixels 39.7 55.3 67.8 83.7 110 153 us, eight 41.1
// 65.5 66.9 91.9 92.3 143.
template <int STRIDE, int EPI, int WY, int WO>
cudaError_t launch_rows(const ConvSimtParams& p, cudaStream_t s) {
  const long groups = (long)(p.cout_packed / (WO * OC)) * p.K, cols = groups * ((p.Wo + 31) / 32);
  auto busiest = [&](long blocks, long warps) { return (blocks + p.sm_count - 1) / p.sm_count * warps; };
  const long fine = busiest(cols * ((p.Ho + 4 * WY - 1) / (4 * WY)), WY * WO);
  const long coarse = busiest(cols * ((p.Ho + 8 * WY - 1) / (8 * WY)), 2 * WY * WO);
  const long eight = busiest(groups * ((p.Wo + 15) / 16) * ((p.Ho + 15) / 16), 2 * WO);
  if (STRIDE == 1 && (eight < std::min(fine, coarse) || (eight == std::min(fine, coarse) && eight >= 16))) return launch_one<1, EPI, 1, WO, 1, 8>(p, s);
  if (coarse <= fine) return launch_one<STRIDE, EPI, 2 * WY, WO, 1>(p, s);
  return launch_one<STRIDE, EPI, WY, WO, 1>(p, s);
}
template <int STRIDE, int EPI>
cudaError_t launch_epi(const ConvSimtParams& p, cudaStream_t s) {
  const int groups = p.cout_packed / OC, split = simt_split(p);
  if (split == 4) return launch_one<STRIDE, EPI, 1, 1, 4>(p, s);
  if (split == 2) return groups % 2 == 0 ? launch_one<STRIDE, EPI, 1, 2, 2>(p, s) : launch_one<STRIDE, EPI, 2, 1, 2>(p, s);
  if (groups % 4 == 0) return launch_rows<STRIDE, EPI, 1, 4>(p, s);
  return groups % 2 == 0 ? launch_rows<STRIDE, EPI, 2, 2>(p, s) : launch_one<STRIDE, EPI, 4, 1, 1>(p, s);
}

}  // namespace

cudaError_t launch_conv_simt(const ConvSimtParams& p, cudaStream_t s) {
  if (p.stride != 1 && p.stride != 2) return cudaErrorInvalidValue;
  switch (p.epilogue) {
    case EPI_RELU_F32_NCHW: return p.stride == 1 ? launch_epi<1, EPI_RELU_F32_NCHW>(p, s) : launch_epi<2, EPI_RELU_F32_NCHW>(p, s);
    case EPI_RELU_BF16_NHWC: return p.stride == 1 ? launch_epi<1, EPI_RELU_BF16_NHWC>(p, s) : launch_epi<2, EPI_RELU_BF16_NHWC>(p, s);
    case EPI_LSTM_F32_NCHW: return p.stride == 1 ? launch_epi<1, EPI_LSTM_F32_NCHW>(p, s) : cudaErrorInvalidValue;
  }
  return cudaErrorInvalidValue;
}

}  // namespace tt
