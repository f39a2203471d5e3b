// Stride-2 encoder layers of the bf16 path with one channel slab (32 or 64 input channels) on the tensor cores: 3x3
// convolution (pad 1, stride 2), bias, ReLU, channels-last bf16 in and out, as an implicit GEMM over tiles of 8 x 16 output pixels.
//
// At stride 2 the nine taps read four parity views of the input (even/odd rows x even/odd columns), each an ordinary
// dense tensor with doubled strides.  Per tile the producer fetches each view ONCE, with its halo (8x16, 9x16, 8x17 and
// 9x17 pixels: 561 pixels instead of nine boxes of 128), and the 1, 2, 2 and 4 taps of a view read it in place: a tap's
// A operand is the view entered (row * width + column) pixels further on, its groups of 8 rows one view row apart.  The
// swizzle is a function of the shared-memory address, so a start in the middle of its pattern needs nothing but the
// address.
//
// Taps are multiplied in their natural order, so the sums are the same bits as with one box per tap.  The views have
// barriers of their own and two buffers each (but for the smallest at 32 channels, where a second would cost the second
// block of the multiprocessor), so the next tile's views travel while this one's are multiplied.  A tile is 64 output
// channels wide: their weights (9 x 64 x 32 or 64 bf16, 36 or 72 KB) stay in shared memory for the whole launch, fetched
// before the wait for the previous kernel.  A block keeps its group of output channels and walks over the tiles.
//
// Against one box per tap a tile's barrier round trips fall from nine to four, and its bytes from 9 x 128 pixel rows and the weights
// to 561 rows.  At 32 channels that wins at every number of tiles.  At 64 it does while a launch has few tiles per block, where
// its time is start-up, first copies and round trips; with many, shared-memory bandwidth decides (an MMA of 64 columns reads
// 6 KB, 48 cycles at 128 bytes a cycle for the 32 it keeps the tensor pipe busy; one of 128 columns 8 KB, 64 for 64), and the
// 128-wide tap-box form of conv_tc.cu does more per byte read: 64 -> 128 channels at 8 full-HD frames take 78 us there and 132 us here.
//
// Warp roles: 0 = views and weights by TMA, 1 = tensor memory and MMA issue, 2..5 = epilogue (TMEM lane quarter = warp
// mod 4; results leave through 2 KB of shared memory per warp and 32 channels, so that four lanes write 64 bytes of a
// pixel).  The whole MMA warp runs the issue loop and one elected lane issues: with uniform control flow the
// operand descriptors stay in uniform registers.
// All waits are bounded (see tc_ptx.cuh).
// Stage times with their event, tap-box form -> this one: one 854x480 stream 12.3 -> 10.3 us (32 -> 64 channels) and 12.3 -> 10.2 us
// (64 -> 128), five 17.0 -> 17.1 and 15.4 -> 14.3 us.
#include "tt_internal.h"
#include "tc_ptx.cuh"

namespace tt {
namespace {

using namespace tc;

constexpr int S2_THREADS = 192;
constexpr int N = 64;                                          // output channels of a tile
constexpr int S2_PW = 8, S2_PH = 16;                          // output tile
// view of a tap: even/even, even rows/odd columns, odd rows/even columns, odd/odd
__host__ __device__ constexpr int s2_view(int tap) { return (tap / 3 != 1 ? 2 : 0) + (tap % 3 != 1 ? 1 : 0); }
__host__ __device__ constexpr int s2_first(int v) { return v == 0 ? 4 : v == 1 ? 3 : v == 2 ? 1 : 0; }   // first and last tap of a view
__host__ __device__ constexpr int s2_last(int v) { return v == 0 ? 4 : v == 1 ? 5 : v == 2 ? 7 : 8; }
__host__ __device__ constexpr int s2_view_w(int v) { return S2_PW + (v & 1); }
__host__ __device__ constexpr int s2_view_h(int v) { return S2_PH + (v >> 1); }

template <int SLAB_C>
struct S2Cfg {
  static constexpr int ROW = SLAB_C * 2;                      // bytes of a pixel's slab
  __host__ __device__ static constexpr int tx(int v) { return s2_view_w(v) * s2_view_h(v) * ROW; }
  __host__ __device__ static constexpr int v_bytes(int v) { return (tx(v) + 1023) / 1024 * 1024; }
  __host__ __device__ static constexpr int bufs(int v) { return SLAB_C == 32 && v == 0 ? 1 : 2; }
  __host__ __device__ static constexpr int v_off(int v) { return v == 0 ? 0 : v_off(v - 1) + bufs(v - 1) * v_bytes(v - 1); }
  static constexpr int PATCH = v_off(4);
  static constexpr int B_BYTES = N * ROW;                     // one tap's weights
  static constexpr int OUT_BYTES = 4 * 2048;
  static constexpr int SMEM = PATCH + 9 * B_BYTES + OUT_BYTES + N * 4 + 256 + 1024 /*alignment slack*/;
  static_assert((SLAB_C == 32 ? 2 : 1) * (SMEM + 1024) <= 228 * 1024, "two blocks per multiprocessor at 32 channels, one at 64");
  static_assert(B_BYTES % 1024 == 0, "weight slabs keep the alignment of the swizzle pattern");
};

template <int SLAB_C>
__global__ void __launch_bounds__(S2_THREADS, SLAB_C == 32 ? 2 : 1) conv_s2_kernel(const __grid_constant__ ConvS2Params p) {
  using Cfg = S2Cfg<SLAB_C>;
  constexpr uint32_t LAYOUT = SLAB_C == 64 ? 2u : 4u;
  constexpr uint32_t IDESC = make_idesc(128, N);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* s_b = smem + Cfg::PATCH;
  uint8_t* s_out = s_b + 9 * Cfg::B_BYTES;
  float* s_bias = reinterpret_cast<float*>(s_out + Cfg::OUT_BYTES);
  uint64_t* vfull = reinterpret_cast<uint64_t*>(s_bias + N);               // [4][2] view landed in a buffer
  uint64_t* vempty = vfull + 8;                                            // [4][2] its taps have read it
  uint64_t* wfull = vempty + 8;                                            // all weights landed
  uint64_t* tfull = wfull + 1;                                             // [2]
  uint64_t* tempty = tfull + 2;                                            // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  // before anything else: a second block of the multiprocessor does not start until the permit to allocate is given up
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"((uint32_t)(2 * N)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    for (int v = 0; v < 8; ++v) {
      mbar_init(smem_u32(vfull + v), 1);
      mbar_init(smem_u32(vempty + v), 1);
      if (v < 4) asm volatile("prefetch.tensormap [%0];" ::"l"(&p.map_v[v]) : "memory");
    }
    mbar_init(smem_u32(wfull), 1);
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(tfull + a), 1);
      mbar_init(smem_u32(tempty + a), 4);
    }
    *abort_flag = 0;
    asm volatile("prefetch.tensormap [%0];" ::"l"(&p.map_b) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const int nt = (int)blockIdx.x % p.n_tiles_n, worker = (int)blockIdx.x / p.n_tiles_n, n_workers = (int)gridDim.x / p.n_tiles_n;
  for (int i = threadIdx.x; i < N; i += S2_THREADS) s_bias[i] = __ldg(p.bias + nt * N + i);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_launch_dependents();   // behind the allocation: a dependent block must not take tensor memory that this grid still needs

  const long long wait_limit = p.wait_limit;
  const int tiles_per_img = p.tiles_x * p.tiles_y, m_tiles = p.K * tiles_per_img;

  if (warp == 0 && lane == 0) {
    // ------------------------------------------------------------------------- views
    mbar_arrive_expect_tx(smem_u32(wfull), 9 * Cfg::B_BYTES);
    for (int i = 0; i < 9; ++i) tma_load_2d(smem_u32(s_b + i * Cfg::B_BYTES), &p.map_b, smem_u32(wfull), i * SLAB_C, nt * N);
    pdl_wait();   // the weights are nobody's output; from here on the previous kernel's results are read
    uint32_t seq = 0;   // tiles so far: buffer seq % 2 in its phase seq / 2 % 2, or a single buffer in phase seq % 2
    bool ok = true;
    for (int m = worker; m < m_tiles && ok; m += n_workers, ++seq) {
      const int img = m / tiles_per_img, rem = m - img * tiles_per_img, ty = rem / p.tiles_x, tx = rem - ty * p.tiles_x;
#pragma unroll
      for (int v = 3; v >= 0; --v) {   // in the order of their first taps
        const uint32_t buf = Cfg::bufs(v) == 2 ? seq & 1u : 0u, phase = Cfg::bufs(v) == 2 ? (seq >> 1) & 1u : seq & 1u;
        const uint32_t bar = smem_u32(vfull + 2 * v + buf);
        ok = ok && mbar_wait(smem_u32(vempty + 2 * v + buf), phase ^ 1u, abort_flag, p.status, WAIT_CONV_S2 + v, wait_limit);
        if (!ok) break;
        mbar_arrive_expect_tx(bar, Cfg::tx(v));
        tma_load_4d(smem_u32(smem + Cfg::v_off(v) + buf * Cfg::v_bytes(v)), &p.map_v[v], bar, 0, tx * S2_PW - (v & 1), ty * S2_PH - (v >> 1), p.img0 + img);
      }
    }
  } else if (warp == 1) {
    // -------------------------------------------------------------------- MMA issuer
    // whole warp, uniform control flow, one elected lane issues; a wait that ran out ends the loop at the end of its tile
    const bool issuer = elect_one();
    uint32_t seq = 0, acc_phase = 0;
    int acc = 0;
    bool ok = true;
    const uint64_t b_desc0 = make_smem_desc(smem_u32(s_b), 8u * Cfg::ROW, LAYOUT);
    ok &= mbar_wait_uniform(smem_u32(wfull), 0u, abort_flag, p.status, WAIT_CONV_S2 + 0x20, wait_limit);
    for (int m = worker; m < m_tiles; m += n_workers) {
      ok &= mbar_wait_uniform(smem_u32(tempty + acc), acc_phase ^ 1u, abort_flag, p.status, WAIT_CONV_S2 + 0x30 + acc, wait_limit);
      tc_fence_after();   // the epilogue's reads of this accumulator come before the MMAs that overwrite it
      const uint32_t d_tmem = tmem_base + (uint32_t)(acc * N);
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const int v = s2_view(i), ky = i / 3, kx = i % 3;
        const uint32_t buf = Cfg::bufs(v) == 2 ? seq & 1u : 0u, phase = Cfg::bufs(v) == 2 ? (seq >> 1) & 1u : seq & 1u;
        if (i == s2_first(v)) ok &= mbar_wait_uniform(smem_u32(vfull + 2 * v + buf), phase, abort_flag, p.status, WAIT_CONV_S2 + 0x40 + v, wait_limit);
        const uint64_t a = make_smem_desc(smem_u32(smem + Cfg::v_off(v)), (uint32_t)(s2_view_w(v) * Cfg::ROW), LAYOUT) +
                           (uint64_t)(((ky == 2 ? s2_view_w(v) : 0) + (kx == 2 ? 1 : 0)) * Cfg::ROW >> 4) + (uint64_t)(buf * (Cfg::v_bytes(v) >> 4));
        const uint64_t b = b_desc0 + (uint64_t)(i * Cfg::B_BYTES >> 4);
        if (issuer) {
#pragma unroll
          for (int k = 0; k < SLAB_C / 16; ++k) umma_bf16(d_tmem, a + (uint64_t)(2 * k), b + (uint64_t)(2 * k), IDESC, (i == 0 && k == 0) ? 0u : 1u);
          if (i == s2_last(v)) umma_commit(smem_u32(vempty + 2 * v + buf));
        }
      }
      ++seq;
      if (__any_sync(0xffffffffu, !ok)) break;
      if (issuer) umma_commit(smem_u32(tfull + acc));
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
  } else if (warp >= 2 && warp < 6) {
    // ---------------------------------------------------------------------- epilogue
    const int quarter = warp & 3;
    uint8_t* mine = s_out + (warp - 2) * 2048;       // 32 pixels x 64 bytes; 16-byte piece c of pixel i at piece c ^ (i / 2 % 4)
    uint32_t acc_phase = 0;
    int acc = 0;
    for (int m = worker; m < m_tiles; m += n_workers) {
      const int img = m / tiles_per_img, rem = m - img * tiles_per_img, ty = rem / p.tiles_x, tx = rem - ty * p.tiles_x;
      // this lane writes piece lane % 4 of the pixels lane / 4 + 8 q of the warp's 32 (4 rows of 8)
      const int x = tx * S2_PW + (lane >> 2), y0 = ty * S2_PH + quarter * 4;
      __nv_bfloat16* out = p.out + (((size_t)img * p.Ho + y0) * p.Wo + x) * p.cout + nt * N + (lane & 3) * 8;
      const bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(tfull + acc), acc_phase, abort_flag, p.status, WAIT_CONV_S2 + 0x60 + acc, wait_limit));
      if (!ok) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * N);
      uint32_t v[2][32];
      tmem_ld32_async(taddr, v[0]);
      tmem_ld32_async(taddr + 32u, v[1]);
      tmem_wait_ld();
      // the accumulator has been read: hand it back to the MMA warp
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(tempty + acc));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4* b4 = reinterpret_cast<const float4*>(s_bias + h * 32);
#pragma unroll
        for (int i = 0; i < 32; i += 8) {
          const float4 ba = b4[i / 4], bb = b4[i / 4 + 1];
          uint4 u;
          u.x = pack_relu_bf16(__uint_as_float(v[h][i + 0]) + ba.x, __uint_as_float(v[h][i + 1]) + ba.y);
          u.y = pack_relu_bf16(__uint_as_float(v[h][i + 2]) + ba.z, __uint_as_float(v[h][i + 3]) + ba.w);
          u.z = pack_relu_bf16(__uint_as_float(v[h][i + 4]) + bb.x, __uint_as_float(v[h][i + 5]) + bb.y);
          u.w = pack_relu_bf16(__uint_as_float(v[h][i + 6]) + bb.z, __uint_as_float(v[h][i + 7]) + bb.w);
          *reinterpret_cast<uint4*>(mine + lane * 64 + (((i >> 3) ^ ((lane >> 1) & 3)) << 4)) = u;
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int px = q * 8 + (lane >> 2);
          const uint4 u = *reinterpret_cast<const uint4*>(mine + px * 64 + (((lane & 3) ^ ((px >> 1) & 3)) << 4));
          if (x < p.Wo && y0 + q < p.Ho) *reinterpret_cast<uint4*>(out + (size_t)q * p.Wo * p.cout + h * 32) = u;
        }
        __syncwarp();
      }
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
  }

  // ------------------------------------------------------------------------------- teardown
  __syncwarp();
  if (*abort_flag) {
    // a wait ran out somewhere: give copies and MMAs in flight time to land before their memory is released
    for (int i = 0; i < 64; ++i) __nanosleep(16000);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)(2 * N)) : "memory");
  }
}

template <int SLAB_C>
cudaError_t launch_t(const ConvS2Params& p, int sm_count, cudaStream_t s) {
  using Cfg = S2Cfg<SLAB_C>;
  auto kern = conv_s2_kernel<SLAB_C>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM);
  if (e != cudaSuccess) return e;
  const int per_sm = (SLAB_C == 32 && !p.one_per_sm) ? 2 : 1;
  const int m_tiles = p.K * p.tiles_x * p.tiles_y;
  int workers = per_sm * sm_count / p.n_tiles_n;
  if (workers < 1) workers = 1;
  if (workers > m_tiles) workers = m_tiles;
  return launch_kernel(kern, workers * p.n_tiles_n, S2_THREADS, Cfg::SMEM, s, p, p.pdl != 0);
}

}  // namespace

// Output channels per tile, or 0 where this kernel does not apply: more than one channel slab.
int conv_s2_block_n(int slab_c, int cin, int cout) { return cin == slab_c && cout % N == 0 ? N : 0; }

// Against the tap-box form, whole ticks of a feed-forward model (us, mean of 360; `rounds` = units per block):
//   32 input channels, two blocks per multiprocessor: never slower.  Rounds 0.5 -1.7, 1.6 -1.5, 2.7 -1.0, 4.3 -0.7, 6.5 -2.0, 9.7 -4.3,
//   13 (eight full-HD streams) -7.6 of 166.  One block, which leaves half of the copies exposed: 1.1 -0.1, 3.2 -1.5, 4.3 +0.3, 7.3 +1.5, 26 +2.0.
//   64 input channels, one block: 0.5 -1.5, 1.6 -1.0, 2.0 +1.9, 2.2 -2.0, 2.7 -1.4, 3.0 +0.4, 3.2 +1.2, 4.1 +2.4, 4.9 +0.4, 6.5 +2.6, 13 +6.1.
bool conv_s2_pays(int slab_c, int units, int sm_count, bool one_per_sm) {
  if (slab_c == 32 && !one_per_sm) return true;
  return units <= (slab_c == 32 ? 4 : 3) * sm_count;
}

void conv_s2_box(int view, int* w, int* h) {
  *w = s2_view_w(view);
  *h = s2_view_h(view);
}

cudaError_t launch_conv_s2(const ConvS2Params& p, int sm_count, cudaStream_t s) {
  if (p.slab_c == 32) return launch_t<32>(p, sm_count, s);
  if (p.slab_c == 64) return launch_t<64>(p, sm_count, s);
  return cudaErrorInvalidValue;
}

}  // namespace tt
