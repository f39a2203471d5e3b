// ConvLSTM step of the bf16 path on the tensor cores, 64-channel slabs: the 3x3 convolution over [x, h] into i/f/g/o gates as an
// implicit GEMM (M = output pixels, N = 4 x hidden, K = 9 taps x channels), gate math, c' and h' in the epilogue.
//
// The output tile is an 8 x 16-pixel patch.  Per 64-channel slab ONE haloed patch (18 rows of 10 pixels, a 4-D TMA box in the ordinary
// 128-byte swizzle) is fetched, and the nine taps read it in place: output pixel (py, px) of tap (ky, kx) is patch row
// (py + ky) * 10 + px + kx, so a tap's A operand is the same shared memory entered (ky * 10 + kx) * 128 bytes further on, its groups of 8
// rows 1280 bytes apart.  The swizzle is a function of the shared-memory address, so a start in the middle of its pattern needs
// nothing but the address.  Weights come one tap and slab at a time through a ring, the first before the wait for the previous kernel.
//
// Bound by the tensor pipe where the rounds of units are full, and there by the clock that the power limit leaves; the bytes that travel from
// L2 into the multiprocessors cost part of that power.  So beyond one round two blocks of a cluster work as a pair: one MMA of 256 rows
// (cta_group::2) takes both blocks' tiles and half of the weight rows from each, 18.6 instead of 34.6 KB into a multiprocessor per 512
// tensor cycles.  1.087 PFLOP of eight full-HD streams: 670 us on single blocks (1.62 PFLOP/s) -> 633 us (1.72 PFLOP/s), tick 1135 -> 1075 us;
// one full-HD stream's tick 179 -> 170 us, five 854x480 streams' 115.3 -> 114.5 us.  One commit that signals both blocks, and the issue loop
// below, make the difference to an earlier pair form (conv_tc.cu's, kept as an option) that was 11-15 % slower than single blocks.
//
// Bound by rounds where they are not full: a multiprocessor holds one block, and 80 units of 256 columns (one 854x480 stream) take as long as
// 148.  A unit is a tile (or a pair's two) x a group of columns, grouped as the launch needs: by 192 (with a remainder of 64 or 128) where that
// still fits the rounds, or by 256 with the last, partly filled round cut into halves.  M128 x N x K16 takes 128, 96 and 64
// cycles at N = 256, 192 and 128; for a narrow group's slab to take less than a wide one's, the whole MMA warp
// runs the issue loop and one elected lane issues (from a single lane's branch a slab takes about 600 cycles at any width).
// ConvLSTM stage with its event, units of 256 -> this: one 854x480 stream 23.6 -> 20.5 us, one full-HD stream 105.5 -> 101.4 us.
// The order of the sums is the same in all forms, so the results are the same bits.
//
// Warp roles (384 threads): 0 = patches by TMA; 10, 11 = weights by TMA, alternate iterations; 1 = tensor memory and MMA
// issue (of a pair: its first block's); 2..9 = epilogue (TMEM lane quarter = warp mod 4, two warps per quarter sharing a unit's columns).
// Two accumulators, so the epilogue of a unit overlaps the next one's products.  A pair's copies complete on its first block's barriers, which
// expect both blocks' bytes; "free" barriers are signalled in both blocks.  All waits are bounded (see tc_ptx.cuh).
#include <algorithm>

#include "tt_internal.h"
#include "tc_ptx.cuh"

namespace tt {
namespace {

using namespace tc;

constexpr int L_THREADS = 384;
constexpr int L_EPI_WARPS = 8, L_EPI_WARP0 = 2;
constexpr int L_PW = 8, L_PH = 16;                       // output tile
constexpr int L_PITCH = 10, L_ROWS = 18;                 // haloed patch
constexpr int L_A_TX = L_ROWS * L_PITCH * 128;
constexpr int L_A_BYTES = (L_A_TX + 1023) / 1024 * 1024;
constexpr int L_A_STAGES = 2;
constexpr int L_MAX_COLS = 4 * 512;

template <bool PAIR>
struct LCfg {
  static constexpr int B_BYTES = (PAIR ? 128 : 256) * 128;   // a block's rows of the widest group, 64 channels each
  static constexpr int B_STAGES = PAIR ? 10 : 5;
  static constexpr int B_STEP = PAIR ? 32 : 64;              // rows of the small weight box
  static constexpr int BAR_BYTES = 256;
  static constexpr int SMEM = B_STAGES * B_BYTES + L_A_STAGES * L_A_BYTES + L_MAX_COLS * 4 + BAR_BYTES + 1024 /*alignment slack*/;
  static_assert(SMEM <= 227 * 1024, "one block per multiprocessor");
  static_assert((2 * B_STAGES + 8) * 8 + 8 <= BAR_BYTES, "barriers");
};

struct Unit {
  int m, col0, n;   // pixel tile, first column, columns
};
// Units in order of tile, then column group; from unit u_full on every group is cut into two.
__device__ __forceinline__ Unit unit_at(const ConvLstmParams& p, int u) {
  Unit t;
  const int v = u - p.u_full, g = v < 0 ? u : p.u_full + (v >> 1);
  t.m = g / p.groups;
  t.col0 = (g - t.m * p.groups) * p.width;
  t.n = min(p.width, p.cols - t.col0);
  if (v >= 0) {
    t.n >>= 1;
    t.col0 += (v & 1) * t.n;
  }
  return t;
}

template <bool PAIR>
__global__ void __launch_bounds__(L_THREADS, 1) conv_lstm_kernel(const __grid_constant__ ConvLstmParams p) {
  using Cfg = LCfg<PAIR>;
  constexpr int L_B_STAGES = Cfg::B_STAGES, L_B_BYTES = Cfg::B_BYTES;
  constexpr int CTAS = PAIR ? 2 : 1;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* s_b = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* s_a = s_b + L_B_STAGES * L_B_BYTES;
  float* s_bias = reinterpret_cast<float*>(s_a + L_A_STAGES * L_A_BYTES);
  uint64_t* bfull = reinterpret_cast<uint64_t*>(s_bias + L_MAX_COLS);   // [L_B_STAGES]
  uint64_t* bempty = bfull + L_B_STAGES;                                // [L_B_STAGES]
  uint64_t* afull = bempty + L_B_STAGES;                                // [2] patch landed
  uint64_t* aempty = afull + 2;                                         // [2] all nine taps have read the patch
  uint64_t* tfull = aempty + 2;                                         // [2]
  uint64_t* tempty = tfull + 2;                                         // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  __shared__ int s_img[4][TT_MAX_STREAMS];                              // h in, c, h out, x in

  // broadcast, so that the compiler knows the roles below to be whole warps
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const long long wait_limit = p.wait_limit;
  const int rank = PAIR ? (int)cluster_ctarank() : 0;
  const int worker = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x, n_workers = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
  const int total = p.u_full + 2 * (p.m_units * p.groups - p.u_full);
  const int slabs = p.slabs[0] + p.slabs[1];
  if (threadIdx.x == 0) {
    for (int s = 0; s < L_B_STAGES; ++s) {
      mbar_init(smem_u32(bfull + s), 1);
      mbar_init(smem_u32(bempty + s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(afull + a), 1);
      mbar_init(smem_u32(aempty + a), 1);
      mbar_init(smem_u32(tfull + a), 1);
      mbar_init(smem_u32(tempty + a), CTAS * L_EPI_WARPS);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&p.map_b) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&p.map_bs) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&p.maps[0]) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&p.maps[1]) : "memory");
  }
  if (warp == 1) {
    if (PAIR) {   // the same warp of both blocks allocates the pair's columns
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  if (threadIdx.x < TT_MAX_STREAMS) {
    s_img[0][threadIdx.x] = p.h_in.v[threadIdx.x];
    s_img[1][threadIdx.x] = p.c_idx.v[threadIdx.x];
    s_img[2][threadIdx.x] = p.h_out.v[threadIdx.x];
    s_img[3][threadIdx.x] = p.x_in.v[threadIdx.x];
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();   // the peer's barriers exist before anything is signalled across the pair
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_launch_dependents();   // behind the allocation: a dependent block must not take tensor memory that this grid still needs

  const int tiles_per_img = p.tiles_x * p.tiles_y;
  if (warp == 0 && lane == 0) {
    // ----------------------------------------------------------------------- patches
    pdl_wait();   // x is the previous kernel's output
    uint32_t stage = 0, phase = 0;
    bool ok = true;
    for (int u = worker; u < total && ok; u += n_workers) {
      // a pair's second block takes the next tile; behind the last tile it computes that one again and stores nothing
      const int m = min(CTAS * unit_at(p, u).m + rank, p.tiles - 1);
      const int img = m / tiles_per_img, rem = m - img * tiles_per_img, ty = rem / p.tiles_x, tx = rem - ty * p.tiles_x;
      const int img_h = s_img[0][img], img_x = s_img[3][img];
      for (int sg = 0; sg < slabs; ++sg) {
        ok = mbar_wait(smem_u32(aempty + stage), phase ^ 1u, abort_flag, p.status, WAIT_CONV_LSTM + 0x10 + (int)stage, wait_limit);
        if (!ok) break;
        const int src = sg < p.slabs[0] ? 0 : 1;
        const int c0 = (src ? sg - p.slabs[0] : sg) * 64, n_img = src ? img_h : img_x;
        if (rank == 0) mbar_arrive_expect_tx(smem_u32(afull + stage), CTAS * L_A_TX);
        if (PAIR) tma_load_4d_pair(smem_u32(s_a + stage * L_A_BYTES), &p.maps[src], map_to_cta(smem_u32(afull + stage), 0u), c0, tx * L_PW - 1, ty * L_PH - 1, n_img);
        else tma_load_4d(smem_u32(s_a + stage * L_A_BYTES), &p.maps[src], smem_u32(afull + stage), c0, tx * L_PW - 1, ty * L_PH - 1, n_img);
        if (++stage == L_A_STAGES) { stage = 0; phase ^= 1u; }
      }
    }
    // The last "free" signals of both buffers, which the MMAs' commits send into both blocks of a pair, arrive before either block leaves:
    // a later commit's signal (an accumulator's) says nothing about when an earlier one's reaches the other block.
    for (int i = 0; PAIR && i < L_A_STAGES && ok; ++i) {
      ok = mbar_wait(smem_u32(aempty + stage), phase ^ 1u, abort_flag, p.status, WAIT_CONV_LSTM + 0x18 + (int)stage, wait_limit);
      if (++stage == L_A_STAGES) { stage = 0; phase ^= 1u; }
    }
  } else if (warp >= L_EPI_WARP0 + L_EPI_WARPS && lane == 0) {
    // ----------------------------------------------------------------------- weights
    // producer j of two owns iterations j, j + 2, ... of the block's sequence (slab-major, tap inside)
    const int j = warp - (L_EPI_WARP0 + L_EPI_WARPS);
    const int iters = slabs * 9, cin = slabs * 64;
    uint32_t stage = (uint32_t)j, phase = 0;
    int it = j;
    bool ok = true;
    for (int u = worker; u < total && ok; u += n_workers) {
      const Unit t = unit_at(p, u);
      for (; it < iters; it += 2) {
        const int sg = it / 9, tap = it - sg * 9;
        ok = mbar_wait(smem_u32(bempty + stage), phase ^ 1u, abort_flag, p.status, WAIT_CONV_LSTM + (int)stage, wait_limit);
        if (!ok) break;
        const uint32_t bar = smem_u32(bfull + stage), dst = smem_u32(s_b + stage * L_B_BYTES);
        const int k0 = tap * cin + sg * 64, rows = t.n / CTAS, r0 = t.col0 + rank * rows;
        if (rank == 0) mbar_arrive_expect_tx(bar, (uint32_t)t.n * 128u);
        if (PAIR) {
          const uint32_t bar0 = map_to_cta(bar, 0u);
          if (t.n == 256) {
            tma_load_2d_pair(dst, &p.map_b, bar0, k0, r0);
          } else {
            for (int i = 0; i < rows; i += Cfg::B_STEP) tma_load_2d_pair(dst + i * 128, &p.map_bs, bar0, k0, r0 + i);
          }
        } else if (t.n == 256) {
          tma_load_2d(dst, &p.map_b, bar, k0, r0);
        } else {
          for (int i = 0; i < rows; i += Cfg::B_STEP) tma_load_2d(dst + i * 128, &p.map_bs, bar, k0, r0 + i);
        }
        stage += 2;
        if (stage >= (uint32_t)L_B_STAGES) { stage -= L_B_STAGES; phase ^= 1u; }
      }
      it -= iters;
    }
    // the last "free" signals of this producer's share of the ring: those its next iterations would wait for, one turn of the ring on
    for (; PAIR && it < L_B_STAGES && ok; it += 2) {
      ok = mbar_wait(smem_u32(bempty + stage), phase ^ 1u, abort_flag, p.status, WAIT_CONV_LSTM + 0x20 + (int)stage, wait_limit);
      stage += 2;
      if (stage >= (uint32_t)L_B_STAGES) { stage -= L_B_STAGES; phase ^= 1u; }
    }
  } else if (warp == 1 && rank == 0) {
    // -------------------------------------------------------------------- MMA issuer (of a pair: its first block)
    const bool issuer = elect_one();
    auto commit = [](uint64_t* bar) {
      if (PAIR) umma_commit_both(smem_u32(bar));
      else umma_commit(smem_u32(bar));
    };
    uint32_t stage = 0, phase = 0, acc_phase = 0, a_stage = 0, a_phase = 0;
    int acc = 0;
    bool ok = true;   // a wait that ran out ends the loop at the end of its unit
    const uint64_t b_desc0 = make_smem_desc(smem_u32(s_b), 1024u, 2u);
    for (int u = worker; u < total; u += n_workers) {
      // (no division in this loop where all groups are as wide)
      const int n = p.even ? (u < p.u_full ? p.width : p.width >> 1) : unit_at(p, u).n;
      const uint32_t idesc = make_idesc(128 * CTAS, 0) | ((uint32_t)(n >> 3) << 17);
      ok &= mbar_wait_uniform(smem_u32(tempty + acc), acc_phase ^ 1u, abort_flag, p.status, WAIT_CONV_LSTM + 0x30 + acc, wait_limit);
      tc_fence_after();   // the epilogue's reads of this accumulator come before the MMAs that overwrite it
      const uint32_t d_tmem = tmem_base + (uint32_t)(acc * 256);
      for (int sg = 0; sg < slabs; ++sg) {
        ok &= mbar_wait_uniform(smem_u32(afull + a_stage), a_phase, abort_flag, p.status, WAIT_CONV_LSTM + 0x40 + (int)a_stage, wait_limit);
        const uint64_t a_patch = make_smem_desc(smem_u32(s_a + a_stage * L_A_BYTES), L_PITCH * 128u, 2u);
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
          ok &= mbar_wait_uniform(smem_u32(bfull + stage), phase, abort_flag, p.status, WAIT_CONV_LSTM + 0x50 + (int)stage, wait_limit);
          const uint64_t a = a_patch + (uint64_t)(((tap / 3) * L_PITCH + tap % 3) * 128 >> 4);
          const uint64_t b = b_desc0 + (uint64_t)stage * (uint64_t)(L_B_BYTES >> 4);
          if (issuer) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {  // 16 bf16 = 32 bytes = 2 descriptor units further on inside the swizzle atom
              const uint32_t more = (tap == 0 && k == 0) ? (sg != 0 ? 1u : 0u) : 1u;
              if (PAIR) umma_bf16_pair(d_tmem, a + (uint64_t)(2 * k), b + (uint64_t)(2 * k), idesc, more);
              else umma_bf16(d_tmem, a + (uint64_t)(2 * k), b + (uint64_t)(2 * k), idesc, more);
            }
            commit(bempty + stage);
            if (tap == 8) commit(aempty + a_stage);
          }
          if (++stage == L_B_STAGES) { stage = 0; phase ^= 1u; }
        }
        if (++a_stage == L_A_STAGES) { a_stage = 0; a_phase ^= 1u; }
      }
      if (__any_sync(0xffffffffu, !ok)) break;
      if (issuer) commit(tfull + acc);
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
  } else if (warp >= L_EPI_WARP0 && warp < L_EPI_WARP0 + L_EPI_WARPS) {
    // ---------------------------------------------------------------------- epilogue
    // the biases are fetched here and not in front of the block's first barrier, where the copies would wait for them
    for (int i = threadIdx.x - 32 * L_EPI_WARP0; i < p.cols; i += 32 * L_EPI_WARPS) s_bias[i] = __ldg(p.bias + i);
    asm volatile("bar.sync 1, 256;" ::: "memory");
    pdl_wait();
    const int quarter = warp & 3, half = (warp - L_EPI_WARP0) >> 2;
    const int row = quarter * 32 + lane, py = row >> 3, px = row & 7;     // row of the 128-row tile = pixel of the patch
    uint32_t acc_phase = 0;
    int acc = 0;
    for (int u = worker; u < total; u += n_workers) {
      const Unit t = unit_at(p, u);
      const int m_own = CTAS * t.m + rank, m = min(m_own, p.tiles - 1);
      const int img = m / tiles_per_img, rem = m - img * tiles_per_img, ty = rem / p.tiles_x, tx = rem - ty * p.tiles_x;
      const int x = tx * L_PW + px, y = ty * L_PH + py;
      const bool valid = x < p.Wm && y < p.Hm && m_own < p.tiles;
      const size_t pix = (size_t)y * p.Wm + x;
      // chunks of 32 columns (8 hidden units x 4 gates), half of them for either of the quarter's two warps
      const int off = half ? t.n >> 1 : 0, chunks = t.n >> 6, odd = (off >> 5) & 1;
      const int col0 = t.col0 + off;

      // the old cell state of this thread's pixel is fetched before the accumulator is waited for: its latency hides under
      // the unit's products
      float c_old[4][8];
      const size_t so = ((size_t)s_img[1][img] * p.Hm * p.Wm + pix) * p.hidden + (col0 >> 2);
      const size_t ho = ((size_t)s_img[2][img] * p.Hm * p.Wm + pix) * p.hidden + (col0 >> 2);
#pragma unroll
      for (int ck = 0; ck < 4; ++ck)
        if (valid && ck < chunks) ld_global_v8(p.c_state + so + ck * 8, c_old[ck]);

      // the warp votes: its lanes leave the loop together or go on to the warp-collective TMEM loads together
      if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(tfull + acc), acc_phase, abort_flag, p.status, WAIT_CONV_LSTM + 0x60 + acc, wait_limit))) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * 256 + off);
      uint32_t hb[8];
#pragma unroll
      for (int ck = 0; ck < 4; ++ck) {
        if (ck < chunks) {
          uint32_t v[32];
          tmem_ld32(taddr + (uint32_t)(ck * 32), v);
          if (valid) {
            // packed column = 4 * unit + gate (i, f, g, o)
            const float4* b4 = reinterpret_cast<const float4*>(s_bias + col0 + ck * 32);
            float c_new[8], h_new[8];
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
              const float4 b = b4[jj];
              const float gi = __uint_as_float(v[4 * jj + 0]) + b.x;
              const float gf = __uint_as_float(v[4 * jj + 1]) + b.y;
              const float gg = __uint_as_float(v[4 * jj + 2]) + b.z;
              const float go = __uint_as_float(v[4 * jj + 3]) + b.w;
              c_new[jj] = fast_sigmoid(gf) * c_old[ck][jj] + fast_sigmoid(gi) * fast_tanh(gg);
              h_new[jj] = fast_sigmoid(go) * fast_tanh(c_new[jj]);
            }
            st_global_v8(p.c_state + so + ck * 8, c_new);
            if (p.h_f32) st_global_v8(p.h_f32 + so + ck * 8, h_new);
            // bf16 copy of h': 8 values are half a sector, so an even chunk of the unit waits for the odd one behind it
            const uint4 hv = make_uint4(pack_bf16(h_new[0], h_new[1]), pack_bf16(h_new[2], h_new[3]), pack_bf16(h_new[4], h_new[5]), pack_bf16(h_new[6], h_new[7]));
            if (((ck + odd) & 1) == 0) {
              hb[0] = hv.x; hb[1] = hv.y; hb[2] = hv.z; hb[3] = hv.w;
              if (ck + 1 == chunks) *reinterpret_cast<uint4*>(p.h_bf16 + ho + ck * 8) = hv;
            } else if (ck == 0) {
              *reinterpret_cast<uint4*>(p.h_bf16 + ho) = hv;
            } else {
              hb[4] = hv.x; hb[5] = hv.y; hb[6] = hv.z; hb[7] = hv.w;
              st_global_v8_b32(p.h_bf16 + ho + (ck - 1) * 8, hb);
            }
          }
        }
      }
      // hand the accumulator back to the MMA warp
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (PAIR) mbar_arrive_cluster(map_to_cta(smem_u32(tempty + acc), 0u));
        else mbar_arrive(smem_u32(tempty + acc));
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
  // neither block of a pair may go while the other can still signal its barriers or have its shared memory read by the pair's MMAs
  if (PAIR) cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    if (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

// Time of a unit in units of one of 256 columns: tensor cycles per slab (512, 384, 256) but no less than the issue loop's
// round of about 300, and the fixed parts.  Units of 128 columns throughout are never the fewest rounds' worth (tried for all widths of up to
// 2048 columns, 1 to 8000 tiles and 1 to 160 multiprocessors): 128 only appears as the half of a last round's units and as a remainder.
constexpr double L_COST_256 = 1.0, L_COST_192 = 0.77, L_COST_128 = 0.58;

struct Grouping {
  int width = 256, u_full = 0;
};
// m_units: tiles (or pairs of tiles) to be shared out over `workers` blocks (or pairs); C: a multiple of 256
Grouping group_columns(int m_units, int C, int workers) {
  Grouping g;
  auto rounds = [&](long units) { return (double)((units + workers - 1) / workers); };
  const long g256 = (long)m_units * (C / 256);
  g.u_full = (int)g256;
  double cost = rounds(g256) * L_COST_256;
  // the last round cut into halves, if that leaves it one round
  const long tail = g256 % workers;
  if (tail > 0 && 2 * tail <= workers) {
    cost = (double)(g256 / workers) * L_COST_256 + L_COST_128;
    g.u_full = (int)(g256 - tail);
  }
  const long units = (long)m_units * ((C + 191) / 192);
  if (rounds(units) * L_COST_192 < cost - 1e-9) { g.width = 192; g.u_full = (int)units; }
  return g;
}

template <bool PAIR>
cudaError_t launch_form(const ConvLstmParams& p, const TensorMap128& whole, const TensorMap128& step, int workers, cudaStream_t s) {
  constexpr int CTAS = PAIR ? 2 : 1;
  auto kern = conv_lstm_kernel<PAIR>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, LCfg<PAIR>::SMEM);
  if (e != cudaSuccess) return e;
  ConvLstmParams q = p;
  q.map_b = whole;
  q.map_bs = step;
  q.m_units = (q.tiles + CTAS - 1) / CTAS;
  const Grouping g = group_columns(q.m_units, q.cols, workers);
  q.width = g.width;
  q.u_full = g.u_full;
  q.groups = (q.cols + q.width - 1) / q.width;
  q.even = q.cols % q.width == 0;
  const long total = q.u_full + 2L * ((long)q.m_units * q.groups - q.u_full);
  return launch_kernel(kern, CTAS * (int)std::min<long>(total, workers), L_THREADS, LCfg<PAIR>::SMEM, s, q, q.pdl != 0, CTAS);
}

}  // namespace

// Pairs where the units of one tile take more than one round.  ConvLSTM stage with its event, single blocks -> pairs (us): one, two, five and eight
// full-HD streams 100.5 -> 94.2, 172 -> 162, 430 -> 397, 686 -> 633; four, six and eight 854x480 streams 45.1 -> 43.0, 57.3 -> 55.3, 71.1 -> 67.6,
// two and three (1.1 and 1.6 rounds) the same.  Within one round copies are not what a block waits for, and the pair's start and
// hand-overs show: one 854x480 stream 65.1 -> 65.3 us a tick.
cudaError_t launch_conv_lstm(const ConvLstmParams& p, const TensorMap128 (&rows)[4], int sm_count, cudaStream_t s) {
  if (p.cols < 256 || p.cols % 256 || p.cols > L_MAX_COLS) return cudaErrorInvalidValue;
  if ((long)p.tiles * (p.cols / 256) > sm_count && sm_count >= 2) return launch_form<true>(p, rows[1], rows[3], sm_count / 2, s);
  return launch_form<false>(p, rows[0], rows[2], sm_count, s);
}

}  // namespace tt
