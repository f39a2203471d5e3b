// Preprocessing and first encoder layer of the bf16 path in one kernel: uint8 RGB frame -> bilinear resize ->
// normalise -> 3x3 convolution (3 -> 32 or 64 channels, pad 1, stride 1 or 2), bias, ReLU -> bf16 channels-last.
// The resized fp32 image is an observable tensor of the context and is still written (unless the caller does not
// want it), but nothing reads it back, and one launch with its start-up and drain is gone.
//
// Bound by the load/store pipe (at two full-HD frames 53 % of the active cycles, most of it through shared memory; 58 % of the issue
// slots), the chain of phases below, and by HBM (8 full-HD frames: 50 MB in, 88 + 236 MB out).  A block of 8 warps takes tiles of 32 x 8 outputs in
// turn, down a column of tiles, and every warp takes part in every phase, so the sampling has all the warps of
// the multiprocessor (three blocks, two at the largest resize factors) at its disposal and the phases of different blocks overlap:
//   stage    the 16-byte aligned byte range of every frame row under the tile's input patch, by bulk copies two
//            tiles ahead;
//   sample   the patch (with halo; zero outside the image = the convolution's padding): a lane per column, a warp per row,
//            positions from two tables, the expressions of the stand-alone kernel, so the fp32 values are the same
//            bits; written out as fp32 and kept as bf16, which is what the contraction takes;
//   gather   a thread per output pixel packs its 27 taps into one 64-byte row of the operand (no-swizzle core-matrix
//            layout, two tiles of 128 rows);
//   MMA      four tcgen05.mma M128 x COUT x K16, issued by one thread;
//   epilogue of the tile before, while the next patch is already being built: bias, ReLU, tile stores by the TMA unit.
// A specialised form (eight sampling warps feeding four gather warps through patch buffers) had been 6 us slower per tick than
// the two kernels at 5 streams of 854x480.  This one, alone under the profiler: 18.8 us against 10.1 + 14.4 us at that size, 9.8 against
// 7.2 + 9.2 us for one stream, 100 against 38 + 61 us for 8 full-HD streams, where only the second launch's gap is won.  All that with the
// output read back from shared memory and stored by the warps, and the resized image stored one column off its 128-byte lines; with tile
// stores and whole lines (both sides in one call): a tick of eight full-HD streams 1049 -> 1034 us, of one 168.4 -> 166.9, of five 854x480 streams
// 111.6 -> 110.7, of one 64.15 -> 63.9.  The biases are operands in the constant bank: from shared memory they took the load/store unit 512 of a tile's 1800 cycles at 64 channels
// (a 128-bit load four cycles, whether its lanes read one address or 32).  This launch in a tick, one, five 854x480 streams 7.44 -> 7.39, 17.0 -> 16.9 us, one, eight full-HD 15.35 -> 15.0,
// 84.8 -> 82.2.
#include <type_traits>

#include "tt_internal.h"
#include "tc_ptx.cuh"
#include "pre_math.cuh"

namespace tt {
namespace {

using namespace tc;
using namespace pre;

constexpr int FF_THREADS = 256, FF_WARPS = 8;
constexpr int FF_PER_SM = 3;                         // most blocks per multiprocessor; before the tile stores (80 registers) 8 full-HD frames took 97 us with three, 107 with four
constexpr int FF_TW = 32, FF_TH = 8;                 // output tile
constexpr int FF_SRC_BUDGET = 48 * 1024;             // shared memory the two buffers of frame rows may take

__host__ __device__ constexpr int ff_patch_w(int stride) { return (FF_TW - 1) * stride + 3; }
__host__ __device__ constexpr int ff_patch_h(int stride) { return (FF_TH - 1) * stride + 3; }
__host__ __device__ constexpr int ff_pitch(int stride) { return stride == 2 ? 68 : 36; }   // bf16 values per patch row

struct Tile {
  int img, tx, ty;
};

// OWN_OUT: output waits for its tile stores in shared memory of its own and not in the operand's.
template <int COUT, int STRIDE, bool OWN_OUT>
__global__ void __launch_bounds__(FF_THREADS, FF_PER_SM) conv_first_fused_kernel(const __grid_constant__ ConvFirstTcParams p) {
  constexpr int PW = ff_patch_w(STRIDE), PH = ff_patch_h(STRIDE), PITCH = ff_pitch(STRIDE);
  constexpr int FULL = PW / 32, EXTRA = PW - 32 * FULL;       // whole warps of patch columns, from the tile's first own column on, and the rest
  constexpr int GROUPS = FF_WARPS / FULL;                     // patch rows sampled at a time
  constexpr int A_BYTES = 2 * 128 * 64;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* s_a = smem;                                        // operand: two tiles of [128 rows][32] bf16
  uint8_t* s_out = s_a + A_BYTES;                             // OWN_OUT: per warp 32 pixels x 32 channels on their way out
  uint8_t* s_b = s_out + (OWN_OUT ? FF_WARPS * 2048 : 0);     // weights in operand layout
  __nv_bfloat16* s_patch = reinterpret_cast<__nv_bfloat16*>(s_b + COUT * 64);    // [3][PH][PITCH]
  uint8_t* s_src = reinterpret_cast<uint8_t*>(s_patch) + ((3 * PH * PITCH * 2 + 15) & ~15);   // [2][src_rows_cap][src_row_cap]
  // per buffer: of every patch row {offsets of its two frame rows in the buffer, bits of the lower one's weight, row of the
  // resized image or -1 outside it}, and the first staged byte column
  __shared__ __align__(16) int4 s_row[2][PH];
  __shared__ int s_b_lo[2];
  __shared__ __align__(8) uint64_t s_bar, s_landed[2];        // accumulator complete; a buffer's frame rows have landed
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  volatile int* abort_flag = &s_abort;

  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  // Before anything else: the next block of the multiprocessor does not start until this one has given up its permit to allocate
  // (allocating behind the first loads let four blocks start up to 4 us one after the other).
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"((uint32_t)(2 * COUT)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const int src_bytes = p.src_rows_cap * p.src_row_cap;
  const int t_begin = (int)blockIdx.x * p.tiles_per_block + min((int)blockIdx.x, p.tiles_left);
  const int n = p.tiles_per_block + ((int)blockIdx.x < p.tiles_left ? 1 : 0);
  // tiles in order of (image, tile column, tile row)
  auto advance = [&](Tile& t) {
    if (++t.ty == p.tiles_y) {
      t.ty = 0;
      if (++t.tx == p.tiles_x) { t.tx = 0; ++t.img; }
    }
  };

  // Byte b of a staged row is the frame's byte (aligned start of that row's range) + b.
  auto stage = [&](const Tile& t, int buf) {
    const uint8_t* frame = p.src_tab ? (const uint8_t*)__ldg((const unsigned long long*)p.src_tab + t.img) : p.src.p[t.img];
    const int x0 = t.tx * FF_TW * STRIDE - 1, y0 = t.ty * FF_TH * STRIDE - 1;
    const int b_lo = __ldg(&p.xtab[max(x0, 0)].x);
    const int span = min(__ldg(&p.xtab[min(x0 + PW - 1, p.W - 1)].x) + 3, 3 * (p.src_w - 1)) + 2 - b_lo;
    const int r_lo = __ldg(&p.ytab[max(y0, 0)].x);
    const int r_hi = min(__ldg(&p.ytab[min(y0 + PH - 1, p.H - 1)].x) + 1, p.src_h - 1);
    const int rows = min(r_hi - r_lo + 1, p.src_rows_cap);
    if (tid >= FF_THREADS - PH) {
      const int r = tid - (FF_THREADS - PH), y = y0 + r;
      int4 e = make_int4(0, 0, 0, -1);
      if (y >= 0 && y < p.H) {
        const int2 ye = __ldg(&p.ytab[y]);
        const int ya = ye.x, yb = min(ye.x + 1, p.src_h - 1);
        // low bits of the address of byte b_lo in source row 0: (that + row * pitch) & 15 is its position in the staged row
        const uint32_t base_lo = (uint32_t)(uintptr_t)frame + (uint32_t)b_lo;
        e = make_int4((ya - r_lo) * p.src_row_cap + (int)((base_lo + (uint32_t)(ya * p.src_pitch)) & 15u),
                      (yb - r_lo) * p.src_row_cap + (int)((base_lo + (uint32_t)(yb * p.src_pitch)) & 15u), ye.y, y);
      }
      s_row[buf][r] = e;
      if (r == 0) s_b_lo[buf] = b_lo;
    }
    // warp w copies rows w, w + 8, ...: one lane and one bulk copy each
    const uint32_t bar = smem_u32(&s_landed[buf]);
    for (int r = warp + FF_WARPS * lane; r < rows; r += FF_WARPS * 32) {
      const uintptr_t first = (uintptr_t)frame + (size_t)(r_lo + r) * p.src_pitch + b_lo;
      const int bytes = min((int)((((uint32_t)first & 15u) + span) & ~15u) + 16, p.src_row_cap);
      bulk_copy(smem_u32(s_src + buf * src_bytes) + r * p.src_row_cap, first & ~(uintptr_t)15, (uint32_t)bytes, bar);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
  };

  const size_t plane = (size_t)p.H * p.W;
  // ONE_ROW: every sample of the frame sits on one of its rows (an axis that is not resized, say), whose blend with the
  // next row is the row itself: it is not fetched.  Decided once for the kernel: a branch per pixel row made the compiler
  // evaluate both sides.
  auto sample = [&](const Tile& t, int buf, auto one_row) {
    constexpr bool ONE_ROW = decltype(one_row)::value;
    const uint32_t* rows = reinterpret_cast<const uint32_t*>(s_src + buf * src_bytes);
    const int b_lo = s_b_lo[buf], x0 = t.tx * FF_TW * STRIDE - 1;
    float* pre_img = p.pre_out + (size_t)(p.img0 + t.img) * 3 * plane;
    // the pixel of patch row e at byte offset xo of the staged rows -> patch entry q; `keep`: also to the resized image.
    // A column outside the image comes with scale and shift zero.
    auto pixel = [&](const int4& e, int xo, float fx, float scale, float shift, __nv_bfloat16* q, bool keep, int x) {
      uint32_t lo0, hi0;
      float o0, o1, o2;
      fetch_pair(rows, e.x + xo, lo0, hi0);
      if (ONE_ROW) {
        sample_row(lo0, hi0, fx, scale, shift, o0, o1, o2);
      } else {
        uint32_t lo1, hi1;
        fetch_pair(rows, e.y + xo, lo1, hi1);
        sample_rows(lo0, hi0, lo1, hi1, fx, __int_as_float(e.z), scale, shift, o0, o1, o2);
      }
      if (keep) {
        float* d = pre_img + (uint32_t)(e.w * p.W + x);
        d[0] = o0;
        d[plane] = o1;
        d[2 * plane] = o2;
      }
      q[0] = __float2bfloat16_rn(o0);
      q[PH * PITCH] = __float2bfloat16_rn(o1);
      q[2 * PH * PITCH] = __float2bfloat16_rn(o2);
    };
    auto zero = [&](__nv_bfloat16* q) { q[0] = q[PH * PITCH] = q[2 * PH * PITCH] = __float2bfloat16_rn(0.f); };
    {
      // the tile's own columns (patch columns 1 .. 32 FULL), so that the 128 bytes a warp stores of the resized image are one line
      const int j = 1 + (warp % FULL) * 32 + lane, x = x0 + j;
      const bool in_x = x < p.W;
      const int2 xe = __ldg(&p.xtab[min(x, p.W - 1)]);
      const int xo = in_x ? xe.x - b_lo : 0;
      const float scale = in_x ? p.scale : 0.f, shift = in_x ? p.shift : 0.f;
      const bool own = p.write_pre && in_x;
#pragma unroll
      for (int k = 0; k < (PH + GROUPS - 1) / GROUPS; ++k) {
        const int r = warp / FULL + k * GROUPS;
        if (r < PH) {
          const int4 e = s_row[buf][r];
          __nv_bfloat16* q = s_patch + r * PITCH + j;
          if (e.w >= 0) pixel(e, xo, __int_as_float(xe.y), scale, shift, q, own && r >= 1 && r <= FF_TH * STRIDE, x);
          else zero(q);
        }
      }
    }
    if (warp == FF_WARPS - 1 && lane < EXTRA * PH) {   // a warp with one row less than the first ones
      // halo columns: the one in front, at stride 1 also the one behind
      const int r = lane / EXTRA, j = lane % EXTRA ? 32 * FULL + 1 : 0, x = x0 + j;
      const int4 e = s_row[buf][r];
      __nv_bfloat16* q = s_patch + r * PITCH + j;
      if (x >= 0 && x < p.W && e.w >= 0) {
        const int2 xe = __ldg(&p.xtab[x]);
        pixel(e, xe.x - b_lo, __int_as_float(xe.y), p.scale, p.shift, q, false, x);
      } else {
        zero(q);
      }
    }
  };

  // thread = output pixel (tid / 32, tid % 32) of the tile = row tid of the operand's two tiles
  auto gather = [&]() {
    const int oy = tid >> 5, ox = tid & 31;
    uint32_t k[14];                                    // taps 2i, 2i + 1 as a pair; tap = channel * 9 + ky * 3 + kx
    const uint16_t* s = reinterpret_cast<const uint16_t*>(s_patch);
    if (STRIDE == 2) {
      const uint32_t* w = reinterpret_cast<const uint32_t*>(s_patch) + (2 * oy) * (PITCH / 2) + ox;
      uint32_t ab[9], c[9];                            // taps (0, 1) and (2, -) of every row of three
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const uint32_t* r = w + ((i / 3) * PH + i % 3) * (PITCH / 2);
        ab[i] = r[0];
        c[i] = r[1];
      }
#pragma unroll
      for (int i = 0; i < 9; i += 2) {                 // rows i, i + 1: taps 3i .. 3i + 5
        k[3 * i / 2] = ab[i];
        if (i + 1 < 9) {
          k[3 * i / 2 + 1] = __byte_perm(c[i], ab[i + 1], 0x5410);
          k[3 * i / 2 + 2] = __byte_perm(ab[i + 1], c[i + 1], 0x5432);
        } else {
          k[13] = c[i] & 0xFFFFu;
        }
      }
    } else {
#pragma unroll
      for (int i = 0; i < 14; ++i) {
        uint32_t v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int tap = 2 * i + h;
          v[h] = tap < 27 ? s[((tap / 9) * PH + oy + (tap % 9) / 3) * PITCH + ox + tap % 3] : 0u;
        }
        k[i] = v[0] | (v[1] << 16);
      }
    }
    uint8_t* dst = s_a + (tid >> 7) * 8192 + ((tid & 127) >> 3) * 512 + (tid & 7) * 16;
    *reinterpret_cast<uint4*>(dst) = make_uint4(k[0], k[1], k[2], k[3]);
    *reinterpret_cast<uint4*>(dst + 128) = make_uint4(k[4], k[5], k[6], k[7]);
    *reinterpret_cast<uint4*>(dst + 256) = make_uint4(k[8], k[9], k[10], k[11]);
    *reinterpret_cast<uint4*>(dst + 384) = make_uint4(k[12], k[13], 0u, 0u);
  };

  uint32_t tmem_base = 0;
  auto epilogue = [&](const Tile& t) {
    tc_fence_after();
    const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * COUT);
    const int y = t.ty * FF_TH + warp, x0 = t.tx * FF_TW;
    // 32 channels of the warp's row of 32 pixels leave as one tile store, which clips what lies outside the map.  They wait for it in 2 KB of
    // the warp's own (OWN_OUT), the first half of 64 channels in the part of the operand that the warp's own gather fills next; without memory of
    // their own all wait there, one half behind the other.  16-byte piece c of pixel i lies at piece c ^ (i / 2 % 4), the swizzle of the store's map.
#pragma unroll
    for (int ck = 0; ck < COUT / 32; ++ck) {
      uint8_t* mine = (OWN_OUT && ck + 1 == COUT / 32 ? s_out : s_a) + warp * 2048;
      uint32_t v[32];
      tmem_ld32(taddr + (uint32_t)(ck * 32), v);
      if (OWN_OUT ? ck == 0 : ck > 0) {   // the stores of the tile before (the half before) have been read
        if (lane == 0) bulk_wait_group_read0();
        __syncwarp();
      }
#pragma unroll
      for (int i = 0; i < 32; i += 8) {
        uint32_t u[4];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int c = i + 4 * q;
          const float* b = p.bias_v + ck * 32 + c;
          u[2 * q] = pack_relu_bf16(__uint_as_float(v[c]) + b[0], __uint_as_float(v[c + 1]) + b[1]);
          u[2 * q + 1] = pack_relu_bf16(__uint_as_float(v[c + 2]) + b[2], __uint_as_float(v[c + 3]) + b[3]);
        }
        *reinterpret_cast<uint4*>(mine + lane * 64 + (((i >> 3) ^ ((lane >> 1) & 3)) << 4)) = make_uint4(u[0], u[1], u[2], u[3]);
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        if (y < p.Ho) tma_store_4d(&p.map_rows, smem_u32(mine), ck * 32, x0, y, p.img0 + t.img);
        bulk_commit_group();
      }
    }
    if (COUT > 32 || !OWN_OUT) {          // the operand's part has been read
      if (lane == 0) {
        if (OWN_OUT) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        else bulk_wait_group_read0();
      }
      __syncwarp();
    }
  };

  Tile cur, ahead, last;
  {
    const int tiles_per_img = p.tiles_x * p.tiles_y;
    cur.img = t_begin / tiles_per_img;
    const int rem = t_begin - cur.img * tiles_per_img;
    cur.tx = rem / p.tiles_y;
    cur.ty = rem - cur.tx * p.tiles_y;
  }
  ahead = last = cur;
  if (tid == 0) {
    mbar_init(smem_u32(&s_bar), 1);
    mbar_init(smem_u32(&s_landed[0]), FF_WARPS);
    mbar_init(smem_u32(&s_landed[1]), FF_WARPS);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (i < n) { stage(ahead, i); advance(ahead); }
  // weights while the first rows are on their way
  for (int i = tid; i < COUT * 4; i += FF_THREADS) reinterpret_cast<uint4*>(s_b)[i] = __ldg(reinterpret_cast<const uint4*>(p.w_packed) + i);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  tmem_base = s_tmem;
  // only now: a dependent block that shares the multiprocessor must not get tensor memory that a block of this grid still has
  // to allocate
  pdl_launch_dependents();

  bool ok = true;
  for (int i = 0; i < n; ++i) {
    // this tile's rows have landed (the barrier at the end of the loop body: the patch has been gathered from)
    ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&s_landed[i & 1]), (uint32_t)(i >> 1) & 1u, abort_flag, p.status, WAIT_CONV_FIRST_FUSED + (i & 1), p.wait_limit));
    if (p.one_row) sample(cur, i & 1, std::true_type{});
    else sample(cur, i & 1, std::false_type{});
    __syncthreads();                                  // the patch is complete, the frame rows have been read
    if (i + 2 < n) { stage(ahead, i & 1); advance(ahead); }
    if (i > 0) {
      // the MMAs of the tile before are done: its accumulator can be read and the operand overwritten
      ok &= __all_sync(0xffffffffu, mbar_wait(smem_u32(&s_bar), (uint32_t)(i - 1) & 1u, abort_flag, p.status, WAIT_CONV_FIRST_FUSED + 0x10, p.wait_limit));
      epilogue(last);
    }
    gather();
    fence_proxy_async_smem();
    tc_fence_before();
    if (__syncthreads_or(!ok)) { ok = false; break; }
    if (tid == 0) {
      tc_fence_after();
      constexpr uint32_t IDESC = make_idesc(128, COUT);
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int k = 0; k < 2; ++k)
          umma_bf16(tmem_base + (uint32_t)(m * COUT), make_smem_desc_lbo(smem_u32(s_a) + m * 8192 + k * 256, 128, 512, 0),
                    make_smem_desc_lbo(smem_u32(s_b) + k * 256, 128, 512, 0), IDESC, k);
      umma_commit(smem_u32(&s_bar));
    }
    last = cur;
    advance(cur);
  }
  if (ok && n > 0) {
    ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&s_bar), (uint32_t)(n - 1) & 1u, abort_flag, p.status, WAIT_CONV_FIRST_FUSED + 0x11, p.wait_limit));
    if (ok) epilogue(last);
  }
  if (lane == 0) bulk_wait_group0();
  __syncwarp();
  if (*abort_flag) {
    for (int i = 0; i < 64; ++i) __nanosleep(16000);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)(2 * COUT)) : "memory");
  }
}

// Dynamic shared memory of a block whose two buffers of frame rows take src_bytes.
template <int COUT, int STRIDE, bool OWN_OUT>
constexpr int ff_smem(int src_bytes) {
  return 2 * 128 * 64 + (OWN_OUT ? FF_WARPS * 2048 : 0) + COUT * 64 + ((3 * ff_patch_h(STRIDE) * ff_pitch(STRIDE) * 2 + 15) & ~15) + src_bytes;
}

// Blocks of a form that a multiprocessor holds, by shared memory: a block takes 1 KB beside its own, and its static variables' up to the
// alignment of the dynamic part.
template <int COUT, int STRIDE, bool OWN_OUT>
constexpr int ff_per_sm(int src_bytes) {
  constexpr int SMEM_SM = 228 * 1024, BESIDE = 1024 + 1024;
  const int n = SMEM_SM / (ff_smem<COUT, STRIDE, OWN_OUT>(src_bytes) + BESIDE);
  return n < FF_PER_SM ? n : FF_PER_SM;
}

template <int COUT, int STRIDE, bool OWN_OUT>
cudaError_t launch_form(const ConvFirstTcParams& p, int src_bytes, int sm_count, cudaStream_t s) {
  auto kern = conv_first_fused_kernel<COUT, STRIDE, OWN_OUT>;
  // the most the form ever takes: the same value whichever context launches
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ff_smem<COUT, STRIDE, OWN_OUT>(FF_SRC_BUDGET));
  if (e != cudaSuccess) return e;
  ConvFirstTcParams q = p;
  q.tiles_x = (p.Wo + FF_TW - 1) / FF_TW;
  q.tiles_y = (p.Ho + FF_TH - 1) / FF_TH;
  const int total = p.K * q.tiles_x * q.tiles_y, slots = ff_per_sm<COUT, STRIDE, OWN_OUT>(src_bytes) * sm_count, grid = total < slots ? total : slots;
  q.tiles_per_block = total / grid;
  q.tiles_left = total % grid;
  return launch_kernel(kern, grid, FF_THREADS, (size_t)ff_smem<COUT, STRIDE, OWN_OUT>(src_bytes), s, q, false);
}

// The frame rows under a patch grow with the resize factor: the output has memory of its own where that costs no block.  Full-HD frames, this layer, one
// more and heads, five / eight streams, us a tick, two blocks with and three without such memory: to 960x540 with 64 channels 116 / 161 and 101 / 135, to
// 856x480 with 32 channels 92 / 117 and 80 / 100.  Where two fit either way (to 768x432, 64 channels) a grid cut for three took 120, cut for two 107.5.
template <int COUT, int STRIDE>
cudaError_t launch_t(const ConvFirstTcParams& p, int sm_count, cudaStream_t s) {
  const int src_bytes = 2 * p.src_rows_cap * p.src_row_cap;
  static_assert(ff_per_sm<COUT, STRIDE, true>(FF_SRC_BUDGET) >= 1, "any staging leaves room for a block");
  if (ff_per_sm<COUT, STRIDE, true>(src_bytes) >= ff_per_sm<COUT, STRIDE, false>(src_bytes)) return launch_form<COUT, STRIDE, true>(p, src_bytes, sm_count, s);
  return launch_form<COUT, STRIDE, false>(p, src_bytes, sm_count, s);
}

}  // namespace

bool conv_first_fused_staging(int stride, int src_w, int src_h, int net_w, int net_h, int* rows_cap, int* row_cap) {
  // Worst-case footprint of a patch: rows = ceil(PH * sh/nh) + 2; bytes per row = 3 * (ceil(PW * sw/nw) + 2) + 15 (alignment
  // at the front) + 15 (at the end) + 12 (the tap fetch reads three whole words from its first byte), rounded up to 16.
  const long ph = ff_patch_h(stride), pw = ff_patch_w(stride);
  const long rows = (ph * src_h + net_h - 1) / net_h + 2, cols = (pw * src_w + net_w - 1) / net_w + 2;
  const long cap = ((3 * cols + 48 + 15) / 16) * 16;
  if (2 * rows * cap > FF_SRC_BUDGET) return false;
  *rows_cap = (int)rows;
  *row_cap = (int)cap;
  return true;
}

cudaError_t launch_conv_first_fused(const ConvFirstTcParams& p, int sm_count, cudaStream_t s) {
  if (p.cout == 32 && p.stride == 1) return launch_t<32, 1>(p, sm_count, s);
  if (p.cout == 32 && p.stride == 2) return launch_t<32, 2>(p, sm_count, s);
  if (p.cout == 64 && p.stride == 1) return launch_t<64, 1>(p, sm_count, s);
  if (p.cout == 64 && p.stride == 2) return launch_t<64, 2>(p, sm_count, s);
  return cudaErrorInvalidValue;
}

}  // namespace tt
