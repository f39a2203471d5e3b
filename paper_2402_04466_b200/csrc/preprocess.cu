// S1: uint8 RGB interleaved frame -> bilinear resize -> normalise -> planar fp32.
//
// A block works down a column of tiles of TILE_W output columns and `tile_rows` rows.  A ninth warp works out where the tiles lie and has the frame rows under a tile
// staged as a byte stream (row pitch 3*W is in general not a multiple of 16) by one bulk copy a row of the aligned range that covers it, a tile ahead; per-thread copies and
// every warp's index arithmetic had been a third of the instructions.  A sampling thread keeps two output columns 32 apart and goes down a run of rows: the two are one
// packed fp32 instruction each step, neighbouring lanes read neighbouring bytes of a staged row (few bank conflicts), a warp's stores are 256 contiguous bytes, and a frame row
// that the row above has already blended horizontally is not fetched again.  A bilinear tap pair (two neighbouring RGB pixels = 6 bytes) is three 32-bit shared loads plus
// funnel shifts; bytes become floats by a byte permute into the mantissa of 2^23.
// Bound by issue and by the start: every block's first tile comes before anything can be sampled (four full-HD frames: launch 2, first rows 3, two tiles 9 us).  Instructions per
// pixel of three channels 117 -> 82, 78 -> 69 % of the issue slots.  Device time, us, of frames in L2, with a column a thread and every thread's own copies / now: four full-HD frames to
// 1280x720 17.6 / 14.4, eight 32.9 / 27.8, one 6.1 / 5.7, eight to 768x432 19.6 / 15.8, four 1280x960 to 640x480 9.2 / 8.2, two 960x540 to 1280x720 9.3 / 8.3 (launches of 2.5 to 3.5 us, one
// tile a block, up to 0.15 longer, for a bulk copy arrives later than a thread's own: three 428x240 to 320x240 3.30 / 3.36); a call among others, frames from memory, in the same order:
// 18.5 / 16.4, 34.8 / 29.1, 8.2 / 8.2, 20.5 / 17.9, 10.3 / 10.3, 10.3 / 10.3 (4.2 / 4.2).
// Not kept: per-thread asynchronous copies by the ninth warp (25 us), three and four tiles in flight of 8 to 16 rows (16.6 to 18.8), five or six blocks with smaller tiles.
#include "tt_internal.h"
#include "pre_math.cuh"
#include "tc_ptx.cuh"

namespace tt {
namespace {

using namespace pre;
using tc::pack2;
using tc::unpack2;
typedef unsigned long long f32x2;   // two fp32 values
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

constexpr int PRE_SAMPLERS = 256, PRE_THREADS = PRE_SAMPLERS + 32, PRE_WARPS = PRE_THREADS / 32, PRE_PER_SM = 4;
constexpr int PRE_MAX_ROWS = 32;             // output rows of a tile
constexpr int PRE_STAGE_BYTES = 26 * 1024;   // staged rows of a tile; two tiles of four blocks fit a multiprocessor
constexpr long long PRE_LAND_CYCLES = 2000000;   // how long a block that has given up a wait stays for copies in flight: about a millisecond
constexpr int PRE_STATIC_BYTES = 2 * (PRE_MAX_ROWS * 16 + 64) + 16;   // the kernel's tables and barriers

struct PreprocessArgs {
  PreprocessParams p;
  int32_t tile_rows, tiles_x, tiles_y;
  int32_t rows_cap, row_cap;                 // staged rows of a tile, bytes of one (a multiple of 16)
  int32_t expire_from = 0x7fffffff;          // the first tile of a block whose wait gives up at once (tests)
  int32_t tiles_per_block, tiles_left;       // the first tiles_left blocks take one tile more
};
static_assert(whole_arguments<PreprocessArgs> && whole_arguments<PreprocessParams>, "kernel arguments");
// What the sampling warps are told of a tile.
struct alignas(16) TileInfo {
  int32_t img, y0, rows, tx;
  int32_t left;              // first frame column
};

// Where a tile lies: image, tile column, first output row and their number, frame, first frame column, last byte of a staged row counted from its first, first frame
// row and their number; sy: of the lane's output row.
struct Place {
  int img, tx, y0, rows;
  const uint8_t* src;
  int left, span, first, src_rows;
  AxisSample sy;
};
// as `count` arrivals at once
__device__ __forceinline__ void mbar_arrive_n(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

// Three channels of a frame row between two of its pixels, for a thread's two columns.  The loads are volatile: a row that is at hand already is not
// fetched all the same.
struct Blend {
  f32x2 r, g, b;
};
struct Taps {
  uint32_t lo, hi;   // bytes R0 G0 B0 R1, G1 B1 . .
};
__device__ __forceinline__ Taps fetch_taps(uint32_t addr) {
  uint32_t w0, w1, w2;
  const uint32_t word = addr & ~3u, sh = addr << 3;   // a funnel shift takes its shift modulo 32
  asm volatile("ld.shared.u32 %0, [%3];\n\tld.shared.u32 %1, [%3+4];\n\tld.shared.u32 %2, [%3+8];" : "=r"(w0), "=r"(w1), "=r"(w2) : "r"(word));
  return {__funnelshift_r(w0, w1, sh), __funnelshift_r(w1, w2, sh)};
}
__device__ __forceinline__ f32x2 magic2(uint32_t a, uint32_t b, uint32_t selector) { return pack2(byte_to_magic(a, selector), byte_to_magic(b, selector)); }
__device__ __forceinline__ Blend blend_row(uint32_t addr_a, uint32_t addr_b, f32x2 fx) {
  const Taps a = fetch_taps(addr_a), b = fetch_taps(addr_b);
  const f32x2 magic = pack2(8388608.0f, 8388608.0f);
  const f32x2 l0 = magic2(a.lo, b.lo, 0x7440), l1 = magic2(a.lo, b.lo, 0x7441), l2 = magic2(a.lo, b.lo, 0x7442);
  return {fma2(fx, sub2(magic2(a.lo, b.lo, 0x7443), l0), sub2(l0, magic)), fma2(fx, sub2(magic2(a.hi, b.hi, 0x7440), l1), sub2(l1, magic)),
          fma2(fx, sub2(magic2(a.hi, b.hi, 0x7441), l2), sub2(l2, magic))};
}

// One output pixel from taps straight in memory, with the frame's rows r0 and r1: the same bits as from staged rows.
__device__ __forceinline__ void direct_pixel(const PreprocessParams& p, const uint8_t* __restrict__ r0, const uint8_t* __restrict__ r1, float fy, float* dst, size_t plane, int x) {
  const AxisSample sx = axis_sample(x, p.src_w, p.net_w);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float p00 = (float)__ldg(r0 + 3 * sx.i0 + c), p01 = (float)__ldg(r0 + 3 * sx.i1 + c);
    const float p10 = (float)__ldg(r1 + 3 * sx.i0 + c), p11 = (float)__ldg(r1 + 3 * sx.i1 + c);
    const float top = p00 + sx.f * (p01 - p00);
    const float bot = p10 + sx.f * (p11 - p10);
    dst[c * plane] = fmaf(top + fy * (bot - top), p.scale, p.shift);
  }
}

// A block's tiles from the i-th on, by one warp and without staging: where a wait for frame rows has run out.  In the copying warp, for the sampling warps' code is as fast
// as without it only there (four full-HD frames 14.6 us; with the call behind their loop 15.3).
template <int TILE_W>
__device__ __noinline__ void sample_unstaged(const PreprocessArgs& a, int t_begin, int i, int n) {
  const PreprocessParams& p = a.p;
  const size_t plane = (size_t)p.net_h * p.net_w;
  for (; i < n; ++i) {
    const int col_tiles = (t_begin + i) / a.tiles_y, img = col_tiles / a.tiles_x, x0 = (col_tiles - img * a.tiles_x) * TILE_W;
    const int y0 = (t_begin + i - col_tiles * a.tiles_y) * a.tile_rows, rows = min(a.tile_rows, p.net_h - y0), cols = min(TILE_W, p.net_w - x0);
    const uint8_t* src = p.src_tab ? p.src_tab[img] : p.src.p[img];
    for (int k = threadIdx.x & 31; k < rows * cols; k += 32) {
      const int y = y0 + k / cols, x = x0 + k % cols;
      const AxisSample sy = axis_sample(y, p.src_h, p.net_h);
      direct_pixel(p, src + (size_t)sy.i0 * p.src_pitch, src + (size_t)sy.i1 * p.src_pitch, sy.f, p.dst + (size_t)img * 3 * plane + (size_t)y * p.net_w + x, plane, x);
    }
  }
}

// ONE_ROW: the height is not resized, so every sample sits on a source row (weight zero for the next one).
template <int TILE_W, bool ONE_ROW>
__global__ void __launch_bounds__(PRE_THREADS, PRE_PER_SM) preprocess_staged_kernel(const __grid_constant__ PreprocessArgs a) {
  constexpr int COLS = TILE_W / 2;                   // threads to a row; a thread's two columns are 32 apart
  constexpr int GROUPS = PRE_SAMPLERS / COLS;        // runs of rows sampled at a time
  extern __shared__ __align__(16) uint8_t s_mem[];   // [2][rows_cap][row_cap]
  __shared__ TileInfo s_tile[2];
  __shared__ __align__(16) int4 s_row[2][PRE_MAX_ROWS];   // per tile row: byte offsets of its two source rows in the buffer, bits of the lower one's weight, whether the upper one is the row above's lower one
  __shared__ __align__(8) uint64_t s_full[2];             // a buffer's frame rows have landed
  // the next kernel of the stream, if it was launched as a programmatic dependent, may start its set-up now;
  // it waits for this grid to finish before it reads the output
  pdl_launch_dependents();
  const PreprocessParams& p = a.p;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int buf_bytes = a.rows_cap * a.row_cap;
  const int t_begin = (int)blockIdx.x * a.tiles_per_block + min((int)blockIdx.x, a.tiles_left);
  const int n = a.tiles_per_block + ((int)blockIdx.x < a.tiles_left ? 1 : 0);
  if (tid == 0) {
    tc::mbar_init(tc::smem_u32(&s_full[0]), PRE_WARPS);
    tc::mbar_init(tc::smem_u32(&s_full[1]), PRE_WARPS);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }

  // Worked out by a whole warp, a lane per row: the i-th tile's place (tiles in order of image, tile column, tile row) ...
  auto place_of = [&](int i) {
    Place t;
    const int tile = t_begin + i, col_tiles = tile / a.tiles_y;
    t.img = col_tiles / a.tiles_x;
    t.tx = col_tiles - t.img * a.tiles_x;
    t.y0 = (tile - col_tiles * a.tiles_y) * a.tile_rows;
    t.rows = min(a.tile_rows, p.net_h - t.y0);
    t.src = p.src_tab ? p.src_tab[t.img] : p.src.p[t.img];
    const AxisSample sx = axis_sample(lane == 0 ? t.tx * TILE_W : min((t.tx + 1) * TILE_W, p.net_w) - 1, p.src_w, p.net_w);
    t.left = __shfl_sync(0xffffffffu, sx.i0, 0);
    t.span = 3 * (__shfl_sync(0xffffffffu, sx.i1, 1) - t.left) + 2;
    t.sy = axis_sample(t.y0 + min(lane, t.rows - 1), p.src_h, p.net_h);
    t.first = __shfl_sync(0xffffffffu, t.sy.i0, 0);
    t.src_rows = __shfl_sync(0xffffffffu, t.sy.i1, t.rows - 1) - t.first + 1;
    return t;
  };
  // ... copies of its frame rows r, r + step, ...: byte b of a staged row is the frame's byte (aligned start of that row's range) + b ...
  auto copy_rows = [&](const Place& t, int buf, int r, int step) {
    const uint32_t bar = tc::smem_u32(&s_full[buf]), dst = tc::smem_u32(s_mem) + (uint32_t)(buf * buf_bytes);
    for (; r < t.src_rows; r += step) {
      const uintptr_t g = (uintptr_t)t.src + (size_t)(t.first + r) * p.src_pitch + 3 * t.left;
      tc::bulk_copy(dst + (uint32_t)(r * a.row_cap), g & ~(uintptr_t)15, ((((uint32_t)g & 15u) + t.span) & ~15u) + 16u, bar);
    }
    __syncwarp();
  };
  // ... and what the sampling warps are told of it.
  auto tell = [&](const Place& t, int buf) {
    const int above = __shfl_up_sync(0xffffffffu, t.sy.i1, 1);
    // low bits of the address of the tile's first column in source row 0: (that + row * pitch) & 15 is its position in the staged row
    const uint32_t base_lo = (uint32_t)(uintptr_t)t.src + 3u * (uint32_t)t.left;
    if (lane < a.tile_rows)
      s_row[buf][lane] = make_int4((t.sy.i0 - t.first) * a.row_cap + (int)((base_lo + (uint32_t)(t.sy.i0 * p.src_pitch)) & 15u),
                                   (t.sy.i1 - t.first) * a.row_cap + (int)((base_lo + (uint32_t)(t.sy.i1 * p.src_pitch)) & 15u), __float_as_int(t.sy.f), above == t.sy.i0);
    if (lane == 0) s_tile[buf] = {t.img, t.y0, t.rows, t.tx, t.left};
  };

  // A warp issues its copies one behind the other: those of the first tile, which everything waits for, are shared out.  Its place
  // is worked out while the barriers are set up (three 428x240 to 320x240 3.44 -> 3.36 us, four full-HD frames 14.57 -> 14.45).
  const Place first = place_of(0);
  __syncthreads();
  copy_rows(first, 0, warp + PRE_WARPS * lane, PRE_WARPS * 32);
  if (lane == 0) tc::mbar_arrive(tc::smem_u32(&s_full[0]));

  if (warp == PRE_WARPS - 1) {
    // ------------------------------------------------------------------------ frame rows
    tell(first, 0);
    __syncthreads();
    for (int i = 1; i <= n; ++i) {
      if (i < n) {
        const Place t = place_of(i);
        copy_rows(t, i & 1, lane, 32);
        if (lane == 0) mbar_arrive_n(tc::smem_u32(&s_full[i & 1]), PRE_WARPS);
        tell(t, i & 1);
      }
      if (__syncthreads_or(0)) {                       // tile i - 1 has been sampled; or a wait has run out: what is in flight may still land, then the rest by this warp
        tc::mbar_wait_limit(tc::smem_u32(&s_full[(i - 1) & 1]), (uint32_t)((i - 1) >> 1) & 1u, PRE_LAND_CYCLES);
        if (i < n) tc::mbar_wait_limit(tc::smem_u32(&s_full[i & 1]), (uint32_t)(i >> 1) & 1u, PRE_LAND_CYCLES);
        sample_unstaged<TILE_W>(a, t_begin, i - 1, n);
        break;
      }
    }
    return;
  }

  // -------------------------------------------------------------------------- samples
  const int col = tid % COLS, grp = tid / COLS;
  const uint32_t plane = (uint32_t)(p.net_h * p.net_w);
  const f32x2 scale = pack2(p.scale, p.scale), shift = pack2(p.shift, p.shift);
  int tx, x, xo_a, xo_b;
  f32x2 fx;
  auto column = [&](int tile_x, int left) {
    tx = tile_x;
    x = tx * TILE_W + 2 * (col & ~31) + (col & 31);
    const AxisSample sa = axis_sample(min(x, p.net_w - 1), p.src_w, p.net_w), sb = axis_sample(min(x + 32, p.net_w - 1), p.src_w, p.net_w);
    xo_a = 3 * (sa.i0 - left);
    xo_b = 3 * (sb.i0 - left);
    fx = pack2(sa.f, sb.f);
  };
  column(first.tx, first.left);                                    // while the first rows are on their way
  __syncthreads();                                     // the first tile has been told of
  for (int i = 0; i < n; ++i) {
    const TileInfo& t = s_tile[i & 1];
    const int img = __shfl_sync(0xffffffffu, t.img, 0), rows = __shfl_sync(0xffffffffu, t.rows, 0);
    if (t.tx != tx) column(t.tx, t.left);
    const bool ok = i < a.expire_from && tc::mbar_wait_limit(tc::smem_u32(&s_full[i & 1]), (uint32_t)(i >> 1) & 1u, p.wait_limit);
    if (ok && x < p.net_w) {
      const uint32_t buf = tc::smem_u32(s_mem) + (uint32_t)((i & 1) * buf_bytes), buf_a = buf + (uint32_t)xo_a, buf_b = buf + (uint32_t)xo_b;
      const bool two = x + 32 < p.net_w;
      float* out = p.dst + (size_t)img * 3 * plane;
      const int share = (rows + GROUPS - 1) / GROUPS, r_begin = grp * share, r_end = min(r_begin + share, rows);
      const int4* e_tab = s_row[i & 1];
      uint32_t o = (uint32_t)((t.y0 + r_begin) * p.net_w + x);
      Blend bot{};
#pragma unroll 1
      for (int r = r_begin; r < r_end; ++r, o += (uint32_t)p.net_w) {
        const int4 e = e_tab[r];
        Blend top = bot;
        if (ONE_ROW || e.w == 0 || r == r_begin) top = blend_row(buf_a + e.x, buf_b + e.x, fx);
        if (!ONE_ROW) {
          bot = blend_row(buf_a + e.y, buf_b + e.y, fx);
          const float f = __int_as_float(e.z);
          const f32x2 fy = pack2(f, f);
          top.r = fma2(fy, sub2(bot.r, top.r), top.r);
          top.g = fma2(fy, sub2(bot.g, top.g), top.g);
          top.b = fma2(fy, sub2(bot.b, top.b), top.b);
        }
        float v[3][2];
        unpack2(fma2(top.r, scale, shift), v[0][0], v[0][1]);
        unpack2(fma2(top.g, scale, shift), v[1][0], v[1][1]);
        unpack2(fma2(top.b, scale, shift), v[2][0], v[2][1]);
        // streaming stores: the image is written once (four 1134x907 frames to 1103x1103, whose rows do not fill whole sectors, 20.3 -> 19.7 us, four full-HD ones to
        // 1280x720 14.9 -> 14.4, eight 27.6 -> 27.8)
        float* d = out + o;
        __stcs(d, v[0][0]);
        __stcs(d + plane, v[1][0]);
        __stcs(d + 2 * (size_t)plane, v[2][0]);
        if (two) {
          __stcs(d + 32, v[0][1]);
          __stcs(d + plane + 32, v[1][1]);
          __stcs(d + 2 * (size_t)plane + 32, v[2][1]);
        }
      }
    }
    if (!ok && p.status) atomicCAS(p.status, 0, tc::WAIT_PREPROCESS + (i & 1));
    if (__syncthreads_or(!ok)) break;                  // the buffer has been read
  }
}

constexpr int DIR_TX = 32, DIR_TY = 8, DIR_OUT_W = DIR_TX * 4;   // threads of a block, 4 outputs each

// Fallback for extreme down-scaling factors whose footprint does not fit in shared memory:
// taps are read straight from global memory (L1-cached byte loads).
__global__ void __launch_bounds__(DIR_TX * DIR_TY) preprocess_direct_kernel(const __grid_constant__ PreprocessParams p) {
  const int n = blockIdx.z;
  const uint8_t* __restrict__ src = p.src_tab ? p.src_tab[n] : p.src.p[n];
  const int yo = blockIdx.y * DIR_TY + threadIdx.y;
  const int xo0 = blockIdx.x * DIR_OUT_W + threadIdx.x * 4;
  if (yo >= p.net_h || xo0 >= p.net_w) return;
  const AxisSample sy = axis_sample(yo, p.src_h, p.net_h);
  const uint8_t* r0 = src + (size_t)sy.i0 * p.src_pitch;
  const uint8_t* r1 = src + (size_t)sy.i1 * p.src_pitch;
  const size_t plane = (size_t)p.net_h * p.net_w;
  float* dst = p.dst + (size_t)n * 3 * plane + (size_t)yo * p.net_w + xo0;
  for (int j = 0; j < 4 && xo0 + j < p.net_w; ++j) direct_pixel(p, r0, r1, sy.f, dst + j, plane, xo0 + j);
}

// Staged rows and bytes per row of a tile in the worst case: rows = ceil(tile_rows * sh/nh) + 2; bytes = 3 * (ceil(cols * sw/nw) + 2) + 15
// (alignment at the front) + 15 (at the end) + 12 (the tap fetch reads three whole words from its first byte), rounded up to 16.
void staging(const PreprocessParams& p, int cols, int tile_rows, long* rows, long* row_cap) {
  *rows = ((long)tile_rows * p.src_h + p.net_h - 1) / p.net_h + 2;
  const long c = ((long)cols * p.src_w + p.net_w - 1) / p.net_w + 2;
  *row_cap = ((3 * c + 48 + 15) / 16) * 16;
}

template <int TILE_W>
cudaError_t launch_staged(const PreprocessParams& p, cudaStream_t s, bool* fits) {
  constexpr int STEP = 256 / TILE_W;
  int sms = 0;
  cudaError_t e = post_sm_count(&sms);
  if (e != cudaSuccess) return e;
  PreprocessArgs a;
  a.p = p;
  a.p.wait_limit = p.wait_limit > 0 ? p.wait_limit : tc::WAIT_LIMIT_CYCLES;
  if (p.wait_limit < 0) a.expire_from = (int)~p.wait_limit;
  a.tiles_x = (p.net_w + TILE_W - 1) / TILE_W;
  // Rows per tile: the busiest block's tiles x (rows to sample, and about two rows' worth for its halo and barriers) is least, and the higher tile of
  // two that come out alike; another height where by it the busiest multiprocessor has at least a tenth less to do, a tile's latency counted as twelve
  // rows.  Device time of frames in L2, us, by rows: four 1280x960 to 640x480 6 10.1, 8 9.0, 10 9.3, 12 8.1, 14 8.2*; four 1920x1080 to 1280x720 16 15.1, 20 14.7,
  // 24 14.3, 26 14.4*; one 320x240 to 1280x960 18 7.5, 22 6.8*, 24 7.0, 28 7.4; heights that leave a run of rows idle are no worse for it, one 640x360 to 427x241 8 3.44,
  // 12 3.18*, 16 3.25 (* chosen).  Of 31 sizes and batches 29 are within 1.5 % of their best height; five 854x480 to 640x480 and three 1280x720 to 700x390 are 8 % from it (one tile a
  // block of 30 and 32 rows 6.25, 22* and 24* 6.7).
  const long slots = (long)PRE_PER_SM * sms;
  struct Height {
    int rows = 0;
    long cap_r = 0, cap_b = 0, tiles = 0, busiest_sm = 0, cost = 0;
  } by_round, by_sm, tallest;
  for (int rows = STEP; rows <= PRE_MAX_ROWS; rows += STEP) {
    Height h;
    h.rows = rows;
    staging(p, TILE_W, rows, &h.cap_r, &h.cap_b);
    if (h.cap_r * h.cap_b > PRE_STAGE_BYTES) break;
    h.tiles = (long)p.K * a.tiles_x * ((p.net_h + rows - 1) / rows);
    h.busiest_sm = (h.tiles / slots * PRE_PER_SM + (h.tiles % slots + sms - 1) / sms) * (rows + 12);
    h.cost = (h.tiles + slots - 1) / slots * (rows + 2);
    if (!by_round.rows || h.cost <= by_round.cost) by_round = h;
    if (!by_sm.rows || h.busiest_sm <= by_sm.busiest_sm) by_sm = h;
    tallest = h;
  }
  // A tile of few rows is mostly halo and latency (resize factors from about three on): taps straight from memory where two rows are the most that fit, and of four beyond three
  // rounds.  Staged / direct, us, one, four and eight frames: 1920x1080 to 480x270 (2 rows) 4.6 / 3.8, 8.3 / 8.4, 11.8 / 13.9; to 608x342 (4) 4.4 / 4.6, 8.9 / 10.0,
  // 13.6 / 17.1; to 640x360 (6) 5.2 / 4.8, 9.0 / 10.7, 13.5 / 17.5; 1280x720 to 320x180 (4, narrow) 3.2 / 3.7, 5.6 / 5.0, 7.6 / 7.8.
  *fits = tallest.rows >= 6 && tallest.rows >= 2 * STEP;
  if (!*fits) *fits = tallest.rows >= 4 && tallest.tiles <= 3 * slots;
  if (!*fits) return cudaSuccess;
  const Height& h = 10 * by_sm.busiest_sm < 9 * by_round.busiest_sm ? by_sm : by_round;
  a.tile_rows = h.rows;
  a.rows_cap = (int)h.cap_r;
  a.row_cap = (int)h.cap_b;
  a.tiles_y = (p.net_h + a.tile_rows - 1) / a.tile_rows;
  const long total = (long)p.K * a.tiles_x * a.tiles_y;
  const int grid = (int)(total < slots ? total : slots);
  a.tiles_per_block = (int)(total / grid);
  a.tiles_left = (int)(total % grid);
  const size_t smem = (size_t)2 * a.rows_cap * a.row_cap;
  auto kern = p.src_h == p.net_h ? preprocess_staged_kernel<TILE_W, true> : preprocess_staged_kernel<TILE_W, false>;
  if (smem + PRE_STATIC_BYTES > 48 * 1024) {   // what a kernel may have of both without asking
    static OncePerContext once;
    e = once([]() {
      const cudaError_t r = cudaFuncSetAttribute(preprocess_staged_kernel<TILE_W, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * PRE_STAGE_BYTES);
      return r != cudaSuccess ? r : cudaFuncSetAttribute(preprocess_staged_kernel<TILE_W, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * PRE_STAGE_BYTES);
    });
    if (e != cudaSuccess) return e;
  }
  kern<<<grid, PRE_THREADS, smem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_preprocess(const PreprocessParams& p, cudaStream_t s) {
  bool fits = false;
  // narrow tiles where the last wide one would be at most half full
  const int over = p.net_w % 128;
  cudaError_t e = over > 0 && over <= 64 ? launch_staged<64>(p, s, &fits) : launch_staged<128>(p, s, &fits);
  if (e != cudaSuccess || fits) return e;
  dim3 grid((p.net_w + DIR_OUT_W - 1) / DIR_OUT_W, (p.net_h + DIR_TY - 1) / DIR_TY, p.K);
  preprocess_direct_kernel<<<grid, dim3(DIR_TX, DIR_TY), 0, s>>>(p);
  return cudaGetLastError();
}

}  // namespace tt
