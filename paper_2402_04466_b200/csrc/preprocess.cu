// S1: uint8 RGB interleaved frame -> bilinear resize -> normalise -> planar fp32.
//
// Bound by instruction issue (78 % of the slots at four full-HD frames, about 117 instructions per pixel of three channels) and by HBM.  A block
// works down a column of tiles of COLS output columns and `tile_rows` rows.  A thread keeps one output column, so the horizontal
// sample position stays in its registers, neighbouring lanes read neighbouring bytes of a staged row (few bank conflicts; with
// four neighbouring outputs per thread every fetch took four to five passes), and a warp's store is 128 contiguous bytes.
// The frame rows under a tile are staged as a byte stream (row pitch 3*W is in general not a multiple of 16) by asynchronous 16-byte
// copies of the aligned range that covers them, while the tile before is sampled.  A bilinear tap pair (two neighbouring RGB pixels = 6
// bytes) is fetched as three 32-bit shared loads plus funnel shifts; bytes become floats by a byte permute into the mantissa of 2^23.
// Four full-HD frames to 1280x720: 24.4 -> 18.45 us a call against a block per 128 x 16 tile (2.8 -> 3.75 TB/s); eight, alone under the profiler: 37.6 -> 34.1.
#include "tt_internal.h"
#include "pre_math.cuh"

namespace tt {
namespace {

using namespace pre;

constexpr int PRE_THREADS = 256, PRE_PER_SM = 4;   // four full-HD frames: 20.5, 18.4, 18.5, 20.5, 22.5, 24.6 us with 2, 3, 4, 5, 6, 8 blocks
constexpr int PRE_MAX_ROWS = 32;             // output rows of a tile
constexpr int PRE_STAGE_BYTES = 26 * 1024;   // staged rows of a tile; two tiles of four blocks fit a multiprocessor
constexpr int PRE_STATIC_BYTES = 2 * PRE_MAX_ROWS * 16;   // the kernel's row tables

struct PreprocessArgs {
  PreprocessParams p;
  float scale, shift;
  int32_t tile_rows, tiles_x, tiles_y;
  int32_t rows_cap, row_cap;                 // staged rows of a tile, bytes of one (a multiple of 16)
  int32_t tiles_per_block, tiles_left;       // the first tiles_left blocks take one tile more
};

struct Tile {
  int img, tx, ty;
};

// ONE_ROW: the height is not resized, so every sample sits on a source row (weight zero for the next one).
template <int COLS, bool ONE_ROW>
__global__ void __launch_bounds__(PRE_THREADS, PRE_PER_SM) preprocess_staged_kernel(const __grid_constant__ PreprocessArgs a) {
  constexpr int GROUPS = PRE_THREADS / COLS;         // rows sampled at a time
  extern __shared__ __align__(16) uint8_t s_mem[];   // [2][rows_cap][row_cap]
  __shared__ __align__(16) int4 s_row[2][PRE_MAX_ROWS];   // per tile row: byte offsets of its two source rows in the buffer, bits of the lower one's weight
  // the next kernel of the stream, if it was launched as a programmatic dependent, may start its set-up now;
  // it waits for this grid to finish before it reads the output
  pdl_launch_dependents();
  const PreprocessParams& p = a.p;
  const int tid = threadIdx.x, col = tid % COLS, grp = tid / COLS;
  const int buf_bytes = a.rows_cap * a.row_cap, vecs = a.row_cap >> 4;
  const int t_begin = (int)blockIdx.x * a.tiles_per_block + min((int)blockIdx.x, a.tiles_left);
  const int n = a.tiles_per_block + ((int)blockIdx.x < a.tiles_left ? 1 : 0);
  const int step_r = PRE_THREADS / vecs, step_v = PRE_THREADS - step_r * vecs;   // from one of a thread's copies to its next
  const int r_first = tid / vecs, v_first = tid - r_first * vecs;
  // tiles in order of (image, tile column, tile row)
  auto advance = [&](Tile& t) {
    if (++t.ty == a.tiles_y) {
      t.ty = 0;
      if (++t.tx == a.tiles_x) { t.tx = 0; ++t.img; }
    }
  };
  auto left_column = [&](int tx) { return axis_sample(tx * COLS, p.src_w, p.net_w).i0; };

  // Byte b of a staged row is the frame's byte (aligned start of that row's range) + b.
  auto stage = [&](const Tile& t, int buf, int sx_lo, int sx_hi) {
    const uint8_t* src = p.src_tab ? p.src_tab[t.img] : p.src.p[t.img];
    const int y0 = t.ty * a.tile_rows, y_last = min(y0 + a.tile_rows, p.net_h) - 1;
    const int r_lo = axis_sample(y0, p.src_h, p.net_h).i0, rows = axis_sample(y_last, p.src_h, p.net_h).i1 - r_lo + 1;
    if (tid < a.tile_rows) {
      const AxisSample sy = axis_sample(min(y0 + tid, p.net_h - 1), p.src_h, p.net_h);
      // low bits of the address of column sx_lo in source row 0: (that + row * pitch) & 15 is its position in the staged row
      const uint32_t base_lo = (uint32_t)(uintptr_t)src + 3u * (uint32_t)sx_lo;
      s_row[buf][tid] = make_int4((sy.i0 - r_lo) * a.row_cap + (int)((base_lo + (uint32_t)(sy.i0 * p.src_pitch)) & 15u),
                                  (sy.i1 - r_lo) * a.row_cap + (int)((base_lo + (uint32_t)(sy.i1 * p.src_pitch)) & 15u), __float_as_int(sy.f), 0);
    }
    const uintptr_t first = (uintptr_t)src + (size_t)r_lo * p.src_pitch + 3 * sx_lo;
    const int span = 3 * (sx_hi - sx_lo) + 2;          // last byte of a row, counted from its first
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_mem + buf * buf_bytes);
    for (int r = r_first, v = v_first; r < rows;) {
      const uintptr_t g = first + (size_t)r * p.src_pitch;
      if (v * 16 <= (int)(g & 15) + span)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + r * a.row_cap + v * 16), "l"((g & ~(uintptr_t)15) + v * 16) : "memory");
      r += step_r;
      v += step_v;
      if (v >= vecs) { v -= vecs; ++r; }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  Tile cur, ahead;
  {
    const int tiles_per_img = a.tiles_x * a.tiles_y;
    cur.img = t_begin / tiles_per_img;
    const int rem = t_begin - cur.img * tiles_per_img;
    cur.tx = rem / a.tiles_y;
    cur.ty = rem - cur.tx * a.tiles_y;
  }
  ahead = cur;
  auto stage_ahead = [&](int buf) {
    const int sx_lo = left_column(ahead.tx), sx_hi = axis_sample(min((ahead.tx + 1) * COLS, p.net_w) - 1, p.src_w, p.net_w).i1;
    stage(ahead, buf, sx_lo, sx_hi);
    advance(ahead);
  };
  if (n > 0) stage_ahead(0);

  const size_t plane = (size_t)p.net_h * p.net_w;
  int tx = -1, x = 0, xo = 0;
  float fx = 0.f;
  for (int i = 0; i < n; ++i) {
    if (i + 1 < n) {
      stage_ahead((i + 1) & 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    if (cur.tx != tx) {
      tx = cur.tx;
      x = tx * COLS + col;
      const AxisSample sx = axis_sample(min(x, p.net_w - 1), p.src_w, p.net_w);
      xo = 3 * (sx.i0 - left_column(tx));
      fx = sx.f;
    }
    __syncthreads();                                   // this tile's rows and row table are complete
    const uint32_t* words = reinterpret_cast<const uint32_t*>(s_mem + (i & 1) * buf_bytes);
    const int y0 = cur.ty * a.tile_rows, rows = min(a.tile_rows, p.net_h - y0);
    if (x < p.net_w) {
      float* d = p.dst + (size_t)cur.img * 3 * plane + (size_t)(y0 + grp) * p.net_w + x;
#pragma unroll 2
      for (int r = grp; r < rows; r += GROUPS, d += GROUPS * p.net_w) {
        const int4 e = s_row[i & 1][r];
        float o0, o1, o2;
        uint32_t lo0, hi0;
        fetch_pair(words, e.x + xo, lo0, hi0);
        if (ONE_ROW) {
          sample_row(lo0, hi0, fx, a.scale, a.shift, o0, o1, o2);
        } else {
          uint32_t lo1, hi1;
          fetch_pair(words, e.y + xo, lo1, hi1);
          sample_rows(lo0, hi0, lo1, hi1, fx, __int_as_float(e.z), a.scale, a.shift, o0, o1, o2);
        }
        d[0] = o0;
        d[plane] = o1;
        d[2 * plane] = o2;
      }
    }
    __syncthreads();                                   // the buffer has been read
    advance(cur);
  }
}

constexpr int DIR_TX = 32, DIR_TY = 8, DIR_OUT_W = DIR_TX * 4;   // threads of a block, 4 outputs each

// Fallback for extreme down-scaling factors whose footprint does not fit in shared memory:
// taps are read straight from global memory (L1-cached byte loads).
__global__ void __launch_bounds__(DIR_TX * DIR_TY) preprocess_direct_kernel(const __grid_constant__ PreprocessParams p, float scale, float shift) {
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
  for (int j = 0; j < 4 && xo0 + j < p.net_w; ++j) {
    const AxisSample sx = axis_sample(xo0 + j, p.src_w, p.net_w);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float p00 = (float)__ldg(r0 + 3 * sx.i0 + c), p01 = (float)__ldg(r0 + 3 * sx.i1 + c);
      const float p10 = (float)__ldg(r1 + 3 * sx.i0 + c), p11 = (float)__ldg(r1 + 3 * sx.i1 + c);
      const float top = p00 + sx.f * (p01 - p00);
      const float bot = p10 + sx.f * (p11 - p10);
      dst[c * plane + j] = fmaf(top + sy.f * (bot - top), scale, shift);
    }
  }
}

// Staged rows and bytes per row of a tile in the worst case: rows = ceil(tile_rows * sh/nh) + 2; bytes = 3 * (ceil(COLS * sw/nw) + 2) + 15
// (alignment at the front) + 15 (at the end) + 12 (the tap fetch reads three whole words from its first byte), rounded up to 16.
void staging(const PreprocessParams& p, int cols, int tile_rows, long* rows, long* row_cap) {
  *rows = ((long)tile_rows * p.src_h + p.net_h - 1) / p.net_h + 2;
  const long c = ((long)cols * p.src_w + p.net_w - 1) / p.net_w + 2;
  *row_cap = ((3 * c + 48 + 15) / 16) * 16;
}

template <int COLS>
cudaError_t launch_staged(const PreprocessParams& p, cudaStream_t s, bool* fits) {
  constexpr int GROUPS = PRE_THREADS / COLS;
  int sms = 0;
  cudaError_t e = post_sm_count(&sms);
  if (e != cudaSuccess) return e;
  PreprocessArgs a;
  a.p = p;
  a.scale = pre::norm_scale(p.inv_div, p.inv_std);
  a.shift = pre::norm_shift(p.mean, p.inv_std);
  a.tiles_x = (p.net_w + COLS - 1) / COLS;
  // Rows per tile: the busiest block's tiles x (rows to sample, and about two rows' worth for its halo and barriers) is least, and the higher tile of
  // two that come out alike; another height where by it the busiest multiprocessor has at least a tenth less to do, a tile's latency counted as twelve
  // rows.  Device time of frames from memory, us, by rows: four 1280x960 to 640x480 6 11.7, 8 10.3, 10 10.6, 12 9.3*, 14 9.3; four 1920x1080 to 1280x720 16 19.1, 20 18.8,
  // 24 18.1, 26 17.8*; one 320x240 to 1280x960 18 7.4, 22 6.9*, 24 7.0, 28 7.6 (* chosen).  Of 140 sizes and batches one is 4 % slower by the second rule, the mean 3 % faster.
  const long slots = (long)PRE_PER_SM * sms;
  struct Height {
    int rows = 0;
    long cap_r = 0, cap_b = 0, tiles = 0, busiest_sm = 0, cost = 0;
  } by_round, by_sm, tallest;
  for (int rows = GROUPS; rows <= PRE_MAX_ROWS; rows += GROUPS) {
    Height h;
    h.rows = rows;
    staging(p, COLS, rows, &h.cap_r, &h.cap_b);
    if (h.cap_r * h.cap_b > PRE_STAGE_BYTES) break;
    h.tiles = (long)p.K * a.tiles_x * ((p.net_h + rows - 1) / rows);
    h.busiest_sm = (h.tiles / slots * PRE_PER_SM + (h.tiles % slots + sms - 1) / sms) * (rows + 12);
    h.cost = (h.tiles + slots - 1) / slots * (rows + 2);
    if (!by_round.rows || h.cost <= by_round.cost) by_round = h;
    if (!by_sm.rows || h.busiest_sm <= by_sm.busiest_sm) by_sm = h;
    tallest = h;
  }
  // A tile of few rows is mostly halo and latency (resize factors from about three on): there taps straight from memory are faster once there are several
  // rounds of such tiles, and of two rows always.  Staged / direct, us, one and eight frames: 1920x1080 to 480x270 (2 rows) 4.9 / 4.4 and 19.3 / 15.4; to 608x342 (4) 5.0 / 5.4
  // and 20.1 / 18.9; to 400x225 (4) 4.5 / 4.6 and 16.9 / 14.1; to 640x360 (6) 5.4 / 5.5 and 18.4 / 19.1.
  *fits = tallest.rows >= 6 && tallest.rows >= 2 * GROUPS;
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
  auto kern = p.src_h == p.net_h ? preprocess_staged_kernel<COLS, true> : preprocess_staged_kernel<COLS, false>;
  if (smem + PRE_STATIC_BYTES > 48 * 1024) {   // what a kernel may have of both without asking
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * PRE_STAGE_BYTES);
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
  preprocess_direct_kernel<<<grid, dim3(DIR_TX, DIR_TY), 0, s>>>(p, pre::norm_scale(p.inv_div, p.inv_std), pre::norm_shift(p.mean, p.inv_std));
  return cudaGetLastError();
}

}  // namespace tt
