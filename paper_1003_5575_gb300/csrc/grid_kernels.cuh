// Gridder (Section 6): V_grid(x, y) = sum_i f(r_i) V_i over the visibilities
// with r_i = |(x, y) - (x_i, y_i)| < r_max, the pixel centres at integer
// coordinates and f a radial gridding convolution function given as a table
// (linear interpolation between samples r_k = k r_max / (n_tab - 1)).
//
// The paper's CUDA gridder is a gather over binned visibilities: the grid is
// cut into bins of B x B pixels (B >= r_max), the visibilities are sorted by
// bin with first/last tables, and the threads of one block (a patch of pixels
// inside one bin) share the visibilities of the bin and its eight neighbours
// through shared memory.  Here:
//   k_grid_sort_pass<false>  one warp per chunk of visibilities counts them per bin
//                   (shared-memory counters)
//   k_grid_bin_totals, k_grid_scan_bins, k_grid_offsets
//                   exclusive scan in (bin, chunk) order over the [chunk][bin]
//                   count table: each chunk's first slot in each bin, and
//                   each bin's first and last
//   k_grid_sort_pass<true>   the same warps place their visibilities, stably:
//                   a lane's rank among the lanes with the same bin
//                   (__match_any_sync) plus the chunk's running count for it
//   k_grid_gather   one CTA per bin, 8 x 8 pixel tiles, several warps a tile (2
//                   pixels per lane); in the dense centre of the u-v plane one
//                   CTA per tile, all of its warps on it.  The warps of a tile
//                   share the 9 bins' sorted list (L2-resident) 32 visibilities at a time: every
//                   lane tests one against the tile's box, the hits' positions
//                   collect in the warp's shared memory, and once 32 are there
//                   their values are fetched together and each costs its
//                   per-pixel work.  Every pixel's sum is deterministic (a tile's
//                   warps are added in order) and every pixel is written exactly
//                   once (no atomics, no memset).
// Measured (512 antennas, 1125^2 pixels, radius 12, 4 values): 591 us before the
// warps of a tile shared its list, values were fetched 32 together, the two
// pixels of a lane became packed operands and the sort's warps were more than 128;
// 233 us now.  The gather is bound by instruction issue and latency (189 us, 61 % of the slots, ALU 42 %),
// the sort by the latency of its five short launches.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace rts {

constexpr int kGridBlock = 256;       // visibilities a counting warp has in flight
constexpr int kGridMaxChunks = 512;   // counting warps, at most: a warp's chunk is the multiple of
                                      // kGridBlock that needs no more (4 warps an SM at 130 000
                                      // visibilities, and a bounded count table)
constexpr int kGridSegs = 8;          // segments of the chunks in the scan
constexpr int kGridWarps = 4;         // counting warps per CTA
constexpr int kGridMaxBins = 8192;    // shared-memory counters per warp
constexpr int kGridPix = 2;           // pixels per gather thread
constexpr int kGridTile = 8;          // gather warp tile: 8 x 8 pixels (kGridPix = 2 per lane)
constexpr int kGridMaxBin = 40;       // at most 5 x 5 tiles (800 threads) per bin
constexpr int kGridMaxPol = 4;
// Dense bins: a tile there has a CTA of its own, or the few CTAs of the u-v
// centre end last (249 us with, 255 without; with a CTA for each tile of
// the whole grid 290: its tables are loaded nine times as often)
constexpr int kGridMaxDense = 128;    // bins whose tiles get a CTA each, at most
constexpr int kGridDenseMin = 2048;   // and the fewest visibilities of such a bin and its neighbours
constexpr int kGridGatherMaxSmem = 100 * 1024;   // 4096 samples, 4 values, 32-pixel bins: 98 320 bytes

// bin of a visibility, or -1 outside [0, n_pix)^2 (NaN compares false)
__device__ __forceinline__ int grid_bin(float2 p, int n_pix, int bin, int nbx) {
  if (!(p.x >= 0.f && p.x < (float)n_pix && p.y >= 0.f && p.y < (float)n_pix)) return -1;
  return ((int)p.y / bin) * nbx + (int)p.x / bin;
}

struct GridSortArgs {
  const float2* xy;         // [n_vis] pixel coordinates
  const float2* vis;        // [n_vis][n_pol]
  int n_vis, n_pol, n_pix, bin, nbx, n_bins, n_chunks, chunk;
  int* counts;              // [n_chunks][n_bins] visibilities of chunk in bin, then exclusive offsets
  int* segs;                // [kGridSegs][n_bins] the same summed over each segment of the chunks
  int* bin_start;           // [n_bins + 1]
  int* dense;               // [1 + kGridMaxDense] count and list of the dense bins, then [n_bins] flags
  int dense_min;            // more visibilities than this in a bin and its neighbours: dense
  float2* sxy;              // [n_vis] sorted positions
  float2* svis;             // [n_vis][n_pol] sorted values
};

// Warp w of the CTA walks chunk blockIdx.x * kGridWarps + w, kGridBlock visibilities
// at a time with all of their loads in flight; SCATTER places them, else it
// counts them.  One warp per 1024 visibilities and a load per step on its
// critical path took 70 us (place) and 27 us (count) at 130 816 visibilities
// and 2 209 bins.
template <bool SCATTER>
__global__ void __launch_bounds__(kGridWarps * 32) k_grid_sort_pass(GridSortArgs a) {
  constexpr int kN = kGridBlock / 32;
  extern __shared__ int s_cnt[];                       // [kGridWarps][n_bins]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunk = blockIdx.x * kGridWarps + warp;
  if (chunk >= a.n_chunks) return;
  int* cnt = s_cnt + (size_t)warp * a.n_bins;
  for (int b = lane; b < a.n_bins; b += 32) cnt[b] = 0;
  __syncwarp();
  const int* first = a.counts + (size_t)chunk * a.n_bins;
  const int i0 = chunk * a.chunk, i1 = min(a.n_vis, i0 + a.chunk);
  const unsigned lt = (1u << lane) - 1u;
  for (int ib = i0; ib < i1; ib += kGridBlock) {
    float2 q[kN];
    int bins[kN], at[kN];
    #pragma unroll
    for (int j = 0; j < kN; ++j) {
      const int i = ib + 32 * j + lane;
      q[j] = i < i1 ? a.xy[i] : make_float2(-1.f, -1.f);
    }
    #pragma unroll
    for (int j = 0; j < kN; ++j) bins[j] = grid_bin(q[j], a.n_pix, a.bin, a.nbx);
    #pragma unroll
    for (int j = 0; j < kN; ++j) {
      const int b = bins[j];
      const unsigned same = __match_any_sync(0xffffffffu, b);
      const int rank = __popc(same & lt);
      at[j] = b >= 0 ? cnt[b] + rank : 0;
      __syncwarp();
      if (b >= 0 && rank == 0) cnt[b] += __popc(same);
      __syncwarp();
    }
    if (SCATTER) {
      #pragma unroll
      for (int j = 0; j < kN; ++j)
        if (bins[j] >= 0) at[j] += __ldg(first + bins[j]);
      #pragma unroll
      for (int j = 0; j < kN; ++j)
        if (bins[j] >= 0) a.sxy[at[j]] = q[j];
      for (int p = 0; p < a.n_pol; ++p) {
        float2 v[kN];
        #pragma unroll
        for (int j = 0; j < kN; ++j)
          if (bins[j] >= 0) v[j] = a.vis[(size_t)(ib + 32 * j + lane) * a.n_pol + p];
        #pragma unroll
        for (int j = 0; j < kN; ++j)
          if (bins[j] >= 0) a.svis[(size_t)at[j] * a.n_pol + p] = v[j];
      }
    }
  }
  if (!SCATTER)
    for (int b = lane; b < a.n_bins; b += 32) a.counts[(size_t)chunk * a.n_bins + b] = cnt[b];
}

// Exclusive scan of counts in (bin, chunk) order, in three steps:
//   k_grid_bin_totals  warp w of a CTA sums 32 bins' counts over the chunks of
//                      segment w (rows read coalesced), the CTA the segments
//   k_grid_scan_bins   one CTA scans the bin totals into bin_start
//   k_grid_offsets     warp w turns the counts of segment w into each chunk's
//                      first slot, 32 chunks' loads in flight, and lists the dense bins:
//                      those with more than dense_min >= 9 n_vis / kGridMaxDense
//                      visibilities in them and their neighbours, so fewer than
//                      kGridMaxDense
__device__ __forceinline__ int2 grid_segment(int n_chunks, int w) {
  const int per = (n_chunks + kGridSegs - 1) / kGridSegs;
  return make_int2(min(n_chunks, w * per), min(n_chunks, (w + 1) * per));
}

__global__ void __launch_bounds__(kGridSegs * 32) k_grid_bin_totals(GridSortArgs a) {
  __shared__ int s_seg[kGridSegs][32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, b = blockIdx.x * 32 + lane;
  const int2 c = grid_segment(a.n_chunks, w);
  int s = 0;
  if (b < a.n_bins) {
    #pragma unroll 32
    for (int k = c.x; k < c.y; ++k) s += a.counts[(size_t)k * a.n_bins + b];
    a.segs[(size_t)w * a.n_bins + b] = s;
  }
  s_seg[w][lane] = s;
  __syncthreads();
  if (w == 0 && b < a.n_bins) {
    for (int k = 1; k < kGridSegs; ++k) s += s_seg[k][lane];
    a.bin_start[b] = s;                               // total for now; start after the scan
  }
}

__global__ void __launch_bounds__(1024) k_grid_scan_bins(GridSortArgs a) {
  __shared__ int s_tot[1024];
  const int per = (a.n_bins + 1023) / 1024;
  const int b0 = min(a.n_bins, (int)threadIdx.x * per), b1 = min(a.n_bins, b0 + per);
  int s = 0;
  for (int b = b0; b < b1; ++b) s += a.bin_start[b];
  s_tot[threadIdx.x] = s;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {              // inclusive Hillis-Steele scan
    const int v = threadIdx.x >= o ? s_tot[threadIdx.x - o] : 0;
    __syncthreads();
    s_tot[threadIdx.x] += v;
    __syncthreads();
  }
  int run = s_tot[threadIdx.x] - s;
  for (int b = b0; b < b1; ++b) {
    const int t = a.bin_start[b];
    a.bin_start[b] = run;
    run += t;
  }
  if (threadIdx.x == 1023) a.bin_start[a.n_bins] = s_tot[1023];
  if (threadIdx.x == 0) a.dense[0] = 0;
}

__global__ void __launch_bounds__(kGridSegs * 32) k_grid_offsets(GridSortArgs a) {
  const int w = threadIdx.x >> 5, b = blockIdx.x * 32 + (threadIdx.x & 31);
  if (b >= a.n_bins) return;
  if (w == 0) {                                     // the list's order changes nothing
    const int bx = b % a.nbx, by = b / a.nbx;
    int near = 0;
    for (int y = max(0, by - 1); y <= min(a.nbx - 1, by + 1); ++y)
      near += a.bin_start[y * a.nbx + min(a.nbx - 1, bx + 1) + 1] - a.bin_start[y * a.nbx + max(0, bx - 1)];
    const bool dense = near > a.dense_min;
    if (dense) a.dense[1 + atomicAdd(a.dense, 1)] = b;
    a.dense[1 + kGridMaxDense + b] = dense;
  }
  const int2 c = grid_segment(a.n_chunks, w);
  int run = a.bin_start[b];
  for (int k = 0; k < w; ++k) run += a.segs[(size_t)k * a.n_bins + b];
  for (int k0 = c.x; k0 < c.y; k0 += 32) {
    int v[32];
    #pragma unroll
    for (int u = 0; u < 32; ++u) v[u] = k0 + u < c.y ? a.counts[(size_t)(k0 + u) * a.n_bins + b] : 0;
    #pragma unroll
    for (int u = 0; u < 32; ++u)
      if (k0 + u < c.y) {
        a.counts[(size_t)(k0 + u) * a.n_bins + b] = run;
        run += v[u];
      }
  }
}

struct GridGatherArgs {
  const float2* sxy;
  const float2* svis;
  const int* bin_start;     // [n_bins + 1]
  const float* gcf;         // [n_tab] (copied to shared memory, one extra sample repeated)
  int n_tab, n_pol, n_pix, bin, nbx, nby;
  float r_max, r2max, tab_scale;   // tab_scale = (n_tab - 1) / r_max
  float2* grid;             // [n_pol][n_pix][n_pix]
  const int* dense;         // see GridSortArgs
};

// warps of a CTA: the tiles of a bin, and as many warps a tile as 1024 threads hold
// (at most 4): the dense u-v centre's tiles set the kernel's time
__host__ __device__ inline int grid_tiles(int bin) {
  const int tpb = (bin + kGridTile - 1) / kGridTile;
  return tpb * tpb;
}
__host__ __device__ inline int grid_split(int bin) {
  const int n = 32 / grid_tiles(bin);
  return n < 1 ? 1 : (n > 4 ? 4 : n);
}
// a warp's workspace: positions and list indices of up to 63 hits, the values of
// 32; then its 64 pixels' sums
__host__ __device__ inline int grid_warp_floats(int n_pol) {
  const int stage = 64 * 3 + 32 * 2 * n_pol, sums = 64 * 2 * n_pol;       // multiples of 4 floats
  return stage > sums ? stage : sums;
}
// table [n_tab + 1] of (sample, step to the next) in whole 16-byte words, then the warps' workspaces
inline size_t grid_gather_smem(int n_tab, int bin, int n_pol) {
  return (size_t)((n_tab + 2) & ~1) * sizeof(float2) +
         (size_t)grid_tiles(bin) * grid_split(bin) * grid_warp_floats(n_pol) * sizeof(float);
}

// sqrt(d2) within an ulp or two (0 and subnormals: 0), by one instruction where
// sqrtf takes several
__device__ __forceinline__ float grid_sqrt(float d2) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d2));
  return r;
}

template <int NPOL>
__global__ void __launch_bounds__(1024, 1) k_grid_gather(GridGatherArgs a) {
  extern __shared__ __align__(16) float2 s_tab[];   // (gcf[t], gcf[t + 1] - gcf[t]), the last sample repeated
  // Tile t of a bin: at (t % tpb, t / tpb); lane l its pixels (l % 8, l / 8) and (l % 8,
  // l / 8 + 4).  The first CTAs take one tile of a dense bin with all of their
  // warps, the others a bin: warp w part w / n_tile of tile w % n_tile
  const int tpb = (a.bin + kGridTile - 1) / kGridTile, n_tile = tpb * tpb, n_warp = blockDim.x >> 5;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool dense = blockIdx.x < kGridMaxDense * n_tile;
  int bid = (int)blockIdx.x - kGridMaxDense * n_tile, tile = warp % n_tile, part = warp / n_tile;
  int split = n_warp / n_tile, next_part = n_tile;              // parts of a tile, warps from one to the next
  if (dense) {
    const int d = blockIdx.x / n_tile;
    if (d >= a.dense[0]) return;
    bid = a.dense[1 + d];
    tile = blockIdx.x % n_tile;
    part = warp;
    split = n_warp;
    next_part = 1;
  } else if (a.dense[1 + kGridMaxDense + bid]) {
    return;
  }
  const int bx = bid % a.nbx, by = bid / a.nbx;
  for (int k = threadIdx.x; k <= a.n_tab; k += blockDim.x) {
    const float f = a.gcf[min(k, a.n_tab - 1)];
    s_tab[k] = make_float2(f, a.gcf[min(k + 1, a.n_tab - 1)] - f);
  }
  __syncthreads();
  float* ws = reinterpret_cast<float*>(s_tab + ((a.n_tab + 2) & ~1)) + (size_t)warp * grid_warp_floats(NPOL);
  float2* s_pos = reinterpret_cast<float2*>(ws);                // [64]
  int* s_idx = reinterpret_cast<int*>(ws + 128);                // [64]
  float2* s_val = reinterpret_cast<float2*>(ws + 192);          // [32][NPOL]
  const int tx = (tile % tpb) * kGridTile, ty = (tile / tpb) * kGridTile;     // tile origin in the bin
  const float x0 = (float)(bx * a.bin + tx), y0 = (float)(by * a.bin + ty);
  const int ix = tx + (lane & 7), px = bx * a.bin + ix;
  int py[kGridPix];
  bool live[kGridPix];
  float2 acc[kGridPix][NPOL];
  #pragma unroll
  for (int u = 0; u < kGridPix; ++u) {
    const int iy = ty + (lane >> 3) + 4 * u;                                  // pixel in the bin
    py[u] = by * a.bin + iy;
    live[u] = ix < a.bin && iy < a.bin && px < a.n_pix && py[u] < a.n_pix;
    #pragma unroll
    for (int k = 0; k < NPOL; ++k) acc[u][k] = make_float2(0.f, 0.f);
  }
  const float fx = (float)px;
  const float2 fy = make_float2((float)py[0], (float)py[1]);
  const float lim0 = live[0] ? a.r2max : -1.f, lim1 = live[1] ? a.r2max : -1.f;
  const float last = (float)(a.n_tab - 1);
  const float ext = (float)(kGridTile - 1);

  int count = 0;                                     // hits waiting in s_pos, s_idx
  // the first n (<= 32) waiting hits: their values together, then pixel by pixel
  auto work = [&](int n) {
    if (lane < n) {
      const float2* g = a.svis + (size_t)s_idx[lane] * NPOL;
      #pragma unroll
      for (int p = 0; p < NPOL; ++p) s_val[lane * NPOL + p] = __ldg(g + p);
    }
    __syncwarp();
    #pragma unroll 2
    for (int h = 0; h < n; ++h) {
      const float2 p = s_pos[h];
      // squared distances rounded as the box test below rounds them: a pixel inside the
      // radius is never outside it for its tile
      const float dx = fx - p.x;
      const float2 dx2 = make_float2(dx, dx), dy = fadd2(fy, make_float2(-p.y, -p.y)), d = ffma2(dx2, dx2, fmul2(dy, dy));
      // table position; its integer part by a round-down addition of 2^23
      float2 at = fmul2(make_float2(grid_sqrt(d.x), grid_sqrt(d.y)), make_float2(a.tab_scale, a.tab_scale));
      at = make_float2(fminf(at.x, last), fminf(at.y, last));
      const float2 m = make_float2(__fadd_rd(at.x, 8388608.f), __fadd_rd(at.y, 8388608.f));
      const float2 w = fadd2(at, fadd2(make_float2(8388608.f, 8388608.f), make_float2(-m.x, -m.y)));
      const float2 e0 = s_tab[__float_as_uint(m.x) & 0x7fffffu], e1 = s_tab[__float_as_uint(m.y) & 0x7fffffu];
      const float f0 = fmaf(w.x, e0.y, e0.x), f1 = fmaf(w.y, e1.y, e1.x);
      const float2 g0 = make_float2(f0, f0), g1 = make_float2(f1, f1);
      // a pixel out of reach takes no part (a value may be infinite or no number)
      float2 v[NPOL];
      if (NPOL == 4) {
        const float4 v01 = reinterpret_cast<const float4*>(s_val)[2 * h], v23 = reinterpret_cast<const float4*>(s_val)[2 * h + 1];
        v[0] = make_float2(v01.x, v01.y); v[1 % NPOL] = make_float2(v01.z, v01.w);
        v[2 % NPOL] = make_float2(v23.x, v23.y); v[3 % NPOL] = make_float2(v23.z, v23.w);
      } else {
        #pragma unroll
        for (int k = 0; k < NPOL; ++k) v[k] = s_val[h * NPOL + k];
      }
      if (d.x < lim0)
        #pragma unroll
        for (int k = 0; k < NPOL; ++k) acc[0][k] = ffma2(g0, v[k], acc[0][k]);
      if (d.y < lim1)
        #pragma unroll
        for (int k = 0; k < NPOL; ++k) acc[1][k] = ffma2(g1, v[k], acc[1][k]);
    }
    __syncwarp();
  };

  // the bin's own 32-visibility steps and its neighbours' in row order; the parts of
  // a tile take them in turn
  int step = 0;
  for (int ny = max(0, by - 1); ny <= min(a.nby - 1, by + 1); ++ny)
    for (int nx = max(0, bx - 1); nx <= min(a.nbx - 1, bx + 1); ++nx) {
      const int nb = ny * a.nbx + nx;
      const int v0 = a.bin_start[nb], v1 = a.bin_start[nb + 1];
      const int n_step = (v1 - v0 + 31) >> 5;
      int k = (part - step % split + split) % split; // this part's first step in the list
      step += n_step;
      float2 next = make_float2(0.f, 0.f);
      if (v0 + 32 * k + lane < v1) next = __ldg(a.sxy + v0 + 32 * k + lane);
      for (; k < n_step; k += split) {
        // lane l tests visibility l of the step against the tile's box; the next step's
        // positions are on their way meanwhile
        const float2 q = next;
        const int i = v0 + 32 * k + lane, in = i + 32 * split;
        if (in < v1) next = __ldg(a.sxy + in);
        bool hit = false;
        if (i < v1) {
          const float ex = fmaxf(fmaxf(x0 - q.x, q.x - (x0 + ext)), 0.f);
          const float ey = fmaxf(fmaxf(y0 - q.y, q.y - (y0 + ext)), 0.f);
          hit = fmaf(ex, ex, ey * ey) < a.r2max;
        }
        const unsigned hits = __ballot_sync(0xffffffffu, hit);
        if (hit) {
          const int at = count + __popc(hits & ((1u << lane) - 1u));
          s_pos[at] = q;
          s_idx[at] = i;
        }
        count += __popc(hits);
        if (count >= 32) {
          __syncwarp();
          work(32);
          // the rest to the front
          count -= 32;
          float2 mp = make_float2(0.f, 0.f);
          int mi = 0;
          if (lane < count) { mp = s_pos[32 + lane]; mi = s_idx[32 + lane]; }
          __syncwarp();
          if (lane < count) { s_pos[lane] = mp; s_idx[lane] = mi; }
        }
        __syncwarp();
      }
    }
  work(count);
  // the parts' sums in order
  float2* sums = reinterpret_cast<float2*>(ws);                 // [2][NPOL][32]
  if (part > 0)
    #pragma unroll
    for (int u = 0; u < kGridPix; ++u)
      #pragma unroll
      for (int k = 0; k < NPOL; ++k) sums[(u * NPOL + k) * 32 + lane] = acc[u][k];
  __syncthreads();
  if (part > 0) return;
  for (int o = 1; o < split; ++o) {
    const float2* s = reinterpret_cast<const float2*>(ws + (size_t)o * next_part * grid_warp_floats(NPOL));
    #pragma unroll
    for (int u = 0; u < kGridPix; ++u)
      #pragma unroll
      for (int k = 0; k < NPOL; ++k) acc[u][k] = fadd2(acc[u][k], s[(u * NPOL + k) * 32 + lane]);
  }
  const size_t plane = (size_t)a.n_pix * a.n_pix;
  #pragma unroll
  for (int u = 0; u < kGridPix; ++u)
    if (live[u])
      #pragma unroll
      for (int k = 0; k < NPOL; ++k) a.grid[k * plane + (size_t)py[u] * a.n_pix + px] = acc[u][k];
}

}  // namespace rts
