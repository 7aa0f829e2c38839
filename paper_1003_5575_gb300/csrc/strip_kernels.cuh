// Per-source arithmetic on a strip (one baseline and time, up to 32 QH channels) by
// one warp on the CUDA cores, and the blocked peel's pass built from it.
//
// The tcgen05 pass forms 64 x 16 x 4 operand values per strip and role whatever
// the strip's length, about 4 900 cycles a strip and role; for short strips the
// 1024 complex multiply-adds a channel themselves are fewer cycles than that.
// Here a warp keeps its strip in registers (lane (h, r): channels 16 q + r of the
// tiles q = h QH .. h QH + QH - 1, two neighbouring tiles packed as one f32x2
// operand) and takes the phasors as products T1_k[q] T2_k[r] of two small tables
// (16 + 2 QH entries a source instead of 32 QH), so a (source, channel) pair
// costs 20 multiply-adds in the subtraction and 17 in the average, two a packed
// instruction.  No step needs another warp: strips of the same baseline share
// its model matrices, nothing else.
//   subtraction  lane = its channels, loop over sources; the model matrix is
//                broadcast from shared memory as packed pairs (-m, -m), (m, m).
//   average      lane = source (32 at a time), loop over channels: the strip goes
//                to shared memory as planes (re of 4 pols | im of 4 pols), read by
//                broadcast; pol pairs are the packed operands and T2 stays in
//                registers.  sum_c R(c) P(c) = sum_q T1[q] sum_r R(16 q + r) T2[r].
#pragma once
#include "block_kernels.cuh"
#include "kahan.cuh"

namespace rts {

constexpr int kStWarps = 8;                // warps of a CTA
constexpr int kStGrp = 32;                 // sources whose tables a warp holds at once
constexpr int kStMaxQh = 8;                // tiles per half warp, at most: 256 channels
// Strips up to here take this pass, and the Taylor cadence's, by default: past 256
// channels a strip no longer fits a warp's registers (the form of block_kernels.cuh
// takes 7.7 ms at 384 channels, tcgen05 3.2).  128 sources, 8 times, this form / tcgen05
// in ms:
//   channels        64           128          160          203          256
//   65 antennas   0.35 / 0.85  0.53 / 0.86  0.77 / 0.86  0.85 / 0.86  0.94 / 0.87
//   128           1.28 / 2.79  1.99 / 2.80  2.89 / 2.81  3.19 / 2.83  3.48 / 2.84
//   512               -        31.2 / 43.6  45.7 / 43.7  50.3 / 43.9  55.0 / 44.2
// With 3 times 65 antennas are ahead here up to 256 (0.39 / 0.44), 128 up to 160.  So from
// 160 channels on, where more than about 20 000 strips fill the tcgen05 form's CTAs, the
// line gives up to 24 % of a pass away; it stood where the former tcgen05 pass (3.75 ms
// at 128 antennas x 256 channels) crossed.  Taylor, 42 sources: 0.84 / 1.02 / 1.60 / 2.51 / 2.79
// ms for 32 / 64 / 128 / 203 / 256 channels, tcgen05 5.0 ms.
constexpr int kStAutoChan = 256;
constexpr int kStMRow = 4;                 // float4 of a source's packed model matrix

// exp(2 pi i x) of a Q0.64 phase whose high word is x: the nearest of 256 table
// angles and a rotation by |d| <= 2 pi / 512 (sin d = d - d^3/6, cos d = 1 - d^2/2, both
// within 1e-9), about 1e-7 absolute; the hardware sin/cos of the same phase is
// within 5e-7, and takes the special-function unit two operations and a conversion
__device__ __forceinline__ float2 phasor_lut(unsigned x, const float2* __restrict__ lut) {
  const unsigned h = x + 0x00800000u;
  const float2 L = lut[h >> 24];
  // the low 24 bits, less the last, minus half of their range, as a float
  const float f = __uint_as_float(0x4B000000u | ((h & 0x00FFFFFFu) >> 1)) - 12582912.0f;
  const float d = f * 2.9258361585343192e-09f;             // 2 pi 2^-31
  const float d2 = d * d, s = fmaf(d * d2, -1.0f / 6.0f, d), c = -0.5f * d2;
  return make_float2(fmaf(L.x, c, fmaf(-L.y, s, L.x)), fmaf(L.y, c, fmaf(L.x, s, L.y)));
}
__device__ __forceinline__ float2 phasor_lut(unsigned long long ph, const float2* lut) {
  return phasor_lut((unsigned)(ph >> 32), lut);
}
// a step rounded to Q0.32: fifteen of them are within 1.1e-8 of a turn's angle
__device__ __forceinline__ unsigned step32(unsigned long long b) { return (unsigned)((b + 0x80000000ull) >> 32); }
__device__ __forceinline__ void lut_fill(float2* lut, int tid, int nthr) {       // [256]
  for (int i = tid; i < 256; i += nthr) {
    float s, c;
    sincospif((float)i * (1.0f / 128.0f), &s, &c);
    lut[i] = make_float2(c, s);
  }
}

// a strip in registers: [pol][pair of tiles], the two tiles' values packed
template <int QH> struct Strip { float2 re[4][QH / 2], im[4][QH / 2]; };

// tables of 32 sources: T2 [32][17] float2, T1 [32][QH + 1] float4 = the pair
// (2 v, 2 v + 1) of tiles as (re, re, im, im); rows padded against bank conflicts
template <int QH> struct StripTables {
  float2 t2[kStGrp][17];
  float4 t1[kStGrp][QH + 1];
};
template <int QH> __host__ __device__ constexpr size_t strip_planes_bytes() { return (size_t)32 * QH * 2 * sizeof(float4); }
// a warp's workspace: tables, planes or (6 KB at most) its sums
template <int QH> __host__ __device__ constexpr size_t strip_warp_bytes() {
  return sizeof(StripTables<QH>) > strip_planes_bytes<QH>()
             ? (sizeof(StripTables<QH>) > 6144 ? sizeof(StripTables<QH>) : 6144)
             : strip_planes_bytes<QH>();
}

// the tables of source `lane` from its phase; np pairs of tiles
template <int QH>
__device__ __forceinline__ void strip_tables(StripTables<QH>& tb, PhaseAB p, int lane, int np, const float2* lut) {
  const unsigned b32 = step32(p.b);
  #pragma unroll
  for (int r = 0; r < 16; ++r) tb.t2[lane][r] = phasor_lut((unsigned)r * b32, lut);
  const unsigned long long step = 16ull * p.b;
  unsigned long long x = p.a;
  #pragma unroll 2
  for (int v = 0; v < np; ++v, x += 2ull * step) {
    const float2 a = phasor_lut(x, lut), b = phasor_lut(x + step, lut);
    tb.t1[lane][v] = make_float4(a.x, b.x, a.y, b.y);
  }
}

// a model matrix entry as the packed pairs (-re, -re), (-im, -im) that strip_subtract reads
__device__ __forceinline__ void strip_pack_model(float4* Mt, int e, float2 m) {
  Mt[e] = make_float4(-m.x, -m.x, -m.y, -m.y);
}

// row x of Jones matrices in a caller's array, aligned to its elements only
__device__ __forceinline__ float4 jones_row(const void* jones, size_t x) {
  const float2* J = static_cast<const float2*>(jones) + 2 * x;
  const float2 a = J[0], b = J[1];
  return make_float4(a.x, a.y, b.x, b.y);
}
// S J_i J_j^H, entry (r, c), rounded to FP32; rows of J as float4
__device__ __forceinline__ float2 model_entry_ff(float4 a, float4 b, float Sh, float Sl) {
  const FF zero = {0.f, 0.f};
  const FF re = ff_fma(a.w, b.w, ff_fma(a.z, b.z, ff_fma(a.y, b.y, ff_fma(a.x, b.x, zero))));
  const FF im = ff_fma(-a.z, b.w, ff_fma(a.w, b.z, ff_fma(-a.x, b.y, ff_fma(a.y, b.x, zero))));
  auto scale = [&](FF v) {
    const float p = __fmul_rn(v.hi, Sh);
    return p + fmaf(v.hi, Sl, fmaf(v.lo, Sh, fmaf(v.hi, Sh, -p)));
  };
  return make_float2(scale(re), scale(im));
}

// R -= sum_{k0 <= k < k1} M_k conj(P_k), M packed [][kStMRow]; kUnroll: sources whose
// loads are in flight together
template <int QH, int kUnroll = QH < 8 ? 2 : 1>
__device__ __forceinline__ void strip_subtract(Strip<QH>& R, const StripTables<QH>& tb, const float4* __restrict__ Mt,
                                               int k0, int k1, int lane) {
  const int r = lane & 15, v0 = (lane >> 4) * (QH / 2);
  #pragma unroll kUnroll
  for (int k = k0; k < k1; ++k) {
    float4 m4[kStMRow];
    #pragma unroll
    for (int i = 0; i < kStMRow; ++i) m4[i] = Mt[k * kStMRow + i];
    const float2 t2 = tb.t2[k][r];
    const float2 tx = make_float2(t2.x, t2.x), ty = make_float2(t2.y, t2.y), nty = make_float2(-t2.y, -t2.y);
    #pragma unroll
    for (int v = 0; v < QH / 2; ++v) {
      const float4 t1 = tb.t1[k][v0 + v];
      const float2 x = make_float2(t1.x, t1.y), y = make_float2(t1.z, t1.w);
      // P = px + i py; npy = -py by the sign bits
      const float2 px = ffma2(x, tx, fmul2(y, nty)), py = ffma2(x, ty, fmul2(y, tx));
      const float2 npy = make_float2(__uint_as_float(__float_as_uint(py.x) ^ 0x80000000u),
                                     __uint_as_float(__float_as_uint(py.y) ^ 0x80000000u));
      #pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 nr = make_float2(m4[e].x, m4[e].y), ni = make_float2(m4[e].z, m4[e].w);
        R.re[e][v] = ffma2(nr, px, ffma2(ni, py, R.re[e][v]));
        R.im[e][v] = ffma2(ni, px, ffma2(nr, npy, R.im[e][v]));
      }
    }
  }
}

// sum_c R(c) P(c) of this lane's source over nq tiles of the planes:
// out = (re 0, re 1), (re 2, re 3), (im 0, im 1), (im 2, im 3)
__device__ __forceinline__ void strip_average(const float4* __restrict__ pre, const float4* __restrict__ pim, int nq,
                                              PhaseAB p, const float2* lut, float2 (&out)[4]) {
  float2 t2[16];
  const unsigned b32 = step32(p.b);
  #pragma unroll
  for (int r = 0; r < 16; ++r) t2[r] = phasor_lut((unsigned)r * b32, lut);
  #pragma unroll
  for (int i = 0; i < 4; ++i) out[i] = make_float2(0.f, 0.f);
  const unsigned long long step = 16ull * p.b;
  unsigned long long ph = p.a;
  #pragma unroll 1
  for (int q = 0; q < nq; ++q, ph += step) {
    // s = u - w + i z: u = sum re tx, w = sum im ty, z = sum re ty + im tx
    float2 u0 = make_float2(0.f, 0.f), u1 = u0, w0 = u0, w1 = u0, z0 = u0, z1 = u0;
    #pragma unroll
    for (int r = 0; r < 16; ++r) {
      const float4 a = pre[16 * q + r], b = pim[16 * q + r];
      const float2 a0 = make_float2(a.x, a.y), a1 = make_float2(a.z, a.w);
      const float2 b0 = make_float2(b.x, b.y), b1 = make_float2(b.z, b.w);
      const float2 tx = make_float2(t2[r].x, t2[r].x), ty = make_float2(t2[r].y, t2[r].y);
      u0 = ffma2(a0, tx, u0); u1 = ffma2(a1, tx, u1);
      w0 = ffma2(b0, ty, w0); w1 = ffma2(b1, ty, w1);
      z0 = ffma2(b0, tx, ffma2(a0, ty, z0)); z1 = ffma2(b1, tx, ffma2(a1, ty, z1));
    }
    const float2 t1 = phasor_lut(ph, lut);
    const float2 x = make_float2(t1.x, t1.x), y = make_float2(t1.y, t1.y), ny = make_float2(-t1.y, -t1.y);
    const float2 s0 = make_float2(u0.x - w0.x, u0.y - w0.y), s1 = make_float2(u1.x - w1.x, u1.y - w1.y);
    out[0] = ffma2(s0, x, ffma2(z0, ny, out[0])); out[1] = ffma2(s1, x, ffma2(z1, ny, out[1]));
    out[2] = ffma2(s0, y, ffma2(z0, x, out[2])); out[3] = ffma2(s1, y, ffma2(z1, x, out[3]));
  }
}

// the strip of lane's channels from / to global memory (channels past n_chan are zero)
template <int QH>
__device__ __forceinline__ void strip_load(Strip<QH>& R, const float4* __restrict__ src, int n_chan, int lane) {
  const int c0 = 16 * (lane >> 4) * QH + (lane & 15);
  #pragma unroll
  for (int u = 0; u < QH; ++u) {
    const int c = c0 + 16 * u;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
    if (c < n_chan) { a = __ldcs(src + 2 * c); b = __ldcs(src + 2 * c + 1); }
    const float re[4] = {a.x, a.z, b.x, b.z}, im[4] = {a.y, a.w, b.y, b.w};
    #pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (u & 1) { R.re[e][u >> 1].y = re[e]; R.im[e][u >> 1].y = im[e]; }
      else { R.re[e][u >> 1].x = re[e]; R.im[e][u >> 1].x = im[e]; }
    }
  }
}
template <int QH>
__device__ __forceinline__ void strip_channel(const Strip<QH>& R, int u, float (&re)[4], float (&im)[4]) {
  #pragma unroll
  for (int e = 0; e < 4; ++e) {
    re[e] = u & 1 ? R.re[e][u >> 1].y : R.re[e][u >> 1].x;
    im[e] = u & 1 ? R.im[e][u >> 1].y : R.im[e][u >> 1].x;
  }
}
template <int QH>
__device__ __forceinline__ void strip_store(const Strip<QH>& R, float4* __restrict__ dst, int n_chan, int lane) {
  const int c0 = 16 * (lane >> 4) * QH + (lane & 15);
  #pragma unroll
  for (int u = 0; u < QH; ++u) {
    const int c = c0 + 16 * u;
    float re[4], im[4];
    strip_channel(R, u, re, im);
    if (c < n_chan) {
      __stcs(dst + 2 * c, make_float4(re[0], im[0], re[1], im[1]));
      __stcs(dst + 2 * c + 1, make_float4(re[2], im[2], re[3], im[3]));
    }
  }
}
// tiles start `PITCH` float4 apart
template <int QH, int PITCH = 16>
__device__ __forceinline__ void strip_planes(const Strip<QH>& R, float4* pre, float4* pim, int n_chan, int lane) {
  const int c0 = 16 * (lane >> 4) * QH + (lane & 15), at = PITCH * (lane >> 4) * QH + (lane & 15);
  #pragma unroll
  for (int u = 0; u < QH; ++u) {
    float re[4], im[4];
    strip_channel(R, u, re, im);
    const bool in = c0 + 16 * u < n_chan;          // channels past the strip hold no data
    pre[at + PITCH * u] = in ? make_float4(re[0], re[1], re[2], re[3]) : make_float4(0.f, 0.f, 0.f, 0.f);
    pim[at + PITCH * u] = in ? make_float4(im[0], im[1], im[2], im[3]) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// Warps of a CTA: `wpb` a baseline (times w, w + wpb, ...), `bpc` baselines.
struct StripGrid { int wpb, bpc; };
__host__ inline StripGrid strip_grid(int n_time) {
  StripGrid g;
  g.wpb = n_time < kStWarps ? n_time : kStWarps;
  g.bpc = kStWarps / g.wpb;
  return g;
}

// dynamic shared memory of the pass: sine table, model matrices, a workspace per
// warp (tables, then planes, then sums), and where a warp takes several times
// its running sums and their compensations [2][8][64]
constexpr size_t kStSumBytes = (size_t)8 * kBlkMax * sizeof(float);
template <int QH> size_t strip_pass_smem(const StripGrid& g, int n_time) {
  return 256 * sizeof(float2) + (size_t)g.bpc * kBlkMax * kStMRow * sizeof(float4) +
         (size_t)g.wpb * g.bpc * (strip_warp_bytes<QH>() + (n_time > g.wpb ? 2 * kStSumBytes : 0));
}

// The pass of the blocked peel (see block_kernels.cuh) on strips of at most 32 QH
// channels.  Bound by instruction issue and the FP32 pipe together: (20 + 17)
// multiply-adds per source and channel of both roles, two a packed instruction, and
// 41 instructions a phasor of the tables; 59 % of the FP32 pipe, 56 % of the issue
// slots and 65 % of the shared-memory pipe measured (128 channels).  Two CTAs an SM
// (<= 128 registers a thread): the loads and tables of one warp hide behind the
// multiply-adds of others.  Against the kernel it replaces on short strips
// (k_block_pass, FP32, one CTA a baseline): 3.9 / 4.2 / 4.6 / 5.9 / 6.2 ms.
// Two sources a lane in the average (half the broadcast reads) gave nothing: the
// registers it takes cost what it saves.
template <int QH, bool SUB, bool ACC>
__global__ void __launch_bounds__(kStWarps * 32, 2) k_block_pass_strip(BlockPassArgs a, int bk, StripGrid g) {
  extern __shared__ __align__(16) unsigned char st_smem[];
  float2* lut = reinterpret_cast<float2*>(st_smem);
  float4* Mt = reinterpret_cast<float4*>(lut + 256);                              // [bpc][64][kStMRow]
  unsigned char* ws0 = reinterpret_cast<unsigned char*>(Mt + (size_t)g.bpc * kBlkMax * kStMRow);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nthr = blockDim.x;
  const bool multi = a.n_time > g.wpb;
  unsigned char* ws = ws0 + (size_t)warp * strip_warp_bytes<QH>();
  float* keep = reinterpret_cast<float*>(ws0 + (size_t)g.wpb * g.bpc * strip_warp_bytes<QH>()) +
                (size_t)warp * 2 * 8 * kBlkMax;                                   // multi only
  StripTables<QH>& tb = *reinterpret_cast<StripTables<QH>*>(ws);
  float4* pre = reinterpret_cast<float4*>(ws);
  float4* pim = pre + 32 * QH;
  const int lb = warp / g.wpb, w = warp - lb * g.wpb;
  const int64_t bl0 = (int64_t)blockIdx.x * g.bpc, bl = bl0 + lb;
  const int nq = (a.n_chan + 15) >> 4, np = (nq + 1) >> 1;
  lut_fill(lut, tid, nthr);
  if (SUB)
    for (int i = tid; i < g.bpc * a.n_sub * 4; i += nthr) {
      const int e = i & 3, k = (i >> 2) % a.n_sub, b = (i >> 2) / a.n_sub;
      if (bl0 + b < a.n_bl)
        strip_pack_model(Mt + ((size_t)b * kBlkMax + k) * kStMRow, e, a.M_sub[((size_t)k * a.n_bl + bl0 + b) * 4 + e]);
    }
  __syncthreads();
  float2 y[2][4];                                    // sums of the sources lane and lane + 32
  #pragma unroll
  for (int s = 0; s < 2; ++s)
    #pragma unroll
    for (int i = 0; i < 4; ++i) y[s][i] = make_float2(0.f, 0.f);
  if (bl < a.n_bl) {
    for (int t = w; t < a.n_time; t += g.wpb) {
      const size_t strip = ((size_t)t * a.n_bl + bl) * a.n_chan * 2;
      const size_t ph = ((size_t)bl * a.n_time + t) * bk;
      {
        Strip<QH> R;
        strip_load(R, a.src + strip, a.n_chan, lane);
        if (SUB) {
          for (int k0 = 0; k0 < a.n_sub; k0 += kStGrp) {
            PhaseAB p;
            p.a = 0; p.b = 0;
            if (k0 + lane < a.n_sub) p = a.ph_sub[ph + k0 + lane];
            __syncwarp();
            strip_tables<QH>(tb, p, lane, np, lut);
            __syncwarp();
            strip_subtract<QH>(R, tb, Mt + ((size_t)lb * kBlkMax + k0) * kStMRow, 0, min(kStGrp, a.n_sub - k0), lane);
          }
          strip_store(R, a.dst + strip, a.n_chan, lane);
          __syncwarp();
        }
        if (ACC) strip_planes(R, pre, pim, a.n_chan, lane);
      }
      if (ACC) {
        __syncwarp();
        #pragma unroll
        for (int s = 0; s < 2; ++s) {
          if (32 * s >= a.n_acc) break;
          PhaseAB p;
          p.a = 0; p.b = 0;
          if (32 * s + lane < a.n_acc) p = a.ph_acc[ph + 32 * s + lane];
          strip_average(pre, pim, nq, p, lut, y[s]);
          if (multi) {                               // compensated sums over the warp's times
            #pragma unroll
            for (int i = 0; i < 8; ++i) {
              float* at = keep + i * kBlkMax + 32 * s + lane;
              float sum = t == w ? 0.f : at[0], comp = t == w ? 0.f : at[8 * kBlkMax];
              kahan_add(sum, comp, i & 1 ? y[s][i >> 1].y : y[s][i >> 1].x);
              at[0] = sum;
              at[8 * kBlkMax] = comp;
            }
          }
        }
        __syncwarp();                                // planes read before the next strip's tables
      }
    }
  }
  if (!ACC) return;
  // the warps' sums [8][64] and compensations at the head of their workspaces, added
  // in warp order with compensation
  float* mine = reinterpret_cast<float*>(ws);
  #pragma unroll
  for (int s = 0; s < 2; ++s)
    #pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int at = i * kBlkMax + 32 * s + lane;
      mine[at] = multi ? keep[at] : (i & 1 ? y[s][i >> 1].y : y[s][i >> 1].x);
      mine[8 * kBlkMax + at] = multi ? keep[8 * kBlkMax + at] : 0.f;
    }
  __syncthreads();
  const float inv = (float)a.inv_n, inv_lo = (float)(a.inv_n - (double)inv);
  for (int i = tid; i < g.bpc * a.n_acc * 8; i += nthr) {
    const int c = i & 7, k = (i >> 3) % a.n_acc, b = (i >> 3) / a.n_acc;      // c = 2 pol + (re, im)
    if (bl0 + b >= a.n_bl) continue;
    // plane of (pol, part): out[0] re 0 1, out[1] re 2 3, out[2] im 0 1, out[3] im 2 3
    const int pl = (c & 1) * 4 + (c >> 1);
    float sum = 0.f, comp = 0.f;
    for (int x = 0; x < g.wpb; ++x) {
      const float* o = reinterpret_cast<const float*>(ws0 + (size_t)(b * g.wpb + x) * strip_warp_bytes<QH>());
      kahan_add(sum, comp, o[pl * kBlkMax + k]);
      comp += o[(8 + pl) * kBlkMax + k];
    }
    // (sum - comp) inv_n, rounded once
    reinterpret_cast<float*>(a.avg)[((size_t)k * a.n_bl + bl0 + b) * 8 + c] =
        fmaf(sum, inv, fmaf(sum, inv_lo, -comp * inv));
  }
}

}  // namespace rts
