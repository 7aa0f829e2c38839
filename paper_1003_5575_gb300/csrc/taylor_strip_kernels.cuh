// The Taylor pass of the blocked schedule (taylor_block_kernels.cuh) on strips of at
// most 256 channels (strip_kernels.cuh): subtract a block's models
// (P0 + x_c P1 + x_c^2 P2) e^{-2 pi i phi} and take the next block's three moments
// mean x_c^n R e^{+2 pi i phi}.  The tcgen05 form spends the operand formation of 64
// sources a strip on 21; here a (source, channel) pair costs 36 multiply-adds in
// the subtraction (the model evaluated at x_c, two packed Horner steps) and 32 in
// the averages: with c = 16 q + r and x_c = u_q + r dx, running sums while r runs
// down give s0 = sum x_r, s1 = sum (r + 1) x_r, s2 = sum (r + 1)(r + 2)/2 x_r of
// x_r = R(16 q + r) T2[r], and sum r x_r = s1 - s0, sum r^2 x_r = 2 s2 - 3 s1 + s0.
// Bound by the FP32 pipe and instruction issue.  At 128 antennas x 128 channels x 8
// times and 50 sources the four passes take 2.15 ms, the tcgen05 form's 7.3; past 256
// channels a strip no longer fits a warp's registers and the tcgen05 form keeps the pass.
#pragma once
#include "strip_kernels.cuh"
#include "taylor_block_kernels.cuh"

namespace rts {

constexpr int kTsModel = 12;               // float4 of a source's packed P0, P1, P2 (entry-major)
constexpr int kTsSums = 24;                // values of a source's three moments

// R -= sum_{k < n} (P0 + x (P1 + x P2)) conj(P_k), Pt packed [n][entry][power]
template <int QH>
__device__ __forceinline__ void taylor_strip_subtract(Strip<QH>& R, const StripTables<QH>& tb,
                                                      const float4* __restrict__ Pt, int n, float x0, float dx, int lane) {
  const int r = lane & 15, h = lane >> 4, v0 = h * (QH / 2);
  #pragma unroll 1
  for (int k = 0; k < n; ++k) {
    const float2 t2 = tb.t2[k][r];
    const float2 tx = make_float2(t2.x, t2.x), ty = make_float2(t2.y, t2.y), nty = make_float2(-t2.y, -t2.y);
    float2 px[QH / 2], py[QH / 2];
    #pragma unroll
    for (int v = 0; v < QH / 2; ++v) {
      const float4 t1 = tb.t1[k][v0 + v];
      const float2 a = make_float2(t1.x, t1.y), b = make_float2(t1.z, t1.w);
      px[v] = ffma2(a, tx, fmul2(b, nty));
      py[v] = ffma2(a, ty, fmul2(b, tx));
    }
    #pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float4 p0 = Pt[(size_t)k * kTsModel + 3 * e], p1 = Pt[(size_t)k * kTsModel + 3 * e + 1],
                   p2 = Pt[(size_t)k * kTsModel + 3 * e + 2];
      const float2 r0 = make_float2(p0.x, p0.y), i0 = make_float2(p0.z, p0.w), r1 = make_float2(p1.x, p1.y);
      const float2 i1 = make_float2(p1.z, p1.w), r2 = make_float2(p2.x, p2.y), i2 = make_float2(p2.z, p2.w);
      #pragma unroll
      for (int v = 0; v < QH / 2; ++v) {
        const float c = (float)(16 * (QH * h + 2 * v) + r);
        const float2 x = make_float2(fmaf(c, dx, x0), fmaf(c + 16.f, dx, x0));
        const float2 nr = ffma2(x, ffma2(x, r2, r1), r0), ni = ffma2(x, ffma2(x, i2, i1), i0);
        const float2 npy = make_float2(__uint_as_float(__float_as_uint(py[v].x) ^ 0x80000000u),
                                       __uint_as_float(__float_as_uint(py[v].y) ^ 0x80000000u));
        R.re[e][v] = ffma2(nr, px[v], ffma2(ni, py[v], R.re[e][v]));
        R.im[e][v] = ffma2(ni, px[v], ffma2(nr, npy, R.im[e][v]));
      }
    }
  }
}

// this lane's source: out[n] = sum_c x_c^n R(c) P(c) as (re 0, re 1), (re 2, re 3), (im ..)
__device__ __forceinline__ void taylor_strip_average(const float4* __restrict__ pre, const float4* __restrict__ pim,
                                                     int nq, float x0, float dx, PhaseAB p, const float2* lut,
                                                     float2 (&out)[3][4]) {
  float2 t2[16];
  const unsigned b32 = step32(p.b);
  #pragma unroll
  for (int r = 0; r < 16; ++r) t2[r] = phasor_lut((unsigned)r * b32, lut);
  #pragma unroll
  for (int n = 0; n < 3; ++n)
    #pragma unroll
    for (int i = 0; i < 4; ++i) out[n][i] = make_float2(0.f, 0.f);
  const unsigned long long step = 16ull * p.b;
  unsigned long long ph = p.a;
  #pragma unroll 1
  for (int q = 0; q < nq; ++q, ph += step) {
    float2 s0[4], s1[4], s2[4];
    #pragma unroll
    for (int i = 0; i < 4; ++i) s0[i] = s1[i] = s2[i] = make_float2(0.f, 0.f);
    #pragma unroll
    for (int r = 15; r >= 0; --r) {
      const float4 a = pre[16 * q + r], b = pim[16 * q + r];
      const float2 a0 = make_float2(a.x, a.y), a1 = make_float2(a.z, a.w);
      const float2 b0 = make_float2(b.x, b.y), b1 = make_float2(b.z, b.w);
      const float2 tx = make_float2(t2[r].x, t2[r].x), ty = make_float2(t2[r].y, t2[r].y);
      const float ny = __uint_as_float(__float_as_uint(t2[r].y) ^ 0x80000000u);
      const float2 nty = make_float2(ny, ny);
      s0[0] = ffma2(a0, tx, ffma2(b0, nty, s0[0]));
      s0[1] = ffma2(a1, tx, ffma2(b1, nty, s0[1]));
      s0[2] = ffma2(a0, ty, ffma2(b0, tx, s0[2]));
      s0[3] = ffma2(a1, ty, ffma2(b1, tx, s0[3]));
      #pragma unroll
      for (int i = 0; i < 4; ++i) {
        s1[i] = fadd2(s1[i], s0[i]);
        s2[i] = fadd2(s2[i], s1[i]);
      }
    }
    const float2 t1 = phasor_lut(ph, lut);
    const float2 x = make_float2(t1.x, t1.x), y = make_float2(t1.y, t1.y), ny = make_float2(-t1.y, -t1.y);
    const float u = fmaf((float)(16 * q), dx, x0);
    // sums of 1, x_c, x_c^2 times x_r over the tile
    float2 m1[4], m2[4];
    #pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 d1 = make_float2(s1[i].x - s0[i].x, s1[i].y - s0[i].y);                        // sum r x_r
      const float2 d2 = make_float2(fmaf(2.f, s2[i].x, fmaf(-3.f, s1[i].x, s0[i].x)),
                                    fmaf(2.f, s2[i].y, fmaf(-3.f, s1[i].y, s0[i].y)));              // sum r^2 x_r
      m1[i] = make_float2(fmaf(u, s0[i].x, dx * d1.x), fmaf(u, s0[i].y, dx * d1.y));
      const float ud = 2.f * u * dx, dd = dx * dx, uu = u * u;
      m2[i] = make_float2(fmaf(uu, s0[i].x, fmaf(ud, d1.x, dd * d2.x)), fmaf(uu, s0[i].y, fmaf(ud, d1.y, dd * d2.y)));
    }
    #pragma unroll
    for (int i = 0; i < 2; ++i) {
      out[0][i] = ffma2(s0[i], x, ffma2(s0[2 + i], ny, out[0][i]));
      out[0][2 + i] = ffma2(s0[i], y, ffma2(s0[2 + i], x, out[0][2 + i]));
      out[1][i] = ffma2(m1[i], x, ffma2(m1[2 + i], ny, out[1][i]));
      out[1][2 + i] = ffma2(m1[i], y, ffma2(m1[2 + i], x, out[1][2 + i]));
      out[2][i] = ffma2(m2[i], x, ffma2(m2[2 + i], ny, out[2][i]));
      out[2][2 + i] = ffma2(m2[i], y, ffma2(m2[2 + i], x, out[2][2 + i]));
    }
  }
}

// sine table, models [bpc][kTayBlk][kTsModel], a workspace per warp, and where a warp
// takes several times its running sums and compensations [2][kTsSums][32]
constexpr size_t kTsSumBytes = (size_t)kTsSums * 32 * sizeof(float);
template <int QH> size_t taylor_strip_smem(const StripGrid& g, int n_time) {
  return 256 * sizeof(float2) + (size_t)g.bpc * kTayBlk * kTsModel * sizeof(float4) +
         (size_t)g.wpb * g.bpc * (strip_warp_bytes<QH>() + (n_time > g.wpb ? 2 * kTsSumBytes : 0));
}

// a.n_sub, a.n_acc <= kTayBlk; phases with a stride of bk sources
template <int QH, bool SUB, bool ACC>
__global__ void __launch_bounds__(kStWarps * 32, 2) k_taylor_pass_strip(BlockPassArgs a, int bk, StripGrid g) {
  extern __shared__ __align__(16) unsigned char st_smem[];
  float2* lut = reinterpret_cast<float2*>(st_smem);
  float4* Pt = reinterpret_cast<float4*>(lut + 256);                              // [bpc][kTayBlk][kTsModel]
  unsigned char* ws0 = reinterpret_cast<unsigned char*>(Pt + (size_t)g.bpc * kTayBlk * kTsModel);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nthr = blockDim.x;
  const bool multi = a.n_time > g.wpb;
  unsigned char* ws = ws0 + (size_t)warp * strip_warp_bytes<QH>();
  float* keep = reinterpret_cast<float*>(ws0 + (size_t)g.wpb * g.bpc * strip_warp_bytes<QH>()) +
                (size_t)warp * 2 * kTsSums * 32;                                  // multi only
  StripTables<QH>& tb = *reinterpret_cast<StripTables<QH>*>(ws);
  float4* pre = reinterpret_cast<float4*>(ws);
  float4* pim = pre + 32 * QH;
  const int lb = warp / g.wpb, w = warp - lb * g.wpb;
  const int64_t bl0 = (int64_t)blockIdx.x * g.bpc, bl = bl0 + lb;
  const int nq = (a.n_chan + 15) >> 4, np = (nq + 1) >> 1;
  lut_fill(lut, tid, nthr);
  if (SUB)
    for (int i = tid; i < g.bpc * a.n_sub * 12; i += nthr) {
      const int x = i % 12, n = x >> 2, e = x & 3, k = (i / 12) % a.n_sub, b = (i / 12) / a.n_sub;
      if (bl0 + b >= a.n_bl) continue;
      const float2 m = a.M_sub[((size_t)(3 * k + n) * a.n_bl + bl0 + b) * 4 + e];
      strip_pack_model(Pt + ((size_t)b * kTayBlk + k) * kTsModel, 3 * e + n, m);
    }
  __syncthreads();
  float2 y[3][4];
  #pragma unroll
  for (int n = 0; n < 3; ++n)
    #pragma unroll
    for (int i = 0; i < 4; ++i) y[n][i] = make_float2(0.f, 0.f);
  auto val = [&](int i) {                            // value i = 8 n + 2 j + part of y
    const float2 v = y[i >> 3][(i & 7) >> 1];
    return i & 1 ? v.y : v.x;
  };
  if (bl < a.n_bl) {
    for (int t = w; t < a.n_time; t += g.wpb) {
      const size_t strip = ((size_t)t * a.n_bl + bl) * a.n_chan * 2;
      const size_t ph = ((size_t)bl * a.n_time + t) * bk;
      auto phase = [&](const PhaseAB* tab, int n) {
        PhaseAB p;
        p.a = 0; p.b = 0;
        if (lane < n) p = tab[ph + lane];
        return p;
      };
      {
        Strip<QH> R;
        strip_load(R, a.src + strip, a.n_chan, lane);
        if (SUB) {
          const PhaseAB p = phase(a.ph_sub, a.n_sub);
          __syncwarp();
          strip_tables<QH>(tb, p, lane, np, lut);
          __syncwarp();
          taylor_strip_subtract<QH>(R, tb, Pt + (size_t)lb * kTayBlk * kTsModel, a.n_sub, a.tx0, a.tdx, lane);
          strip_store(R, a.dst + strip, a.n_chan, lane);
          __syncwarp();
        }
        if (ACC) strip_planes(R, pre, pim, a.n_chan, lane);
      }
      if (ACC) {
        __syncwarp();
        taylor_strip_average(pre, pim, nq, a.tx0, a.tdx, phase(a.ph_acc, a.n_acc), lut, y);
        if (multi) {                                 // compensated sums over the warp's times
          #pragma unroll
          for (int i = 0; i < kTsSums; ++i) {
            float* at = keep + i * 32 + lane;
            float sum = t == w ? 0.f : at[0], comp = t == w ? 0.f : at[kTsSums * 32];
            kahan_add(sum, comp, val(i));
            at[0] = sum;
            at[kTsSums * 32] = comp;
          }
        }
        __syncwarp();                                // planes read before the next strip's tables
      }
    }
  }
  if (!ACC) return;
  // the warps' sums [kTsSums][32] (and compensations) at the head of their workspaces,
  // added in warp order with compensation
  float* mine = reinterpret_cast<float*>(ws);
  #pragma unroll
  for (int i = 0; i < kTsSums; ++i) {
    mine[i * 32 + lane] = multi ? keep[i * 32 + lane] : val(i);
    if (multi) mine[(kTsSums + i) * 32 + lane] = keep[(kTsSums + i) * 32 + lane];
  }
  __syncthreads();
  const float inv = (float)a.inv_n, inv_lo = (float)(a.inv_n - (double)inv);
  for (int i = tid; i < g.bpc * a.n_acc * kTsSums; i += nthr) {
    const int c = i % kTsSums, n = c >> 3, o = c & 7, k = (i / kTsSums) % a.n_acc, b = (i / kTsSums) / a.n_acc;
    if (bl0 + b >= a.n_bl) continue;
    // output o = 2 pol + (re, im) of moment n: value 8 n + 4 (re, im) + pol
    const int at = (8 * n + (o & 1) * 4 + (o >> 1)) * 32 + k;
    float sum = 0.f, comp = 0.f;
    for (int x = 0; x < g.wpb; ++x) {
      const float* s = reinterpret_cast<const float*>(ws0 + (size_t)(b * g.wpb + x) * strip_warp_bytes<QH>());
      kahan_add(sum, comp, s[at]);
      if (multi) comp += s[kTsSums * 32 + at];
    }
    reinterpret_cast<float*>(a.avg)[((size_t)(3 * k + n) * a.n_bl + bl0 + b) * 8 + o] =
        fmaf(sum, inv, fmaf(sum, inv_lo, -comp * inv));
  }
}

}  // namespace rts
