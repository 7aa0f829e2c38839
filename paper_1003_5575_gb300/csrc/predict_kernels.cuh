// Model prediction: vis (+)= sum over a chunk of sources of
// S_k J_i J_j^H exp(-2 pi i phi_k).  The FP32 sums over sources are compensated (term by
// term in k_predict_mixed, eight terms at a time in k_predict_strip), so a
// 1000-source prediction stays within a few ulp of the exact sum.
#pragma once
#include "stream_kernels.cuh"
#include "kahan.cuh"
#include "strip_kernels.cuh"

namespace rts {


constexpr int kPredictChunk = 32;

struct PredictArgs {
  void* vis;
  const double* uvw;
  const int2* bl_ant;
  const double* freq_c;
  const double* src;         // device [n_src][3] (l, m, S) of this chunk
  const void* jones;         // device [n_src][n_ant][4] (cube precision) of this chunk
  int n_src;                 // <= kPredictChunk
  int n_ant, n_chan, n_time;
  int64_t n_bl;
  double nu0_c, dnu_c;
  int accumulate;
};

__device__ inline SrcDir dev_dir(const double* s) {
  SrcDir d; d.l = s[0]; d.m = s[1]; d.S = s[2];
  double r2 = d.l * d.l + d.m * d.m;
  d.nm1 = -r2 / (1.0 + sqrt(1.0 - r2));
  return d;
}

__global__ void __launch_bounds__(kStreamThreads) k_predict_mixed(PredictArgs a) {
  extern __shared__ unsigned long long s_ab[];      // [n_time][n_src][2]
  __shared__ float2 s_M[kPredictChunk][4];    // -S_k J_i J_j^H
  const int64_t bl = blockIdx.x;
  const int2 ij = a.bl_ant[bl];
  for (int q = threadIdx.x; q < a.n_time * a.n_src; q += blockDim.x) {
    const int t = q / a.n_src, k = q - t * a.n_src;
    SrcDir d = dev_dir(a.src + 3 * k);
    double tau = delay_m(a.uvw, a.n_ant, t, ij.x, ij.y, d);
    s_ab[2 * q] = frac_q64(tau * a.nu0_c);
    s_ab[2 * q + 1] = frac_q64(tau * a.dnu_c);
  }
  for (int k = threadIdx.x; k < a.n_src; k += blockDim.x) {
    const float2* J = static_cast<const float2*>(a.jones) + (size_t)k * a.n_ant * 4;
    M22<double2> Ji, Jj;
    #pragma unroll
    for (int e = 0; e < 4; ++e) {
      float2 p = J[(size_t)ij.x * 4 + e], q = J[(size_t)ij.y * 4 + e];
      Ji.e[e] = make_double2(p.x, p.y); Jj.e[e] = make_double2(q.x, q.y);
    }
    M22<double2> P = mmul_h(Ji, Jj);
    const double S = a.src[3 * k + 2];
    #pragma unroll
    for (int e = 0; e < 4; ++e) s_M[k][e] = make_float2((float)(-S * P.e[e].x), (float)(-S * P.e[e].y));
  }
  __syncthreads();
  float4* vis = static_cast<float4*>(a.vis);
  const int n_s = a.n_time * a.n_chan;
  TCWalk w;
  w.init(threadIdx.x, a.n_chan);
  for (int s = threadIdx.x; s < n_s; s += kStreamThreads, w.next()) {
    const size_t idx = (((size_t)w.t * a.n_bl + bl) * a.n_chan + w.c) * 2;
    float sum[8], comp[8];
    if (a.accumulate) {
      const float4 x0 = vis[idx], x1 = vis[idx + 1];
      sum[0] = x0.x; sum[1] = x0.y; sum[2] = x0.z; sum[3] = x0.w;
      sum[4] = x1.x; sum[5] = x1.y; sum[6] = x1.z; sum[7] = x1.w;
    } else {
      #pragma unroll
      for (int e = 0; e < 8; ++e) sum[e] = 0.f;
    }
    #pragma unroll
    for (int e = 0; e < 8; ++e) comp[e] = 0.f;
    for (int k = 0; k < a.n_src; ++k) {
      const unsigned long long A = s_ab[2 * (w.t * a.n_src + k)];
      const unsigned long long B = s_ab[2 * (w.t * a.n_src + k) + 1];
      const float2 ph = phasor_f(q64_to_turns(A + (unsigned long long)w.c * B));
      #pragma unroll
      for (int e = 0; e < 4; ++e) {
        // term = M exp(-2 pi i phi) = M conj(ph); s_M holds -M
        const float2 nm = s_M[k][e];
        const float tr = -(nm.x * ph.x + nm.y * ph.y);
        const float ti = -(nm.y * ph.x - nm.x * ph.y);
        kahan_add(sum[2 * e], comp[2 * e], tr);
        kahan_add(sum[2 * e + 1], comp[2 * e + 1], ti);
      }
    }
    vis[idx] = make_float4(sum[0], sum[1], sum[2], sum[3]);
    vis[idx + 1] = make_float4(sum[4], sum[5], sum[6], sum[7]);
  }
}

// The FP32 prediction on strips (strip_kernels.cuh): a warp accumulates one
// (baseline, time, 32 QH channels) strip in registers, a launch takes up to
// kPredictStripSrc sources in two groups.  Against one hardware sin/cos and a
// compensated sum per (source, channel), about 60 instructions, it issues about
// 16: phasors as products of table entries, packed multiply-adds, sums compensated
// every kPredictSum sources: the remainder of the sum's rounding stays in the
// registers that the next sources are added up in (three packed operations, no
// third set of registers).  The cube is added exactly and the result rounded once.
// Model matrices by float-float products (as their FP64
// evaluation, rounded to FP32); phases as differences of the antennas' Q0.64
// phases (k_block_ant_phases).  Bound by instruction issue and the FP32 pipe: 20
// multiply-adds per source and channel, two an instruction.  100 sources into
// 128 antennas x 256 channels x 8 times: 2.00 ms, k_predict_mixed 4.01 ms; error
// against 64 bits 1.05e-7 of the rms (largest 0.9e-6) and 1.98e-7 (1.3e-6); with plain sums of
// 32 sources 1.88 ms, 1.86e-7 and 2.6e-6, compensated every four 2.17 ms.  Strips of 128
// channels (QH = 4): 64 registers hold the sum and its remainder.
constexpr int kPredictStripSrc = 2 * kStGrp;
constexpr int kPredictSum = 8;             // sources whose terms are added in plain FP32
// Antenna phases a handle keeps for predictions, at most: 1 KB per antenna and time,
// 4 MB for 512 antennas and 8 times.  Longer cubes (more than 131 072 antenna-times),
// and handles whose device has no room for them, take k_predict_mixed, which needs none.
constexpr size_t kPredictAphBytes = (size_t)128 << 20;

template <int QH> size_t predict_strip_smem(const StripGrid& g) {
  return 256 * sizeof(float2) + (size_t)g.bpc * kPredictStripSrc * kStMRow * sizeof(float4) +
         (size_t)g.wpb * g.bpc * sizeof(StripTables<QH>);
}

// a.n_src <= kPredictStripSrc; aph [n_time][n_ant][kPredictStripSrc]; n_tile tiles of 32 QH channels
template <int QH>
__global__ void __launch_bounds__(kStWarps * 32, 2) k_predict_strip(PredictArgs a, const PhaseAB* __restrict__ aph,
                                                                   StripGrid g, int n_tile) {
  extern __shared__ __align__(16) unsigned char ps_smem[];
  float2* lut = reinterpret_cast<float2*>(ps_smem);
  float4* Mt = reinterpret_cast<float4*>(lut + 256);                     // [bpc][kPredictStripSrc][kStMRow]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nthr = blockDim.x;
  StripTables<QH>& tb =
      reinterpret_cast<StripTables<QH>*>(Mt + (size_t)g.bpc * kPredictStripSrc * kStMRow)[warp];
  const int lb = warp / g.wpb, w = warp - lb * g.wpb;
  const int64_t bl0 = (int64_t)blockIdx.x * g.bpc, bl = bl0 + lb;
  lut_fill(lut, tid, nthr);
  for (int i = tid; i < g.bpc * a.n_src * 4; i += nthr) {
    const int e = i & 3, k = (i >> 2) % a.n_src, b = (i >> 2) / a.n_src;
    if (bl0 + b >= a.n_bl) continue;
    const int2 ij = a.bl_ant[bl0 + b];
    const size_t at = (size_t)k * a.n_ant;
    const double S = a.src[3 * k + 2];
    const float Sh = (float)S, Sl = (float)(S - (double)Sh);
    const float2 m = model_entry_ff(jones_row(a.jones, 2 * (at + ij.x) + (e >> 1)),
                                    jones_row(a.jones, 2 * (at + ij.y) + (e & 1)), Sh, Sl);
    strip_pack_model(Mt + ((size_t)b * kPredictStripSrc + k) * kStMRow, e, make_float2(-m.x, -m.y));
  }
  __syncthreads();
  if (bl >= a.n_bl) return;
  const int2 ij = a.bl_ant[bl];
  const int n_strip = a.n_time * n_tile;
  for (int s = w; s < n_strip; s += g.wpb) {
    const int t = s / n_tile, c0 = (s - t * n_tile) * 32 * QH, nc = min(32 * QH, a.n_chan - c0);
    const int np = (((nc + 15) >> 4) + 1) >> 1;
    Strip<QH> S, R;                            // the sum is S + R, R what S's rounding left and the present sources
    #pragma unroll
    for (int e = 0; e < 4; ++e)
      #pragma unroll
      for (int v = 0; v < QH / 2; ++v) S.re[e][v] = S.im[e][v] = R.re[e][v] = R.im[e][v] = make_float2(0.f, 0.f);
    for (int k0 = 0; k0 < a.n_src; k0 += kStGrp) {
      PhaseAB p;
      p.a = 0; p.b = 0;
      if (k0 + lane < a.n_src) {
        const PhaseAB pi = aph[((size_t)t * a.n_ant + ij.x) * kPredictStripSrc + k0 + lane];
        const PhaseAB pj = aph[((size_t)t * a.n_ant + ij.y) * kPredictStripSrc + k0 + lane];
        p.b = pi.b - pj.b;
        p.a = pi.a - pj.a + (unsigned long long)c0 * p.b;
      }
      __syncwarp();
      strip_tables<QH>(tb, p, lane, np, lut);
      __syncwarp();
      const int n_grp = min(kStGrp, a.n_src - k0);
      #pragma unroll 1
      for (int k1 = 0; k1 < n_grp; k1 += kPredictSum) {
        strip_subtract<QH>(R, tb, Mt + ((size_t)lb * kPredictStripSrc + k0) * kStMRow, k1, min(k1 + kPredictSum, n_grp), lane);
        #pragma unroll
        for (int e = 0; e < 4; ++e)
          #pragma unroll
          for (int v = 0; v < QH / 2; ++v) {
            kahan_carry2(S.re[e][v], R.re[e][v]);
            kahan_carry2(S.im[e][v], R.im[e][v]);
          }
      }
    }
    float4* vis = static_cast<float4*>(a.vis) + (((size_t)t * a.n_bl + bl) * a.n_chan + c0) * 2;
    const int cl = 16 * (lane >> 4) * QH + (lane & 15);
    #pragma unroll
    for (int u = 0; u < QH; ++u) {
      const int c = cl + 16 * u;
      if (c >= nc) continue;
      float re[4], im[4], lr[4], li[4];
      strip_channel(S, u, re, im);
      strip_channel(R, u, lr, li);
      float4 x0 = make_float4(0.f, 0.f, 0.f, 0.f), x1 = x0;
      if (a.accumulate) { x0 = __ldcs(vis + 2 * c); x1 = __ldcs(vis + 2 * c + 1); }
      auto sum = [](float x, float s, float r) {           // x + s + r, rounded once (an infinite x stays one)
        const FF o = ff_two_sum(x, s);
        return isfinite(o.hi) ? o.hi + (o.lo + r) : o.hi;
      };
      __stcs(vis + 2 * c, make_float4(sum(x0.x, re[0], lr[0]), sum(x0.y, im[0], li[0]), sum(x0.z, re[1], lr[1]),
                                     sum(x0.w, im[1], li[1])));
      __stcs(vis + 2 * c + 1, make_float4(sum(x1.x, re[2], lr[2]), sum(x1.y, im[2], li[2]), sum(x1.z, re[3], lr[3]),
                                         sum(x1.w, im[3], li[3])));
    }
  }
}

__global__ void __launch_bounds__(kStreamThreads) k_predict_fp64(PredictArgs a) {
  extern __shared__ double s_tau64[];               // [n_time][n_src]
  __shared__ double2 s_M64[kPredictChunk][4];
  const int64_t bl = blockIdx.x;
  const int2 ij = a.bl_ant[bl];
  for (int q = threadIdx.x; q < a.n_time * a.n_src; q += blockDim.x) {
    const int t = q / a.n_src, k = q - t * a.n_src;
    SrcDir d = dev_dir(a.src + 3 * k);
    s_tau64[q] = delay_m(a.uvw, a.n_ant, t, ij.x, ij.y, d);
  }
  for (int k = threadIdx.x; k < a.n_src; k += blockDim.x) {
    const double2* J = static_cast<const double2*>(a.jones) + (size_t)k * a.n_ant * 4;
    M22<double2> Ji, Jj;
    #pragma unroll
    for (int e = 0; e < 4; ++e) { Ji.e[e] = J[(size_t)ij.x * 4 + e]; Jj.e[e] = J[(size_t)ij.y * 4 + e]; }
    M22<double2> P = mmul_h(Ji, Jj);
    const double S = a.src[3 * k + 2];
    #pragma unroll
    for (int e = 0; e < 4; ++e) s_M64[k][e] = make_double2(S * P.e[e].x, S * P.e[e].y);
  }
  __syncthreads();
  double2* vis = static_cast<double2*>(a.vis);
  const int n_s = a.n_time * a.n_chan;
  TCWalk w;
  w.init(threadIdx.x, a.n_chan);
  for (int s = threadIdx.x; s < n_s; s += kStreamThreads, w.next()) {
    const size_t idx = (((size_t)w.t * a.n_bl + bl) * a.n_chan + w.c) * 4;
    double2 x[4];
    #pragma unroll
    for (int e = 0; e < 4; ++e) x[e] = a.accumulate ? vis[idx + e] : make_double2(0.0, 0.0);
    for (int k = 0; k < a.n_src; ++k) {
      double2 ph = phasor_d(s_tau64[w.t * a.n_src + k] * a.freq_c[w.c]);
      #pragma unroll
      for (int e = 0; e < 4; ++e) x[e] = cadd(x[e], cmulc(s_M64[k][e], ph));
    }
    #pragma unroll
    for (int e = 0; e < 4; ++e) vis[idx + e] = x[e];
  }
}

}  // namespace rts
