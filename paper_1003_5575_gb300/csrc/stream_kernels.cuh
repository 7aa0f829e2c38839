// Streaming kernels over the visibility cube vis[t][bl][c][4]:
//   rotate + average      (the average step of one source)
//   subtract + average    (subtract source k, average for source k+1, one pass)
//   subtract              (last source)
// One CTA per baseline: its N_t strips of N_c contiguous visibilities are read
// with coalesced 16-byte loads (consecutive threads = consecutive channels) and
// its average is reduced in the CTA (warp shuffles, FP64 across warps), so no
// atomics and a deterministic result.
#pragma once
#include "common.cuh"

namespace rts {

constexpr int kStreamThreads = 256;
constexpr int kStreamBatch = 4;   // visibilities in flight per thread

struct StreamArgs {
  const void* src;          // cube read
  void* dst;                // cube written (may equal src)
  const double* uvw;        // [n_time][n_ant][3]
  const int2* bl_ant;       // [n_bl] (i, j)
  const double* freq_c;     // [n_chan] nu_c / c_light (per metre), FP64 path only
  int n_ant, n_chan, n_time;
  int64_t n_bl;
  double nu0_c, dnu_c;      // nu_0 / c and dnu / c (per metre)
  SrcDir sub;               // source subtracted
  const double2* Jsub;      // its FP64 Jones [n_ant][4]
  SrcDir acc;               // source averaged
  void* avg;                // [n_bl][4] complex (cube precision)
  double inv_n;             // 1 / (n_time n_chan)
};

// ---------------------------------------------------------------------------
// reductions

template <int N>
__device__ inline void block_sum_f32_to_f64(float (&v)[N], double* s_red /* [32][N] */,
                                            double (&out)[N]) {
  #pragma unroll
  for (int k = 0; k < N; ++k)
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0)
    #pragma unroll
    for (int k = 0; k < N; ++k) s_red[warp * N + k] = (double)v[k];
  __syncthreads();
  if (threadIdx.x == 0) {
    const int nw = blockDim.x >> 5;
    #pragma unroll
    for (int k = 0; k < N; ++k) {
      double s = 0.0;
      for (int w = 0; w < nw; ++w) s += s_red[w * N + k];
      out[k] = s;
    }
  }
}

// (t, c) walk of one thread: s = t*n_chan + c advanced by kStreamThreads
struct TCWalk {
  int t, c, dt, dc, n_chan;
  __device__ inline void init(int s0, int n_chan_) {
    n_chan = n_chan_;
    t = s0 / n_chan; c = s0 - t * n_chan;
    dt = kStreamThreads / n_chan; dc = kStreamThreads - dt * n_chan;
  }
  __device__ inline void next() {
    c += dc; t += dt;
    if (c >= n_chan) { c -= n_chan; ++t; }
  }
};

// ---------------------------------------------------------------------------
// mixed precision: complex64 cube, Q0.64 phases, FP32 arithmetic

// x -= M * exp(-2 pi i phi)  on the 4 complex of one visibility
__device__ inline void sub_model(float4& x0, float4& x1, const float2 (&M)[4], float2 ph) {
  // ph = exp(+2 pi i phi); model term M * conj(ph)
  x0.x -= M[0].x * ph.x + M[0].y * ph.y;  x0.y -= M[0].y * ph.x - M[0].x * ph.y;
  x0.z -= M[1].x * ph.x + M[1].y * ph.y;  x0.w -= M[1].y * ph.x - M[1].x * ph.y;
  x1.x -= M[2].x * ph.x + M[2].y * ph.y;  x1.y -= M[2].y * ph.x - M[2].x * ph.y;
  x1.z -= M[3].x * ph.x + M[3].y * ph.y;  x1.w -= M[3].y * ph.x - M[3].x * ph.y;
}
// acc += x * exp(+2 pi i phi)
__device__ inline void acc_rot(float (&a)[8], const float4& x0, const float4& x1, float2 ph) {
  a[0] += x0.x * ph.x - x0.y * ph.y;  a[1] += x0.x * ph.y + x0.y * ph.x;
  a[2] += x0.z * ph.x - x0.w * ph.y;  a[3] += x0.z * ph.y + x0.w * ph.x;
  a[4] += x1.x * ph.x - x1.y * ph.y;  a[5] += x1.x * ph.y + x1.y * ph.x;
  a[6] += x1.z * ph.x - x1.w * ph.y;  a[7] += x1.z * ph.y + x1.w * ph.x;
}

__device__ inline void model_matrix_f(const double2* __restrict__ J, int n_ant, int i, int j,
                                      double S, float2 (&M)[4]) {
  M22<double2> Ji, Jj;
  #pragma unroll
  for (int e = 0; e < 4; ++e) { Ji.e[e] = J[(size_t)i * 4 + e]; Jj.e[e] = J[(size_t)j * 4 + e]; }
  M22<double2> P = mmul_h(Ji, Jj);
  #pragma unroll
  for (int e = 0; e < 4; ++e) M[e] = make_float2((float)(S * P.e[e].x), (float)(S * P.e[e].y));
}

template <bool SUB, bool ACC>
__global__ void __launch_bounds__(kStreamThreads, 3) k_stream_mixed(StreamArgs a) {
  extern __shared__ unsigned long long s_ph[];   // [n_time][4]: A_sub B_sub A_acc B_acc
  __shared__ float2 s_M[4];
  __shared__ double s_red[(kStreamThreads / 32) * 8];
  const int64_t bl = blockIdx.x;
  const int2 ij = a.bl_ant[bl];
  for (int t = threadIdx.x; t < a.n_time; t += blockDim.x) {
    if (SUB) {
      double tau = delay_m(a.uvw, a.n_ant, t, ij.x, ij.y, a.sub);
      s_ph[4 * t + 0] = frac_q64(tau * a.nu0_c);
      s_ph[4 * t + 1] = frac_q64(tau * a.dnu_c);
    }
    if (ACC) {
      double tau = delay_m(a.uvw, a.n_ant, t, ij.x, ij.y, a.acc);
      s_ph[4 * t + 2] = frac_q64(tau * a.nu0_c);
      s_ph[4 * t + 3] = frac_q64(tau * a.dnu_c);
    }
  }
  if (SUB && threadIdx.x == 0) {
    float2 M[4];
    model_matrix_f(a.Jsub, a.n_ant, ij.x, ij.y, a.sub.S, M);
    #pragma unroll
    for (int e = 0; e < 4; ++e) s_M[e] = M[e];
  }
  __syncthreads();
  float2 M[4];
  if (SUB) {
    #pragma unroll
    for (int e = 0; e < 4; ++e) M[e] = s_M[e];
  }
  float acc[8];
  #pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = 0.f;

  const float4* src = static_cast<const float4*>(a.src);   // may alias dst (in place)
  float4* dst = static_cast<float4*>(a.dst);
  const int n_s = a.n_time * a.n_chan;
  TCWalk w;
  w.init(threadIdx.x, a.n_chan);
  for (int s0 = threadIdx.x; s0 < n_s; s0 += kStreamBatch * kStreamThreads) {
    float4 x0[kStreamBatch], x1[kStreamBatch];
    int tt[kStreamBatch], cc[kStreamBatch];
    size_t idx[kStreamBatch];
    #pragma unroll
    for (int u = 0; u < kStreamBatch; ++u) {
      tt[u] = w.t; cc[u] = w.c;
      idx[u] = (((size_t)w.t * a.n_bl + bl) * a.n_chan + w.c) * 2;
      if (s0 + u * kStreamThreads < n_s) {
        x0[u] = __ldcs(src + idx[u]);
        x1[u] = __ldcs(src + idx[u] + 1);
      }
      w.next();
    }
    #pragma unroll
    for (int u = 0; u < kStreamBatch; ++u) {
      if (s0 + u * kStreamThreads < n_s) {
        if (SUB) {
          const unsigned long long A = s_ph[4 * tt[u]], B = s_ph[4 * tt[u] + 1];
          float2 ph = phasor_f(q64_to_turns(A + (unsigned long long)cc[u] * B));
          sub_model(x0[u], x1[u], M, ph);
          __stcs(dst + idx[u], x0[u]);
          __stcs(dst + idx[u] + 1, x1[u]);
        }
        if (ACC) {
          const unsigned long long A = s_ph[4 * tt[u] + 2], B = s_ph[4 * tt[u] + 3];
          float2 ph = phasor_f(q64_to_turns(A + (unsigned long long)cc[u] * B));
          acc_rot(acc, x0[u], x1[u], ph);
        }
      }
    }
  }
  if (ACC) {
    double tot[8];
    block_sum_f32_to_f64<8>(acc, s_red, tot);
    if (threadIdx.x == 0) {
      float4* out = static_cast<float4*>(a.avg) + bl * 2;
      out[0] = make_float4((float)(tot[0] * a.inv_n), (float)(tot[1] * a.inv_n),
                           (float)(tot[2] * a.inv_n), (float)(tot[3] * a.inv_n));
      out[1] = make_float4((float)(tot[4] * a.inv_n), (float)(tot[5] * a.inv_n),
                           (float)(tot[6] * a.inv_n), (float)(tot[7] * a.inv_n));
    }
  }
}

// ---------------------------------------------------------------------------
// plain FP64: complex128 cube, FP64 sincospi, FP64 arithmetic
//
// GB300 retires about 1.7 FP64 fused multiply-adds a cycle and SM (19 cycles a
// warp instruction), so the pass is bound by how many it issues: 32 a sample
// are the two roles' four complex multiply-adds each, written as fused chains;
// two sincospi a sample would be about 80 more.  Where the channels are uniform
// to FP64 rounding the phasor is therefore a product of table entries instead
// (4 more a role): channel c = R q + r has e^{2 pi i tau nu_c / c} = T1[q] T2[r]
// with T1[q] = e^{2 pi i tau (nu_0 + R q dnu) / c}, T2[r] = e^{2 pi i tau r dnu / c},
// and, because tau_ij = tau_i - tau_j, each table of a baseline is the product
// T_i conj(T_j) of its antennas' tables, which k_fp64_ant_tables forms once per
// source ([n_time][n_ant][Q + R]).  At 128 antennas x 128 channels x 8 times x 50
// sources the whole cadence, solves included, went from 111 ms to 34.1.  Other
// frequency lists (uniform to 1e-9 only) keep one sincospi per sample and role
// (k_stream_fp64).

constexpr size_t kFp64TableBytes = 32 * 1024;    // a CTA's baseline tables, at most (but one time's)

// R of the tables: about sqrt(n_chan), a power of two, at most kFp64Threads
__host__ inline int fp64_table_r(int n_chan) {
  int r = 1;
  while (r * r < n_chan && r < 128) r *= 2;
  return r;
}

// [n_time][n_ant][Q + R]: T1 then T2 of one source direction.  The delays are those of
// u_i - u_0: only differences of coordinates mean anything, so their origin may be far
// from the array, and from a geocentric one (6.4e6 m) the phases of u_i itself are off by
// up to 8.6e-10 radian.  Differences, delay, frequency and their product are pairs of
// doubles: an antenna's error is common to all of its baselines and so goes whole into
// its gains, where a baseline's own rounding averages out.  *_lo: what nu0 / c and
// dnu / c leave after their rounding.
struct Fp64Freq { double nu0, nu0_lo, dnu, dnu_lo; };
__global__ void __launch_bounds__(256) k_fp64_ant_tables(const double* __restrict__ uvw, SrcDir d, int n_ant,
                                                        int n_time, int Q, int R, Fp64Freq f,
                                                        double2* __restrict__ tab) {
  const int n_e = Q + R;
  const int64_t n = (int64_t)n_time * n_ant * n_e;
  // hi + lo = a + b
  auto two_sum = [](double a, double b, double& lo) {
    const double s = a + b, bb = s - a;
    lo += (a - (s - bb)) + (b - bb);
    return s;
  };
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
    const int64_t ta = x / n_e;
    const int e = (int)(x - ta * n_e);
    const double *u = uvw + ta * 3, *u0 = uvw + ta / n_ant * n_ant * 3;
    double tl = 0.0, th = 0.0;
    const double dir[3] = {d.l, d.m, d.nm1};
    #pragma unroll
    for (int i = 0; i < 3; ++i) {
      double dl = 0.0;
      const double dh = two_sum(u[i], -u0[i], dl), p = __dmul_rn(dh, dir[i]);
      tl += fma(dh, dir[i], -p) + dl * dir[i];
      th = two_sum(th, p, tl);
    }
    const double k = (double)(e < Q ? R * e : e - Q), s = __dmul_rn(k, f.dnu);
    double fl = fma(k, f.dnu, -s) + k * f.dnu_lo, fh = s;
    if (e < Q) {
      fl += f.nu0_lo;
      fh = two_sum(f.nu0, s, fl);
    }
    const double p = __dmul_rn(th, fh);
    tab[x] = phasor_d((p - rint(p)) + (fma(th, fh, -p) + fma(th, fl, tl * fh)));
  }
}

struct Fp64Tables {
  const double2* sub;       // [n_time][n_ant][Q + R] of the subtracted source
  const double2* acc;       // of the averaged source
  int Q, R, lr;             // R = 1 << lr
  int n_t;                  // times whose baseline tables a CTA holds at once
};

// -S J_i J_j^H of the subtracted source, one entry a thread
__device__ __forceinline__ void fp64_model(const StreamArgs& a, int2 ij, int tid, double2* s_M) {
  if (tid < 4) {
    const int r = tid >> 1, c = tid & 1;
    const double2 *Ji = a.Jsub + (size_t)ij.x * 4 + 2 * r, *Jj = a.Jsub + (size_t)ij.y * 4 + 2 * c;
    const double2 m = cadd(cmulc(Ji[0], Jj[0]), cmulc(Ji[1], Jj[1]));
    s_M[tid] = make_double2(-a.sub.S * m.x, -a.sub.S * m.y);
  }
}
// a CTA's averages: warp totals by halving exchanges (9 additions a lane for the 8 sums),
// then one thread a sum adds the warps' in warp order
template <int WARPS>
__device__ __forceinline__ void fp64_average(const StreamArgs& a, int64_t bl, double (&acc)[8], double (*s_red)[8]) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const double v = warp_reduce_scatter8d(acc, lane);
  if ((lane & 3) == 0) s_red[warp][lane >> 2] = v;
  __syncthreads();
  if (tid < 8) {
    double t = 0.0;
    #pragma unroll
    for (int w = 0; w < WARPS; ++w) t += s_red[w][tid];
    static_cast<double*>(a.avg)[bl * 8 + tid] = t * a.inv_n;
  }
}

// The pass from phasor tables.  A thread owns channel offset r of one time and walks
// the tiles q, so T2[r] is applied once a (time, r) on each side of the walk: to the
// model before it and to the sums after it; a sample then takes 32 multiply-adds
// (36 with a walk of 8 tiles), where the product of both tables for every sample
// took 40.  Threads: groups of R offsets, each a (time, part of the tiles).
constexpr int kFp64Threads = 128;
template <bool SUB, bool ACC>
__global__ void __launch_bounds__(kFp64Threads) k_stream_fp64_tab(StreamArgs a, Fp64Tables tb) {
  extern __shared__ __align__(16) unsigned char s_f64[];
  double2* s_tab = reinterpret_cast<double2*>(s_f64);            // [n_t][sub, acc][Q]
  __shared__ double2 s_M[4];
  __shared__ double s_red[kFp64Threads / 32][8];
  const int64_t bl = blockIdx.x;
  const int2 ij = a.bl_ant[bl];
  const int tid = threadIdx.x, r = tid & (tb.R - 1), g = tid >> tb.lr, G = kFp64Threads >> tb.lr;
  if (SUB) fp64_model(a, ij, tid, s_M);
  double acc[8];
  #pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = 0.0;
  const double2* src = static_cast<const double2*>(a.src);
  double2* dst = static_cast<double2*>(a.dst);
  const int n_e = tb.Q + tb.R;
  for (int t0 = 0; t0 < a.n_time; t0 += tb.n_t) {
    const int nt = min(tb.n_t, a.n_time - t0);
    if (t0) __syncthreads();                 // the previous times' tables are read
    for (int x = tid; x < nt * 2 * tb.Q; x += kFp64Threads) {
      const int row = x / tb.Q, e = x - row * tb.Q;
      if ((row & 1) ? !ACC : !SUB) continue;
      const double2* tab = (row & 1) ? tb.acc : tb.sub;
      const size_t at = (size_t)(t0 + (row >> 1)) * a.n_ant;
      s_tab[x] = cmulc(tab[(at + ij.x) * n_e + e], tab[(at + ij.y) * n_e + e]);
    }
    __syncthreads();
    const int parts = max(1, G / nt);
    for (int it = g; it < nt * parts; it += G) {
      const int t = it % nt, part = it / nt;
      const size_t ti = ((size_t)(t0 + t) * a.n_ant + ij.x) * n_e + tb.Q + r, tj = ti + (size_t)(ij.y - ij.x) * n_e;
      double2 A[4], s[4];
      if (SUB) {
        const double2 z = cmulc(tb.sub[ti], tb.sub[tj]);
        #pragma unroll
        for (int e = 0; e < 4; ++e) A[e] = cmulc(s_M[e], z);
      }
      if (ACC) {
        #pragma unroll
        for (int e = 0; e < 4; ++e) s[e] = make_double2(0.0, 0.0);
      }
      const double2* T = s_tab + (size_t)2 * t * tb.Q;
      const size_t row = ((size_t)(t0 + t) * a.n_bl + bl) * a.n_chan;
      #pragma unroll 2
      for (int q = part; q < tb.Q; q += parts) {
        const int c = (q << tb.lr) + r;
        if (c >= a.n_chan) break;
        const size_t idx = (row + c) * 4;
        double2 x[4];
        #pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = src[idx + e];
        if (SUB) {
          const double2 z = T[q];
          #pragma unroll
          for (int e = 0; e < 4; ++e) {       // x += A conj(z)
            x[e].x = fma(A[e].x, z.x, fma(A[e].y, z.y, x[e].x));
            x[e].y = fma(A[e].y, z.x, fma(-A[e].x, z.y, x[e].y));
            dst[idx + e] = x[e];
          }
        }
        if (ACC) {
          const double2 z = T[tb.Q + q];
          #pragma unroll
          for (int e = 0; e < 4; ++e) {
            s[e].x = fma(x[e].x, z.x, fma(-x[e].y, z.y, s[e].x));
            s[e].y = fma(x[e].x, z.y, fma(x[e].y, z.x, s[e].y));
          }
        }
      }
      if (ACC) {
        const double2 z = cmulc(tb.acc[ti], tb.acc[tj]);
        #pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc[2 * e] = fma(s[e].x, z.x, fma(-s[e].y, z.y, acc[2 * e]));
          acc[2 * e + 1] = fma(s[e].x, z.y, fma(s[e].y, z.x, acc[2 * e + 1]));
        }
      }
    }
  }
  if (ACC) fp64_average<kFp64Threads / 32>(a, bl, acc, s_red);
}

// The pass on any frequency list: one sincospi a sample and role.
template <bool SUB, bool ACC>
__global__ void __launch_bounds__(kStreamThreads) k_stream_fp64(StreamArgs a) {
  extern __shared__ __align__(16) unsigned char s_f64[];
  double* s_tau = reinterpret_cast<double*>(s_f64);              // [n_time][2]: tau_sub, tau_acc
  __shared__ double2 s_M[4];
  __shared__ double s_red[kStreamThreads / 32][8];
  const int64_t bl = blockIdx.x;
  const int2 ij = a.bl_ant[bl];
  const int tid = threadIdx.x;
  for (int t = tid; t < a.n_time; t += kStreamThreads) {
    if (SUB) s_tau[2 * t] = delay_m(a.uvw, a.n_ant, t, ij.x, ij.y, a.sub);
    if (ACC) s_tau[2 * t + 1] = delay_m(a.uvw, a.n_ant, t, ij.x, ij.y, a.acc);
  }
  if (SUB) fp64_model(a, ij, tid, s_M);
  __syncthreads();
  double2 M[4];
  if (SUB) {
    #pragma unroll
    for (int e = 0; e < 4; ++e) M[e] = s_M[e];
  }
  double acc[8];
  #pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = 0.0;
  const double2* src = static_cast<const double2*>(a.src);
  double2* dst = static_cast<double2*>(a.dst);
  const int n_s = a.n_time * a.n_chan;
  TCWalk w;
  w.init(tid, a.n_chan);
  for (int s = tid; s < n_s; s += kStreamThreads, w.next()) {
    const size_t idx = (((size_t)w.t * a.n_bl + bl) * a.n_chan + w.c) * 4;
    double2 x[4];
    #pragma unroll
    for (int e = 0; e < 4; ++e) x[e] = src[idx + e];
    if (SUB) {
      const double2 ph = phasor_d(s_tau[2 * w.t] * a.freq_c[w.c]);          // exp(+2 pi i phi)
      #pragma unroll
      for (int e = 0; e < 4; ++e) {           // x += (-M) conj(ph)
        x[e].x = fma(M[e].x, ph.x, fma(M[e].y, ph.y, x[e].x));
        x[e].y = fma(M[e].y, ph.x, fma(-M[e].x, ph.y, x[e].y));
        dst[idx + e] = x[e];
      }
    }
    if (ACC) {
      const double2 ph = phasor_d(s_tau[2 * w.t + 1] * a.freq_c[w.c]);
      #pragma unroll
      for (int e = 0; e < 4; ++e) {
        acc[2 * e] = fma(x[e].x, ph.x, fma(-x[e].y, ph.y, acc[2 * e]));
        acc[2 * e + 1] = fma(x[e].x, ph.y, fma(x[e].y, ph.x, acc[2 * e + 1]));
      }
    }
  }
  if (ACC) fp64_average<kStreamThreads / 32>(a, bl, acc, s_red);
}

}  // namespace rts
