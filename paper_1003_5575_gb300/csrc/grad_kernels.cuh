// Adjoint of the multi-source predict step.
//
//   R = V - sum_k M_k exp(-2 pi i phi_k),  M_k = S_k J_i J_j^H,  L = sum ||R||_F^2
//   G_k  = sum_{t,c} R exp(+2 pi i phi_k)
//   H^l_k = sum_{t,c} R exp(+2 pi i phi_k) dphi_k/dl,  dphi/dl = (u - w l/n) nu_c / c
//   (H^m_k likewise with v, m)
//   dL/dJ_i += -2 S G J_j,  dL/dJ_j += -2 S G^H J_i    (dL/dRe + i dL/dIm)
//   dL/dS   += -2 Re tr(G^H J_i J_j^H)
//   dL/dl   += -4 pi Im tr(H^lH M),  dL/dm likewise.
//
// Kernel 1, one CTA per (baseline, chunk of sources): for each time and
// channel tile it forms R for every channel of the tile in shared memory
// (all K sources subtracted, phasors computed, never stored) and adds |R|^2 to
// the loss; then threads = (source, channel group) accumulate
// H0 = sum_c R e^{+i phi} and H1 = sum_c c R e^{+i phi}, from which
// G += H0 and H^l += (u - w l/n)(nu_0/c H0 + dnu/c H1).  Per (source,
// baseline) it stores G and the three scalar contributions (FP64).
// With WEIGHTED the channel weight of the position derivative is a table
// (d phi/d shift = a_p wchan[c], used by the offset fit's frequency law) and
// H^l = (u - w l/n) sum_c wchan[c] R e^{+i phi}.
// Kernels 2-4 reduce those per antenna / per source / for the loss in a fixed
// order, so the result is deterministic (no atomics).
#pragma once
#include <algorithm>
#include <string>
#include <type_traits>

#include "common.cuh"
#include "kahan.cuh"
#include "strip_kernels.cuh"

namespace rts {

constexpr int kGradThreads = 512;
constexpr int kGradTile = 512;        // channels per shared-memory tile
constexpr int kGradChunk = 512;       // sources per CTA in the backward phase
constexpr size_t kGradMaxSmem = 227 * 1024;

struct __align__(16) DirQ { double x, y, z, w; };   // (l, m, n - 1, S) of one source

struct GradWorkspace {
  int cap_src = 0;
  int64_t n_bl = 0;
  double2* G = nullptr;     // [K][n_bl][4]
  double* gsc = nullptr;    // [K][n_bl][3] (dl, dm, dS contributions)
  double* loss_bl = nullptr;// [n_bl]
  DirQ* dir = nullptr;   // [K] (l, m, nm1, S)
  PhaseAB* aph = nullptr;   // [n_time][n_ant][kp] antenna phases (k_grad_strip), kp = K rounded up to 32
  int aph_src = 0;          // kp, at most (0: no room for them, or never used)
  float4* lmn = nullptr;    // [kp] l / n and m / n, each as a pair of floats
  double* wchan = nullptr;  // [n_chan] per-channel weight of the position derivative (offsets)
};

struct GradArgs {
  const void* vis;
  const void* jones;        // [K][n_ant][4] cube precision
  const DirQ* dir;       // [K] (l, m, n-1, S)
  const double* uvw;
  const int2* bl_ant;
  const double* freq_c;
  const double* wchan;      // WEIGHTED: d phi / d(shift) = a_p wchan[c]; else a_p nu_c / c
  double2* G;
  double* gsc;
  double* loss_bl;
  int n_src, n_ant, n_chan, n_time;
  int64_t n_bl;
  double nu0_c, dnu_c;
};

__global__ void k_grad_dirs(const double* __restrict__ src, int n, DirQ* __restrict__ dir, float4* __restrict__ lmn) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) {
    double l = src[3 * k], m = src[3 * k + 1], S = src[3 * k + 2];
    double r2 = l * l + m * m;
    const double nm1 = -r2 / (1.0 + sqrt(1.0 - r2));
    dir[k] = DirQ{l, m, nm1, S};
    const double ln = l / (1.0 + nm1), mn = m / (1.0 + nm1);
    const float lh = (float)ln, mh = (float)mn;
    lmn[k] = make_float4(lh, (float)(ln - (double)lh), mh, (float)(mn - (double)mh));
  }
}

template <typename T>
__device__ inline typename cplx_of<T>::type load_j(const void* jones, size_t idx) {
  using C = typename cplx_of<T>::type;
  return static_cast<const C*>(jones)[idx];
}

// exp(+2 pi i phi) for channel c of source k at the current time
template <bool MIXED>
__device__ inline typename cplx_of<typename std::conditional<MIXED, float, double>::type>::type
grad_phasor(unsigned long long A, unsigned long long B, double tau, const double* freq_c, int c) {
  if constexpr (MIXED) {
    return phasor_f(q64_to_turns(A + (unsigned long long)c * B));
  } else {
    return phasor_d(tau * freq_c[c]);
  }
}

// per (source k, baseline bl): G, and the (dl, dm, dS) contributions
//   dL/dl = -4 pi S Im tr(H^lH J_i J_j^H), dL/dm likewise, dL/dS = -2 Re tr(G^H J_i J_j^H)
template <typename T>
__device__ inline void grad_store(const GradArgs& a, int k, int64_t bl, int2 ij, const double (&G)[8],
                                  const double (&Hl)[8], const double (&Hm)[8]) {
  using C = typename cplx_of<T>::type;
  M22<double2> Ji, Jj, Gm, Hlm, Hmm;
  #pragma unroll
  for (int e = 0; e < 4; ++e) {
    C p = load_j<T>(a.jones, ((size_t)k * a.n_ant + ij.x) * 4 + e);
    C q = load_j<T>(a.jones, ((size_t)k * a.n_ant + ij.y) * 4 + e);
    Ji.e[e] = make_double2(p.x, p.y); Jj.e[e] = make_double2(q.x, q.y);
    Gm.e[e] = make_double2(G[2 * e], G[2 * e + 1]);
    Hlm.e[e] = make_double2(Hl[2 * e], Hl[2 * e + 1]);
    Hmm.e[e] = make_double2(Hm[2 * e], Hm[2 * e + 1]);
    a.G[((size_t)k * a.n_bl + bl) * 4 + e] = Gm.e[e];
  }
  const double S = a.dir[k].w;
  M22<double2> P = mmul_h(Ji, Jj);                 // J_i J_j^H
  // tr(X^H Y) = sum_e conj(X_e) Y_e
  double2 tG = make_double2(0, 0), tl = make_double2(0, 0), tm = make_double2(0, 0);
  #pragma unroll
  for (int e = 0; e < 4; ++e) {
    tG = cadd(tG, cconjmul(Gm.e[e], P.e[e]));
    tl = cadd(tl, cconjmul(Hlm.e[e], P.e[e]));
    tm = cadd(tm, cconjmul(Hmm.e[e], P.e[e]));
  }
  const double four_pi = 12.566370614359172953850573533118;
  double* o = a.gsc + ((size_t)k * a.n_bl + bl) * 3;
  o[0] = -four_pi * S * tl.y;
  o[1] = -four_pi * S * tm.y;
  o[2] = -2.0 * tG.x;
}

template <bool MIXED, bool WEIGHTED>
__global__ void __launch_bounds__(kGradThreads) k_grad_sweep(GradArgs a) {
  using T = typename std::conditional<MIXED, float, double>::type;
  using C = typename cplx_of<T>::type;
  extern __shared__ __align__(16) unsigned char g_smem[];
  // layout (16-byte aligned pieces first):
  //   R tile [kGradTile][4] C | M [K][4] C | part [threads][16] T | A, B [K] u64 | tau [K] double
  C* sR = reinterpret_cast<C*>(g_smem);
  C* sM = sR + kGradTile * 4;
  T* sPart = reinterpret_cast<T*>(sM + (size_t)a.n_src * 4);
  unsigned long long* sA = reinterpret_cast<unsigned long long*>(sPart + (size_t)kGradThreads * 16);
  unsigned long long* sB = sA + a.n_src;
  double* sTau = reinterpret_cast<double*>(sB + a.n_src);
  __shared__ double s_uvw[3];
  __shared__ double s_loss[kGradThreads / 32];

  const int64_t bl = blockIdx.x;
  const int2 ij = a.bl_ant[bl];
  const int k0 = blockIdx.y * kGradChunk;
  const int kc = max(1, min(kGradChunk, a.n_src - k0));   // sources of this CTA's backward phase
  const int groups = max(1, kGradThreads / kc);
  const int my_k = threadIdx.x % kc, my_g = threadIdx.x / kc;
  const bool bw = my_g < groups && k0 + my_k < a.n_src;

  // model matrices of all sources on this baseline
  for (int k = threadIdx.x; k < a.n_src; k += blockDim.x) {
    M22<double2> Ji, Jj;
    #pragma unroll
    for (int e = 0; e < 4; ++e) {
      C p = load_j<T>(a.jones, ((size_t)k * a.n_ant + ij.x) * 4 + e);
      C q = load_j<T>(a.jones, ((size_t)k * a.n_ant + ij.y) * 4 + e);
      Ji.e[e] = make_double2(p.x, p.y); Jj.e[e] = make_double2(q.x, q.y);
    }
    M22<double2> P = mmul_h(Ji, Jj);
    const double S = a.dir[k].w;
    #pragma unroll
    for (int e = 0; e < 4; ++e) sM[(size_t)k * 4 + e] = cmk<C>(S * P.e[e].x, S * P.e[e].y);
  }
  double G[8], Hl[8], Hm[8];
  #pragma unroll
  for (int e = 0; e < 8; ++e) { G[e] = 0.0; Hl[e] = 0.0; Hm[e] = 0.0; }
  double loss = 0.0;
  double lk_n = 0.0, mk_n = 0.0;
  if (bw) {
    const DirQ d = a.dir[k0 + my_k];
    const double n = 1.0 + d.z;
    lk_n = d.x / n; mk_n = d.y / n;
  }

  for (int t = 0; t < a.n_time; ++t) {
    __syncthreads();                              // previous users of sA/sB/sTau/s_uvw done
    for (int k = threadIdx.x; k < a.n_src; k += blockDim.x) {
      SrcDir d; d.l = a.dir[k].x; d.m = a.dir[k].y; d.nm1 = a.dir[k].z; d.S = a.dir[k].w;
      double tau = delay_m(a.uvw, a.n_ant, t, ij.x, ij.y, d);
      sTau[k] = tau;
      if (MIXED) { sA[k] = frac_q64(tau * a.nu0_c); sB[k] = frac_q64(tau * a.dnu_c); }
    }
    if (threadIdx.x < 3)
      s_uvw[threadIdx.x] = a.uvw[((size_t)t * a.n_ant + ij.x) * 3 + threadIdx.x] -
                           a.uvw[((size_t)t * a.n_ant + ij.y) * 3 + threadIdx.x];
    for (int c0 = 0; c0 < a.n_chan; c0 += kGradTile) {
      const int nc = min(kGradTile, a.n_chan - c0);
      __syncthreads();                            // tables ready; previous tile consumed
      // forward: R for each channel of the tile
      for (int cl = threadIdx.x; cl < nc; cl += blockDim.x) {
        const int c = c0 + cl;
        const C* v = static_cast<const C*>(a.vis) + (((size_t)t * a.n_bl + bl) * a.n_chan + c) * 4;
        C r[4];
        #pragma unroll
        for (int e = 0; e < 4; ++e) r[e] = v[e];
        for (int k = 0; k < a.n_src; ++k) {
          C ph = grad_phasor<MIXED>(sA[k], sB[k], sTau[k], a.freq_c, c);
          #pragma unroll
          for (int e = 0; e < 4; ++e) r[e] = csub(r[e], cmulc(sM[(size_t)k * 4 + e], ph));
        }
        #pragma unroll
        for (int e = 0; e < 4; ++e) {
          sR[cl * 4 + e] = r[e];
          loss += (double)r[e].x * r[e].x + (double)r[e].y * r[e].y;
        }
      }
      __syncthreads();
      // backward: partial H0, H1 over this thread's channel group
      if (bw) {
        const int k = k0 + my_k;
        T h0[8], h1[8];
        #pragma unroll
        for (int e = 0; e < 8; ++e) { h0[e] = T(0); h1[e] = T(0); }
        for (int cl = my_g; cl < nc; cl += groups) {
          const int c = c0 + cl;
          C ph = grad_phasor<MIXED>(sA[k], sB[k], sTau[k], a.freq_c, c);
          const T cw = WEIGHTED ? (T)a.wchan[c] : (T)c;
          #pragma unroll
          for (int e = 0; e < 4; ++e) {
            C x = cmul(sR[cl * 4 + e], ph);
            h0[2 * e] += x.x; h0[2 * e + 1] += x.y;
            h1[2 * e] += cw * x.x; h1[2 * e + 1] += cw * x.y;
          }
        }
        T* part = sPart + (size_t)threadIdx.x * 16;
        #pragma unroll
        for (int e = 0; e < 8; ++e) { part[e] = h0[e]; part[8 + e] = h1[e]; }
      }
      __syncthreads();
      if (bw && my_g == 0) {
        double H0[8], H1[8];
        #pragma unroll
        for (int e = 0; e < 8; ++e) { H0[e] = 0.0; H1[e] = 0.0; }
        for (int g = 0; g < groups; ++g) {
          const T* part = sPart + (size_t)(g * kc + my_k) * 16;
          #pragma unroll
          for (int e = 0; e < 8; ++e) { H0[e] += (double)part[e]; H1[e] += (double)part[8 + e]; }
        }
        const double wl = s_uvw[0] - s_uvw[2] * lk_n;
        const double wm = s_uvw[1] - s_uvw[2] * mk_n;
        #pragma unroll
        for (int e = 0; e < 8; ++e) {
          const double hn = WEIGHTED ? H1[e] : a.nu0_c * H0[e] + a.dnu_c * H1[e];
          G[e] += H0[e];
          Hl[e] += wl * hn;
          Hm[e] += wm * hn;
        }
      }
    }
  }
  // loss of this baseline (chunk 0 only)
  if (blockIdx.y == 0) {
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if ((threadIdx.x & 31) == 0) s_loss[threadIdx.x >> 5] = loss;
  }
  __syncthreads();
  if (blockIdx.y == 0 && threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < kGradThreads / 32; ++w) s += s_loss[w];
    a.loss_bl[bl] = s;
  }
  if (bw && my_g == 0) grad_store<T>(a, k0 + my_k, bl, ij, G, Hl, Hm);
}

// The FP32 adjoint on strips (strip_kernels.cuh).  One CTA per baseline; a warp
// takes one (time, tile of 256 channels) strip of it through both halves:
//   forward   R = V - sum_k M_k conj(T1_k[q] T2_k[r]) in registers, lane = its
//             channels, 32 sources' phasor tables at a time in shared memory;
//   backward  lane = source, R read by broadcast from shared-memory planes:
//             sum_c R(c) P_k(c) = sum_q T1_k[q] s_q,  s_q = sum_r x_r, x_r = R(16q + r) T2_k[r],
//             sum_c c R(c) P_k(c) = sum_q T1_k[q] [(c0 + 16q - 1) s_q + a_q],
//             a_q = sum_r (r + 1) x_r, the running sum of the suffix sums while r
//             runs down from 15 (c0 the tile's first channel).
// A (source, channel) pair costs 20 multiply-adds in the forward half and 24 in
// the backward one, two a packed instruction; the FP32 pipe bounds it (66 % busy,
// 56 % of the issue slots, at 100 sources, 128 antennas x 256 channels x 8 times).
// Where a lane had stood for each (source, channel) with every phasor and sum formed
// apart (62 instructions a pair) that size took 5.96 ms, this takes 3.27; 300
// sources, 512 antennas x 768 channels x 8 times with the reductions: 607 and 463 ms.
// The last group's lanes share out the tiles when 16 sources or fewer are left (100
// sources: a quarter of the backward half was idle lanes).  The
// position derivative is contracted with M per strip (one number instead of two
// complex 2x2 sums a direction).  After each group of 32 sources the CTA's warps
// meet once and their ten sums a source are added, in warp order, to compensated
// FP32 totals (two stages, so that one barrier a group is enough).
constexpr int kGsQh = 8;
constexpr int kGsTile = 32 * kGsQh;       // channels of a strip
constexpr int kGsPitch = 17;              // float4 from tile to tile: the lanes of several tiles read other banks
constexpr int kGsMaxWarps = 12;           // of one CTA an SM: 168 registers a thread
constexpr int kGsPairWarps = 8;           // of each of two: 128 registers
constexpr size_t kGsPairSmem = 112 * 1024;
// Two CTAs of 8 warps against one of 12: 463 and 470 ms at 300 sources, where the
// totals leave shared memory to make room for the second; at 100 sources two CTAs,
// the sharing of the last group and k_grad_jones's reduction took 4.57 ms to 3.56
constexpr int kGsVals = 10;               // per source: G (8), l, m
// No more sources fit (64 bytes of models a source in 112 KB for one of two CTAs, 144 with
// the totals in 225 KB): the antenna phases are kept for no more
constexpr int kGsMaxSrc = 1600;

__host__ __device__ inline int grad_kp(int n_src) { return (n_src + kStGrp - 1) / kStGrp * kStGrp; }
template <bool WEIGHTED> __host__ __device__ constexpr size_t grad_strip_warp_bytes() {
  constexpr size_t planes = (size_t)4 * kGsQh * kGsPitch * sizeof(float4);
  return (planes > strip_warp_bytes<kGsQh>() ? planes : strip_warp_bytes<kGsQh>()) + (WEIGHTED ? kGsTile * sizeof(float) : 0);
}
// sine table | model matrices [Kp][kStMRow] float4 | (tot) totals and compensations
// [2][kGsVals][Kp] | two stages [2][warps][kGsVals][32] | a workspace per warp
template <bool WEIGHTED> inline size_t grad_strip_smem(int n_src, int warps, bool tot) {
  const size_t kp = grad_kp(n_src);
  return 256 * sizeof(float2) + kp * kStMRow * sizeof(float4) + (tot ? 2 * kGsVals * kp * sizeof(float) : 0) +
         (size_t)warps * (2 * kGsVals * kStGrp * sizeof(float) + grad_strip_warp_bytes<WEIGHTED>());
}
// Warps of a CTA: as few rounds over the baseline's strips as `most` gives, then
// as few warps as those rounds need; fewer where the sources' tables leave no
// room in `room` bytes.  0: they do not fit.
template <bool WEIGHTED>
inline int grad_strip_warps(int n_src, int n_chan, int n_time, int most, size_t room, bool tot) {
  const int64_t strips = (int64_t)n_time * ((n_chan + kGsTile - 1) / kGsTile);
  const int64_t rounds = (strips + most - 1) / most;
  int w = (int)((strips + rounds - 1) / rounds);
  const int least = w < 4 ? w : 4;
  while (w >= least && grad_strip_smem<WEIGHTED>(n_src, w, tot) > room) --w;
  return w >= least ? w : 0;
}

// the antennas' Q0.64 phases of every source (of u_i - u_0: see k_block_ant_phases), [n_time][n_ant][kp]
__global__ void __launch_bounds__(256) k_grad_ant_phases(const DirQ* __restrict__ dir, int n_src, int kp,
                                                        const double* __restrict__ uvw, int n_ant, int n_time,
                                                        double nu0_c, double dnu_c, PhaseAB* __restrict__ aph) {
  const int64_t n = (int64_t)n_time * n_ant * kp;
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
    const int64_t ti = x / kp;
    const int k = (int)(x - ti * kp);
    PhaseAB p;
    p.a = 0; p.b = 0;
    if (k < n_src) {
      SrcDir d;
      d.l = dir[k].x; d.m = dir[k].y; d.nm1 = dir[k].z;
      const int t = (int)(ti / n_ant);
      const double tau = delay_m(uvw, n_ant, t, (int)(ti - (int64_t)t * n_ant), 0, d);
      p.a = frac_q64(tau * nu0_c);
      p.b = frac_q64(tau * dnu_c);
    }
    aph[x] = p;
  }
}

// sums of this lane's source over a strip's planes: y0 = sum R P, y1 = sum w R P with
// w the channel number (WEIGHTED: the table wt), as (re 0, re 1), (re 2, re 3), (im ..)
template <bool WEIGHTED>
__device__ __forceinline__ void grad_strip_average(const float4* __restrict__ pre, const float4* __restrict__ pim,
                                                   const float* __restrict__ wt, int nq, int c0, int part,
                                                   int parts, PhaseAB p, const float2* lut, float2 (&y0)[4], float2 (&y1)[4]) {
  float2 t2[16];
  #pragma unroll
  for (int r = 0; r < 16; ++r) t2[r] = phasor_lut((unsigned long long)r * p.b, lut);
  #pragma unroll
  for (int i = 0; i < 4; ++i) y0[i] = y1[i] = make_float2(0.f, 0.f);
  const unsigned long long step = (unsigned long long)(16 * parts) * p.b;
  unsigned long long ph = p.a + (unsigned long long)(16 * part) * p.b;
  pre += kGsPitch * part;
  pim += kGsPitch * part;
  #pragma unroll 1
  for (int q = part; q < nq; q += parts, ph += step, pre += kGsPitch * parts, pim += kGsPitch * parts) {
    float2 s0[4], s1[4];
    #pragma unroll
    for (int i = 0; i < 4; ++i) s0[i] = s1[i] = make_float2(0.f, 0.f);
    #pragma unroll
    for (int r = 15; r >= 0; --r) {
      const float4 a = pre[r], b = pim[r];
      const float2 a0 = make_float2(a.x, a.y), a1 = make_float2(a.z, a.w);
      const float2 b0 = make_float2(b.x, b.y), b1 = make_float2(b.z, b.w);
      const float2 tx = make_float2(t2[r].x, t2[r].x), ty = make_float2(t2[r].y, t2[r].y);
      const float ny = __uint_as_float(__float_as_uint(t2[r].y) ^ 0x80000000u);
      const float2 nty = make_float2(ny, ny);
      if (WEIGHTED) {
        const float w = wt[16 * q + r];
        const float2 w2 = make_float2(w, w);
        const float2 x[4] = {ffma2(a0, tx, fmul2(b0, nty)), ffma2(a1, tx, fmul2(b1, nty)),
                             ffma2(a0, ty, fmul2(b0, tx)), ffma2(a1, ty, fmul2(b1, tx))};
        #pragma unroll
        for (int i = 0; i < 4; ++i) {
          s0[i] = fadd2(s0[i], x[i]);
          s1[i] = ffma2(x[i], w2, s1[i]);
        }
      } else {
        s0[0] = ffma2(a0, tx, ffma2(b0, nty, s0[0]));
        s0[1] = ffma2(a1, tx, ffma2(b1, nty, s0[1]));
        s0[2] = ffma2(a0, ty, ffma2(b0, tx, s0[2]));
        s0[3] = ffma2(a1, ty, ffma2(b1, tx, s0[3]));
        #pragma unroll
        for (int i = 0; i < 4; ++i) s1[i] = fadd2(s1[i], s0[i]);
      }
    }
    if (!WEIGHTED) {
      const float cw = (float)(c0 + 16 * q - 1);
      const float2 c2 = make_float2(cw, cw);
      #pragma unroll
      for (int i = 0; i < 4; ++i) s1[i] = ffma2(s0[i], c2, s1[i]);
    }
    const float2 t1 = phasor_lut(ph, lut);
    const float2 x = make_float2(t1.x, t1.x), y = make_float2(t1.y, t1.y), ny = make_float2(-t1.y, -t1.y);
    #pragma unroll
    for (int i = 0; i < 2; ++i) {
      y0[i] = ffma2(s0[i], x, ffma2(s0[2 + i], ny, y0[i]));
      y0[2 + i] = ffma2(s0[i], y, ffma2(s0[2 + i], x, y0[2 + i]));
      y1[i] = ffma2(s1[i], x, ffma2(s1[2 + i], ny, y1[i]));
      y1[2 + i] = ffma2(s1[i], y, ffma2(s1[2 + i], x, y1[2 + i]));
    }
  }
  for (int o = 32 / parts; o < 32; o <<= 1)          // the parts of a source
    #pragma unroll
    for (int i = 0; i < 4; ++i) {
      y0[i] = fadd2(y0[i], make_float2(__shfl_xor_sync(0xffffffffu, y0[i].x, o), __shfl_xor_sync(0xffffffffu, y0[i].y, o)));
      y1[i] = fadd2(y1[i], make_float2(__shfl_xor_sync(0xffffffffu, y1[i].x, o), __shfl_xor_sync(0xffffffffu, y1[i].y, o)));
    }
}

template <bool WEIGHTED, int WARPS, bool TOT>
__global__ void __launch_bounds__(WARPS * 32, WARPS == kGsPairWarps ? 2 : 1) k_grad_strip(GradArgs a, const PhaseAB* __restrict__ aph,
                                                                   const float4* __restrict__ lmn) {
  extern __shared__ __align__(16) unsigned char g_smem[];
  const int K = a.n_src, kp = grad_kp(K);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nthr = blockDim.x, nw = nthr >> 5;
  const int64_t bl = blockIdx.x;
  float2* lut = reinterpret_cast<float2*>(g_smem);
  float4* Mt = reinterpret_cast<float4*>(lut + 256);                           // [kp][kStMRow]
  float* tot = reinterpret_cast<float*>(Mt + (size_t)kp * kStMRow);             // [2][kGsVals][kp]
  float* stage = tot + (TOT ? (size_t)2 * kGsVals * kp : 0);                    // [2][nw][kGsVals][32]
  // value v's total and compensation of source k: in shared memory, or (TOT false) in
  // the words of this baseline's own results
  auto total = [&](int v, int k) -> float* {
    if (TOT) return tot + v * kp + k;
    const size_t at = (size_t)k * a.n_bl + bl;
    return v < 8 ? reinterpret_cast<float*>(a.G + at * 4) + v : reinterpret_cast<float*>(a.gsc + at * 3) + (v - 8);
  };
  auto total_comp = [&](int v, int k) -> float* {
    if (TOT) return tot + (kGsVals + v) * kp + k;
    return total(v, k) + (v < 8 ? 8 : 2);
  };
  unsigned char* ws = reinterpret_cast<unsigned char*>(stage + (size_t)2 * nw * kGsVals * kStGrp) +
                      (size_t)warp * grad_strip_warp_bytes<WEIGHTED>();
  StripTables<kGsQh>& tb = *reinterpret_cast<StripTables<kGsQh>*>(ws);
  float4* pre = reinterpret_cast<float4*>(ws);
  float4* pim = pre + 2 * kGsQh * kGsPitch;
  float* wt = reinterpret_cast<float*>(ws + grad_strip_warp_bytes<false>());         // WEIGHTED only
  __shared__ double s_loss[WARPS];
  const int2 ij = a.bl_ant[bl];
  lut_fill(lut, tid, nthr);
  for (int i = tid; i < kp * 4; i += nthr) {
    const int k = i >> 2, e = i & 3;
    float2 m = make_float2(0.f, 0.f);
    if (k < K) {
      const double S = a.dir[k].w;
      const float Sh = (float)S, Sl = (float)(S - (double)Sh);
      const size_t at = (size_t)k * a.n_ant;
      m = model_entry_ff(jones_row(a.jones, 2 * (at + ij.x) + (e >> 1)), jones_row(a.jones, 2 * (at + ij.y) + (e & 1)),
                         Sh, Sl);
    }
    strip_pack_model(Mt + (size_t)k * kStMRow, e, m);
  }
  __syncthreads();
  const int n_tile = (a.n_chan + kGsTile - 1) / kGsTile, n_strip = a.n_time * n_tile;
  const float nu0 = (float)a.nu0_c, dnu = (float)a.dnu_c;
  FF loss = {0.f, 0.f};
  int buf = 0;
  for (int s0 = 0; s0 < n_strip; s0 += nw) {
    const int s = s0 + warp, n_act = min(nw, n_strip - s0);
    const bool active = warp < n_act;
    const int t = active ? s / n_tile : 0, c0 = active ? (s - t * n_tile) * kGsTile : 0;
    const int nc = min(kGsTile, a.n_chan - c0), nq = (nc + 15) >> 4, np = (nq + 1) >> 1;
    const size_t ai = ((size_t)t * a.n_ant + ij.x) * kp, aj = ((size_t)t * a.n_ant + ij.y) * kp;
    auto phase = [&](int k) {                  // of source k at channel c0
      const PhaseAB x = aph[ai + k], y = aph[aj + k];
      PhaseAB p;
      p.b = x.b - y.b;
      p.a = x.a - y.a + (unsigned long long)c0 * p.b;
      return p;
    };
    // baseline (u, v, w) at t as float pairs
    FF u3[3];
    #pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double u = a.uvw[((size_t)t * a.n_ant + ij.x) * 3 + i] - a.uvw[((size_t)t * a.n_ant + ij.y) * 3 + i];
      u3[i].hi = (float)u;
      u3[i].lo = (float)(u - (double)u3[i].hi);
    }
    if (active) {
      Strip<kGsQh> R;
      strip_load(R, static_cast<const float4*>(a.vis) + (((size_t)t * a.n_bl + bl) * a.n_chan + c0) * 2, nc, lane);
      for (int k0 = 0; k0 < K; k0 += kStGrp) {
        const PhaseAB p = phase(k0 + lane);
        __syncwarp();
        strip_tables<kGsQh>(tb, p, lane, np, lut);
        __syncwarp();
        strip_subtract<kGsQh>(R, tb, Mt + (size_t)k0 * kStMRow, 0, min(kStGrp, K - k0), lane);
      }
      __syncwarp();
      strip_planes<kGsQh, kGsPitch>(R, pre, pim, nc, lane);
      const int cl = 16 * (lane >> 4) * kGsQh + (lane & 15);
      #pragma unroll
      for (int u = 0; u < kGsQh; ++u) {
        float re[4], im[4], l2 = 0.f;
        strip_channel(R, u, re, im);
        #pragma unroll
        for (int e = 0; e < 4; ++e) l2 = fmaf(re[e], re[e], fmaf(im[e], im[e], l2));
        if (cl + 16 * u < nc) {
          const FF x = ff_two_sum(loss.hi, l2);
          loss.hi = x.hi;
          loss.lo += x.lo;
        }
        if (WEIGHTED) wt[cl + 16 * u] = cl + 16 * u < nc ? (float)a.wchan[c0 + cl + 16 * u] : 0.f;
      }
      __syncwarp();
    }
    for (int k0 = 0; k0 < K; k0 += kStGrp, buf ^= 1) {
      float* st = stage + (size_t)buf * nw * kGsVals * kStGrp;
      if (active) {
        float2 y0[4], y1[4];
        // a group of 16 sources or fewer: several lanes a source, each some of the tiles
        const int n = K - k0, parts = n > 16 ? 1 : n > 8 ? 2 : n > 4 ? 4 : 8, kl = lane & (32 / parts - 1);
        grad_strip_average<WEIGHTED>(pre, pim, wt, nq, c0, lane / (32 / parts), parts, phase(k0 + kl), lut, y0, y1);
        float* o = st + (size_t)warp * kGsVals * kStGrp + lane;
        #pragma unroll
        for (int i = 0; i < 4; ++i) {
          o[(2 * i) * kStGrp] = y0[i].x;
          o[(2 * i + 1) * kStGrp] = y0[i].y;
        }
        // z = Im sum_e conj(h_e) M_e, h = sum R P (d phi / d shift) / a_p
        const float4* m = Mt + (size_t)(k0 + kl) * kStMRow;      // (-re, -re, -im, -im)
        FF z = {0.f, 0.f};
        #pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float hr0 = e & 1 ? y0[e >> 1].y : y0[e >> 1].x, hi0 = e & 1 ? y0[2 + (e >> 1)].y : y0[2 + (e >> 1)].x;
          const float hr1 = e & 1 ? y1[e >> 1].y : y1[e >> 1].x, hi1 = e & 1 ? y1[2 + (e >> 1)].y : y1[2 + (e >> 1)].x;
          const float hr = WEIGHTED ? hr1 : fmaf(nu0, hr0, dnu * hr1), hi = WEIGHTED ? hi1 : fmaf(nu0, hi0, dnu * hi1);
          const float4 me = m[e];
          z = ff_fma(-hr, me.z, z);                    // hr Im M
          z = ff_fma(hi, me.x, z);                     // - hi Re M
        }
        const float zf = z.hi + z.lo;
        const float4 ln = lmn[k0 + kl];                // l / n, m / n as float pairs
        auto arm = [&](FF u, float qh, float ql) {      // u - w q
          FF v = ff_fma(-u3[2].hi, qh, u);
          v.lo -= fmaf(u3[2].hi, ql, u3[2].lo * qh);
          return v.hi + v.lo;
        };
        o[8 * kStGrp] = arm(u3[0], ln.x, ln.y) * zf;
        o[9 * kStGrp] = arm(u3[1], ln.z, ln.w) * zf;
      }
      __syncthreads();
      for (int i = tid; i < kGsVals * kStGrp; i += nthr) {
        const int v = i / kStGrp, k = k0 + (i & (kStGrp - 1));
        if (!TOT && k >= K) continue;
        float *ps = total(v, k), *pc = total_comp(v, k);
        float sum = s0 ? *ps : 0.f, comp = s0 ? *pc : 0.f;
        for (int w = 0; w < n_act; ++w) kahan_add(sum, comp, st[(size_t)w * kGsVals * kStGrp + i]);
        *ps = sum;
        *pc = comp;
      }
    }
  }
  double l = isfinite(loss.hi) ? (double)loss.hi + (double)loss.lo : (double)loss.hi;     // lo of an infinite sum is no number
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if (lane == 0) s_loss[warp] = l;
  __syncthreads();
  if (tid == 0) {
    double x = 0.0;
    for (int w = 0; w < nw; ++w) x += s_loss[w];
    a.loss_bl[bl] = x;
  }
  // G, and the (dl, dm, dS) contributions: -4 pi z, -2 Re tr(G^H J_i J_j^H)
  const double four_pi = 12.566370614359172953850573533118;
  for (int k = tid; k < K; k += nthr) {
    // totals in plane order re 0 1 2 3 (values 0 .. 3), im 0 1 2 3 (values 4 .. 7)
    double2* Go = a.G + ((size_t)k * a.n_bl + bl) * 4;
    const size_t at = (size_t)k * a.n_ant;
    float sum[kGsVals], comp[kGsVals];
    #pragma unroll
    for (int v = 0; v < kGsVals; ++v) { sum[v] = *total(v, k); comp[v] = *total_comp(v, k); }
    if (!TOT) asm volatile("" ::: "memory");         // read before the same words take the results
    FF tg = {0.f, 0.f};
    #pragma unroll
    for (int e = 0; e < 4; ++e) {
      Go[e] = make_double2((double)sum[e] - (double)comp[e], (double)sum[4 + e] - (double)comp[4 + e]);
      const float2 pe = model_entry_ff(jones_row(a.jones, 2 * (at + ij.x) + (e >> 1)),
                                       jones_row(a.jones, 2 * (at + ij.y) + (e & 1)), 1.f, 0.f);
      tg = ff_fma(sum[e], pe.x, tg);
      tg = ff_fma(sum[4 + e], pe.y, tg);
      tg.lo -= fmaf(comp[e], pe.x, comp[4 + e] * pe.y);
    }
    double* o = a.gsc + ((size_t)k * a.n_bl + bl) * 3;
    o[0] = -four_pi * ((double)sum[8] - (double)comp[8]);
    o[1] = -four_pi * ((double)sum[9] - (double)comp[9]);
    o[2] = -2.0 * ((double)tg.hi + (double)tg.lo);
  }
}

// Bound by FP64 arithmetic: 32 fused multiply-adds a baseline and a reduction that
// halves the values with the lanes (9 additions a lane; a full tree a value took
// 40, and the kernel 355 us at 128 antennas and 100 sources).
// dL/dJ for antenna p of source k: -2 S [sum_{q>p} G(pq) J_q + sum_{q<p} G(qp)^H J_q]
template <bool MIXED>
__global__ void __launch_bounds__(128) k_grad_jones(const double2* __restrict__ G,
                                                    const void* __restrict__ jones,
                                                    const DirQ* __restrict__ dir,
                                                    void* __restrict__ gJ, int n_ant, int64_t n_bl) {
  using T = typename std::conditional<MIXED, float, double>::type;
  using C = typename cplx_of<T>::type;
  __shared__ double s_red[4 * 8];
  const int p = blockIdx.x, k = blockIdx.y;
  double acc[8];
  #pragma unroll
  for (int e = 0; e < 8; ++e) acc[e] = 0.0;
  const double2* Gk = G + (size_t)k * n_bl * 4;
  for (int q = threadIdx.x; q < n_ant; q += 128) {
    if (q == p) continue;
    double2 g[4];
    if (p < q) {
      const double2* s = Gk + bl_index(n_ant, p, q) * 4;
      g[0] = s[0]; g[1] = s[1]; g[2] = s[2]; g[3] = s[3];
    } else {
      const double2* s = Gk + bl_index(n_ant, q, p) * 4;
      g[0] = cconj(s[0]); g[1] = cconj(s[2]); g[2] = cconj(s[1]); g[3] = cconj(s[3]);
    }
    double2 J[4];
    #pragma unroll
    for (int e = 0; e < 4; ++e) {
      C v = load_j<T>(jones, ((size_t)k * n_ant + q) * 4 + e);
      J[e] = make_double2(v.x, v.y);
    }
    auto mac = [](double2 x, double2 y, double& re, double& im) {
      re = fma(x.x, y.x, fma(-x.y, y.y, re));
      im = fma(x.x, y.y, fma(x.y, y.x, im));
    };
    #pragma unroll
    for (int e = 0; e < 4; ++e) {
      mac(g[2 * (e >> 1)], J[e & 1], acc[2 * e], acc[2 * e + 1]);
      mac(g[2 * (e >> 1) + 1], J[2 + (e & 1)], acc[2 * e], acc[2 * e + 1]);
    }
  }
  const int lane = threadIdx.x & 31;
  const double tot = warp_reduce_scatter8d(acc, lane);          // value (lane >> 2) & 7
  if ((lane & 3) == 0) s_red[(threadIdx.x >> 5) * 8 + (lane >> 2)] = tot;
  __syncthreads();
  if (threadIdx.x == 0) {
    const double f = -2.0 * dir[k].w;
    C* out = static_cast<C*>(gJ) + ((size_t)k * n_ant + p) * 4;
    #pragma unroll
    for (int e = 0; e < 4; ++e) {
      double re = 0.0, im = 0.0;
      for (int w = 0; w < 4; ++w) { re += s_red[w * 8 + 2 * e]; im += s_red[w * 8 + 2 * e + 1]; }
      out[e] = cmk<C>(f * re, f * im);
    }
  }
}

// per-source (dl, dm, dS) and the loss, summed over baselines in a fixed order
__global__ void __launch_bounds__(256) k_grad_sum(const double* __restrict__ v, int64_t n, int stride,
                                                  int width, double* __restrict__ out) {
  __shared__ double s[256 * 3];
  const double* base = v + (size_t)blockIdx.x * n * stride;
  double acc[3] = {0.0, 0.0, 0.0};
  for (int64_t i = threadIdx.x; i < n; i += 256)
    for (int w = 0; w < width; ++w) acc[w] += base[i * stride + w];
  for (int w = 0; w < width; ++w) s[w * 256 + threadIdx.x] = acc[w];
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o)
      for (int w = 0; w < width; ++w) s[w * 256 + threadIdx.x] += s[w * 256 + threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int w = 0; w < width; ++w) out[(size_t)blockIdx.x * width + w] = s[w * 256];
}

inline void grad_free(GradWorkspace& w) {
  if (w.G) cudaFree(w.G);
  if (w.gsc) cudaFree(w.gsc);
  if (w.loss_bl) cudaFree(w.loss_bl);
  if (w.dir) cudaFree(w.dir);
  if (w.wchan) cudaFree(w.wchan);
  if (w.aph) cudaFree(w.aph);
  if (w.lmn) cudaFree(w.lmn);
  w = GradWorkspace();
}

inline int grad_fail(std::string& err, cudaError_t e, const char* what) {
  err = std::string(what) + ": " + cudaGetErrorString(e);
  return e == cudaErrorMemoryAllocation ? -2 : -3;
}

// Allocates its workspace on first use (G and per-baseline terms for up to
// max_src sources: (64 + 24) bytes per source and baseline, and with strip
// 16 bytes per antenna, time and source of up to kGsMaxSrc) and keeps it.
// strip: the handle's sweep may be k_grad_strip; without room for its phases it is
// k_grad_sweep, which needs none.
inline int grad_prepare(GradWorkspace& w, bool strip, int n_src, const double* src, int n_ant, int n_time,
                        int64_t n_bl, int max_src, cudaStream_t s, std::string& err) {
  cudaError_t e;
  if (!w.loss_bl) {
    w.cap_src = max_src; w.n_bl = n_bl;
    // the most any call may take, once a handle (every handle sets the same)
    auto room = [&](auto kernel) {
      return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGradMaxSmem - 1024) != cudaSuccess;
    };
    if (strip && (room(k_grad_strip<false, kGsPairWarps, true>) || room(k_grad_strip<false, kGsPairWarps, false>) ||
                  room(k_grad_strip<false, kGsMaxWarps, true>) || room(k_grad_strip<true, kGsPairWarps, true>) ||
                  room(k_grad_strip<true, kGsPairWarps, false>) || room(k_grad_strip<true, kGsMaxWarps, true>)))
      return grad_fail(err, cudaGetLastError(), "cudaFuncSetAttribute");
    if ((e = cudaMalloc(&w.G, (size_t)max_src * n_bl * 4 * sizeof(double2))) != cudaSuccess ||
        (e = cudaMalloc(&w.gsc, (size_t)max_src * n_bl * 3 * sizeof(double))) != cudaSuccess ||
        (e = cudaMalloc(&w.loss_bl, (size_t)n_bl * sizeof(double))) != cudaSuccess ||
        (e = cudaMalloc(&w.dir, (size_t)max_src * sizeof(DirQ))) != cudaSuccess ||
        (e = cudaMalloc(&w.lmn, (size_t)grad_kp(max_src) * sizeof(float4))) != cudaSuccess ||
        (e = cudaMemsetAsync(w.lmn, 0, (size_t)grad_kp(max_src) * sizeof(float4), s)) != cudaSuccess) {
      int rc = grad_fail(err, e, "cudaMalloc(gradient workspace)");
      grad_free(w);
      return rc;
    }
    if (strip) {
      w.aph_src = std::min(grad_kp(max_src), kGsMaxSrc);
      if (cudaMalloc(&w.aph, (size_t)n_time * n_ant * w.aph_src * sizeof(PhaseAB)) != cudaSuccess) {
        cudaGetLastError();
        w.aph = nullptr;
        w.aph_src = 0;
      }
    }
  }
  if (n_src > 0) k_grad_dirs<<<(n_src + 127) / 128, 128, 0, s>>>(src, n_src, w.dir, w.lmn);
  return 0;
}

inline size_t grad_smem_bytes(bool mixed, int n_src) {
  const size_t esz = mixed ? sizeof(float2) : sizeof(double2);
  const size_t tsz = mixed ? sizeof(float) : sizeof(double);
  return (size_t)kGradTile * 4 * esz + (size_t)n_src * (2 * 8 + 8 + 4 * esz) +
         (size_t)kGradThreads * 16 * tsz;
}

// the fused loss + adjoint sweep (one launch)
inline int grad_sweep(GradWorkspace& w, bool mixed, const void* vis, int n_src, const void* jones,
                      const double* uvw, const int2* bl_ant, const double* freq_c, int n_ant,
                      int n_chan, int n_time, int64_t n_bl, double nu0_c, double dnu_c,
                      cudaStream_t s, std::string& err, const double* wchan = nullptr,
                      bool direct = false) {
  cudaError_t e;
  GradArgs a;
  a.vis = vis; a.jones = jones; a.dir = w.dir; a.uvw = uvw; a.bl_ant = bl_ant; a.freq_c = freq_c;
  a.wchan = wchan;
  a.G = w.G; a.gsc = w.gsc; a.loss_bl = w.loss_bl;
  a.n_src = n_src; a.n_ant = n_ant; a.n_chan = n_chan; a.n_time = n_time; a.n_bl = n_bl;
  a.nu0_c = nu0_c; a.dnu_c = dnu_c;
  if (mixed && !direct && w.aph && grad_kp(n_src) <= w.aph_src) {
    // two CTAs an SM where they have more warps than one, with the totals in shared
    // memory if that leaves them all of their warps
    auto fit = [&](int most, size_t room, bool tot) {
      return wchan ? grad_strip_warps<true>(n_src, n_chan, n_time, most, room, tot)
                   : grad_strip_warps<false>(n_src, n_chan, n_time, most, room, tot);
    };
    int warps = fit(kGsMaxWarps, kGradMaxSmem - 2048, true);
    const int two_tot = fit(kGsPairWarps, kGsPairSmem, true), two = fit(kGsPairWarps, kGsPairSmem, false);
    const bool pair = 2 * two > warps, tot = !pair || two_tot == two;
    if (pair) warps = two;
    if (warps > 0) {
      const size_t smem = wchan ? grad_strip_smem<true>(n_src, warps, tot) : grad_strip_smem<false>(n_src, warps, tot);
      if (n_src > 0)
        k_grad_ant_phases<<<1024, 256, 0, s>>>(w.dir, n_src, grad_kp(n_src), uvw, n_ant, n_time, nu0_c, dnu_c, w.aph);
      auto launch = [&](auto kernel) { kernel<<<(unsigned)n_bl, 32 * warps, smem, s>>>(a, w.aph, w.lmn); };
      if (!pair) wchan ? launch(k_grad_strip<true, kGsMaxWarps, true>) : launch(k_grad_strip<false, kGsMaxWarps, true>);
      else if (tot) wchan ? launch(k_grad_strip<true, kGsPairWarps, true>) : launch(k_grad_strip<false, kGsPairWarps, true>);
      else wchan ? launch(k_grad_strip<true, kGsPairWarps, false>) : launch(k_grad_strip<false, kGsPairWarps, false>);
      if ((e = cudaGetLastError()) != cudaSuccess) return grad_fail(err, e, "gradient sweep launch");
      return 0;
    }
  }
  const size_t smem = grad_smem_bytes(mixed, n_src);
  const int chunks = n_src > 0 ? (n_src + kGradChunk - 1) / kGradChunk : 1;
  if (smem > kGradMaxSmem) {
    err = "too many sources for the gradient kernel's shared memory";
    return -1;
  }
  const dim3 grid((unsigned)n_bl, (unsigned)chunks);
  auto launch = [&](auto kernel) -> cudaError_t {
    cudaError_t r = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (r == cudaSuccess) kernel<<<grid, kGradThreads, smem, s>>>(a);
    return r;
  };
  if (mixed) e = wchan ? launch(k_grad_sweep<true, true>) : launch(k_grad_sweep<true, false>);
  else e = wchan ? launch(k_grad_sweep<false, true>) : launch(k_grad_sweep<false, false>);
  if (e != cudaSuccess) return grad_fail(err, e, "cudaFuncSetAttribute");
  if ((e = cudaGetLastError()) != cudaSuccess) return grad_fail(err, e, "gradient sweep launch");
  return 0;
}

// per-antenna dL/dJ, per-source (dl, dm, dS) and the loss; returns launches made
inline int grad_reduce(GradWorkspace& w, bool mixed, int n_src, const void* jones, double* loss,
                       void* gJ, double* gsrc, int n_ant, int64_t n_bl, cudaStream_t s,
                       std::string& err, int* launches) {
  cudaError_t e;
  int n = 0;
  if (n_src > 0 && gJ) {
    const dim3 gj((unsigned)n_ant, (unsigned)n_src);
    if (mixed) k_grad_jones<true><<<gj, 128, 0, s>>>(w.G, jones, w.dir, gJ, n_ant, n_bl);
    else k_grad_jones<false><<<gj, 128, 0, s>>>(w.G, jones, w.dir, gJ, n_ant, n_bl);
    ++n;
  }
  if (n_src > 0 && gsrc) { k_grad_sum<<<n_src, 256, 0, s>>>(w.gsc, n_bl, 3, 3, gsrc); ++n; }
  k_grad_sum<<<1, 256, 0, s>>>(w.loss_bl, n_bl, 1, 1, loss);
  ++n;
  *launches = n;
  if ((e = cudaGetLastError()) != cudaSuccess) return grad_fail(err, e, "gradient reduction launch");
  return 0;
}

}  // namespace rts
