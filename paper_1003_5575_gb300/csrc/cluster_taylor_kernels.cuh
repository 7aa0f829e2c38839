// The solve of one source's Taylor gains (taylor_kernels.cuh) by one thread-block
// cluster: its n_iter sweeps and slope-rotation steps in one launch, where three
// launches a sweep spend most of their time in one thread's FP64 chain (an FP64
// instruction occupies its sub-partition for 64 cycles whatever its lanes).
//
// CTAs, antenna slots, the exchange of iterates through st.async and the bounded
// waits are those of cluster_solve_kernels.cuh.  What differs:
//
// One set of sums serves both the rotation step and the next sweep.  With X = [G H]
// the iterate before its rotation, each antenna's warp sums over its partners
//   U0G = sum M0 G_q, U1G = sum M1 G_q, U2G = sum M2 G_q, U1H = sum M1 H_q, U2H = sum M2 H_q,
// and every CTA the Gram matrices P = sum G^H G, Q = sum G^H H, R = sum H^H H.
//   rotation: the gradient and Hessian sums over baselines reduce to sums over
//     antennas.  With the other antennas' Gram sums P', Q', R' (own term out) and the
//     residual row sums (mu_1 = mu_3 = 0: the channels are symmetric about the centre)
//       W^G = U2G - S (mu_2 G P' + mu_4 H Q'^H),  W^H = U2H - S (mu_2 G Q' + mu_4 H R'),
//       sum_{p<q} Re<rho, F_a> = 1/2 Re tr(Y B_a),   Y = sum_p W^G^H G,
//       sum_{p<q} Re<rho, D_a> = -1/2 Im tr(Z B_a),  Z = sum_p (W^H^H G - W^G^H H),
//       sum_{p<q} Re<D_a, D_b> = 1/2 Re sum_p [tr(B_a P B_b R') + tr(B_a R B_b P')
//                                  - tr(B_a Q B_b Q') - tr(B_a Q^H B_b Q'^H)],
//     18 numbers added over the cluster by one more exchange; every warp then takes
//     the 4x4 step itself.
//   next sweep: the partners' rotated slopes H + i G K enter linearly,
//       A = [U0G + U1H + i U1G K,  U1G + U2H + i U2G K],
//       Q' -> Q' + i P' K,  R' -> R' + i Q'^H K - i K Q' + K P' K.
// Precision: products FP32; a lane's few partners are summed in FP32 and
// everything after that (lanes, the others' Gram sums, W, the normal matrix, the
// iterate) in float-float arithmetic (about 47 bits).  The 4x4 systems of the
// sweep and of the step are solved in FP32 and refined once from a float-float
// residual; where a pivot is below 1e-3 of its scale they are solved in FP64.
// Measured (128 antennas, 20 sweeps): 165 us a source where the launches took 606
// (20 sweeps of 12.8 us, 19 row sums of 12.0 and 19 steps of 5.4, and their gaps);
// error of the gains and slopes of a 50-source cadence of 128 channels against 64 bits
// 1.5e-6 and 3.5e-6 with the launches, 1.4e-7 and 3.8e-7 here.  In cycles an iteration: row sums 4 200, Gram sums 1 300, the step's sums
// 3 100, the step 3 000 (one lane an entry of its matrix, the CTAs' sums pairwise; every
// lane doing all of it took 3 800), normal matrix 1 250, solve 2 000, exchange 1 600.
// The rows of all antennas have to fit the cluster's shared memory, up to about
// 175 antennas; larger arrays keep the launches (k_als_taylor_sweep).
#pragma once
#include "cluster_solve_kernels.cuh"
#include "taylor_kernels.cuh"

namespace rts {

struct FFC { FF re, im; };               // complex float-float

__device__ __forceinline__ FF ff_neg(FF a) { a.hi = -a.hi; a.lo = -a.lo; return a; }
__device__ __forceinline__ FF ff_norm(FF a) {              // hi the rounding of the sum (|lo| small)
  FF r;
  r.hi = __fadd_rn(a.hi, a.lo);
  r.lo = __fadd_rn(a.lo, -__fsub_rn(r.hi, a.hi));
  return r;
}
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
  FF r;
  r.hi = __fmul_rn(a.hi, b.hi);
  r.lo = fmaf(a.hi, b.hi, -r.hi) + fmaf(a.hi, b.lo, a.lo * b.hi);
  return r;
}
__device__ __forceinline__ FF ff_of(double x) {
  FF r;
  r.hi = (float)x;
  r.lo = (float)(x - (double)r.hi);
  return r;
}
__device__ __forceinline__ float ff_f(FF a) { return a.hi + a.lo; }
__device__ __forceinline__ double ff_d(FF a) { return (double)a.hi + (double)a.lo; }
// s + a b, b float-float
__device__ __forceinline__ FF ff_mac(float a, FF b, FF s) {
  FF r = ff_fma(a, b.hi, s);
  r.lo = fmaf(a, b.lo, r.lo);
  return r;
}
// s + g p (complex), p float-float
__device__ __forceinline__ FFC ffc_mac(float2 g, FFC p, FFC s) {
  s.re = ff_mac(-g.y, p.im, ff_mac(g.x, p.re, s.re));
  s.im = ff_mac(g.y, p.re, ff_mac(g.x, p.im, s.im));
  return s;
}
__device__ __forceinline__ FFC ffc_zero() {
  const FF z = {0.f, 0.f};
  return FFC{z, z};
}

struct ClusterTaylorArgs {
  const float2* mom;       // [3][n_bl][4] channel moments of the source
  double S;
  double mu0, mu2, mu4;    // mean_c x_c^n
  int rotate;              // take the slope-rotation steps (three channels or more)
  int n_ant, n_iter, apc;
  int64_t n_bl;
  double2* X;              // [n_ant][8] solution (G then H)
  float2* Xf;              // [n_ant][8] its FP32 rounding
  float2* gain;            // [n_ant][4] G and
  float2* slope;           // [n_ant][4] H of the source, FP32
  double* norms;           // [n_ant][4] dn, nn, non-finite
  int* status;
  double* rel;
};

constexpr int kCtRot = 18;               // rotation sums: Re<rho,F> 4, Re<rho,D> 4, Re<D,D> 10

// rows [apc][3][2][n_ant] float4, iterates [2][4][n_ant] float4 (rows of G, rows of H)
inline size_t cluster_taylor_smem(int n_ant, int apc) { return ((size_t)6 * apc + 8) * n_ant * sizeof(float4); }

// o (8 reals) += m x, rows as float4
__device__ __forceinline__ void ct_mm(float* o, float4 m0, float4 m1, float4 x0, float4 x1) {
  o[0] = fmaf(m0.x, x0.x, o[0]); o[0] = fmaf(-m0.y, x0.y, o[0]); o[0] = fmaf(m0.z, x1.x, o[0]); o[0] = fmaf(-m0.w, x1.y, o[0]);
  o[1] = fmaf(m0.x, x0.y, o[1]); o[1] = fmaf(m0.y, x0.x, o[1]); o[1] = fmaf(m0.z, x1.y, o[1]); o[1] = fmaf(m0.w, x1.x, o[1]);
  o[2] = fmaf(m0.x, x0.z, o[2]); o[2] = fmaf(-m0.y, x0.w, o[2]); o[2] = fmaf(m0.z, x1.z, o[2]); o[2] = fmaf(-m0.w, x1.w, o[2]);
  o[3] = fmaf(m0.x, x0.w, o[3]); o[3] = fmaf(m0.y, x0.z, o[3]); o[3] = fmaf(m0.z, x1.w, o[3]); o[3] = fmaf(m0.w, x1.z, o[3]);
  o[4] = fmaf(m1.x, x0.x, o[4]); o[4] = fmaf(-m1.y, x0.y, o[4]); o[4] = fmaf(m1.z, x1.x, o[4]); o[4] = fmaf(-m1.w, x1.y, o[4]);
  o[5] = fmaf(m1.x, x0.y, o[5]); o[5] = fmaf(m1.y, x0.x, o[5]); o[5] = fmaf(m1.z, x1.y, o[5]); o[5] = fmaf(m1.w, x1.x, o[5]);
  o[6] = fmaf(m1.x, x0.z, o[6]); o[6] = fmaf(-m1.y, x0.w, o[6]); o[6] = fmaf(m1.z, x1.z, o[6]); o[6] = fmaf(-m1.w, x1.w, o[6]);
  o[7] = fmaf(m1.x, x0.w, o[7]); o[7] = fmaf(m1.y, x0.z, o[7]); o[7] = fmaf(m1.z, x1.w, o[7]); o[7] = fmaf(m1.w, x1.z, o[7]);
}

// Gram matrices of one antenna: P = G^H G (P00, P11, re P01, im P01), Q = G^H H (8),
// R = H^H H (4); g0, g1 the rows of G, h0, h1 of H
__device__ __forceinline__ void ct_gram(float (&o)[16], float4 g0, float4 g1, float4 h0, float4 h1) {
  auto herm = [](float* v, float4 a, float4 b) {          // rows a, b of A: A^H A
    v[0] = fmaf(a.x, a.x, fmaf(a.y, a.y, fmaf(b.x, b.x, b.y * b.y)));
    v[1] = fmaf(a.z, a.z, fmaf(a.w, a.w, fmaf(b.z, b.z, b.w * b.w)));
    v[2] = fmaf(a.x, a.z, fmaf(a.y, a.w, fmaf(b.x, b.z, b.y * b.w)));
    v[3] = fmaf(a.x, a.w, fmaf(-a.y, a.z, fmaf(b.x, b.w, -b.y * b.z)));
  };
  auto cc = [](float* v, float ax, float ay, float bx, float by, float cx, float cy, float dx, float dy) {
    v[0] = fmaf(ax, bx, fmaf(ay, by, fmaf(cx, dx, cy * dy)));              // conj(a) b + conj(c) d
    v[1] = fmaf(ax, by, fmaf(-ay, bx, fmaf(cx, dy, -cy * dx)));
  };
  herm(o, g0, g1);
  cc(o + 4, g0.x, g0.y, h0.x, h0.y, g1.x, g1.y, h1.x, h1.y);
  cc(o + 6, g0.x, g0.y, h0.z, h0.w, g1.x, g1.y, h1.z, h1.w);
  cc(o + 8, g0.z, g0.w, h0.x, h0.y, g1.z, g1.w, h1.x, h1.y);
  cc(o + 10, g0.z, g0.w, h0.z, h0.w, g1.z, g1.w, h1.z, h1.w);
  herm(o + 12, h0, h1);
}

// One entry of x = b C^-1 in FP32 (schur_solve4_entry's scheme); false where a
// pivot is below 1e-3 of its scale
__device__ inline bool ct_schur4f(const float2 (&C)[4][4], const float2 (&b)[4], int col, float2* x) {
  auto inv2h = [](float a00, float2 a01, float a11, float2 (&o)[2][2]) {
    const float det = a00 * a11 - (a01.x * a01.x + a01.y * a01.y), id = __frcp_rn(det);
    o[0][0] = make_float2(a11 * id, 0.f);
    o[1][1] = make_float2(a00 * id, 0.f);
    o[0][1] = make_float2(-a01.x * id, -a01.y * id);
    o[1][0] = make_float2(-a01.x * id, a01.y * id);
    return det;
  };
  float2 Ai[2][2], Si[2][2], T[2][2], Sc[2][2];
  const float detA = inv2h(C[0][0].x, C[0][1], C[1][1].x, Ai);
  bool ok = C[0][0].x > 0.f && detA > 1e-3f * C[0][0].x * C[1][1].x;
  #pragma unroll
  for (int r = 0; r < 2; ++r)
    #pragma unroll
    for (int c = 0; c < 2; ++c) T[r][c] = cadd(cmul(Ai[r][0], C[0][2 + c]), cmul(Ai[r][1], C[1][2 + c]));
  #pragma unroll
  for (int r = 0; r < 2; ++r)
    #pragma unroll
    for (int c = 0; c < 2; ++c)
      Sc[r][c] = csub(C[2 + r][2 + c], cadd(cmul(cconj(C[0][2 + r]), T[0][c]), cmul(cconj(C[1][2 + r]), T[1][c])));
  const float detS = inv2h(Sc[0][0].x, Sc[0][1], Sc[1][1].x, Si);
  ok = ok && Sc[0][0].x > 1e-3f * C[2][2].x && Sc[1][1].x > 1e-3f * C[3][3].x && detS > 1e-3f * Sc[0][0].x * Sc[1][1].x;
  float2 Rh[2], Xh[2], Rg[2];
  #pragma unroll
  for (int k = 0; k < 2; ++k) Rh[k] = csub(b[2 + k], cadd(cmul(b[0], T[0][k]), cmul(b[1], T[1][k])));
  #pragma unroll
  for (int c = 0; c < 2; ++c) Xh[c] = cadd(cmul(Rh[0], Si[0][c]), cmul(Rh[1], Si[1][c]));
  #pragma unroll
  for (int k = 0; k < 2; ++k) Rg[k] = csub(b[k], cadd(cmul(Xh[0], cconj(C[k][2])), cmul(Xh[1], cconj(C[k][3]))));
  const float2 x0 = cadd(cmul(Rg[0], Ai[0][0]), cmul(Rg[1], Ai[1][0]));
  const float2 x1 = cadd(cmul(Rg[0], Ai[0][1]), cmul(Rg[1], Ai[1][1]));
  *x = col == 0 ? x0 : (col == 1 ? x1 : (col == 2 ? Xh[0] : Xh[1]));
  return ok;
}

// The rotation step k = -h^-1 g from the 18 sums (float-float): h in 2x2 blocks,
// solved in FP32 and refined once, or in FP64 where a pivot is below 1e-3 of
// the largest diagonal entry.  Returns whether the step is taken.
__device__ inline bool ct_step(FF t, int lane, FF c4, FF c2, FF (&k)[4]) {
  auto from = [](FF v, int src) { return FF{__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src)}; };
  // lanes 0 .. 9: entry (0,0) (0,1) (0,2) (0,3) (1,1) (1,2) (1,3) (2,2) (2,3) (3,3) of the matrix,
  // c4 s[8 + lane] - c2 sub; lanes 10 .. 13: c2 s[4 ..], minus the gradient
  const int i = lane < 14 ? lane : 13;
  const bool is_h = i < 10;
  const FF first = from(t, is_h ? 8 + i : i - 6);
  const FF b1 = from(t, (int)((0x0003213200ull >> (4 * i)) & 15u)), b2 = from(t, 1);
  const float f1 = is_h ? (float)((0x2021121102ull >> (4 * i)) & 15u) : 0.f, f2 = i == 7 || i == 9 ? 2.f : 0.f;
  const FF sub = ff_add(FF{f1 * b1.hi, f1 * b1.lo}, FF{f2 * b2.hi, f2 * b2.lo});
  const FF mine = ff_norm(ff_add(ff_mul(is_h ? c4 : c2, first), ff_neg(ff_mul(c2, sub))));
  float h[14];
  #pragma unroll
  for (int j = 0; j < 14; ++j) h[j] = __shfl_sync(0xffffffffu, mine.hi, j);
  const float dmax = fmaxf(fmaxf(h[0], h[4]), fmaxf(h[7], h[9]));
  if (!(dmax > 0.f)) return false;
  const float h00 = h[0], h01 = h[1], h02 = h[2], h03 = h[3], h11 = h[4], h12 = h[5], h13 = h[6];
  const float detA = h00 * h11 - h01 * h01, idA = __frcp_rn(detA);
  const float A00 = h11 * idA, A01 = -h01 * idA, A11 = h00 * idA;
  const float T00 = A00 * h02 + A01 * h12, T01 = A00 * h03 + A01 * h13;
  const float T10 = A01 * h02 + A11 * h12, T11 = A01 * h03 + A11 * h13;
  const float S00 = h[7] - (h02 * T00 + h12 * T10), S01 = h[8] - (h02 * T01 + h12 * T11);
  const float S11 = h[9] - (h03 * T01 + h13 * T11);
  const float detS = S00 * S11 - S01 * S01, idS = __frcp_rn(detS), tol = 1e-3f * dmax;
  if (h00 > tol && detA > tol * h00 && S00 > tol && detS > tol * S00) {
    auto solve = [&](const float (&r)[4], float (&x)[4]) {
      const float u0 = r[2] - (T00 * r[0] + T10 * r[1]), u1 = r[3] - (T01 * r[0] + T11 * r[1]);
      x[2] = (S11 * u0 - S01 * u1) * idS;
      x[3] = (S00 * u1 - S01 * u0) * idS;
      const float w0 = r[0] - (h02 * x[2] + h03 * x[3]), w1 = r[1] - (h12 * x[2] + h13 * x[3]);
      x[0] = A00 * w0 + A01 * w1;
      x[1] = A01 * w0 + A11 * w1;
    };
    float r[4] = {h[10], h[11], h[12], h[13]}, x[4], d[4];
    solve(r, x);
    // lane u & 3: the residual of row u, whose entries sit on lanes 0 1 2 3 | 1 4 5 6 | 2 5 7 8 | 3 6 8 9
    const unsigned row = lane & 2 ? (lane & 1 ? 0x9863u : 0x8752u) : (lane & 1 ? 0x6541u : 0x3210u);
    FF res = from(mine, 10 + (lane & 3));
    #pragma unroll
    for (int j = 0; j < 4; ++j) res = ff_mac(-x[j], from(mine, (int)((row >> (4 * j)) & 15u)), res);
    const float rf = ff_f(res);
    #pragma unroll
    for (int j = 0; j < 4; ++j) r[j] = __shfl_sync(0xffffffffu, rf, j);
    solve(r, d);
    #pragma unroll
    for (int j = 0; j < 4; ++j) k[j] = ff_two_sum(x[j], d[j]);
    return true;
  }
  // FP64 (the pivot test itself at 1e-6 of the largest diagonal entry)
  double H[10], r[4];
  #pragma unroll
  for (int j = 0; j < 10; ++j) H[j] = ff_d(from(mine, j));
  #pragma unroll
  for (int j = 0; j < 4; ++j) r[j] = ff_d(from(mine, 10 + j));
  const double dm = fmax(fmax(H[0], H[4]), fmax(H[7], H[9])), tol64 = 1e-6 * dm;
  const double dA = H[0] * H[4] - H[1] * H[1], iA = 1.0 / dA;
  const double a00 = H[4] * iA, a01 = -H[1] * iA, a11 = H[0] * iA;
  const double t00 = a00 * H[2] + a01 * H[5], t01 = a00 * H[3] + a01 * H[6];
  const double t10 = a01 * H[2] + a11 * H[5], t11 = a01 * H[3] + a11 * H[6];
  const double s00 = H[7] - (H[2] * t00 + H[5] * t10), s01 = H[8] - (H[2] * t01 + H[5] * t11);
  const double s11 = H[9] - (H[3] * t01 + H[6] * t11), dS = s00 * s11 - s01 * s01;
  if (!(H[0] > tol64 && dA > tol64 * H[0] && s00 > tol64 && dS > tol64 * s00)) return false;
  const double iS = 1.0 / dS, u0 = r[2] - (t00 * r[0] + t10 * r[1]), u1 = r[3] - (t01 * r[0] + t11 * r[1]);
  const double k2 = (s11 * u0 - s01 * u1) * iS, k3 = (s00 * u1 - s01 * u0) * iS;
  const double w0 = r[0] - (H[2] * k2 + H[3] * k3), w1 = r[1] - (H[5] * k2 + H[6] * k3);
  k[0] = ff_of(a00 * w0 + a01 * w1);
  k[1] = ff_of(a01 * w0 + a11 * w1);
  k[2] = ff_of(k2);
  k[3] = ff_of(k3);
  return true;
}

__global__ void __launch_bounds__(kClThreads, 1) k_cluster_taylor(ClusterTaylorArgs a) {
  extern __shared__ __align__(16) unsigned char cl_smem[];
  const int n = a.n_ant;
  float4* rows = reinterpret_cast<float4*>(cl_smem);                 // [apc][3][2][n]
  float4* Xb = rows + (size_t)6 * a.apc * n;                          // [2][4][n]
  __shared__ FF s_tot[kClMaxSlots][40];      // U0G, U1G, U2G, U1H, U2H
  __shared__ FF s_gram[kClMaxSlots][16];     // per warp
  __shared__ FF s_oth[kClMaxSlots][24];      // P', Q', R' as full 2x2 (re, im)
  __shared__ FFC s_C[kClMaxSlots][16];
  __shared__ FFC s_B[kClMaxSlots][8];
  __shared__ float2 s_W[kClMaxSlots][8];
  __shared__ float s_r[kClMaxSlots][kCtRot];
  __shared__ __align__(16) FF s_rsum[kCtRot];
  __shared__ __align__(16) FF s_red[2][kClMaxCta][kCtRot];
  __shared__ __align__(8) uint64_t s_bar[2], s_rbar[2];
  __shared__ int s_bad;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nthr = blockDim.x;
  const int rank = (int)cluster_rank(), CS = (int)cluster_size();
  const int slot = warp, p = rank + slot * CS;
  const bool live = p < n;
  if (tid == 0) {
    s_bad = 0;
    for (int i = 0; i < 2; ++i) {
      tc05::mbar_init(&s_bar[i], 1);
      tc05::mbar_init(&s_rbar[i], 1);
    }
  }
  float4* row = rows + (size_t)6 * slot * n;           // [3][2][n]
  if (live)
    for (int q = lane; q < n; q += 32)
      #pragma unroll
      for (int m = 0; m < 3; ++m) {
        float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0;
        if (q != p) {
          const float4* P4 = reinterpret_cast<const float4*>(a.mom + ((size_t)m * a.n_bl + bl_index(n, min(p, q), max(p, q))) * 4);
          r0 = __ldcg(P4);
          r1 = __ldcg(P4 + 1);
          if (q < p) {                               // M_pq = M_qp^H
            const float4 t0 = r0, t1 = r1;
            r0 = make_float4(t0.x, -t0.y, t1.x, -t1.y);
            r1 = make_float4(t0.z, -t0.w, t1.z, -t1.w);
          }
        }
        row[(2 * m) * n + q] = r0;
        row[(2 * m + 1) * n + q] = r1;
      }
  for (int i = tid; i < 4 * n; i += nthr)             // G = I, H = 0
    Xb[i] = i < n ? make_float4(1.f, 0.f, 0.f, 0.f) : (i < 2 * n ? make_float4(0.f, 0.f, 1.f, 0.f)
                                                                  : make_float4(0.f, 0.f, 0.f, 0.f));
  __syncthreads();
  cluster_sync();
  volatile int* bad = &s_bad;
  // this lane's destinations: rows (lane & 1) of G and of H in CTA lane >> 1
  const uint32_t dst_rank = (uint32_t)(lane >> 1);
  const bool sends = live && (int)dst_rank < CS;
  const uint32_t my_row = tc05::smem_u32(Xb) + (uint32_t)((lane & 1) * n + p) * 16u;
  const uint32_t dst_row = sends ? cluster_map(my_row, dst_rank) : 0u;
  const uint32_t dst_bar = sends ? cluster_map(tc05::smem_u32(&s_bar[0]), dst_rank) : 0u;
  const FF fS = ff_of(a.S), fmu0S = ff_of(a.mu0 * a.S), fmu2S = ff_of(a.mu2 * a.S), fmu4S = ff_of(a.mu4 * a.S);
  const FF c4 = ff_of(2.0 * a.S * a.S * a.mu4), c2 = ff_of(2.0 * a.S);
  // lanes 0 .. 7: entry e of X_p = [G H] (row er, column ec of 4), the rotated iterate
  const int e = lane & 7, er = (e & 3) >> 1, ec = (e < 4 ? 0 : 2) + (e & 1);
  FFC X = ffc_zero(), Xprev = X;
  if (e == 0 || e == 3) X.re.hi = 1.f;
  int n_red = 0;

  for (int it = 1; it <= a.n_iter + 1; ++it) {
    const bool fin = it == a.n_iter + 1;               // only the last iterate's rotation is left
    const bool rot = a.rotate && it >= 3;              // X^(it - 1) takes a step
    if (fin && !rot) break;
    const float4* Xc = Xb + (size_t)((it - 1) & 1) * 4 * n;
    if (tid == 0) {
      if (!fin) mbar_expect(&s_bar[it & 1], (uint32_t)n * 64u);
      if (rot) mbar_expect(&s_rbar[n_red & 1], (uint32_t)(CS * kCtRot * sizeof(FF)));
    }
    // ---- row sums of this warp's antenna
    {
      float u[48];
      #pragma unroll
      for (int i = 0; i < 48; ++i) u[i] = 0.f;
      if (live)
        for (int q = lane; q < n; q += 32) {
          const float4 g0 = Xc[q], g1 = Xc[n + q], h0 = Xc[2 * n + q], h1 = Xc[3 * n + q];
          float4 m0 = row[q], m1 = row[n + q];
          ct_mm(u, m0, m1, g0, g1);
          m0 = row[2 * n + q]; m1 = row[3 * n + q];
          ct_mm(u + 8, m0, m1, g0, g1);
          ct_mm(u + 24, m0, m1, h0, h1);
          m0 = row[4 * n + q]; m1 = row[5 * n + q];
          ct_mm(u + 16, m0, m1, g0, g1);
          ct_mm(u + 32, m0, m1, h0, h1);
        }
      #pragma unroll
      for (int b = 0; b < 3; ++b) {
        float v[16];
        #pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = u[16 * b + i];
        const FF t = warp_reduce_scatter16ff(v, lane);
        if ((lane & 1) == 0 && 16 * b + (lane >> 1) < 40) s_tot[slot][16 * b + (lane >> 1)] = t;
      }
    }
    // ---- Gram sums over all antennas, then the others' of this antenna
    {
      float v[16];
      #pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = 0.f;
      for (int q = tid; q < n; q += nthr) {
        float o[16];
        ct_gram(o, Xc[q], Xc[n + q], Xc[2 * n + q], Xc[3 * n + q]);
        #pragma unroll
        for (int i = 0; i < 16; ++i) v[i] += o[i];
      }
      const FF t = warp_reduce_scatter16ff(v, lane);
      if ((lane & 1) == 0) s_gram[warp][lane >> 1] = t;
    }
    __syncthreads();
    const int pc = live ? p : 0;
    const float4 g0 = Xc[pc], g1 = Xc[n + pc], h0 = Xc[2 * n + pc], h1 = Xc[3 * n + pc];
    float own[16];
    ct_gram(own, g0, g1, h0, h1);
    {
      const int i = lane & 15, nw = nthr >> 5;
      FF t = s_gram[0][i];
      for (int w = 1; w < nw; ++w) t = ff_add(t, s_gram[w][i]);
      float mine = own[0];
      #pragma unroll
      for (int j = 1; j < 16; ++j) mine = i == j ? own[j] : mine;
      const FF m = {-mine, 0.f};
      t = ff_norm(ff_add(t, m));
      // 2x2 layout: Hermitian P and R from (00, 11, re 01, im 01)
      if (lane < 16) {
        FF* o = s_oth[slot];
        const FF z = {0.f, 0.f};
        const int k = i & 3, base = i < 4 ? 0 : 16;
        if (i >= 4 && i < 12) o[8 + i - 4] = t;
        else if (k == 0) { o[base] = t; o[base + 1] = z; }
        else if (k == 1) { o[base + 6] = t; o[base + 7] = z; }
        else if (k == 2) { o[base + 2] = t; o[base + 4] = t; }
        else { o[base + 3] = t; o[base + 5] = ff_neg(t); }
      }
      __syncwarp();
    }
    auto oth = [&](int m, int r, int c) {               // entry (r, c) of P', Q', R' (m = 0, 1, 2)
      const FF* o = s_oth[slot] + 8 * m + 2 * (2 * r + c);
      return FFC{o[0], o[1]};
    };
    auto othf = [&](int m, int r, int c) {
      const FF* o = s_oth[slot] + 8 * m + 2 * (2 * r + c);
      return make_float2(o[0].hi, o[1].hi);
    };
    auto herm = [&](FFC v) { v.im = ff_neg(v.im); return v; };
    // ---- the rotation step of X^(it - 1)
    FF k[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    const float2 G[4] = {make_float2(g0.x, g0.y), make_float2(g0.z, g0.w), make_float2(g1.x, g1.y), make_float2(g1.z, g1.w)};
    const float2 H[4] = {make_float2(h0.x, h0.y), make_float2(h0.z, h0.w), make_float2(h1.x, h1.y), make_float2(h1.z, h1.w)};
    if (rot) {
      {
        // lanes 0 .. 3: W^G, lanes 4 .. 7: W^H, entry (er, c)
        const int c = e & 1, hi = e >> 2;
        FFC t2 = ffc_zero(), t4 = t2;
        #pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float2 gg = er ? (j ? G[3] : G[2]) : (j ? G[1] : G[0]), hh = er ? (j ? H[3] : H[2]) : (j ? H[1] : H[0]);
          t2 = ffc_mac(gg, oth(hi, j, c), t2);                          // G P' or G Q'
          t4 = ffc_mac(hh, hi ? oth(2, j, c) : herm(oth(1, c, j)), t4);   // H R' or H Q'^H
        }
        const FF* U = s_tot[slot] + (hi ? 32 : 16) + 2 * (2 * er + c);
        const FF wr = ff_add(U[0], ff_neg(ff_add(ff_mul(fmu2S, t2.re), ff_mul(fmu4S, t4.re))));
        const FF wi = ff_add(U[1], ff_neg(ff_add(ff_mul(fmu2S, t2.im), ff_mul(fmu4S, t4.im))));
        if (lane < 8) s_W[slot][e] = make_float2(ff_f(wr), ff_f(wi));
      }
      __syncwarp();
      float val[kCtRot];
      {
        const float2* W = s_W[slot];
        // Y = W^G^H G, Z = W^H^H G - W^G^H H
        float2 Y[4], Z[4];
        #pragma unroll
        for (int i = 0; i < 2; ++i)
          #pragma unroll
          for (int j = 0; j < 2; ++j) {
            Y[2 * i + j] = cadd(cconjmul(W[i], G[j]), cconjmul(W[2 + i], G[2 + j]));
            Z[2 * i + j] = csub(cadd(cconjmul(W[4 + i], G[j]), cconjmul(W[6 + i], G[2 + j])),
                                cadd(cconjmul(W[i], H[j]), cconjmul(W[2 + i], H[2 + j])));
          }
        val[0] = Y[0].x; val[1] = Y[3].x; val[2] = Y[1].x + Y[2].x; val[3] = Y[2].y - Y[1].y;
        val[4] = -Z[0].y; val[5] = -Z[3].y; val[6] = -(Z[1].y + Z[2].y); val[7] = Z[2].x - Z[1].x;
        // sum of tr(B_a X B_b Y) over (P, R'), (R, P'), -(Q, Q'), -(Q^H, Q'^H)
        #pragma unroll
        for (int i = 8; i < kCtRot; ++i) val[i] = 0.f;
        #pragma unroll
        for (int m = 0; m < 4; ++m) {
          float2 x[4], y[4];
          #pragma unroll
          for (int r = 0; r < 2; ++r)
            #pragma unroll
            for (int c = 0; c < 2; ++c) {
              const float* h4 = own + (m == 0 ? 0 : 12);
              float2 v;
              if (m < 2) v = r == c ? make_float2(h4[r], 0.f) : make_float2(h4[2], r ? -h4[3] : h4[3]);
              else v = m == 2 ? make_float2(own[4 + 2 * (2 * r + c)], own[5 + 2 * (2 * r + c)])
                              : make_float2(own[4 + 2 * (2 * c + r)], -own[5 + 2 * (2 * c + r)]);
              x[2 * r + c] = v;
              y[2 * r + c] = m < 2 ? othf(m == 0 ? 2 : 0, r, c) : (m == 2 ? othf(1, r, c) : cconj(othf(1, c, r)));
            }
          const float sg = m < 2 ? 1.f : -1.f;
          auto pr = [&](int i, int j) { return make_float2(sg * (x[i].x * y[j].x - x[i].y * y[j].y), sg * (x[i].x * y[j].y + x[i].y * y[j].x)); };
          const float2 p00 = pr(0, 0), p12 = pr(1, 2), p02 = pr(0, 2), p10 = pr(1, 0), p33 = pr(3, 3), p23 = pr(2, 3),
                       p31 = pr(3, 1), p22 = pr(2, 2), p30 = pr(3, 0), p03 = pr(0, 3), p11 = pr(1, 1);
          val[8] += p00.x;                              // (0, 0)
          val[9] += p12.x;                              // (0, 1)
          val[10] += p02.x + p10.x;                     // (0, 2)
          val[11] += p02.y - p10.y;                     // (0, 3): Re(-i a + i b) = Im a - Im b
          val[12] += p33.x;                             // (1, 1)
          val[13] += p23.x + p31.x;                     // (1, 2)
          val[14] += p23.y - p31.y;                     // (1, 3)
          val[15] += p22.x + p30.x + p03.x + p11.x;     // (2, 2)
          val[16] += (p22.y + p03.y) - (p30.y + p11.y); // (2, 3)
          val[17] += p30.x + p03.x - p22.x - p11.x;     // (3, 3)
        }
      }
      if (lane == 0)
        #pragma unroll
        for (int i = 0; i < kCtRot; ++i) s_r[slot][i] = live ? 0.5f * val[i] : 0.f;
      __syncthreads();
      if (tid < kCtRot) {
        FF v[kClMaxSlots];
        #pragma unroll
        for (int q = 0; q < kClMaxSlots; ++q) v[q] = FF{q < a.apc ? s_r[q][tid] : 0.f, 0.f};
        #pragma unroll
        for (int o = kClMaxSlots / 2; o >= 1; o >>= 1)
          #pragma unroll
          for (int q = 0; q < o; ++q) v[q] = ff_add(v[q], v[q + o]);
        const FF t = v[0];
        s_rsum[tid] = ff_norm(t);
      }
      __syncthreads();
      const int rb = n_red & 1;
      constexpr int kPieces = kCtRot * (int)sizeof(FF) / 16;
      for (int i = tid; i < kPieces * CS && !*bad; i += nthr) {
        const uint32_t dr = (uint32_t)(i / kPieces);
        const int piece = i % kPieces;
        const float4 v = reinterpret_cast<const float4*>(s_rsum)[piece];
        cluster_send16(cluster_map(tc05::smem_u32(reinterpret_cast<float4*>(s_red[rb][rank]) + piece), dr), v,
                       cluster_map(tc05::smem_u32(&s_rbar[rb]), dr));
      }
      cluster_wait(&s_rbar[rb], (uint32_t)(n_red >> 1) & 1u, bad);
      ++n_red;
      FF t = {0.f, 0.f};
      if (lane < kCtRot) {                             // the CTAs' sums, pairwise
        FF v[kClMaxCta];
        #pragma unroll
        for (int r = 0; r < kClMaxCta; ++r) v[r] = r < CS ? s_red[rb][r][lane] : t;
        #pragma unroll
        for (int o = kClMaxCta / 2; o >= 1; o >>= 1)
          #pragma unroll
          for (int r = 0; r < o; ++r) v[r] = ff_add(v[r], v[r + o]);
        t = v[0];
      }
      __syncwarp();
      if (!ct_step(t, lane, c4, c2, k)) {
        const FF z = {0.f, 0.f};
        k[0] = k[1] = k[2] = k[3] = z;
      }
      // H += i G K, K = [k0, k2 - i k3; k2 + i k3, k1] (own rotated iterate, lanes 4 .. 7)
      if (e >= 4) {
        const int c = e & 1;
        const FF zf = {0.f, 0.f};
        const FFC K0 = c ? FFC{k[2], ff_neg(k[3])} : FFC{k[0], zf}, K1 = c ? FFC{k[1], zf} : FFC{k[2], k[3]};
        FFC gk = ffc_mac(er ? G[2] : G[0], K0, ffc_zero());
        gk = ffc_mac(er ? G[3] : G[1], K1, gk);
        X.re = ff_norm(ff_add(X.re, ff_neg(gk.im)));
        X.im = ff_norm(ff_add(X.im, gk.re));
      }
    }
    if (fin) break;
    // ---- the sweep: right-hand sides and normal matrix from the rotated sums
    const float2 Kf[4] = {make_float2(k[0].hi, 0.f), make_float2(k[2].hi, -k[3].hi), make_float2(k[2].hi, k[3].hi),
                          make_float2(k[1].hi, 0.f)};
    auto cmi = [](float2 x) { return make_float2(-x.y, x.x); };                // i x
    {
      const int c = e & 1, hi = e >> 2, at = 2 * (2 * er + c);
      const FF* T = s_tot[slot];
      FFC b;
      b.re = ff_add(T[(hi ? 8 : 0) + at], T[(hi ? 32 : 24) + at]);             // U0G + U1H, U1G + U2H
      b.im = ff_add(T[(hi ? 8 : 0) + at + 1], T[(hi ? 32 : 24) + at + 1]);
      const FF* U = T + (hi ? 16 : 8) + 4 * er;                                // row er of U1G, U2G
      #pragma unroll
      for (int j = 0; j < 2; ++j) b = ffc_mac(cmi(j ? (c ? Kf[3] : Kf[2]) : (c ? Kf[1] : Kf[0])), FFC{U[2 * j], U[2 * j + 1]}, b);
      b.re = ff_norm(b.re);
      b.im = ff_norm(b.im);
      if (lane < 8) s_B[slot][(er << 2) + ec] = b;
    }
    {
      // entry (R, Cc) of S [mu0 P + mu2 R'', mu2 (Q'' + Q''^H); ., mu2 P + mu4 R'']
      const int t = lane & 15, R = t >> 2, Cc = t & 3, bi = R >> 1, bj = Cc >> 1, i = R & 1, j = Cc & 1;
      float2 Pf[4], Qf[4];
      #pragma unroll
      for (int x = 0; x < 4; ++x) { Pf[x] = othf(0, x >> 1, x & 1); Qf[x] = othf(1, x >> 1, x & 1); }
      float2 PK[4];
      #pragma unroll
      for (int r = 0; r < 2; ++r)
        #pragma unroll
        for (int c = 0; c < 2; ++c) PK[2 * r + c] = cadd(cmul(Pf[2 * r], Kf[c]), cmul(Pf[2 * r + 1], Kf[2 + c]));
      FFC v;
      if (bi != bj) {
        // Q'' = Q' + i P' K; block (0, 1) and its Hermitian transpose are equal
        const float2 d0 = cmi(i ? (j ? PK[3] : PK[2]) : (j ? PK[1] : PK[0]));
        const float2 d1 = cconj(cmi(j ? (i ? PK[3] : PK[2]) : (i ? PK[1] : PK[0])));
        const FFC q0 = oth(1, i, j), q1 = herm(oth(1, j, i));
        v.re = ff_add(q0.re, q1.re);
        v.im = ff_add(q0.im, q1.im);
        const FF dr = ff_two_sum(d0.x, d1.x), di = ff_two_sum(d0.y, d1.y);
        v.re = ff_mul(fmu2S, ff_norm(ff_add(v.re, dr)));
        v.im = ff_mul(fmu2S, ff_norm(ff_add(v.im, di)));
      } else {
        // R'' = R' + i Q'^H K - i K Q' + K P' K
        float2 d = make_float2(0.f, 0.f);
        #pragma unroll
        for (int m = 0; m < 2; ++m) {
          const float2 qh = cconj(i ? (m ? Qf[3] : Qf[1]) : (m ? Qf[2] : Qf[0]));       // Q'^H [i][m] = conj(Q'[m][i])
          const float2 kj = m ? (j ? Kf[3] : Kf[2]) : (j ? Kf[1] : Kf[0]);               // K [m][j]
          const float2 ki = i ? (m ? Kf[3] : Kf[2]) : (m ? Kf[1] : Kf[0]);               // K [i][m]
          const float2 qj = m ? (j ? Qf[3] : Qf[2]) : (j ? Qf[1] : Qf[0]);               // Q' [m][j]
          const float2 pk = m ? (j ? PK[3] : PK[2]) : (j ? PK[1] : PK[0]);               // (P' K) [m][j]
          d = cadd(d, cmi(csub(cmul(qh, kj), cmul(ki, qj))));
          d = cadd(d, cmul(ki, pk));
        }
        FFC r = oth(2, i, j);
        const FF dr = {d.x, 0.f}, di = {d.y, 0.f};
        r.re = ff_norm(ff_add(r.re, dr));
        r.im = ff_norm(ff_add(r.im, di));
        const FFC pp = oth(0, i, j);
        v.re = ff_add(ff_mul(bi ? fmu2S : fmu0S, pp.re), ff_mul(bi ? fmu4S : fmu2S, r.re));
        v.im = ff_add(ff_mul(bi ? fmu2S : fmu0S, pp.im), ff_mul(bi ? fmu4S : fmu2S, r.im));
      }
      v.re = ff_norm(v.re);
      v.im = ff_norm(v.im);
      if (i == j && bi == bj) { v.im.hi = 0.f; v.im.lo = 0.f; }
      if (lane < 16) s_C[slot][t] = v;
    }
    __syncwarp();
    {
      float2 C[4][4], b[4], x0, d0;
      #pragma unroll
      for (int i = 0; i < 16; ++i) C[i >> 2][i & 3] = make_float2(s_C[slot][i].re.hi, s_C[slot][i].im.hi);
      #pragma unroll
      for (int c = 0; c < 4; ++c) b[c] = make_float2(s_B[slot][4 * er + c].re.hi, s_B[slot][4 * er + c].im.hi);
      const bool ok = ct_schur4f(C, b, ec, &x0);
      FFC Xn;
      if (__all_sync(0xffffffffu, ok || !live)) {
        // residual of this lane's row: b - x C, entry ec
        FFC r = s_B[slot][4 * er + ec];
        #pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int src = (u < 2 ? 0 : 4) + 2 * er + (u & 1);              // lane of entry (er, u)
          const float2 xu = make_float2(__shfl_sync(0xffffffffu, x0.x, src), __shfl_sync(0xffffffffu, x0.y, src));
          r = ffc_mac(make_float2(-xu.x, -xu.y), s_C[slot][4 * u + ec], r);
        }
        const float2 rf = make_float2(ff_f(r.re), ff_f(r.im));
        float2 rr[4];
        #pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int src = (u < 2 ? 0 : 4) + 2 * er + (u & 1);
          rr[u] = make_float2(__shfl_sync(0xffffffffu, rf.x, src), __shfl_sync(0xffffffffu, rf.y, src));
        }
        ct_schur4f(C, rr, ec, &d0);
        Xn.re = ff_two_sum(x0.x, d0.x);
        Xn.im = ff_two_sum(x0.y, d0.y);
      } else {
        double2 Cd[4][4], bd[4], xd;
        #pragma unroll
        for (int i = 0; i < 16; ++i) Cd[i >> 2][i & 3] = make_double2(ff_d(s_C[slot][i].re), ff_d(s_C[slot][i].im));
        #pragma unroll
        for (int c = 0; c < 4; ++c) bd[c] = make_double2(ff_d(s_B[slot][4 * er + c].re), ff_d(s_B[slot][4 * er + c].im));
        if (!schur_solve4_entry(Cd, bd, ec, &xd)) xd = make_double2(NAN, NAN);
        Xn.re = ff_of(xd.x);
        Xn.im = ff_of(xd.y);
      }
      Xprev = X;
      if ((it & 1) == 0) {
        Xn.re = ff_norm(ff_add(Xn.re, X.re));
        Xn.im = ff_norm(ff_add(Xn.im, X.im));
        Xn.re.hi *= 0.5f; Xn.re.lo *= 0.5f; Xn.im.hi *= 0.5f; Xn.im.lo *= 0.5f;
      }
      X = Xn;
    }
    // ---- row lane & 1 of G and of H to CTA lane >> 1
    {
      const int g = 2 * (lane & 1);
      float4 vg, vh;
      vg.x = __shfl_sync(0xffffffffu, X.re.hi, g);     vg.y = __shfl_sync(0xffffffffu, X.im.hi, g);
      vg.z = __shfl_sync(0xffffffffu, X.re.hi, g + 1); vg.w = __shfl_sync(0xffffffffu, X.im.hi, g + 1);
      vh.x = __shfl_sync(0xffffffffu, X.re.hi, g + 4); vh.y = __shfl_sync(0xffffffffu, X.im.hi, g + 4);
      vh.z = __shfl_sync(0xffffffffu, X.re.hi, g + 5); vh.w = __shfl_sync(0xffffffffu, X.im.hi, g + 5);
      const uint32_t bb = (uint32_t)(it & 1);
      if (sends && !*bad) {
        cluster_send16(dst_row + bb * 64u * (uint32_t)n, vg, dst_bar + 8u * bb);
        cluster_send16(dst_row + bb * 64u * (uint32_t)n + 32u * (uint32_t)n, vh, dst_bar + 8u * bb);
      }
      cluster_wait(&s_bar[bb], (uint32_t)((it - 1) >> 1) & 1u, bad);
    }
  }
  // ---- the solution and the last sweep's norms
  if (live) {
    const double2 Xd = make_double2(ff_d(X.re), ff_d(X.im)), Xo = make_double2(ff_d(Xprev.re), ff_d(Xprev.im));
    const double dx = Xd.x - Xo.x, dy = Xd.y - Xo.y;
    double dn = dx * dx + dy * dy, nn = Xd.x * Xd.x + Xd.y * Xd.y;
    int nf = !(isfinite(Xd.x) && isfinite(Xd.y));
    #pragma unroll
    for (int o = 1; o <= 4; o <<= 1) {
      dn += __shfl_xor_sync(0xffffffffu, dn, o);
      nn += __shfl_xor_sync(0xffffffffu, nn, o);
      nf |= __shfl_xor_sync(0xffffffffu, nf, o);
    }
    if (lane < 8) {
      const float2 Xs = make_float2((float)Xd.x, (float)Xd.y);
      a.X[(size_t)p * 8 + e] = Xd;
      a.Xf[(size_t)p * 8 + e] = Xs;
      *(e < 4 ? a.gain + (size_t)p * 4 + e : a.slope + (size_t)p * 4 + (e - 4)) = Xs;
      if (e == 0) {
        a.norms[4 * p] = dn;
        a.norms[4 * p + 1] = nn;
        a.norms[4 * p + 2] = (double)nf;
      }
    }
  }
  if (*bad) __nanosleep(100000);
  cluster_sync();
  if (rank == 0 && warp == 0) cluster_status(a.norms, n, lane, *bad, a.status, a.rel);
  cluster_sync();
  if (*bad && tid == 0) *a.status = kSolveStatusTimeout;
}

}  // namespace rts
