// Solve of a group of sources of the blocked peel by one thread-block cluster.
//
// The chain of a source (corrected average, n_iter Jacobi sweeps) is bound by
// how fast every antenna's new Jones matrix reaches every other antenna.
// Between the CTAs of a grid that is a global barrier and a trip through L2
// (about 5 600 cycles a sweep in k_block_solve); between the CTAs of a cluster
// it is one store into the other CTA's shared memory that also counts itself
// in on that CTA's mbarrier.  For arrays whose rows fit in the shared memory of
// one cluster the chain therefore runs in one cluster of at most 16 CTAs, and
// the in-block corrections, which one cluster is too narrow for, are split in
// two: before each group of kClGroup sources k_cluster_prep takes the terms of
// all earlier sources of the block out of the group's averages with the whole
// GPU, and the cluster only adds the terms of the group's own sources.  The
// same kernel lays both out for the cluster as full antenna matrices (V_qp =
// V_pq^H, D_qp = conj(D_pq)): gathered from the baseline-ordered tables a row
// cost 14 scattered loads a partner pair, 8 us a source at 128 antennas.
//
// A CTA owns the antennas p = rank + slot CS.  Per source q of the group:
//   rows: V_pq of its antennas in shared memory, with the terms
//     S_j D_jq J_p J_q^H of the group's solved sources j < q taken out.
//   sweeps: one warp a slot, each lane the partners lane + 32 u, up to kClChain terms
//     added in FP32 one after another; of the warp's shuffle tree the first level in
//     FP32, the others float-float, the total rounded once.  (k_block_solve: trees of 32
//     FP32 terms, their totals in FP64, rounded once; in units of a term's rounding
//     157 there and 146 here at 128 antennas, 287 and 282 at 256.)  The warp solves the
//     2x2 system (each lane the row it sends) and lane (rank,
//     row) stores one 16-byte row of J_p into CTA `rank` with st.async, which
//     completes 16 bytes of that CTA's mbarrier transaction count; a CTA starts
//     the next sweep when all n_ant matrices have arrived.  Iterates alternate
//     between two buffers and two mbarriers: a CTA sends sweep g + 1 only after
//     it has received every matrix of sweep g, which every CTA sends after its
//     last read of the buffer that sweep g + 1 overwrites, and after its wait for
//     sweep g - 1, so no store can reach a buffer still read or a barrier phase
//     still open.  That holds for warps that send; a warp whose slot has no antenna
//     sends nothing, so nobody would wait for it and the phase it waits for could be two
//     behind: it reads no iterate and waits for none of the sweeps' barriers (it meets the
//     others at the last sweep's CTA barriers and at the cluster barrier).
//   last sweep: a partner's terms in FP32, everything after that in float-float (about 47
//     bits; an FP64 tree cost 5 us a source here), the 2x2 solve, the averaging
//     and the relative change in FP64 against the FP32 previous iterate.
// Measured (GB300, 20 sweeps): 35 us a source at 128 antennas where k_block_solve
// took 87 (its barriers alone 54), 27 against 83 at 65, 22 against 80 at 32.  At 128
// antennas a sweep is about 2 700 cycles: 1 000 of FP32 terms, 400 of the tree,
// 300 of the 2x2 solve and 1 000 of the exchange.  Error of the gains against 64 bits,
// 61 sources on 65 antennas x 203 channels x 3 times / 50 on 128 x 128 x 8 (8 seeds):
// 2.4e-7 / 1.9e-7, with k_block_solve's schedule 3.3e-7 / 2.6e-7; with the corrections
// of a group summed in FP32 3.8e-7 / 2.7e-7.
// Every wait is bounded (kSolveWaitNs).  A CTA whose wait ran out keeps its
// control flow, but waits and sends no more and marks the group's statuses
// kSolveStatusTimeout; no CTA exits before the last cluster barrier, so no store
// can meet an exited CTA.
#pragma once
#include "kahan.cuh"
#include "solve_kernels.cuh"
#include "tc05.cuh"

namespace rts {

constexpr int kClThreads = 512;            // at most (a warp per slot)
constexpr int kClGroup = 8;                // sources per launch
constexpr int kClMaxCta = 16;
constexpr int kClChain = 4;                // partners whose terms a lane adds one after another
constexpr int kClMaxSlots = 16;            // antennas per CTA, at most
constexpr int kClSlots = 8;                // and as many where more CTAs can be had: two warps a
                                           // sub-partition; the exchange costs the same whatever the CTAs

// terms (s, j), j < s, of a group's sources
__host__ __device__ constexpr int cl_pair(int s, int j) { return s * (s - 1) / 2 + j; }
constexpr int kClPairs = kClGroup * (kClGroup - 1) / 2;

struct ClusterSolveArgs {
  const float4* V;         // [kClGroup][n_ant][2][n_ant] averages, corrected for the sources before the group
  const float2* D;         // [kClPairs][n_ant][n_ant] closed-form averages D_jq of the group's sources
  const double* src;       // [n_src][3] (l, m, S)
  int s0;                  // first source of the block
  int q0, n_grp;           // first source of the group in the block, sources in it (<= kClGroup)
  int n_ant;
  int64_t n_bl;
  int n_iter;
  int apc;                 // antenna slots per CTA: ceil(n_ant / cluster size)
  float2* M;               // [BK][n_bl][4] model matrices of the block (written)
  double* part;            // [BK][n_ant][4] per antenna, last sweep: dn, nn, non-finite
  int* status;             // [n_src]
  double* rel;             // [n_src]
  float2* jones;           // [n_src][n_ant][4]
};

// dynamic shared memory: rows [apc][2][n_ant] float4, two iterates and the
// group's solved matrices [2 + kClGroup][2][n_ant] float4
inline size_t cluster_solve_smem(int n_ant, int apc) {
  return ((size_t)apc + 2 + kClGroup) * 2 * n_ant * sizeof(float4);
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// the address in CTA `rank` of the cluster that corresponds to this CTA's shared address
__device__ __forceinline__ uint32_t cluster_map(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// 16 bytes into a CTA of the cluster; they count on the mbarrier `bar` of the same CTA
__device__ __forceinline__ void cluster_send16(uint32_t dst, float4 v, uint32_t bar) {
  asm volatile(
      "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst),
      "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc05::smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, 20000;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(tc05::smem_u32(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
// wait for a phase unless the CTA has given up; sets *bad when the limit runs out
__device__ __forceinline__ void cluster_wait(uint64_t* bar, uint32_t parity, volatile int* bad) {
  if (mbar_try_cluster(bar, parity)) return;
  const unsigned long long t0 = global_ns();
  for (unsigned spin = 0; !mbar_try_cluster(bar, parity); ++spin) {
    if (*bad) return;
    if (spin > kSolveMaxSpins || global_ns() - t0 > kSolveWaitNs) {
      *bad = 1;
      return;
    }
  }
}

__device__ __forceinline__ FF ff_shfl_xor(FF x, int o) {
  FF r;
  r.hi = __shfl_xor_sync(0xffffffffu, x.hi, o);
  r.lo = __shfl_xor_sync(0xffffffffu, x.lo, o);
  return r;
}
// the last four levels of the sums below
__device__ __forceinline__ FF warp_reduce_scatter8ff(FF (&w)[8], int lane) {
  #pragma unroll
  for (int o = 8, n = 8; o >= 2; o >>= 1, n >>= 1) {
    const bool upper = (lane & o) != 0;
    #pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const FF send = upper ? w[i] : w[i + n / 2], keep = upper ? w[i + n / 2] : w[i];
      w[i] = ff_add(keep, ff_shfl_xor(send, o));
    }
  }
  return ff_add(w[0], ff_shfl_xor(w[0], 1));
}

// Reduce 16 floats over the 32 lanes of a warp (each level exchanges half of the
// remaining values with the partner lane) with the last four levels, whose sums are
// the large ones, in float-float; afterwards lane L holds the warp total of value
// index L >> 1, rounded once
__device__ __forceinline__ float warp_reduce_scatter16c(float (&v)[16], int lane) {
  {
    const bool upper = (lane & 16) != 0;
    #pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float send = upper ? v[i] : v[i + 8], keep = upper ? v[i + 8] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
  }
  FF w[4];
  {
    const bool upper = (lane & 8) != 0;
    #pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float send = upper ? v[i] : v[i + 4], keep = upper ? v[i + 4] : v[i];
      w[i] = ff_two_sum(keep, __shfl_xor_sync(0xffffffffu, send, 8));
    }
  }
  #pragma unroll
  for (int o = 4, n = 4; o >= 2; o >>= 1, n >>= 1) {
    const bool upper = (lane & o) != 0;
    #pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const FF send = upper ? w[i] : w[i + n / 2], keep = upper ? w[i + n / 2] : w[i];
      w[i] = ff_add(keep, ff_shfl_xor(send, o));
    }
  }
  const FF t = ff_add(w[0], ff_shfl_xor(w[0], 1));
  return t.hi + t.lo;
}
// the same of 16 floats, all levels in float-float
__device__ __forceinline__ FF warp_reduce_scatter16ff(const float (&v)[16], int lane) {
  FF w[8];
  {
    const bool upper = (lane & 16) != 0;
    #pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float send = upper ? v[i] : v[i + 8], keep = upper ? v[i + 8] : v[i];
      w[i] = ff_two_sum(keep, __shfl_xor_sync(0xffffffffu, send, 16));
    }
  }
  return warp_reduce_scatter8ff(w, lane);
}
// the same of 12 float-float values (and four zeros)
__device__ __forceinline__ FF warp_reduce_scatter12ff(const FF (&v)[12], int lane) {
  const FF zero = {0.f, 0.f};
  FF w[8];
  const bool upper = (lane & 16) != 0;
  #pragma unroll
  for (int i = 0; i < 8; ++i) {
    const FF hi = i < 4 ? v[i + 8] : zero;
    const FF send = upper ? v[i] : hi, keep = upper ? hi : v[i];
    w[i] = ff_add(keep, ff_shfl_xor(send, 16));
  }
  return warp_reduce_scatter8ff(w, lane);
}

// A group's input from the block's tables: V_s = A_s - sum_{j<q0} M_j D_js of its
// sources s = q0 .. q0 + n_grp - 1 and their own terms D_js (j >= q0), both as full
// antenna matrices.  Four threads a baseline, two targets each: M_j is read once
// for both, and the four threads' reads of it meet in the same 32 bytes.  Bound
// by L2 (M_j and D_jk once each, the matrices' stores).
// It is resident while the launch before it writes M, so M is read from L2 and through
// no pointer that promises read-only data (D_jk, the averages and the antenna pairs
// are older than both launches).
__global__ void __launch_bounds__(128) k_cluster_prep(const float2* __restrict__ Ablk, int q0, int n_grp,
                                                     const float2* Mblk, const float2* __restrict__ Dtab,
                                                     const int2* __restrict__ bl_ant, int n_ant, int64_t n_bl,
                                                     float4* V, float2* D) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t bl = idx >> 2;
  const int g0 = 2 * (int)(idx & 3);
  if (bl >= n_bl || g0 >= n_grp) {
    grid_next_may_start();
    return;
  }
  const bool two = g0 + 1 < n_grp;
  const int ka = q0 + g0, kb = two ? ka + 1 : ka;
  const float2* Da = Dtab + dir_index(n_bl, bl, 0, ka);
  const float2* Db = Dtab + dir_index(n_bl, bl, 0, kb);
  const float4* M4 = reinterpret_cast<const float4*>(Mblk) + 2 * bl;
  const int2 ij = bl_ant[bl];
  grid_previous_done();                      // the group before it has written its models
  grid_next_may_start();
  const int64_t up = (int64_t)ij.x * n_ant + ij.y, lo = (int64_t)ij.y * n_ant + ij.x, nn = (int64_t)n_ant * n_ant;
  // sums of eight terms in FP32, added to A - (those before) in float-float: near the
  // phase centre and on short baselines the terms add up to many times the difference
  FF va[8], vb[8];
  auto load = [&](int s, FF (&v)[8]) {
    const float4* A = reinterpret_cast<const float4*>(Ablk + ((size_t)(q0 + s) * n_bl + bl) * 4);
    const float4 a0 = A[0], a1 = A[1];
    const float x[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
    #pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = FF{x[e], 0.f};
  };
  load(g0, va);
  load(two ? g0 + 1 : g0, vb);
  auto cfma = [](float2 acc, float2 m, float2 d) {
    acc.x = fmaf(m.x, d.x, fmaf(-m.y, d.y, acc.x));
    acc.y = fmaf(m.x, d.y, fmaf(m.y, d.x, acc.y));
    return acc;
  };
  auto less = [](FF (&v)[8], const float2 (&t)[4]) {
    #pragma unroll
    for (int e = 0; e < 4; ++e) {
      const FF x = ff_two_sum(v[2 * e].hi, -t[e].x), y = ff_two_sum(v[2 * e + 1].hi, -t[e].y);
      v[2 * e] = FF{x.hi, v[2 * e].lo + x.lo};
      v[2 * e + 1] = FF{y.hi, v[2 * e + 1].lo + y.lo};
    }
  };
  for (int j0 = 0; j0 < q0; j0 += kClGroup) {              // q0: a multiple of kClGroup
    float2 ta[4], tb[4];
    #pragma unroll
    for (int e = 0; e < 4; ++e) ta[e] = tb[e] = make_float2(0.f, 0.f);
    #pragma unroll
    for (int j = j0; j < j0 + kClGroup; ++j) {
      const float4 m0 = __ldcg(M4 + (size_t)j * n_bl * 2), m1 = __ldcg(M4 + (size_t)j * n_bl * 2 + 1);
      const float2 m[4] = {make_float2(m0.x, m0.y), make_float2(m0.z, m0.w), make_float2(m1.x, m1.y),
                           make_float2(m1.z, m1.w)};
      const float2 da = __ldg(Da + j), db = __ldg(Db + j);
      #pragma unroll
      for (int e = 0; e < 4; ++e) {
        ta[e] = cfma(ta[e], m[e], da);
        tb[e] = cfma(tb[e], m[e], db);
      }
    }
    less(va, ta);
    less(vb, tb);
  }
  auto put = [&](int s, const FF (&v)[8], const float2* Dk) {
    const float4 a0 = make_float4(v[0].hi + v[0].lo, v[1].hi + v[1].lo, v[2].hi + v[2].lo, v[3].hi + v[3].lo);
    const float4 a1 = make_float4(v[4].hi + v[4].lo, v[5].hi + v[5].lo, v[6].hi + v[6].lo, v[7].hi + v[7].lo);
    // [p][plane][q]: planes of entries (0, 1) and (2, 3); V_qp = V_pq^H below the diagonal
    float4* Vs = V + (size_t)s * 2 * nn;
    Vs[(int64_t)ij.x * 2 * n_ant + ij.y] = a0;
    Vs[(int64_t)ij.x * 2 * n_ant + n_ant + ij.y] = a1;
    Vs[(int64_t)ij.y * 2 * n_ant + ij.x] = make_float4(a0.x, -a0.y, a1.x, -a1.y);
    Vs[(int64_t)ij.y * 2 * n_ant + n_ant + ij.x] = make_float4(a0.z, -a0.w, a1.z, -a1.w);
    for (int j = 0; j < s; ++j) {
      const float2 d = __ldg(Dk + q0 + j);
      D[cl_pair(s, j) * nn + up] = d;
      D[cl_pair(s, j) * nn + lo] = make_float2(d.x, -d.y);
    }
  };
  put(g0, va, Da);
  if (two) put(g0 + 1, vb, Db);
}

// normal-equation terms of one partner: A += V J (8 reals), C += J^H J (c00,
// c11, re c01, im c01), entries row-major, complex interleaved.  J is near the identity:
// the products with its small entries first, so that a partner's own sum (v = 0) is
// rounded once at its full size
__device__ __forceinline__ void als_terms(float (&v)[16], const float4 v0, const float4 v1, const float4 j0,
                                          const float4 j1) {
  auto row = [](float* a, float4 m, float4 j0, float4 j1) {
    a[0] = fmaf(m.z, j1.x, a[0]); a[0] = fmaf(-m.w, j1.y, a[0]); a[0] = fmaf(-m.y, j0.y, a[0]); a[0] = fmaf(m.x, j0.x, a[0]);
    a[1] = fmaf(m.z, j1.y, a[1]); a[1] = fmaf(m.w, j1.x, a[1]); a[1] = fmaf(m.x, j0.y, a[1]); a[1] = fmaf(m.y, j0.x, a[1]);
    a[2] = fmaf(m.x, j0.z, a[2]); a[2] = fmaf(-m.y, j0.w, a[2]); a[2] = fmaf(-m.w, j1.w, a[2]); a[2] = fmaf(m.z, j1.z, a[2]);
    a[3] = fmaf(m.x, j0.w, a[3]); a[3] = fmaf(m.y, j0.z, a[3]); a[3] = fmaf(m.z, j1.w, a[3]); a[3] = fmaf(m.w, j1.z, a[3]);
  };
  row(v, v0, j0, j1);
  row(v + 4, v1, j0, j1);
  v[8] = fmaf(j1.x, j1.x, v[8]); v[8] = fmaf(j1.y, j1.y, v[8]); v[8] = fmaf(j0.y, j0.y, v[8]); v[8] = fmaf(j0.x, j0.x, v[8]);
  v[9] = fmaf(j0.z, j0.z, v[9]); v[9] = fmaf(j0.w, j0.w, v[9]); v[9] = fmaf(j1.w, j1.w, v[9]); v[9] = fmaf(j1.z, j1.z, v[9]);
  v[10] = fmaf(j0.y, j0.w, v[10]); v[10] = fmaf(j1.y, j1.w, v[10]); v[10] = fmaf(j0.x, j0.z, v[10]); v[10] = fmaf(j1.x, j1.z, v[10]);
  v[11] = fmaf(-j0.y, j0.z, v[11]); v[11] = fmaf(j1.x, j1.w, v[11]); v[11] = fmaf(j0.x, j0.w, v[11]); v[11] = fmaf(-j1.y, j1.z, v[11]);
}

// a partner's terms added to a lane's float-float sums
__device__ __forceinline__ void als_terms_ff(FF (&sum)[12], const float4 v0, const float4 v1, const float4 j0,
                                             const float4 j1) {
  float v[16];
  #pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = 0.f;
  als_terms(v, v0, v1, j0, j1);
  #pragma unroll
  for (int i = 0; i < 12; ++i) {
    const FF t = ff_two_sum(sum[i].hi, v[i]);
    sum[i].hi = t.hi;
    sum[i].lo += t.lo;
  }
}

// one source's status and last relative change from its per-antenna norms
// [n_ant][4] (dn, nn, non-finite), by one warp
__device__ __forceinline__ void cluster_status(const double* norms, int n_ant, int lane, int bad, int* status,
                                               double* rel) {
  double dn = 0.0, nn = 0.0, nf = 0.0;
  for (int p = lane; p < n_ant; p += 32) {
    dn += __ldcg(norms + 4 * p);
    nn += __ldcg(norms + 4 * p + 1);
    nf += __ldcg(norms + 4 * p + 2);
  }
  #pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    dn += __shfl_xor_sync(0xffffffffu, dn, o);
    nn += __shfl_xor_sync(0xffffffffu, nn, o);
    nf += __shfl_xor_sync(0xffffffffu, nf, o);
  }
  if (lane == 0) {
    const double r = sqrt(dn / nn);
    *status = bad ? kSolveStatusTimeout : (nf != 0.0 || !isfinite(r)) ? -4 : (r > 1e-6 ? 1 : 0);
    *rel = r;
  }
}

// one launch: one cluster of gridDim.x CTAs of 32 apc threads
__global__ void __launch_bounds__(kClThreads, 1) k_cluster_solve(ClusterSolveArgs a) {
  extern __shared__ __align__(16) unsigned char cl_smem[];
  const int n_ant = a.n_ant;
  float4* rows = reinterpret_cast<float4*>(cl_smem);               // [apc][2][n_ant]
  float4* Jb = rows + (size_t)a.apc * 2 * n_ant;                    // [2][2][n_ant] iterates
  float4* Jsol = Jb + (size_t)4 * n_ant;                            // [kClGroup][2][n_ant] solved
  __shared__ double s_tot64[kClMaxSlots][12];
  __shared__ float4 s_Jn[kClMaxSlots][2];
  __shared__ __align__(8) uint64_t s_bar[2];
  __shared__ int s_bad;
  __shared__ float s_S[kClGroup];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nthr = blockDim.x;
  const int rank = (int)cluster_rank(), CS = (int)cluster_size();
  const int slot = warp, my_p = rank + slot * CS;
  const bool live = my_p < n_ant;
  if (tid == 0) {
    s_bad = 0;
    tc05::mbar_init(&s_bar[0], 1);
    tc05::mbar_init(&s_bar[1], 1);
  }
  if (tid < a.n_grp) s_S[tid] = (float)a.src[3 * (a.s0 + a.q0 + tid) + 2];
  __syncthreads();
  cluster_sync();                          // every CTA's barriers exist before any store to them
  grid_previous_done();                    // V and D are written
  volatile int* bad = &s_bad;
  // this lane's destination: row (lane & 1) of the warp's antenna in CTA lane >> 1
  const uint32_t dst_rank = (uint32_t)(lane >> 1);
  const bool sends = live && (int)dst_rank < CS;
  const uint32_t my_row = tc05::smem_u32(Jb) + (uint32_t)((lane & 1) * n_ant + my_p) * 16u;
  const uint32_t dst_row = sends ? cluster_map(my_row, dst_rank) : 0u;          // in buffer 0
  const uint32_t dst_bar = sends ? cluster_map(tc05::smem_u32(&s_bar[0]), dst_rank) : 0u;
  const uint32_t buf_bytes = (uint32_t)n_ant * 32u;
  uint32_t g = 0;                          // sweeps done, over all sources: buffer and barrier g & 1

  for (int q = 0; q < a.n_grp; ++q) {
    const int kq = a.q0 + q, k = a.s0 + kq;
    // ---- the warp's antenna's row: planes (entries 0, 1 | 2, 3), V_pp = 0; two
    // partners' loads in flight a lane
    if (live) {
      const float4* V0 = a.V + ((size_t)q * n_ant + my_p) * 2 * n_ant;
      const float2* D0 = a.D + (size_t)cl_pair(q, 0) * n_ant * n_ant + (size_t)my_p * n_ant;
      float4* row0 = rows + (size_t)slot * 2 * n_ant;
      float4* row1 = row0 + n_ant;
      for (int qb = lane; qb < n_ant; qb += 64) {
        float4 r0[2], r1[2];
        float2 d[2][kClGroup - 1];
        #pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int qq = qb + 32 * u;
          if (qq < n_ant) {
            r0[u] = __ldcg(V0 + qq);
            r1[u] = __ldcg(V0 + n_ant + qq);
            #pragma unroll
            for (int j = 0; j < kClGroup - 1; ++j)
              if (j < q) d[u][j] = __ldcg(D0 + (size_t)j * n_ant * n_ant + qq);
          }
        }
        #pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int qq = qb + 32 * u;
          if (qq >= n_ant) break;
          float4 t0 = make_float4(0.f, 0.f, 0.f, 0.f), t1 = t0;
          #pragma unroll
          for (int j = 0; j < kClGroup - 1; ++j) {
            if (j < q) {
              // S_j D J_p J_q^H: w_rm = S_j D J_p[r][m], entry (r, c) = sum_m w_rm conj(J_q[c][m])
              const float S = s_S[j];
              const float4* Jj = Jsol + (size_t)2 * j * n_ant;
              const float4 i0 = Jj[my_p], i1 = Jj[n_ant + my_p], k0 = Jj[qq], k1 = Jj[n_ant + qq];
              const float2 sd = make_float2(S * d[u][j].x, S * d[u][j].y);
              const float2 w00 = cmul(sd, make_float2(i0.x, i0.y)), w01 = cmul(sd, make_float2(i0.z, i0.w));
              const float2 w10 = cmul(sd, make_float2(i1.x, i1.y)), w11 = cmul(sd, make_float2(i1.z, i1.w));
              auto put = [](float& re, float& im, float2 w, float kx, float ky) {      // += w conj(k)
                re = fmaf(w.x, kx, fmaf(w.y, ky, re));
                im = fmaf(w.y, kx, fmaf(-w.x, ky, im));
              };
              put(t0.x, t0.y, w00, k0.x, k0.y); put(t0.x, t0.y, w01, k0.z, k0.w);
              put(t0.z, t0.w, w00, k1.x, k1.y); put(t0.z, t0.w, w01, k1.z, k1.w);
              put(t1.x, t1.y, w10, k0.x, k0.y); put(t1.x, t1.y, w11, k0.z, k0.w);
              put(t1.z, t1.w, w10, k1.x, k1.y); put(t1.z, t1.w, w11, k1.z, k1.w);
            }
          }
          r0[u] = make_float4(r0[u].x - t0.x, r0[u].y - t0.y, r0[u].z - t0.z, r0[u].w - t0.w);
          r1[u] = make_float4(r1[u].x - t1.x, r1[u].y - t1.y, r1[u].z - t1.z, r1[u].w - t1.w);
          const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
          row0[qq] = qq == my_p ? z : r0[u];
          row1[qq] = qq == my_p ? z : r1[u];
        }
      }
    }
    const double Sd = a.src[3 * k + 2];
    const float Sf = (float)Sd;
    __syncwarp();                          // a warp sums the row that it staged

    for (int it = 1; it <= a.n_iter; ++it, ++g) {
      const bool first = it == 1, last = it == a.n_iter, average = (it & 1) == 0;
      const uint32_t b = g & 1u;
      const float4* Jo = Jb + (size_t)(b ^ 1u) * 2 * n_ant;       // previous iterate (not on the first sweep)
      if (tid == 0) mbar_expect(&s_bar[b], buf_bytes);
      const float4* row0 = rows + (size_t)slot * 2 * n_ant;
      const float4* row1 = row0 + n_ant;
      auto iterate = [&](int qq, float4& j0, float4& j1) {
        j0 = first ? make_float4(1.f, 0.f, 0.f, 0.f) : Jo[qq];
        j1 = first ? make_float4(0.f, 0.f, 1.f, 0.f) : Jo[n_ant + qq];
        if (qq == my_p) j0 = j1 = make_float4(0.f, 0.f, 0.f, 0.f);     // C excludes q = p
      };
      float4 Jn = make_float4(0.f, 0.f, 0.f, 0.f);                 // the row this lane sends
      if (!last) {
        float v[16];
        #pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = 0.f;
        if (live)
          for (int q0 = lane; q0 < n_ant; q0 += 32 * kClChain) {
            float w[16];
            #pragma unroll
            for (int i = 0; i < 16; ++i) w[i] = 0.f;
            #pragma unroll
            for (int u = 0; u < kClChain; ++u) {
              const int qq = q0 + 32 * u;
              if (qq >= n_ant) break;
              float4 j0, j1;
              iterate(qq, j0, j1);
              als_terms(w, row0[qq], row1[qq], j0, j1);
            }
            #pragma unroll
            for (int i = 0; i < 12; ++i) v[i] += w[i];
          }
        const float wsum = warp_reduce_scatter16c(v, lane);
        // lane L holds the total of value L >> 1: this lane's row of A, and C
        const int at = 8 * (lane & 1);
        const float2 A0 = make_float2(__shfl_sync(0xffffffffu, wsum, at), __shfl_sync(0xffffffffu, wsum, at + 2));
        const float2 A1 = make_float2(__shfl_sync(0xffffffffu, wsum, at + 4), __shfl_sync(0xffffffffu, wsum, at + 6));
        const float c00 = __shfl_sync(0xffffffffu, wsum, 16), c11 = __shfl_sync(0xffffffffu, wsum, 18);
        const float2 c01 = make_float2(__shfl_sync(0xffffffffu, wsum, 20), __shfl_sync(0xffffffffu, wsum, 22));
        if (live) {
          // row r = lane & 1 of A C^-1 / S
          const float sc = solve_recip((c00 * c11 - (c01.x * c01.x + c01.y * c01.y)) * Sf);
          const float2 i00 = make_float2(c11 * sc, 0.f), i10 = make_float2(-c01.x * sc, c01.y * sc);
          const float2 i01 = make_float2(-c01.x * sc, -c01.y * sc), i11 = make_float2(c00 * sc, 0.f);
          const float2 x = cadd(cmul(A0, i00), cmul(A1, i10)), y = cadd(cmul(A0, i01), cmul(A1, i11));
          Jn = make_float4(x.x, x.y, y.x, y.y);
          if (average) {
            const float4 o = Jo[(lane & 1) * n_ant + my_p];
            Jn = make_float4(0.5f * (Jn.x + o.x), 0.5f * (Jn.y + o.y), 0.5f * (Jn.z + o.z), 0.5f * (Jn.w + o.w));
          }
        }
      } else {
        FF sum[12];
        #pragma unroll
        for (int i = 0; i < 12; ++i) sum[i].hi = sum[i].lo = 0.f;
        if (live)
          for (int qq = lane; qq < n_ant; qq += 32) {
            float4 j0, j1;
            iterate(qq, j0, j1);
            als_terms_ff(sum, row0[qq], row1[qq], j0, j1);
          }
        const FF wsum = warp_reduce_scatter12ff(sum, lane);
        if ((lane & 1) == 0 && (lane >> 1) < 12) s_tot64[slot][lane >> 1] = (double)wsum.hi + (double)wsum.lo;
        __syncthreads();
        // the FP64 solves of all slots, one entry a lane of the first warps
        if (warp < (4 * a.apc + 31) / 32) {
          const int s = tid >> 2, e = tid & 3, p = rank + s * CS;
          const bool lv = s < a.apc && p < n_ant;
          double dn = 0.0, nn = 0.0;
          int nf = 0;
          if (lv) {
            const float2 eye = make_float2(e == 0 || e == 3 ? 1.f : 0.f, 0.f);
            const float2 o = first ? eye
                                   : reinterpret_cast<const float2*>(Jo + (size_t)(e >> 1) * n_ant + p)[e & 1];
            double2 Jd = solve_entry<double>(s_tot64[s], Sd, e);
            if (average) Jd = make_double2(0.5 * (Jd.x + (double)o.x), 0.5 * (Jd.y + (double)o.y));
            const double dx = Jd.x - (double)o.x, dy = Jd.y - (double)o.y;
            dn = dx * dx + dy * dy;
            nn = Jd.x * Jd.x + Jd.y * Jd.y;
            nf = !(isfinite(Jd.x) && isfinite(Jd.y));
            const float2 Jf = make_float2((float)Jd.x, (float)Jd.y);
            a.jones[((size_t)k * n_ant + p) * 4 + e] = Jf;
            reinterpret_cast<float2*>(&s_Jn[s][e >> 1])[e & 1] = Jf;
          }
          #pragma unroll
          for (int o = 1; o <= 2; o <<= 1) {
            dn += __shfl_xor_sync(0xffffffffu, dn, o);
            nn += __shfl_xor_sync(0xffffffffu, nn, o);
            nf |= __shfl_xor_sync(0xffffffffu, nf, o);
          }
          if (lv && e == 0) {
            double* pt = a.part + ((size_t)kq * n_ant + p) * 4;
            pt[0] = dn;
            pt[1] = nn;
            pt[2] = (double)nf;
          }
        }
        __syncthreads();
        if (live) Jn = s_Jn[slot][lane & 1];
      }
      if (sends && !*bad) {
        // the last sweep's matrices go to the group's solved ones
        const uint32_t off = last ? (uint32_t)(4 + 2 * q) * (uint32_t)n_ant * 16u : b * (uint32_t)n_ant * 32u;
        cluster_send16(dst_row + off, Jn, dst_bar + 8u * b);
      }
      if (live) cluster_wait(&s_bar[b], (g >> 1) & 1u, bad);
    }
  }

  // ---- every CTA's norms are written and no store is in flight past this barrier;
  // warp 0 of CTA q % CS takes source q's status, the others form the group's
  // model matrices from the rows p < q of their antennas
  grid_next_may_start();
  if (*bad) __nanosleep(100000);
  cluster_sync();
  if (warp == 0)
    for (int q = rank; q < a.n_grp; q += CS)
      cluster_status(a.part + (size_t)(a.q0 + q) * n_ant * 4, n_ant, lane, *bad, a.status + a.s0 + a.q0 + q,
                     a.rel + a.s0 + a.q0 + q);
  const int n_warp = nthr >> 5;
  const bool busy = n_warp > 1 && rank < a.n_grp;        // warp 0 is at the statuses
  if (!(busy && warp == 0))
    for (int x = warp - (busy ? 1 : 0); x < a.apc * a.n_grp; x += n_warp - (busy ? 1 : 0)) {
      const int s = x / a.n_grp, j = x - s * a.n_grp, p = rank + s * CS;
      if (p >= n_ant) continue;
      const float S = s_S[j];
      const float4* Jj = Jsol + (size_t)2 * j * n_ant;
      const float4 p0 = Jj[p], p1 = Jj[n_ant + p];
      for (int qq = p + 1 + lane; qq < n_ant; qq += 32) {
        float2 M[4];
        block_model4(p0, p1, Jj[qq], Jj[n_ant + qq], S, M);
        float4* d = reinterpret_cast<float4*>(a.M + ((size_t)(a.q0 + j) * a.n_bl + bl_index(n_ant, p, qq)) * 4);
        d[0] = make_float4(M[0].x, M[0].y, M[1].x, M[1].y);
        d[1] = make_float4(M[2].x, M[2].y, M[3].x, M[3].y);
      }
    }
  cluster_sync();
  if (*bad && tid < a.n_grp) a.status[a.s0 + a.q0 + tid] = kSolveStatusTimeout;
}

// The solve of one source's averages with FP64 iterates (k_als_sweep's arithmetic)
// by one cluster: 20 launches of 6.6 us and their gaps become one launch.  As
// k_cluster_solve, but every sweep's sums over partners are float-float (a
// partner's product and its lane's first are FP32, as a k_als_sweep thread's
// are), and the 2x2 solve, the iterate and its averaging FP64; the sweeps' terms
// read the FP32 rounding of the iterate.  An FP64 instruction occupies its
// sub-partition for 64 cycles whatever its lanes, so all slots' solves run as
// lanes of one or two warps.  Measured (128 antennas, 20 sweeps): 66 us where the
// launches took 137; the call with its status read 185 and 110 us.  A sweep: terms
// 1 830 cycles, reduction 870, FP64 solve 2 010, exchange 1 040.
struct ClusterAlsArgs {
  const float2* avg;       // [n_bl][4]
  double S;
  int n_ant, n_iter, apc;
  double2* J;              // [n_ant][4] FP64 solution
  float2* jones;           // [n_ant][4] its FP32 rounding
  double* norms;           // [n_ant][4] dn, nn, non-finite of the last sweep
  int* status;             // of this source
  double* rel;
};

inline size_t cluster_als_smem(int n_ant, int apc) { return ((size_t)apc + 2) * 2 * n_ant * sizeof(float4); }

__global__ void __launch_bounds__(kClThreads, 1) k_cluster_als(ClusterAlsArgs a) {
  extern __shared__ __align__(16) unsigned char cl_smem[];
  const int n_ant = a.n_ant;
  float4* rows = reinterpret_cast<float4*>(cl_smem);               // [apc][2][n_ant]
  float4* Jb = rows + (size_t)a.apc * 2 * n_ant;                    // [2][2][n_ant] iterates
  __shared__ double s_tot64[kClMaxSlots][12];
  __shared__ float4 s_Jn[kClMaxSlots][2];
  __shared__ __align__(8) uint64_t s_bar[2];
  __shared__ int s_bad;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = (int)cluster_rank(), CS = (int)cluster_size();
  const int slot = warp, my_p = rank + slot * CS;
  const bool live = my_p < n_ant;
  if (tid == 0) {
    s_bad = 0;
    tc05::mbar_init(&s_bar[0], 1);
    tc05::mbar_init(&s_bar[1], 1);
  }
  float4* row0 = rows + (size_t)slot * 2 * n_ant;
  float4* row1 = row0 + n_ant;
  if (live)
    for (int qq = lane; qq < n_ant; qq += 32) {
      float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0;
      if (qq != my_p) {
        const float4* P = reinterpret_cast<const float4*>(a.avg + bl_index(n_ant, min(my_p, qq), max(my_p, qq)) * 4);
        r0 = P[0];
        r1 = P[1];
        if (qq < my_p) {                   // V_pq = V_qp^H
          const float4 t0 = r0, t1 = r1;
          r0 = make_float4(t0.x, -t0.y, t1.x, -t1.y);
          r1 = make_float4(t0.z, -t0.w, t1.z, -t1.w);
        }
      }
      row0[qq] = r0;
      row1[qq] = r1;
    }
  __syncthreads();
  cluster_sync();                          // every CTA's barriers exist before any store to them
  volatile int* bad = &s_bad;
  const uint32_t dst_rank = (uint32_t)(lane >> 1);
  const bool sends = live && (int)dst_rank < CS;
  const uint32_t my_row = tc05::smem_u32(Jb) + (uint32_t)((lane & 1) * n_ant + my_p) * 16u;
  const uint32_t dst_row = sends ? cluster_map(my_row, dst_rank) : 0u;
  const uint32_t dst_bar = sends ? cluster_map(tc05::smem_u32(&s_bar[0]), dst_rank) : 0u;
  // the FP64 solver's lanes: entry e of slot s
  const int s = tid >> 2, e = tid & 3, ps = rank + s * CS;
  const bool solver = warp < (4 * a.apc + 31) / 32, lv = s < a.apc && ps < n_ant;
  double2 Jd = make_double2(e == 0 || e == 3 ? 1.0 : 0.0, 0.0);    // this lane's iterate

  for (int it = 1; it <= a.n_iter; ++it) {
    const bool first = it == 1, last = it == a.n_iter;
    const uint32_t b = (uint32_t)(it - 1) & 1u;
    const float4* Jo = Jb + (size_t)(b ^ 1u) * 2 * n_ant;
    if (tid == 0) mbar_expect(&s_bar[b], (uint32_t)n_ant * 32u);
    FF sum[12];
    #pragma unroll
    for (int i = 0; i < 12; ++i) sum[i].hi = sum[i].lo = 0.f;
    if (live)
      for (int qq = lane; qq < n_ant; qq += 32) {
        float4 j0 = first ? make_float4(1.f, 0.f, 0.f, 0.f) : Jo[qq];
        float4 j1 = first ? make_float4(0.f, 0.f, 1.f, 0.f) : Jo[n_ant + qq];
        if (qq == my_p) j0 = j1 = make_float4(0.f, 0.f, 0.f, 0.f);   // C excludes q = p
        als_terms_ff(sum, row0[qq], row1[qq], j0, j1);
      }
    const FF wsum = warp_reduce_scatter12ff(sum, lane);
    if ((lane & 1) == 0 && (lane >> 1) < 12) s_tot64[slot][lane >> 1] = (double)wsum.hi + (double)wsum.lo;
    __syncthreads();
    double2 Jp = Jd;
    if (solver && lv) {
      // entry (r, c) of A C^-1 / S: C^-1 = [c11 -c01; -conj(c01) c00] / det
      const double* t = s_tot64[s];
      const int r = e >> 1;
      const double c00 = t[8], c11 = t[9], cx = t[10], cy = t[11];
      const double ax = t[4 * r], ay = t[4 * r + 1], bx = t[4 * r + 2], by = t[4 * r + 3];
      const double sc = 1.0 / (fma(c00, c11, -fma(cx, cx, cy * cy)) * a.S);
      double2 num;
      if (e & 1) num = make_double2(fma(bx, c00, -fma(ax, cx, -ay * cy)), fma(by, c00, -fma(ax, cy, ay * cx)));
      else num = make_double2(fma(ax, c11, -fma(bx, cx, by * cy)), fma(ay, c11, -fma(by, cx, -bx * cy)));
      if (it & 1) Jd = make_double2(num.x * sc, num.y * sc);
      else Jd = make_double2(0.5 * fma(num.x, sc, Jp.x), 0.5 * fma(num.y, sc, Jp.y));
      reinterpret_cast<float2*>(&s_Jn[s][r])[e & 1] = make_float2((float)Jd.x, (float)Jd.y);
    }
    __syncthreads();
    if (sends && !*bad) cluster_send16(dst_row + b * (uint32_t)n_ant * 32u, s_Jn[slot][lane & 1], dst_bar + 8u * b);
    if (last && solver) {
      const double dx = Jd.x - Jp.x, dy = Jd.y - Jp.y;
      double dn = dx * dx + dy * dy, nn = Jd.x * Jd.x + Jd.y * Jd.y;
      int nf = lv && !(isfinite(Jd.x) && isfinite(Jd.y));
      #pragma unroll
      for (int o = 1; o <= 2; o <<= 1) {
        dn += __shfl_xor_sync(0xffffffffu, dn, o);
        nn += __shfl_xor_sync(0xffffffffu, nn, o);
        nf |= __shfl_xor_sync(0xffffffffu, nf, o);
      }
      if (lv) {
        a.J[(size_t)ps * 4 + e] = Jd;
        a.jones[(size_t)ps * 4 + e] = make_float2((float)Jd.x, (float)Jd.y);
        if (e == 0) {
          a.norms[4 * ps] = dn;
          a.norms[4 * ps + 1] = nn;
          a.norms[4 * ps + 2] = (double)nf;
        }
      }
    }
    cluster_wait(&s_bar[b], ((uint32_t)(it - 1) >> 1) & 1u, bad);
  }
  if (*bad) __nanosleep(100000);
  cluster_sync();
  if (rank == 0 && warp == 0) cluster_status(a.norms, n_ant, lane, *bad, a.status, a.rel);
  cluster_sync();
  if (*bad && tid == 0) *a.status = kSolveStatusTimeout;
}

}  // namespace rts
