// Blocked peel pass on the 5th-generation tensor cores, transposed form: the
// same pass as k_block_pass (subtract the solved sources of block b from one
// (baseline, time step) strip of channels, average the directions of block b+1),
// with both contractions as tcgen05.mma kind::tf32 GEMMs whose operands the
// CUDA cores form in O(sources x 16) or O(sources x channels / 16) work.
//
// The phasor of source k at channel c = 16 q + r factors as
//   P_k(c) = T1_k[q] T2_k[r],  T1_k[q] = e^{2 pi i (A_k + 16 q B_k)},  T2_k[r] = e^{2 pi i r B_k},
// and T1 once more as V_k[q % 8] U_k[q / 8], so a source and role need at most 30 table
// phasors (16 + 8 + 6) for any strip; T1 is their product.
//
// subtraction  R(16 q + r, e) -= sum_k a_k(r, e) conj(T1_k[q]),  a_k(r, e) = M_k(e) conj(T2_k[r])
//   A_s: 128 rows m = 8 r + 2 e + o, row o = 0 the real parts of a_k, o = 1 the
//   imaginary ones, K = 64 sources, written by the threads into TMEM.  B_s: rows
//   q the real parts of T1, rows NQ + q the imaginary ones (NQ: the 16-channel
//   tiles, rounded up to 16), K = 64, in shared memory.  The four real products
//   of a complex one are thus the two halves of N on two neighbouring rows: a
//   lane adds its own re half and, by one shuffle, its neighbour's im half.
// average      A_k(e) += sum_r T2_k[r] H_k(r, e),  H_k(r, e) = sum_q T1_k[q] R(16 q + r, e)
//   A_a: 128 rows 2 k + o (re or im of T1_k), K = NQ, in TMEM.  B_a: 128 rows
//   8 r + 2 e + o' (re or im of the new residual), K = NQ, written by the
//   subtraction's epilogue (4 tiles a 16-byte store).  The 16-term T2
//   contraction of a row's products runs on the CUDA cores as packed
//   multiply-adds; a thread's sums over the time steps are compensated and
//   the rows o and the column groups meet once a baseline.
// Writing the operands in their real parts once, instead of the 2 x 2 real form of
// one of them, halves what the CUDA cores form and split; the tensor cores do
// the same work.
//
// TF32 keeps 11 significand bits, so every operand is split x = hi + lo and
// each product takes three MMAs, hi*hi + lo*hi + hi*lo.  The tensor cores'
// FP32 accumulation does not round to nearest, so an accumulator takes at most 4
// k-steps; the epilogues add them in FP32 with round-to-nearest.
//
// One CTA per SM (~225 KB of shared memory, all 512 TMEM columns): 16 compute
// warps, 4 warps whose lane 0 issues one accumulator's MMAs (an issuing thread
// stalls while its MMAs are accepted); the last of these also moves the strips
// and phases by bulk asynchronous copies (a fifth such warp would leave 80
// registers a thread).  A step of a compute warp:
//   C1  A_a into TMEM; the last step's T2 contraction; the next step's tables (all
//       sources)
//   ----  the step's only barrier among the compute warps
//   C2  residual into the strip and B_a
//   C3  the next step's B_s and A_s
//   C4  the average's accumulators into registers
// with operands handed to the issuers by one arrival a warp (after C2: B_a and
// the strip; after C4: A_s, B_s and the accumulators read), so the warps drift
// apart and fill each other's latencies, the subtraction's MMAs run beside C4 and
// C1 and the average's beside C3.  What a warp may overwrite early is safe
// because it has waited for the MMAs of the step, which need every warp's
// arrival.  Every wait is bounded (a wait that runs out sets *err and stops the
// pass, which the status read reports, after the copies in flight have been
// waited for and TMEM is freed).
// Bound by the CUDA cores' phases (issue 62 % of the slots, shared-memory pipe 57 %,
// ALU pipe 40 %, tensor pipe 31 %; without any MMA a step takes 5 % less).  A step of both
// roles at 768 channels, 64 sources: about 7 200 cycles (the 2 x 2 form with five barriers
// a step: 9 700); a cadence of 512 antennas x 768 channels x 8 times x 1000 sources went
// from 722 to 582 ms, its passes from 559 to 418 (24.6 ms each).  Steps on the way: real
// parts and one barrier 496 ms of passes, constant offsets, polled waits and loads before
// stores 472, A_a before the barrier 418.  Phasors by polynomials instead of the sine
// table: no gain.
// Limits: at most 64 sources per role, n_chan <= kTc5MaxChan.
#pragma once
#include "block_kernels.cuh"
#include "kahan.cuh"
#include "strip_kernels.cuh"
#include "tc05.cuh"

namespace rts {

constexpr int kTc5Compute = 512;             // 16 compute warps (4 per TMEM lane quarter)
constexpr int kTc5Issuers = 4;               // and 4 warps whose lane 0 issues one accumulator's MMAs
constexpr int kTc5Threads = kTc5Compute + 32 * kTc5Issuers;
constexpr int kTc5Src = 64;                  // sources per role
constexpr int kTc5BaselinesPerCta = 16;      // baselines a CTA peels one after another: its set-up
                                             // and first operands are paid once for them
constexpr int kTc5MaxChan = 768;             // NQ <= 48
constexpr uint32_t kTc5MaxPolls = 1u << 17;  // mbarrier polls (each up to 20 us) before giving up
constexpr uint32_t kTc5MaxSpins = 1u << 26;  // polls that return at once (about a second)
// TMEM columns.  Subtraction: accumulator (g, part) at (2 g + part) NQ (< 192); A_s
// hi and lo at [384, 512).  Average: accumulator g at 128 g (< 256); A_a hi at
// [256, 256 + NQ), lo after it (< 352).
constexpr uint32_t kTc5ColAa = 256;
constexpr uint32_t kTc5ColAsHi = 384;
constexpr uint32_t kTc5ColAsLo = 448;
constexpr uint32_t kTc5Cols = 512;

// phasor tables of one step, in floats: x and y planes
constexpr int kTc5Row = 68, kTc5VRow = 72, kTc5ARow = 12;      // row strides, chosen against bank conflicts
struct Tc05Tab {
  float sx[16][kTc5Row], sy[16][kTc5Row];    // T2 of the subtracted sources [r][k]
  float svx[8][kTc5VRow], svy[8][kTc5VRow];  // V of the subtracted sources [q % 8][k]
  float sux[6][kTc5VRow], suy[6][kTc5VRow];  // U [q / 8][k]
  float avx[kTc5Src][kTc5ARow], avy[kTc5Src][kTc5ARow];         // V of the averaged sources [k][q % 8]
  float2 au[6][kTc5Src];                     // U [q / 8][k]
};
// T2 of the averaged sources as T2[4 c + r] = P[r] Q[c]: P, then Q, as [4][k]
struct Tc05T2 { float2 pq[8][kTc5Src]; };
// a baseline's model matrices: re, im and -re as [e][k]
struct Tc05Model { float m[3][4][kTc5Row]; };

// shared-memory layout (byte offsets) for NQ 16-channel tiles (16, 32 or 48)
struct Tc05Smem {
  int strip, bs_hi, bs_lo, ba_hi, ba_lo, tab, t2, model, ph, lut, bar, total;
  __host__ __device__ constexpr explicit Tc05Smem(int NQ)
      : strip(0), bs_hi(0), bs_lo(0), ba_hi(0), ba_lo(0), tab(0), t2(0), model(0), ph(0), lut(0), bar(0), total(0) {
    int o = 0;
    strip = o; o += 2 * 16 * NQ * 32;            // two strips [16 NQ channels][4 pol][re, im]
    bs_hi = o; o += 2 * NQ * kTc5Src * 4;        // B_s [2 NQ rows][64 K], K-major
    bs_lo = o; o += 2 * NQ * kTc5Src * 4;
    ba_hi = o; o += 128 * NQ * 4;                // B_a [128 rows][NQ K], K-major
    ba_lo = o; o += 128 * NQ * 4;
    tab = o;   o += 2 * (int)sizeof(Tc05Tab);
    t2 = o;    o += 3 * (int)sizeof(Tc05T2);     // the last step's is read while the next step's is written
    model = o; o += 2 * (int)sizeof(Tc05Model);
    ph = o;    o += 2 * 2 * kTc5Src * 16;        // phases of two time steps [2][sub 64, avg 64]
    lut = o;   o += 256 * 8;
    bar = o;   o += 80;                          // mbarriers (sub MMAs done, avg MMAs done, strip 0, strip 1,
                                                 // sub operands ready, avg operands ready, phases 0, phases 1),
                                                 // TMEM address
    total = o;
  }
};

inline int tc05_nq(int n_chan) { return (((n_chan + 15) >> 4) + 15) & ~15; }
inline size_t tc05_pass_smem(int n_chan) { return (size_t)Tc05Smem(tc05_nq(n_chan)).total; }
static_assert(sizeof(Tc05Tab) % 16 == 0 && sizeof(Tc05Model) % 16 == 0, "16-byte rows");

// TF32 rounding (to nearest, ties away from zero, as cvt.rna.tf32.f32 for
// finite x below the FP32 maximum) by two integer operations
__device__ __forceinline__ uint32_t tc05_tf32(float x) { return (__float_as_uint(x) + 0x1000u) & 0xFFFFE000u; }
// x = hi + lo, hi the TF32 rounding of x, lo the exact remainder (the MMA reads
// lo truncated to TF32: error below 2^-21 |x|)
__device__ __forceinline__ float2 tc05_split(float x) {
  const float hi = __uint_as_float(tc05_tf32(x));
  return make_float2(hi, x - hi);
}
__device__ __forceinline__ void tc05_split2(float2 x, float2& hi, float2& lo) {
  hi = make_float2(__uint_as_float(tc05_tf32(x.x)), __uint_as_float(tc05_tf32(x.y)));
  lo = ffma2(make_float2(-1.f, -1.f), hi, x);
}
// the same for |x| <= 1: hi is x rounded to a multiple of 2^-11 (11 bits up to 1), by
// an addition that leaves no bits below
__device__ __forceinline__ void tc05_split2_unit(float2 x, float2& hi, float2& lo) {
  hi = fadd2(fadd2(x, make_float2(6144.f, 6144.f)), make_float2(-6144.f, -6144.f));
  lo = ffma2(make_float2(-1.f, -1.f), hi, x);
}

// NQ (16, 32 or 48): the strip's tiles of 16 channels, rounded up to 16; a template
// parameter so that every shared-memory offset is a constant (the registers that
// held them spilled)
template <int NQ, bool SUB, bool ACC>
__global__ void __launch_bounds__(kTc5Threads, 1) k_block_pass_tc05(BlockPassArgs a, int bk, int nb, int* err) {
  using namespace tc05;
  constexpr int QW = NQ >> 2;               // tiles per column-group warp: 4, 8 or 12
  constexpr int nacc = NQ > 32 ? 2 : 1;     // the average's accumulators
  constexpr int n16 = 16 * NQ;
  const uint32_t strip_bytes = (uint32_t)a.n_chan * 32u;
  constexpr Tc05Smem L(NQ);
  extern __shared__ __align__(1024) unsigned char tc05_smem[];
  float* strip0 = reinterpret_cast<float*>(tc05_smem + L.strip);
  unsigned char* bs_hi = tc05_smem + L.bs_hi;
  unsigned char* bs_lo = tc05_smem + L.bs_lo;
  unsigned char* ba_hi = tc05_smem + L.ba_hi;
  unsigned char* ba_lo = tc05_smem + L.ba_lo;
  Tc05Tab* tabs = reinterpret_cast<Tc05Tab*>(tc05_smem + L.tab);
  Tc05T2* t2s = reinterpret_cast<Tc05T2*>(tc05_smem + L.t2);
  Tc05Model* models = reinterpret_cast<Tc05Model*>(tc05_smem + L.model);
  PhaseAB* ph = reinterpret_cast<PhaseAB*>(tc05_smem + L.ph);
  float2* lut = reinterpret_cast<float2*>(tc05_smem + L.lut);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(tc05_smem + L.bar);      // see Tc05Smem::bar
  uint32_t* tslot = reinterpret_cast<uint32_t*>(tc05_smem + L.bar + 64);
  volatile int& s_bad = *reinterpret_cast<volatile int*>(tc05_smem + L.bar + 68);

  // baselines bl0 .. bl0 + nbl - 1, their time steps one after another: step g
  // is time g % n_time of baseline bl0 + g / n_time
  const int64_t bl0 = (int64_t)blockIdx.x * nb;
  const int nbl = (int)min((int64_t)nb, a.n_bl - bl0), n_steps = nbl * a.n_time;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, qtr = warp & 3, cg = warp >> 2;
  const uint32_t lane_base = (uint32_t)(32 * qtr) << 16;
  const bool compute = tid < kTc5Compute;

  if (warp == 0) tmem_alloc(tslot, kTc5Cols);
  if (tid == 0) {
    mbar_init(&mbar[0], kTc5Issuers);        // one commit per issuer
    mbar_init(&mbar[1], 2 * nacc);           // one commit per issuer of the average
    mbar_init(&mbar[2], 1);
    mbar_init(&mbar[3], 1);
    mbar_init(&mbar[4], kTc5Compute / 32);   // one arrival per compute warp
    mbar_init(&mbar[5], kTc5Compute / 32);
    mbar_init(&mbar[6], 1);
    mbar_init(&mbar[7], 1);
    s_bad = *reinterpret_cast<volatile int*>(err);    // a pass in which some CTA's wait ran out does no more work
  }
  // a baseline's model matrices, entry tid: loaded here, stored by put_model
  auto get_model = [&](int64_t bl) {
    const int s = tid >> 2;
    return s < a.n_sub ? a.M_sub[((size_t)s * a.n_bl + bl) * 4 + (tid & 3)] : make_float2(0.f, 0.f);
  };
  auto put_model = [&](int slot, float2 v) {
    float (*m)[4][kTc5Row] = models[slot].m;
    const int s = tid >> 2, e = tid & 3;
    m[0][e][s] = v.x;
    m[1][e][s] = v.y;
    m[2][e][s] = -v.x;
  };
  if (compute) {
    lut_fill(lut, tid, kTc5Compute);
    // padding channels of both strips stay zero (the copies never write them)
    for (int i = tid; i < (n16 - a.n_chan) * 8; i += kTc5Compute) {
      strip0[a.n_chan * 8 + i] = 0.f;
      strip0[(n16 + a.n_chan) * 8 + i] = 0.f;
    }
    if (SUB && tid < 4 * kTc5Src) put_model(0, get_model(bl0));
    // phases of sources beyond bk stay zero (the copies bring bk per role)
    for (int i = tid; i < 4 * kTc5Src; i += kTc5Compute) {
      ph[i].a = 0;
      ph[i].b = 0;
    }
  }
  fence_smem_async();                        // the zero fills precede the bulk copies into the same words
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tslot;

  // a bounded mbarrier wait that also gives up once another thread has raised s_bad; it
  // polls (a wait that suspends the thread cost 3 % of the pass in wake-ups)
  auto wait_or_bad = [&](uint64_t* bar, uint32_t parity) {
    for (uint32_t it = 0; it < kTc5MaxSpins; ++it) {
      if (mbar_test(bar, parity)) return true;
      if ((it & 1023u) == 1023u && s_bad) return false;
    }
    return false;
  };

  if (!compute) {
    // ---- the MMAs: lane 0 of warp 16 + i issues the products of k-half g = i / 2
    // with half i % 2 of B's rows.  An accumulator takes the cross terms (lo*hi,
    // hi*lo) of its k-steps first, then their hi*hi products
    const int i = warp - kTc5Compute / 32, g = i >> 1, part = i & 1;
    if (lane == 0) {
      const bool copies = i == kTc5Issuers - 1;                 // this thread also moves the data
      int strips = 0, phases = 0;                               // steps whose loads have been issued
      auto load_strip = [&]() {                                 // ring slot: step & 1
        const int b = strips & 1, t = strips % a.n_time;
        const int64_t bl = bl0 + strips / a.n_time;
        mbar_expect_tx(&mbar[2 + b], strip_bytes);
        bulk_load(strip0 + (size_t)b * n16 * 8, a.src + ((size_t)t * a.n_bl + bl) * a.n_chan * 2, strip_bytes,
                  &mbar[2 + b]);
        ++strips;
      };
      auto load_phases = [&]() {
        const int b = phases & 1, t = phases % a.n_time;
        const int64_t bl = bl0 + phases / a.n_time;
        const uint32_t bytes = (uint32_t)bk * sizeof(PhaseAB);
        mbar_expect_tx(&mbar[6 + b], (SUB ? bytes : 0u) + (ACC ? bytes : 0u));
        const size_t at = ((size_t)bl * a.n_time + t) * bk;
        if (SUB) bulk_load(ph + 2 * kTc5Src * b, a.ph_sub + at, bytes, &mbar[6 + b]);
        if (ACC) bulk_load(ph + 2 * kTc5Src * b + kTc5Src, a.ph_acc + at, bytes, &mbar[6 + b]);
        ++phases;
      };
      if (copies) {
        for (int u = 0; u < 2 && u < n_steps; ++u) {
          load_phases();
          load_strip();
        }
      }
      const uint64_t row = (uint64_t)(16 * NQ * part);          // both operands: 256 NQ bytes a half
      const uint64_t dbs_hi = desc_kmajor(smem_u32(bs_hi), 128, 2048) + row;
      const uint64_t dbs_lo = desc_kmajor(smem_u32(bs_lo), 128, 2048) + row;
      const uint64_t dba_hi = desc_kmajor(smem_u32(ba_hi), 128, 32 * NQ) + row;
      const uint64_t dba_lo = desc_kmajor(smem_u32(ba_lo), 128, 32 * NQ) + row;
      const uint32_t id_s = idesc_tf32(128, NQ), id_a = idesc_tf32(128, 64);
      const int ks = nacc == 2 ? 3 : NQ >> 3;                   // k-steps of an average accumulator
      for (int t = 0; t < n_steps; ++t) {
        if (SUB) {
          if (!wait_or_bad(&mbar[4], (uint32_t)t & 1u)) break;
          fence_after_sync();
          #pragma unroll
          for (int j = 0; j < 12; ++j) {
            const int s = 4 * g + (j & 3);
            const uint32_t acol = tmem + (j < 4 ? kTc5ColAsLo : kTc5ColAsHi) + 8 * s;   // lo(A) for j < 4, else hi(A)
            const uint64_t bd = (j >= 4 && j < 8 ? dbs_lo : dbs_hi) + 16 * s;
            mma_ts(tmem + i * NQ, acol, bd, id_s, j != 0);
          }
          commit(&mbar[0]);
          if (copies && t >= 1 && t + 1 < n_steps) {
            bulk_wait_read();                // the residual of step t - 1 has left the buffer
            load_strip();
          }
        }
        if (copies || (ACC && g < nacc)) {
          if (!wait_or_bad(&mbar[5], (uint32_t)t & 1u)) break;
          fence_after_sync();
        }
        if (ACC && g < nacc) {
          #pragma unroll
          for (int j = 0; j < 3; ++j)
            for (int x = 0; x < ks; ++x) {
              const int s = ks * g + x;
              const uint32_t acol = tmem + kTc5ColAa + (j == 0 ? NQ : 0) + 8 * s;
              const uint64_t bd = (j == 1 ? dba_lo : dba_hi) + 16 * s;
              mma_ts(tmem + 128 * g + 64 * part, acol, bd, id_a, j + x != 0);
            }
          commit(&mbar[1]);
        }
        if (copies) {
          if (SUB) {
            bulk_store(a.dst + ((size_t)(t % a.n_time) * a.n_bl + bl0 + t / a.n_time) * a.n_chan * 2,
                       strip0 + (size_t)(t & 1) * n16 * 8, strip_bytes);
            bulk_commit();
          }
          if (t + 2 < n_steps) {
            load_phases();
            if (!SUB) load_strip();
          }
        }
      }
      if (copies) {
        // loads still in flight after a failed wait must land before the CTA's shared
        // memory goes away (bounded); stores are waited for unconditionally
        for (int u = max(0, strips - 2); u < strips; ++u)
          mbar_wait(&mbar[2 + (u & 1)], (uint32_t)(u >> 1) & 1u, kTc5MaxPolls);
        for (int u = max(0, phases - 2); u < phases; ++u)
          mbar_wait(&mbar[6 + (u & 1)], (uint32_t)(u >> 1) & 1u, kTc5MaxPolls);
        bulk_wait_all();
      }
    }
  } else {
    // ---- the compute warps
    bool fail = false;                       // this thread's; the warps agree on it at csync
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      if (!wait_or_bad(bar, parity)) {
        fail = true;
        s_bad = 1;
        atomicExch(err, 1);
      }
      __syncwarp();
    };
    // the compute warps' own barrier; true once any thread's wait has run out
    auto csync = [&]() {
      uint32_t bad;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, 1, %2, p;\n\t"
          "selp.u32 %0, 1, 0, q;\n\t}"
          : "=r"(bad) : "r"((uint32_t)fail), "r"(kTc5Compute) : "memory");
      return bad != 0;
    };
    // this warp's shared-memory, TMEM writes and TMEM reads are done: one arrival (the
    // lanes meet again: the TMEM instructions that follow take a whole warp)
    auto warp_arrive = [&](uint64_t* bar) {
      fence_smem_async();
      fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar);
      __syncwarp();
    };
    auto phase_slot = [&](int t) { return ph + 2 * kTc5Src * (t & 1); };   // [sub 64][avg 64]

    // step t's tables, thread (k, g): all phasors, then all stores (a store to shared
    // memory between them would hold back the next table load).  Phases as Q0.32
    // multiples of rounded steps, within 6e-9 of a radian
    auto fill_tables = [&](int t) {
      const PhaseAB* p0 = phase_slot(t);
      const int k = tid & 63, g = tid >> 6;
      const bool u = 8 * g < NQ;
      float2 z[7];
      if (SUB) {
        const PhaseAB p = p0[k];
        const unsigned b = step32(p.b);
        z[0] = phasor_lut((unsigned)g * b, lut);
        z[1] = phasor_lut((unsigned)(g + 8) * b, lut);
        z[2] = phasor_lut(step32(p.a) + (unsigned)g * step32(p.b << 4), lut);
        if (u) z[3] = phasor_lut((unsigned)g * step32(p.b << 7), lut);
      }
      if (ACC) {
        const PhaseAB p = p0[kTc5Src + k];
        z[4] = phasor_lut(step32(p.a) + (unsigned)g * step32(p.b << 4), lut);
        if (u) z[5] = phasor_lut((unsigned)g * step32(p.b << 7), lut);
        z[6] = phasor_lut((unsigned)(g < 4 ? g : 4 * (g - 4)) * step32(p.b), lut);
      }
      Tc05Tab& T = tabs[t & 1];
      if (SUB) {
        T.sx[g][k] = z[0].x; T.sy[g][k] = z[0].y;
        T.sx[g + 8][k] = z[1].x; T.sy[g + 8][k] = z[1].y;
        T.svx[g][k] = z[2].x; T.svy[g][k] = z[2].y;
        if (u) { T.sux[g][k] = z[3].x; T.suy[g][k] = z[3].y; }
      }
      if (ACC) {
        T.avx[k][g] = z[4].x; T.avy[k][g] = z[4].y;
        if (u) T.au[g][k] = z[5];
        t2s[t % 3].pq[g][k] = z[6];
      }
    };
    // B_s of step t: thread (q % 8 = lane % 8, a pair of sources) takes every second
    // group of 8 tiles; its 8-byte stores cover whole 128-byte lines per half warp
    auto bs_fill = [&](int t) {
      const Tc05Tab& T = tabs[t & 1];
      const int ql = lane & 7, k = 2 * ((lane >> 3) + 4 * (warp & 7));
      const float2 vx = *reinterpret_cast<const float2*>(&T.svx[ql][k]);
      const float2 vy = *reinterpret_cast<const float2*>(&T.svy[ql][k]);
      const float2 nvy = make_float2(-vy.x, -vy.y);
      const int o = kmaj_byte(ql, k, kTc5Src);
      float2 ux[3], uy[3];
      #pragma unroll
      for (int u = 0; u < 3; ++u) {
        const int j = (warp >> 3) + 2 * u;
        if (8 * j < NQ) {
          ux[u] = *reinterpret_cast<const float2*>(&T.sux[j][k]);
          uy[u] = *reinterpret_cast<const float2*>(&T.suy[j][k]);
        }
      }
      #pragma unroll
      for (int u = 0; u < 3; ++u) {
        const int j = (warp >> 3) + 2 * u;
        if (8 * j < NQ) {
          float2 hi, lo;
          tc05_split2_unit(ffma2(vx, ux[u], fmul2(nvy, uy[u])), hi, lo);
          *reinterpret_cast<float2*>(bs_hi + o + j * 2048) = hi;
          *reinterpret_cast<float2*>(bs_lo + o + j * 2048) = lo;
          tc05_split2_unit(ffma2(vx, uy[u], fmul2(vy, ux[u])), hi, lo);
          *reinterpret_cast<float2*>(bs_hi + o + j * 2048 + NQ * 256) = hi;
          *reinterpret_cast<float2*>(bs_lo + o + j * 2048 + NQ * 256) = lo;
        }
      }
    };
    // A_s of step t, warp (qtr, cg): rows 32 qtr + lane = 8 r + 2 e + o, sources 16 cg ..:
    // re or im of M conj(T2) = (re, im or im, -re of M) . T2
    auto as_store = [&](int t, int slot) {
      const Tc05Tab& T = tabs[t & 1];
      const int r = 4 * qtr + (lane >> 3), e = (lane >> 1) & 3, o = lane & 1;
      const float* mp = models[slot].m[o][e];
      const float* mq = models[slot].m[o + 1][e];
      uint32_t vh[16], vl[16];
      #pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int k = 16 * cg + 4 * h;
        const float4 p = *reinterpret_cast<const float4*>(mp + k), q = *reinterpret_cast<const float4*>(mq + k);
        const float4 x = *reinterpret_cast<const float4*>(&T.sx[r][k]), y = *reinterpret_cast<const float4*>(&T.sy[r][k]);
        float2 hi, lo;
        tc05_split2(ffma2(make_float2(p.x, p.y), make_float2(x.x, x.y),
                         fmul2(make_float2(q.x, q.y), make_float2(y.x, y.y))), hi, lo);
        vh[4 * h] = __float_as_uint(hi.x); vh[4 * h + 1] = __float_as_uint(hi.y);
        vl[4 * h] = __float_as_uint(lo.x); vl[4 * h + 1] = __float_as_uint(lo.y);
        tc05_split2(ffma2(make_float2(p.z, p.w), make_float2(x.z, x.w),
                         fmul2(make_float2(q.z, q.w), make_float2(y.z, y.w))), hi, lo);
        vh[4 * h + 2] = __float_as_uint(hi.x); vh[4 * h + 3] = __float_as_uint(hi.y);
        vl[4 * h + 2] = __float_as_uint(lo.x); vl[4 * h + 3] = __float_as_uint(lo.y);
      }
      tmem_st16(tmem + lane_base + kTc5ColAsHi + 16 * cg, vh);
      tmem_st16(tmem + lane_base + kTc5ColAsLo + 16 * cg, vl);
    };
    // A_a of step t: rows 2 k + o, the warp's tiles q = cg QW ..: re or im of V U
    auto aa_store = [&](int t) {
      const Tc05Tab& T = tabs[t & 1];
      const int k = 16 * qtr + (lane >> 1), o = lane & 1, q0 = cg * QW;
      float4 x[3], y[3];
      float2 u[3];
      #pragma unroll
      for (int ch = 0; ch < 3; ++ch)
        if (4 * ch < QW) {
          const int q = q0 + 4 * ch;
          u[ch] = T.au[q >> 3][k];
          x[ch] = *reinterpret_cast<const float4*>(&T.avx[k][q & 7]);
          y[ch] = *reinterpret_cast<const float4*>(&T.avy[k][q & 7]);
        }
      #pragma unroll
      for (int ch = 0; ch < 3; ++ch) {
        if (4 * ch < QW) {
          const int q = q0 + 4 * ch;
          const float fa = o ? u[ch].y : u[ch].x, fb = o ? u[ch].x : -u[ch].y;
          const float2 a2 = make_float2(fa, fa), b2 = make_float2(fb, fb);
          float2 h0, l0, h1, l1;
          tc05_split2_unit(ffma2(make_float2(x[ch].x, x[ch].y), a2, fmul2(make_float2(y[ch].x, y[ch].y), b2)), h0, l0);
          tc05_split2_unit(ffma2(make_float2(x[ch].z, x[ch].w), a2, fmul2(make_float2(y[ch].z, y[ch].w), b2)), h1, l1);
          const uint32_t vh[4] = {__float_as_uint(h0.x), __float_as_uint(h0.y), __float_as_uint(h1.x), __float_as_uint(h1.y)};
          const uint32_t vl[4] = {__float_as_uint(l0.x), __float_as_uint(l0.y), __float_as_uint(l1.x), __float_as_uint(l1.y)};
          tmem_st4(tmem + lane_base + kTc5ColAa + q, vh);
          tmem_st4(tmem + lane_base + kTc5ColAa + NQ + q, vl);
        }
      }
    };
    // residual values x[u] = R(16 (q + u) + r, e).o, u = 0..3, into B_a: row 8 r + 2 e + o
    const int row_m = 32 * qtr + lane;
    const int ba_off = kmaj_byte(row_m, cg * QW, NQ);
    auto ba_put4 = [&](int ch, const float (&x)[4]) {
      float2 h0, l0, h1, l1;
      tc05_split2(make_float2(x[0], x[1]), h0, l0);
      tc05_split2(make_float2(x[2], x[3]), h1, l1);
      *reinterpret_cast<float4*>(ba_hi + ba_off + 128 * ch) = make_float4(h0.x, h0.y, h1.x, h1.y);
      *reinterpret_cast<float4*>(ba_lo + ba_off + 128 * ch) = make_float4(l0.x, l0.y, l1.x, l1.y);
    };
    // subtraction epilogue: rows 8 r + 2 e + o of lane, tiles q = cg QW ..; the strip
    // word (16 q + r) 8 + 2 e + o of the 32 lanes is 32 consecutive words.  The strip is
    // read before the wait for the MMAs, and a chunk of the accumulators while the
    // one before it is worked on
    auto strip_read = [&](const float* strip, float (&w)[12]) {
      #pragma unroll
      for (int u = 0; u < 12; ++u)
        if ((u & ~3) < QW) w[u] = strip[(16 * (cg * QW + u) + (row_m >> 3)) * 8 + (lane & 7)];
    };
    auto sub_epilogue = [&](float* strip, const float (&w)[12]) {
      const int r = row_m >> 3, q0 = cg * QW;
      const float sgn = lane & 1 ? 1.f : -1.f;   // re: a_re T_re + a_im T_im; im: a_im T_re - a_re T_im
      const uint32_t base = tmem + lane_base + q0;
      float v[2][4][4];
      #pragma unroll
      for (int i = 0; i < 4; ++i) tmem_ld4(base + i * NQ, v[0][i]);
      #pragma unroll
      for (int ch = 0; ch < 3; ++ch)
        if (4 * ch < QW) {
          __syncwarp();                      // the lanes part at the strip's ragged end
          tmem_wait_ld();
          if (ch < 2 && 4 * (ch + 1) < QW) {
            #pragma unroll
            for (int i = 0; i < 4; ++i) tmem_ld4(base + i * NQ + 4 * (ch + 1), v[(ch + 1) & 1][i]);
          }
          float x[4];
          #pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int c = 16 * (q0 + 4 * ch + u) + r;
            const float (&d)[4][4] = v[ch & 1];
            const float d1 = d[0][u] + d[2][u];
            const float d2 = __shfl_xor_sync(0xffffffffu, d[1][u] + d[3][u], 1);
            x[u] = 0.f;
            if (c < a.n_chan) {
              x[u] = fmaf(sgn, d2, w[4 * ch + u] - d1);
              strip[c * 8 + (lane & 7)] = x[u];
            }
          }
          if (ACC) ba_put4(ch, x);
        }
    };
    // first pass: B_a straight from the strip
    auto ba_from_strip = [&](const float* strip) {
      const int r = row_m >> 3, q0 = cg * QW;
      #pragma unroll
      for (int ch = 0; ch < 3; ++ch)
        if (4 * ch < QW) {
          float x[4];
          #pragma unroll
          for (int u = 0; u < 4; ++u) x[u] = strip[(16 * (q0 + 4 * ch + u) + r) * 8 + (lane & 7)];
          ba_put4(ch, x);
        }
    };
    // H of the last step: [4 rr + e] = this row's sums with (re, im) of R at r = 4 cg + rr
    float2 H[16];
    float2 ks[4], kn[4];                     // sums over the time steps of sum_r T2 H and minus their compensations
    #pragma unroll
    for (int e = 0; e < 4; ++e) ks[e] = kn[e] = make_float2(0.f, 0.f);
    auto contract = [&](int t) {
      const float2 (&T)[8][kTc5Src] = t2s[t % 3].pq;
      const int k = 16 * qtr + (lane >> 1);
      const float2 q = T[4 + cg][k];
      float2 s1[4], s2[4];
      #pragma unroll
      for (int rr = 1; rr < 4; ++rr) {       // P[0] = 1
        const float2 p = T[rr][k];
        #pragma unroll
        for (int e = 0; e < 4; ++e) {
          s1[e] = ffma2(make_float2(p.x, p.x), H[4 * rr + e], rr == 1 ? H[e] : s1[e]);
          s2[e] = rr == 1 ? fmul2(make_float2(p.y, p.y), H[4 * rr + e]) : ffma2(make_float2(p.y, p.y), H[4 * rr + e], s2[e]);
        }
      }
      const float2 neg = make_float2(-1.f, -1.f);
      #pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 v = make_float2(s1[e].x - s2[e].y, s1[e].y + s2[e].x);
        const float2 y = fadd2(make_float2(fmaf(v.x, q.x, -v.y * q.y), fmaf(v.x, q.y, v.y * q.x)), kn[e]);
        const float2 s = fadd2(ks[e], y);
        kn[e] = ffma2(neg, ffma2(neg, ks[e], s), y);
        ks[e] = s;
      }
    };
    // a baseline's averages: rows o = 0 and 1 (T1's real and imaginary parts) meet by
    // a shuffle, the column groups in B_a's words (free until C2)
    float4* fl = reinterpret_cast<float4*>(ba_hi);                 // [4 cg][64 k][4 e] (re, re lo, im, im lo)
    auto flush_put = [&]() {
      const int k = 16 * qtr + (lane >> 1);
      #pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float sx = __shfl_xor_sync(0xffffffffu, ks[e].x, 1), sy = __shfl_xor_sync(0xffffffffu, ks[e].y, 1);
        const float nx = __shfl_xor_sync(0xffffffffu, kn[e].x, 1), ny = __shfl_xor_sync(0xffffffffu, kn[e].y, 1);
        const FF re = ff_two_sum(ks[e].x, -sy), im = ff_two_sum(ks[e].y, sx);
        if (!(lane & 1))
          fl[(cg * kTc5Src + k) * 4 + e] = make_float4(re.hi, re.lo + (kn[e].x - ny), im.hi, im.lo + (kn[e].y + nx));
        ks[e] = kn[e] = make_float2(0.f, 0.f);
      }
    };
    const float inv = (float)a.inv_n, inv_lo = (float)(a.inv_n - (double)inv);
    auto flush_out = [&](int64_t bl) {
      const int k = tid >> 3, i = tid & 7;   // value i = (re, im) of pol i / 2
      const float2* f = reinterpret_cast<const float2*>(fl) + k * 8 + i;
      FF s = {f[0].x, f[0].y};
      #pragma unroll
      for (int c = 1; c < 4; ++c) {
        const float2 v = f[c * kTc5Src * 8];
        const FF x = ff_two_sum(s.hi, v.x);
        s.hi = x.hi;
        s.lo += x.lo + v.y;
      }
      if (k < a.n_acc)
        reinterpret_cast<float*>(a.avg)[((size_t)k * a.n_bl + bl) * 8 + i] =
            fmaf(s.hi, inv, fmaf(s.hi, inv_lo, s.lo * inv));
    };

    // the first step's operands
    wait(&mbar[6], 0);
    fill_tables(0);
    bool bad = csync();
    if (SUB && !bad) {
      bs_fill(0);
      as_store(0, 0);
      tmem_wait_st();
      warp_arrive(&mbar[4]);
    }
    // Half of the warps form B_s before A_s: phases that load different pipes run beside
    // each other.  (No branch on the warp around A_s or A_a: TMEM instructions under a
    // condition that the compiler cannot see to be a warp's gave wrong operands.)
    const bool odd = cg & 1;
    int tt = 0, ib = 0;                      // step t is time tt of baseline bl0 + ib
    for (int t = 0; t < n_steps && !bad; ++t) {
      const bool next = t + 1 < n_steps, last_tt = tt + 1 == a.n_time;
      float* strip = strip0 + (size_t)(t & 1) * n16 * 8;
      // ---- C1
      const bool new_model = SUB && next && last_tt && tid < 4 * kTc5Src;
      float2 m = make_float2(0.f, 0.f);
      if (new_model) m = get_model(bl0 + ib + 1);
      if (ACC) aa_store(t);
      if (ACC && t > 0) contract(t - 1);
      if (next) {
        wait(&mbar[6 + ((t + 1) & 1)], (uint32_t)((t + 1) >> 1) & 1u);
        fill_tables(t + 1);
      }
      if (new_model) put_model((ib + 1) & 1, m);
      const bool flush = ACC && tt == 0 && t > 0;       // the previous baseline is complete
      if (flush) flush_put();
      bad = csync();
      if (bad) break;
      if (flush) {
        flush_out(bl0 + ib - 1);
        bad = csync();
        if (bad) break;
      }
      // ---- C2
      wait(&mbar[2 + (t & 1)], (uint32_t)(t >> 1) & 1u);
      if (SUB) {
        float w[12];
        strip_read(strip, w);
        wait(&mbar[0], (uint32_t)t & 1u);
        fence_after_sync();
        sub_epilogue(strip, w);
      } else {
        ba_from_strip(strip);
      }
      if (ACC) tmem_wait_st();
      warp_arrive(&mbar[5]);
      // ---- C3
      if (next) {
        if (SUB) {
          if (odd) bs_fill(t + 1);
          as_store(t + 1, (ib + (last_tt ? 1 : 0)) & 1);
          if (!odd) bs_fill(t + 1);
        }
      }
      // ---- C4
      if (ACC) {
        wait(&mbar[1], (uint32_t)t & 1u);
        fence_after_sync();
        const uint32_t base = tmem + lane_base + 32 * cg;
        #pragma unroll
        for (int h = 0; h < 2; ++h) {
          float v[16], w[16];
          tmem_ld16(base + 16 * h, v);
          if (nacc == 2) tmem_ld16(base + 128 + 16 * h, w);
          tmem_wait_ld();
          #pragma unroll
          for (int i = 0; i < 8; ++i) {
            H[8 * h + i] = make_float2(v[2 * i], v[2 * i + 1]);
            if (nacc == 2) H[8 * h + i] = fadd2(H[8 * h + i], make_float2(w[2 * i], w[2 * i + 1]));
          }
        }
      }
      if (SUB && next) {
        tmem_wait_st();
        warp_arrive(&mbar[4]);
      }
      if (last_tt) { tt = 0; ++ib; }
      else ++tt;
    }
    if (ACC && !bad) {                       // the last baseline
      contract(n_steps - 1);
      flush_put();
      bad = csync();
      if (!bad) flush_out(bl0 + nbl - 1);
    }
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  if (warp == 0) tmem_dealloc(tmem, kTc5Cols);
}

}  // namespace rts
