// gemm_tc.cu -- kernel (c), tensor-core forms (bs = 64 and 128): BF16 error-free
// slice splits (3 or 4 slices) and FP16 with per-leaf power-of-two scaling;
// and their kernel (d), the pass that finishes the output leaves in FP64 and
// takes their norms.
//
// Each leaf product of Algorithm 1 ("C = AB" at the lowest level) is a real
// 64 x 64 x 64 contraction on tcgen05.  Operands are split at plan time
// (prep.cu, layout in tcforms.cuh):
//   BF16 split : every row of an A leaf and column of a B leaf as S = 3 or 4
//                BF16 slices on a grid set by the line's largest element
//                (slices.cuh); the slice products with index sum < S are
//                formed.  For one output element the products of one index
//                sum are integers on a common grid, so the K = 64 sum of
//                index sum 0 (and 1 for S = 4) is exact in its own FP32
//                accumulator; the smaller rest shares one accumulator.
//   FP16 scaled: a' = a 2^eA with max|a'| in [2^14, 2^15) per leaf,
//                a' = h0 + h1 (f16), likewise b'; products h0 g0, h0 g1, h1 g0
//                into one accumulator.
// Every step's accumulators are scaled back by the step's power of two
// (exact) and drained into registers: the FP16 form adds them to one FP32
// accumulator per output element; the BF16 forms keep a two-float (hi + lo)
// accumulator, adding each exact accumulator with an error-free TwoSum and
// the rest into lo.  The epilogue stores the pairs as they are; the finishing
// pass writes hi + lo in FP64 and the leaf norms, away from the GEMM, because
// this part issues FP64 instructions at two per clock per SM and an epilogue
// busy with them stops draining the accumulators the next MMAs need.
//
// 128 x 128 leaves.  A unit is one output leaf; its four 64 x 64 quadrants
// are the children, and every kept product runs as two K-half steps over the
// tile-split operand terms (prep.cu, steps.cu): the same steps and MMAs.
//
// Quads.  The four output leaves (2I + h, 2J + c) of a quadtree node one level
// above the leaves are computed together: at each k the A operand of term s is
// [A(2I,k)_s; A(2I+1,k)_s] (M = 128) and the B operand of term t is
// [B(k,2J)_t | B(k,2J+1)_t] (N = 128), so one step loads two A and two B leaves
// for up to four leaf products.  The steps of each quad (the four kept-product
// runs merged by k, with the leaves to load and each child's scale) are listed
// at plan time, so the kernel reads them sequentially.  A product whose norm
// test failed (or whose leaf is absent) is still formed by the MMA over the
// whole tile, but its quadrant is discarded by the epilogue; an operand leaf no
// kept product of the step needs is not loaded (its stale contents reach only
// discarded quadrants: each output element depends on one A row and one B
// column).  The 4-slice form stages each step in two K-halves (64 KB each,
// three in flight) so that its 128 KB of operands per step still pipeline.
// Accumulators are 128 x 128 FP32 slots of TMEM; four slots rotate (acc_slot below),
// so the MMAs of the next step start as soon as the epilogue has drained the slots
// they reuse.
//
// Warp roles (one CTA per SM, persistent; quads are claimed one at a time
// from a global counter in Morton order, so the quads in flight on all SMs
// form one narrow window whose A rows and B columns are shared in L2):
//   warp 0     TMA producer: claims the next quad for all roles (a ring of 4
//              in shared memory), ring of NS stages, one 1-D bulk copy per
//              leaf and stage (the leaf's K-part with all its pre-swizzled,
//              atom-interleaved terms), mbarriers.
//   warp 1     allocates 512 TMEM columns and issues the MMAs of each step.
//   warps 2-3  idle (they fill the first warpgroup, see the register split)
//   warps 4-11 epilogue: warps 4-7 column 0, warps 8-11 column 1; TMEM lane =
//              output row (warp w reads lanes 32 (w mod 4) ..); writes the
//              output rows as two-float pairs.
// No atomics on C: one CTA owns each output quad; k runs in ascending order.
// Every wait is bounded; on timeout the CTA sets the error word and leaves.
//
// What bounds it: per step the MMAs (64 cycles each: 10, 6 or 3 terms x 4 K pieces,
// 2560 / 1536 / 768 cycles), the FP32 pipe of the epilogue (about 1980 / 1050 / 130
// cycles where all four children are kept) and the copies (up to 128 / 96 / 64 KB
// through L2) all come within a factor of two of one another, and every hand-over
// between them is a look at a barrier in shared memory that takes some 250 cycles
// beside the operand reads.  Measured on the 3-D lattices (GEMM only, CUDA events),
// with the waits taken out of each role's way as the comments below say: 4 slices,
// n = 65536, tau = 1e-6, 115.6 -> 93 ms (1.42 PFLOP/s executed, one-column steps
// counted at half width: 83 % of the chip's power-limited rate); 3 slices, n = 16384, 8.19 -> 6.37 ms; FP16 with 128-leaves,
// n = 20000, tau = 1e-4, 7.67 -> 5.80 ms.  With single parts left out the first takes
// 68 ms (MMAs alone), 51 (copies alone), 80 (without epilogue), 85 (without copies).
#include "convert.cuh"
#include "internal.cuh"
#include "ptx.cuh"
#include "tcforms.cuh"

namespace spamm {

// ------------------------------------------------------------------- GEMM
// Three warpgroups: warpgroup 0 holds the producer (warp 0) and the MMA issuer
// (warp 1; warps 2-3 idle), warpgroups 1-2 the epilogue (warps 4-11).  The
// launch gives every thread 168 registers (384 x 168 = 64512 of 65536); the
// control warpgroup then gives up 96 of them per thread and the epilogue
// takes 48 more, enough for its two-float accumulators and one slot's columns:
// 128 x 72 + 256 x 216 = 64512, the launch total, so the increase never waits.
// (-Xptxas -v: the 4-slice kernel spills 48 bytes, the other two none.)
constexpr int kQuadThreads = 384;
constexpr uint32_t kLaunchRegs = 168, kCtlRegs = 72, kEpiRegs = 216;
static_assert(128 * kCtlRegs + 256 * kEpiRegs == kQuadThreads * kLaunchRegs, "register split must match the launch");
static_assert(kQuadThreads * kLaunchRegs <= 65536, "launch registers exceed the register file");
constexpr int kQuadBufs = 4;  // rotating TMEM accumulator slots of 128 FP32 columns
constexpr int kQuadQ = 4;     // ring of claimed quads shared by the three roles
// Ring of step scales, written by the producer (eight steps at a time) and read by
// the epilogue.  The producer's copies are at most the stages ahead of the MMAs, and
// these at most four steps (one per slot) ahead of the epilogue, so fewer than
// 8 + 6 + 4 entries are in use and one is read before it is reused.
constexpr int kScaleRing = 32;
// Steps before the end of a unit at which the next one is claimed.  Neighbouring
// units read the same leaves at the same k, so they share them in L2 only while they
// run side by side: claimed a whole unit ahead, their starts scatter over a unit's
// length (the copies alone of the 4-slice form on the n = 65536 lattice 72 ms instead
// of 54); claimed at the unit's end, its look-ups leave the stages empty.
constexpr int kClaimAhead = 5;

// One stage: two A and two B leaves, every term of a step (whole-K forms) or
// of one K-part of it.  A region: leaf 2I's part (all terms, atom-interleaved,
// tcforms.cuh) then leaf 2I+1's; B region at BREG: leaves 2J, 2J+1 likewise.
// Term s of the 128-row A operand [A(2I,k)_s; A(2I+1,k)_s] starts at s x atom
// with TERMS x atom between 8-row groups, and the same for B.
template <int PREC>
struct QuadLayout {
  using Cfg = FormCfg<PREC>;
  static constexpr uint32_t TILE = kTerm / Cfg::KPARTS;            // one term's part of one leaf
  static constexpr uint32_t LPART = (uint32_t)Cfg::TERMS * TILE;   // one leaf's part, all terms
  static constexpr uint32_t ATOM = term_atom<Cfg::KPARTS>();
  static constexpr uint32_t SBO = (uint32_t)Cfg::TERMS * ATOM;
  static constexpr int SPS = Cfg::KPARTS;      // stages per step
  static constexpr int KS = 4 / Cfg::KPARTS;   // K = 16 MMAs per stage
  static constexpr uint32_t BREG = 2 * LPART;
  static constexpr uint32_t STAGE = 2 * BREG;
  static constexpr size_t SMEM = 1024 + (size_t)Cfg::NS * STAGE;
  // high word of every operand's matrix descriptor (stride, version, swizzle)
  __device__ static constexpr uint32_t desc_hi() {
    return (uint32_t)((Cfg::KPARTS == 1   ? sw128_kmajor_desc(0, SBO)
                       : Cfg::KPARTS == 2 ? sw64_kmajor_desc(0, SBO)
                                          : sw32_kmajor_desc(0, SBO)) >>
                      32);
  }
};

double quad_step_flops(spamm_prec prec) {
  const int terms = prec == SPAMM_PREC_BF16_SPLIT ? 3 : (prec == SPAMM_PREC_BF16_SPLIT4 ? 4 : 2);
  return (double)(terms * (terms + 1) / 2) * 2.0 * 128.0 * 128.0 * 64.0;
}

// Accumulator slots.  A step's accumulator a < NACC - 1 takes the term products
// of index sum a (exact), the last one every larger sum.  kQuadBufs slots of 128
// FP32 columns rotate so that a step's first MMAs never wait for the previous
// step's last drain: the last accumulator (the longest in use, committed at the
// end of its step) alternates between slots 0 and 1, the others between 2 and 3;
// with three accumulators sums 0 and 1 swap slots 2 and 3 every step.  `use` is
// how often the slot was used before.
template <int NACC>
__device__ __forceinline__ void acc_slot(uint32_t n, int a, uint32_t* slot, uint32_t* use) {
  if constexpr (NACC == 1) {
    *slot = n & 3u;
    *use = n >> 2;
  } else if (a == NACC - 1) {
    *slot = n & 1u;
    *use = n >> 1;
  } else if constexpr (NACC == 2) {
    *slot = 2u + (n & 1u);
    *use = n >> 1;
  } else {
    *slot = 2u + ((n + (uint32_t)a + 1u) & 1u);
    *use = n;
  }
}
static_assert(kQuadBufs == 4, "acc_slot rotates four slots");

// The order of one stage's MMAs: K = 16 piece `ks` of A term i against B term j,
// and how the tensor core's buffer for A serves it.  A 128 x 128 x 16 MMA reads
// 8 KB of operands in the 64 cycles it computes, all that shared memory delivers
// (128 B per clock), beside the copies into the next stage; where consecutive
// MMAs use the same A piece, the first keeps it in the buffer (fill) and the
// others read only B.  The sum in an accumulator that is not exact depends on the
// order, so that is fixed: the smaller products (the larger index sum) first, each
// product whole, A's last term first.  (4 slices with each A term against all its B
// terms, 16 reads of A instead of 32, is as fast and 7e-4 further off.)  The exact
// products go wherever their accumulators are in use for the shortest time, as the
// four slots are what the next step waits for: last in the first K-part, where they
// ride on the A of the smallest index sum that shares an accumulator, and first in
// the last one.  At the end of the last part instead they cost the 4-slice form 104 ms
// for 93 (n = 65536), the 3-slice form 6.63 for 6.37 (n = 16384).
struct MmaOrder {
  int n = 0;
  uint8_t i[48] = {}, j[48] = {}, ks[48] = {}, collect[48] = {};
  __host__ __device__ constexpr void add(int i_, int j_, int ks_, int collect_) {
    i[n] = (uint8_t)i_;
    j[n] = (uint8_t)j_;
    ks[n] = (uint8_t)ks_;
    collect[n] = (uint8_t)collect_;
    ++n;
  }
};
template <int PREC>
__host__ __device__ constexpr MmaOrder mma_order(bool last_part) {
  constexpr int T = FormCfg<PREC>::TERMS, KS = 4 / FormCfg<PREC>::KPARTS;
  MmaOrder o;
  if (last_part && T > 2)  // the exact products
    for (int i = 0; i < T - 2; ++i)
      for (int ks = 0; ks < KS; ++ks)
        for (int j = 0; j < T - 2 - i; ++j)
          o.add(i, j, ks, i == T - 3 ? kCollectNone : j == 0 ? kCollectFill : kCollectLast);
  for (int g = T - 1; g >= (T > 2 ? T - 2 : 0); --g)
    for (int i = g; i >= 0; --i)
      for (int ks = 0; ks < KS; ++ks) {
        const int exact = !last_part && g == T - 2 && i < g ? g - i : 0;  // exact products that ride on this A
        o.add(i, g - i, ks, exact ? kCollectFill : kCollectNone);
        for (int j = exact - 1; j >= 0; --j) o.add(i, j, ks, j == 0 ? kCollectLast : kCollectUse);
      }
  return o;
}

// Issues one stage's MMAs into the step's accumulator slots.  ready(a): waits until
// slot a may be overwritten, called before the first MMA into it; ahead(): called
// a few MMAs before the end, while the tensor core still has work queued (it takes
// about five MMAs ahead), to look at the barriers the next stage needs -- a wait
// on a barrier in shared memory takes some 250 cycles beside the operand reads, and
// the tensor core would run dry; done(a): after the last MMA into slot a.
constexpr int kAhead = 4;
template <int PREC, bool FIRST, bool LAST, class Ready, class Ahead, class Done>
__device__ __forceinline__ bool issue_stage(uint32_t tbase, const uint32_t (&slot)[3], uint32_t a_s, uint32_t b_s,
                                            uint32_t idesc, Ready ready, Ahead ahead, Done done) {
  using Cfg = FormCfg<PREC>;
  using Lay = QuadLayout<PREC>;
  constexpr uint32_t HI = Lay::desc_hi();
  constexpr MmaOrder O = mma_order<PREC>(LAST);
  const uint32_t alo = desc_lo(a_s), blo = desc_lo(b_s);
  bool fresh[3] = {FIRST, FIRST, FIRST};
  int left[3] = {0, 0, 0};
#pragma unroll
  for (int q = 0; q < O.n; ++q) ++left[O.i[q] + O.j[q] < Cfg::NACC - 1 ? O.i[q] + O.j[q] : Cfg::NACC - 1];
#pragma unroll
  for (int q = 0; q < O.n; ++q) {
    const int a = O.i[q] + O.j[q] < Cfg::NACC - 1 ? O.i[q] + O.j[q] : Cfg::NACC - 1;
    if (fresh[a] && !ready(a)) return false;
    if (q == O.n - kAhead) ahead();
    umma_f16(tbase + slot[a] * 128u, alo + ((O.i[q] * Lay::ATOM + 32u * O.ks[q]) >> 4),
             blo + ((O.j[q] * Lay::ATOM + 32u * O.ks[q]) >> 4), HI, idesc, fresh[a] ? 0u : 1u, O.collect[q]);
    fresh[a] = false;
    if (LAST && --left[a] == 0) done(a);
  }
  return true;
}

// Eight pairs of adjacent output elements at a time: (hi, lo) += v sc with an
// error-free TwoSum of hi and v sc (the product is exact: sc is a power of two),
// in the packed FP32x2 instructions, each lane rounding like the scalar
// round-to-nearest operation; hi + lo gains v sc up to the rounding of lo.  Seven
// instructions per pair (the products ride in the two FMAs), taken across the
// eight pairs one operation after the other: a packed instruction issues every
// two cycles and its result is ready after four, so a single pair's chain would
// leave the pipe idle half of the time (measured with two warps per scheduler:
// 1165 cycles per 64 columns in eight instructions pair by pair, 920 like this,
// the pipe's rate).
__device__ __forceinline__ void two_sum_x8(uint64_t* hi, uint64_t* lo, const uint32_t* v, uint64_t sc2) {
  uint64_t x[8], s[8], nb[8], t[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) x[q] = pack_x2(v[2 * q], v[2 * q + 1]);
#pragma unroll
  for (int q = 0; q < 8; ++q) s[q] = fma_x2(x[q], sc2, hi[q]);
#pragma unroll
  for (int q = 0; q < 8; ++q) nb[q] = sub_x2(hi[q], s[q]);  // -(s - hi)
#pragma unroll
  for (int q = 0; q < 8; ++q) t[q] = add_x2(s[q], nb[q]);
#pragma unroll
  for (int q = 0; q < 8; ++q) nb[q] = fma_x2(x[q], sc2, nb[q]);  // v sc - (s - hi)
#pragma unroll
  for (int q = 0; q < 8; ++q) t[q] = sub_x2(hi[q], t[q]);  // hi - (s - (s - hi))
#pragma unroll
  for (int q = 0; q < 8; ++q) t[q] = add_x2(t[q], nb[q]);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    hi[q] = s[q];
    lo[q] = add_x2(lo[q], t[q]);
  }
}

// What the producer tells the other roles about a claimed unit.
struct UnitInfo {
  double* out[4];  // first element of each child's 64 x 64 output, null where absent
  int32_t nstep;   // -1: no more units
  int32_t ld;      // row length of the output leaves
};

template <int PREC>
__global__ void __launch_bounds__(kQuadThreads, 1)
    gemm_quad_kernel(BatchDev batch, unsigned long long* __restrict__ work, int* __restrict__ err) {
  using Cfg = FormCfg<PREC>;
  using Lay = QuadLayout<PREC>;
  constexpr int NS = Cfg::NS, NACC = Cfg::NACC, NB = kQuadBufs, SPS = Lay::SPS;
  constexpr uint32_t LEAF = leaf_bytes<PREC>(), STAGE = Lay::STAGE, BREG = Lay::BREG, LP = Lay::LPART;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[NS], empty[NS], tfull[NB], tempty[NB], qfull[kQuadQ], qempty[kQuadQ];
  __shared__ UnitInfo qinfo[kQuadQ];
  __shared__ __align__(16) float4 sscale[kScaleRing];  // step n's scales at n mod kScaleRing
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < NB; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 8);  // the eight epilogue warps, one arrival each
    }
    for (int q = 0; q < kQuadQ; ++q) {
      mbar_init(&qfull[q], 1);
      mbar_init(&qempty[q], 9);  // the MMA issuer and the eight epilogue warps
    }
    fence_mbar_init();
    abort_flag = 0;
  }
  if (warp == 1) {
    tmem_alloc(&tmem_base, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = tmem_base;
  volatile int* abortp = &abort_flag;
  if (warp < 4) {
    regs_dec<kCtlRegs>();  // every warp of warpgroup 0, at this one instruction
    if (warp == 0) {
      // ---------------- TMA producer; claims the quads (Morton order, first come first served) for all
      // roles.  Step records are read eight at a time, lanes 4 i .. 4 i + 3 holding the four leaf indices
      // (and scales) of step i, which these lanes then copy: no shuffles, and one load per eight steps,
      // well ahead of its use.  The next unit is claimed and looked up during the current one's last
      // steps, each dependent load one step before it is used.
      struct Unit {
        const int32_t* rec;  // records of eight words: a0, a1, b0, b1, four scales
        const uint8_t* term; // this lane's operand: A (lanes 0, 1 mod 4) or B
        int32_t nstep;       // -1: no more units
      };
      const int sub = lane >> 2, leafn = lane & 3;  // this lane's step of eight and its leaf in it
      uint32_t t = 0, n = 0;       // stages filled, steps listed
      uint32_t s = 0, ephase = 1;  // the stage to fill, and the phase of `empty` that frees it (from the second fill on)
      bool ok = true;
      // The next unit (number c of this CTA), in three parts.
      unsigned long long claimed = 0;
      const PlanDev* npl = nullptr;
      int64_t nQ = 0, nq0 = 0, nq1 = 0;
      int32_t ngrp = 0, nidx = -1, nscl = 0;  // nidx, nscl: its first eight records
      Unit next{nullptr, nullptr, -1};
      auto load = [&](const Unit& u, int32_t j, int32_t* idx, int32_t* scl) {
        const bool in = j + sub < u.nstep;
        const int32_t* r = u.rec + 8 * (int64_t)(j + sub) + leafn;
        *idx = in ? __ldg(r) : -1;
        *scl = in ? __ldg(r + 4) : 0;
      };
      auto advance = [&](int part, uint32_t c) {
        if (part == 0) {  // claim it
          if (lane == 0) claimed = atomicAdd(work, 1ull);
        } else if (part == 1) {  // find its plan, start reading its step range and outputs
          const int64_t un = (int64_t)__shfl_sync(0xffffffffu, claimed, 0);
          npl = nullptr;
          if (un < batch.nunits) {
            const int r = plan_of(batch.ubegin, batch.nplans, un);
            npl = batch.plans + r;
            const int64_t Qc = un - batch.ubegin[r];
            nQ = npl->uorder ? npl->uorder[Qc] : npl->ufirst + Qc;
            nq0 = npl->qstart[nQ];
            nq1 = npl->qstart[nQ + 1];
            ngrp = npl->tc_bs == 128 ? 0 : npl->quads[4 * nQ + leafn];
          }
        } else {  // enter it in the ring (not announced yet), start reading its first records
          next.nstep = -1;
          if (npl) {
            next.nstep = (int32_t)(nq1 - nq0);
            next.rec = reinterpret_cast<const int32_t*>(npl->qsteps) + 8 * nq0;
            next.term = leafn < 2 ? npl->termsA : npl->termsB;
          }
          load(next, 0, &nidx, &nscl);
          ok = ok && (c < kQuadQ || mbar_wait_or_abort(&qempty[c % kQuadQ], ((c / kQuadQ) - 1) & 1u, abortp));
          ok = __all_sync(0xffffffffu, ok);
          if (ok && lane < 4) {
            UnitInfo& info = qinfo[c % kQuadQ];
            if (npl) {  // lane c: child c; the four quadrants of output leaf Q, or up to four output leaves
              const bool big = npl->tc_bs == 128;
              info.out[lane] = ngrp < 0 ? nullptr
                               : big    ? npl->cpool + nQ * 16384 + (lane >> 1) * 8192 + (lane & 1) * 64
                                        : npl->cpool + (int64_t)ngrp * 4096;
              if (lane == 0) info.ld = big ? 128 : 64;
            }
            if (lane == 0) info.nstep = next.nstep;
          }
          __syncwarp();
        }
      };
      for (int part = 0; part < 3; ++part) advance(part, 0);
      for (uint32_t c = 0; ok; ++c) {
        const Unit cur = next;
        int32_t idx = nidx, scl = nscl;
        if (lane == 0) mbar_arrive(&qfull[c % kQuadQ]);
        if (cur.nstep < 0) break;
        int part = 0;
        for (int32_t jb = 0; jb < cur.nstep && ok; jb += 8) {
          int32_t idx2, scl2;
          load(cur, jb + 8, &idx2, &scl2);
          const unsigned used = __ballot_sync(0xffffffffu, idx >= 0);
          const uint8_t* src = cur.term + (int64_t)idx * LEAF;
          reinterpret_cast<int32_t*>(&sscale[(n + sub) % kScaleRing])[leafn] = scl;
          __syncwarp();  // ordered before the arrivals below, which the epilogue's waits follow
          const int m = min(8, cur.nstep - jb);
          for (int i = 0; i < m && ok; ++i, ++n) {
            const uint32_t bytes = (uint32_t)__popc((used >> (4 * i)) & 15u) * LP;
#pragma unroll
            for (int h = 0; h < SPS; ++h) {
              if (t >= NS) ok = __all_sync(0xffffffffu, mbar_wait_or_abort(&empty[s], ephase, abortp));
              if (!ok) break;
              if (sub == i) {  // one copy per leaf: its part h, every term
                if (leafn == 0) mbar_arrive_expect_tx(&full[s], bytes);
                if (idx >= 0) bulk_g2s(smem + s * STAGE + (uint32_t)leafn * LP, src + (int64_t)h * LP, LP, &full[s]);
              }
              ++t;
              if (++s == NS) {
                s = 0;
                ephase ^= 1u;
              }
            }
            if (ok && part < 3 && cur.nstep - (jb + i) <= kClaimAhead) advance(part++, c + 1);
          }
          idx = idx2;
          scl = scl2;
        }
        while (part < 3 && ok) advance(part++, c + 1);
      }
      if (lane == 0) {
        if (!ok) {
          atomicOr(err, DEV_ERR_TIMEOUT);
          *abortp = 1;
        }
        // leave no bulk copy in flight: the last fill of every stage has landed
        for (uint32_t k = (t > NS ? t - NS : 0); k < t; ++k) mbar_wait_bounded(&full[k % NS], (k / NS) & 1u);
      }
    } else if (warp == 1) {
      // ---------------- MMA issuer (one elected lane)
      if (elect_one()) {
        constexpr int A0 = mma_order<PREC>(SPS == 1).i[0] + mma_order<PREC>(SPS == 1).j[0] < NACC - 1
                               ? mma_order<PREC>(SPS == 1).i[0] + mma_order<PREC>(SPS == 1).j[0]
                               : NACC - 1;  // the accumulator a step touches first
        const uint32_t smem0 = smem_u32(smem);
        uint32_t n = 0;                  // steps started
        uint32_t s = 0, sphase = 0;      // stage, and the phase of its next fill
        uint32_t last = 0, lphase = 0;   // the last committed stage and its phase
        bool any = false, stop = false;
        bool saw_full = false, saw_slot = false;  // the next stage / its first slot, seen ready ahead
        for (uint32_t c = 0; !stop; ++c) {
          const uint32_t qs = c % kQuadQ;
          if (!mbar_wait_or_abort(&qfull[qs], (c / kQuadQ) & 1u, abortp)) {
            stop = true;
            break;
          }
          const int32_t nstep = qinfo[qs].nstep;
          mbar_arrive(&qempty[qs]);
          if (nstep < 0) break;
          for (int32_t j = 0; j < nstep && !stop; ++j, ++n) {
            uint32_t idesc = 0, doff = 0, boff = 0;  // the step's width and columns (its first stage sets them)
            uint32_t slot[3] = {0, 0, 0}, use[3] = {0, 0, 0};
#pragma unroll
            for (int a = 0; a < NACC; ++a) acc_slot<NACC>(n, a, &slot[a], &use[a]);
            uint32_t nslot, nuse;  // the next step's first slot
            acc_slot<NACC>(n + 1, A0, &nslot, &nuse);
            auto ready = [&](int a) {
              if (use[a] == 0) return true;
              if (a == A0 && saw_slot) {
                tc_fence_after();
                return true;
              }
              if (!mbar_wait_or_abort(&tempty[slot[a]], (use[a] - 1u) & 1u, abortp)) return false;
              tc_fence_after();
              return true;
            };
            auto done = [&](int a) { umma_commit(&tfull[slot[a]]); };
#pragma unroll
            for (int h = 0; h < SPS; ++h) {
              if (!saw_full && !mbar_wait_or_abort(&full[s], sphase, abortp)) {
                stop = true;
                break;
              }
              tc_fence_after();
              // Split forms: a step whose kept products lie in one output column runs
              // half-width MMAs on that column's B leaf (a quarter of the steps on the 3-D
              // lattices): 4 slices, n = 65536, 97 -> 92 ms, 3 slices, n = 16384, 6.75 -> 6.61 ms.
              // FP16, bound by its copies, was 1.5 % slower for the look at the scales.
              if constexpr (NACC == 1) {
                idesc = umma_idesc_f16(Cfg::AB, 128, 128);
              } else if (h == 0) {
                const float4 sc = sscale[n % kScaleRing];
                const bool c0 = sc.x != 0.f || sc.z != 0.f, c1 = sc.y != 0.f || sc.w != 0.f;
                idesc = c0 && c1 ? umma_idesc_f16(Cfg::AB, 128, 128) : umma_idesc_f16(Cfg::AB, 128, 64);
                doff = c0 ? 0u : 64u;
                boff = c0 ? 0u : LP;
              }
              const uint32_t a_s = smem0 + s * STAGE, b_s = a_s + BREG + boff;
              const uint32_t s1 = s + 1 == NS ? 0 : s + 1, p1 = s + 1 == NS ? sphase ^ 1u : sphase;
              bool sf = false, ss = false;
              auto ahead = [&] {
                sf = mbar_test_wait(&full[s1], p1);
                if (h == SPS - 1) ss = nuse > 0 && mbar_test_wait(&tempty[nslot], (nuse - 1u) & 1u);
              };
              bool ok;
              if (SPS == 1)
                ok = issue_stage<PREC, true, true>(tbase + doff, slot, a_s, b_s, idesc, ready, ahead, done);
              else if (h == 0)
                ok = issue_stage<PREC, true, false>(tbase + doff, slot, a_s, b_s, idesc, ready, ahead, done);
              else if (h == SPS - 1)
                ok = issue_stage<PREC, false, true>(tbase + doff, slot, a_s, b_s, idesc, ready, ahead, done);
              else
                ok = issue_stage<PREC, false, false>(tbase + doff, slot, a_s, b_s, idesc, ready, ahead, done);
              umma_commit(&empty[s]);
              saw_full = sf;
              saw_slot = ss;
              any = true;
              last = s;
              lphase = sphase;
              s = s1;
              sphase = p1;
              if (!ok) {
                stop = true;
                break;
              }
            }
          }
        }
        if (stop) {
          atomicOr(err, DEV_ERR_TIMEOUT);
          *abortp = 1;
        }
        // leave no MMA in flight: everything issued before the last commit has completed
        if (any) mbar_wait_bounded(&empty[last], lphase);
      }
    }
  } else {
    regs_inc<kEpiRegs>();
    // ---------------- epilogue: warps 4..11; column c = (warp - 4) / 4; TMEM lane = output row.  Each
    // warp goes its own way (its own arrivals on the unit ring and the slots), so one warp's output
    // stores overlap the others' sums.
    const int col = (warp - 4) >> 2;
    const int quarter = warp & 3;
    const int lrow = 32 * quarter + lane;
    const int half = lrow >> 6, row = lrow & 63;
    const int child = 2 * half + col;  // warp-uniform
    const uint32_t taddr0 = tbase + ((uint32_t)(32 * quarter) << 16) + 64u * (uint32_t)col;
    uint32_t n = 0;     // steps drained
    bool seen = false;  // the next accumulator was seen complete ahead
    // FP16: one FP32 accumulator per element; BF16 splits: (hi, lo) pairs of
    // adjacent elements packed for the FP32x2 instructions
    constexpr int NHI = NACC == 1 ? 64 : 1, NPK = NACC == 1 ? 1 : 32;
    float hi[NHI];
    uint64_t hi2[NPK], lo2[NPK];
    bool failed = false;
    for (uint32_t c = 0; !failed; ++c) {
      const uint32_t qs = c % kQuadQ;
      bool ok = true;
      if (lane == 0) ok = mbar_wait_or_abort(&qfull[qs], (c / kQuadQ) & 1u, abortp);
      if (!__shfl_sync(0xffffffffu, ok ? 1 : 0, 0)) {
        failed = true;
        break;
      }
      const int32_t nstep = qinfo[qs].nstep, ld = qinfo[qs].ld;
      double* const outp = qinfo[qs].out[child];
      __syncwarp();
      if (lane == 0) mbar_arrive(&qempty[qs]);
      if (nstep < 0) break;
#pragma unroll
      for (int i = 0; i < NHI; ++i) hi[i] = 0.f;
#pragma unroll
      for (int i = 0; i < NPK; ++i) hi2[i] = lo2[i] = 0ull;
      auto wait_full = [&](uint32_t b, uint32_t use) {
        bool done = true;
        if (lane == 0) done = mbar_wait_or_abort(&tfull[b], use & 1u, abortp);
        return __shfl_sync(0xffffffffu, done ? 1 : 0, 0) != 0;
      };
      auto release = [&](uint32_t b) {  // one arrival per warp, after all its lanes' loads
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[b]);
      };
      // 32 of the slot's columns, added to the accumulators of columns 32 hh ..
      auto add_up = [&](int hh, const uint32_t (&v)[32], bool exact, float sc) {
        const uint64_t sc2 = ((uint64_t)__float_as_uint(sc) << 32) | __float_as_uint(sc);
        if constexpr (NACC == 1) {
#pragma unroll
          for (int i = 0; i < 32; ++i) hi[32 * hh + i] = fmaf(__uint_as_float(v[i]), sc, hi[32 * hh + i]);
        } else if (exact) {  // an exact accumulator: TwoSum into (hi, lo)
          two_sum_x8(hi2 + 16 * hh, lo2 + 16 * hh, v, sc2);
          two_sum_x8(hi2 + 16 * hh + 8, lo2 + 16 * hh + 8, v + 16, sc2);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            lo2[16 * hh + i] = fma_x2(pack_x2(v[2 * i], v[2 * i + 1]), sc2, lo2[16 * hh + i]);
        }
      };
      // One step: its accumulators in the order the MMAs commit them.  A slot's 64 columns of this
      // thread's row are loaded in two halves and handed back to the MMAs before they are added up; the
      // next accumulator's halves are loaded as soon as the registers of this one's are free, so their
      // way from tensor memory passes behind the sums.
      auto step = [&]() {
        uint32_t b, use;
        acc_slot<NACC>(n, 0, &b, &use);
        if (!seen && !wait_full(b, use)) return false;
        seen = false;
        tc_fence_after();
        const float sc = reinterpret_cast<const float*>(&sscale[n % kScaleRing])[child];
        if (sc == 0.f) {  // no kept product of this warp's child at this k
          release(b);
#pragma unroll
          for (int a = 1; a < NACC; ++a) {
            acc_slot<NACC>(n, a, &b, &use);
            if (!wait_full(b, use)) return false;
            release(b);
          }
          return true;
        }
        uint32_t va[32], vb[32];
        tmem_ld32_async(taddr0 + b * 128u, va);
        tmem_ld32_async(taddr0 + b * 128u + 32u, vb);
#pragma unroll
        for (int a = 0; a < NACC; ++a) {
          tmem_wait32(va);  // waits for every load in flight
          tmem_wait32(vb);
          release(b);
          add_up(0, va, a < NACC - 1, sc);
          if (a + 1 < NACC) {
            acc_slot<NACC>(n, a + 1, &b, &use);
            if (!wait_full(b, use)) return false;
            tc_fence_after();
            tmem_ld32_async(taddr0 + b * 128u, va);
          } else {
            acc_slot<NACC>(n + 1, 0, &b, &use);
            seen = __all_sync(0xffffffffu, mbar_test_wait(&tfull[b], use & 1u));
          }
          add_up(1, vb, a < NACC - 1, sc);
          if (a + 1 < NACC) tmem_ld32_async(taddr0 + b * 128u + 32u, vb);
        }
        return true;
      };
      for (int32_t j = 0; j < nstep; ++j, ++n) {
        if (!step()) {
          failed = true;
          break;
        }
      }
      if (failed) break;
      // output row `row` of this warp's child, unconverted: each element's 8-byte
      // slot receives its two-float pair (hi, lo) (FP16: (hi, 0)); the finishing
      // pass (tc_finish_kernel) turns the slots into FP64 and takes the leaf
      // norms, so no FP64 instruction runs here, where it would hold up the
      // draining of the accumulators the next quad's MMAs wait for.  32 bytes
      // (one sector) per lane and store, 16 where the caller's allocator gave the pool an
      // address between sectors.
      if (outp) {
        double* out = outp + row * ld;
        const bool wide = (reinterpret_cast<uintptr_t>(outp) & 31) == 0;  // rows are a multiple of 512 bytes
#pragma unroll
        for (int q = 0; q < 64; q += 4) {
          if constexpr (NACC == 1)
            store_32(out + q, wide, __float_as_uint(hi[q]), 0u, __float_as_uint(hi[q + 1]), 0u,
                     __float_as_uint(hi[q + 2]), 0u, __float_as_uint(hi[q + 3]), 0u);
          else
            store_32(out + q, wide, (uint32_t)hi2[q / 2], (uint32_t)lo2[q / 2], (uint32_t)(hi2[q / 2] >> 32),
                     (uint32_t)(lo2[q / 2] >> 32), (uint32_t)hi2[q / 2 + 1], (uint32_t)lo2[q / 2 + 1],
                     (uint32_t)(hi2[q / 2 + 1] >> 32), (uint32_t)(lo2[q / 2 + 1] >> 32));
        }
      }
    }
    if (failed && lane == 0) {
      atomicOr(err, DEV_ERR_TIMEOUT);
      *abortp = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tbase, 512);
  }
}

static unsigned gemm_grid(spamm_ctx ctx, int64_t nunits) {
  int64_t grid = ctx->gemm_sm_limit > 0 ? ctx->gemm_sm_limit : ctx->num_sms;
  if (grid > nunits) grid = nunits;
  return (unsigned)(grid < 1 ? 1 : grid);
}

template <int PREC>
static void launch_quads(spamm_ctx ctx, const BatchDev& b) {
  if (b.nunits == 0) return;
  const size_t smem = QuadLayout<PREC>::SMEM;
  // the register split in the kernel assumes exactly kLaunchRegs per thread at
  // launch: with fewer, the epilogue's increase could never be granted
  // (checked once per context)
  if (!(ctx->tc_ready >> PREC & 1)) {
    cudaFuncAttributes attr;
    CK(cudaFuncGetAttributes(&attr, gemm_quad_kernel<PREC>));
    if (attr.numRegs != (int)kLaunchRegs || attr.maxThreadsPerBlock < kQuadThreads)
      fail(SPAMM_E_CUDA, "tensor-core kernel built with an unexpected register count; refusing to launch");
    CK(cudaFuncSetAttribute(gemm_quad_kernel<PREC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    ctx->tc_ready |= 1 << PREC;
  }
  gemm_quad_kernel<PREC><<<gemm_grid(ctx, b.nunits), kQuadThreads, smem, ctx->stream>>>(b, b.work, ctx->d_err);
  CK_LAUNCH("gemm_quad_kernel");
}

// ------------------------------------------------------------------ finish
// Kernel (d) for the tensor-core forms: every 8-byte slot of an output leaf
// holds the two-float pair (hi, lo) the GEMM's epilogue left there (FP16: lo =
// 0); the slot becomes the FP64 value hi + lo (FP16: the exact conversion of hi
// alone), and the leaf's squared Frobenius norm is
// accumulated with one FMA per element in the order of kernel (a) -- lane l
// takes the 16-byte pairs l, l + 32, ..., a butterfly combines the lanes -- so
// the stored norm equals kernel (a) applied to the finished leaf, bit for bit.
// One warp per leaf, eight leaves per block.  The FMA of the norm is the only FP64
// instruction (two per clock and SM): the pair is added in integer arithmetic, exact
// where the floats' exponents are within 28 of one another (the others take the
// FP64 addition, one rounding), so HBM bounds both forms: 418,979 leaves of the split
// forms (27.5 GB) 7.3 -> 4.5 ms, 51,491 leaves 0.78 -> 0.52 ms.
// Eight 16-byte pieces per lane are read before the first is written back: the
// writes go to where the reads come from, so the compiler keeps their order and a
// lane would wait for memory at every piece.  4088 leaves (134 MB, FP16 form): 313 ->
// 45 us, 20023 leaves of 128 x 128 (2.6 GB) 1.50 -> 0.78 ms; with 64 leaves per block a few
// thousand leaves kept a third of the SMs busy.  All outputs of a batch in one launch:
// a leaf's chain of additions takes 20 us however few leaves there are, and eight
// outputs (n = 1000 .. 5000) took 272 us one after the other; in one launch their
// batch takes 2.76 ms instead of 2.88.
constexpr int64_t kFinishLeavesPerBlock = 8;

template <bool TWO>
__global__ void __launch_bounds__(256) tc_finish_kernel(const __grid_constant__ OutBatch out, int bs) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t e = (int64_t)bs * bs;
  const int pairs = bs * bs / 2;
  for (int64_t u = (int64_t)blockIdx.x * kFinishLeavesPerBlock + warp; u < out.total;
       u += (int64_t)gridDim.x * kFinishLeavesPerBlock) {
    const int r = out.n > 1 ? plan_of(out.first, out.n, u) : 0;
    const OutLeaves C = out.n > 1 ? out.tab[r] : out.only;
    const int64_t q = out.n > 1 ? u - out.first[r] : u;
    uint4* leaf = reinterpret_cast<uint4*>(C.pool + q * e);
    double s = 0.0;
    for (int i = lane; i < pairs; i += 32 * 8) {
      uint64_t x[8][2];  // (hi, lo) of elements 2i and 2i + 1, then their values' bits
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const uint4 w = leaf[i + 32 * u];
        x[u][0] = (uint64_t)w.y << 32 | w.x;
        x[u][1] = (uint64_t)w.w << 32 | w.z;
      }
      unsigned rest = 0;  // pairs left to the FP64 addition (a branch of its own: rare, and
                          // predicated it would take the pipe's time all the same)
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        uint64_t& b = x[u >> 1][u & 1];
        const uint32_t hi = (uint32_t)b, lo = (uint32_t)(b >> 32);
        if (!TWO)
          b = f32_to_f64_bits(hi);
        else if (f32_pair_sum_covers(hi, lo))
          b = f32_pair_sum_bits(hi, lo);
        else
          rest |= 1u << u;
      }
      if (TWO && __any_sync(0xffffffffu, rest != 0)) {
#pragma unroll 1
        for (int u = 0; u < 16; ++u)
          if (rest >> u & 1u) {
#pragma unroll
            for (int k = 0; k < 16; ++k)
              if (k == u) {
                uint64_t& b = x[k >> 1][k & 1];
                b = (uint64_t)__double_as_longlong(
                    __dadd_rn(__longlong_as_double((long long)f32_to_f64_bits((uint32_t)b)),
                              __longlong_as_double((long long)f32_to_f64_bits((uint32_t)(b >> 32)))));
              }
          }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const double x0 = __longlong_as_double((long long)x[u][0]), x1 = __longlong_as_double((long long)x[u][1]);
        s = __fma_rn(x0, x0, s);
        s = __fma_rn(x1, x1, s);
        leaf[i + 32 * u] = make_uint4((uint32_t)x[u][0], (uint32_t)(x[u][0] >> 32), (uint32_t)x[u][1],
                                      (uint32_t)(x[u][1] >> 32));
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) {
      C.sq[q] = s;
      C.slot[q] = q;
    }
  }
}

void tc_finish(spamm_ctx ctx, spamm_prec prec, const OutBatch& out, int bs) {
  if (out.total <= 0) return;
  const int64_t nblk = (out.total + kFinishLeavesPerBlock - 1) / kFinishLeavesPerBlock;
  const unsigned grid = (unsigned)(nblk < (1ll << 30) ? nblk : (1ll << 30));
  if (prec == SPAMM_PREC_FP16_SCALED)
    tc_finish_kernel<false><<<grid, 256, 0, ctx->stream>>>(out, bs);
  else
    tc_finish_kernel<true><<<grid, 256, 0, ctx->stream>>>(out, bs);
  CK_LAUNCH("tc_finish_kernel");
}

void gemm_tc_batch(spamm_ctx ctx, spamm_prec prec, const BatchDev& b) {
  switch (prec) {
    case SPAMM_PREC_BF16_SPLIT: launch_quads<SPAMM_PREC_BF16_SPLIT>(ctx, b); break;
    case SPAMM_PREC_BF16_SPLIT4: launch_quads<SPAMM_PREC_BF16_SPLIT4>(ctx, b); break;
    case SPAMM_PREC_FP16_SCALED: launch_quads<SPAMM_PREC_FP16_SCALED>(ctx, b); break;
    default: fail(SPAMM_E_INVALID_ARG, "not a tensor-core precision form");
  }
}

}  // namespace spamm
