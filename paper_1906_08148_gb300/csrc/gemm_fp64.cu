// gemm_fp64.cu -- kernel (c), FP64 form.
//
// C_ij = sum over the kept k (ascending) of A_ik B_kj (Algorithm 1, "C = AB"
// at the lowest level, run batched over the task list as Section 4.4
// describes).  A work unit is a TILE x TILE sub-tile of an output leaf.  The units
// of every plan in a batch form one work list; persistent CTAs claim them from an
// atomic counter (the large leaves in order of decreasing kept-product count, so
// the last claims are short).  Every output element is computed by one CTA, so
// there are no atomics on C and the k order is fixed: results do not depend on the
// schedule, the tile or the batch.  The leaf norms (kernel (d)) are kernel (a) on
// the finished leaves, in one launch for the batch (out_sqnorm_kernel), so they do not
// depend on the tile either (one FMA per element against bs per element and product here).
//
// Bound by the FP64 pipe (two FMAs per clock and SM): a 64 x 64 x 64 product takes an
// SM 63 us, so what is lost is lost at the end, when some SMs still work on their
// last units.  Tiles are 64 x 64 (32 x 32 leaves whole) where a launch holds many units
// per SM, and a quarter of that where it does not (launch_fp64): 1744 leaves of 32 x 32
// (26,440 products, 1.38 ms at the pipe's rate) 1.54 -> 1.44 ms; 100 leaves (932 products)
// 94 -> 78 us.
//
// Operand panels are staged in shared memory by 1-D TMA bulk copies issued by one
// warp, double-buffered on mbarriers; the product is register-tiled DFMA (FP64 has
// no tcgen05 kind; DFMA measures faster than the FP64 mma.sync path on this part).
// A 32 x 32 leaf is staged whole (one copy per operand); other tiles in K-panels of
// KP = 32 (A's panel as row segments of 256 bytes, B's as 32 row segments, one copy
// where they are contiguous), so three CTAs of 64 x 64 tiles share an SM (64 KB of
// shared memory each).
#include "internal.cuh"
#include "ptx.cuh"

namespace spamm {

constexpr int kGemmThreads = 256;
// sort key of an output leaf: kUnitKeyMax - its kept-product count (at most
// 2^16, the leaf grid side), so an ascending stable sort puts the longest first
constexpr int kUnitKeyBits = 18;
constexpr int64_t kUnitKeyMax = (int64_t)1 << 17;

template <int BS, int KP, int TILE>
__global__ void __launch_bounds__(kGemmThreads)
    gemm_fp64_kernel(BatchDev batch, int nq, unsigned long long* __restrict__ work, int* __restrict__ err) {
  constexpr int LEAF = BS * BS;
  constexpr int NP = BS / KP;                    // K-panels per leaf product
  constexpr int NQ = (BS / TILE) * (BS / TILE);  // work units (sub-tiles) per output leaf
  constexpr int PANEL = TILE * KP;               // doubles in one A panel (and one B panel)
  constexpr uint32_t PANEL_BYTES = PANEL * sizeof(double);
  constexpr int TM = TILE / 16;  // per-thread tile TM x TM: rows tr + 16 i, cols tc + 16 j
  static_assert(BS % TILE == 0 && BS % KP == 0 && TILE % 16 == 0 && KP % 2 == 0, "tile shape");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  double* sA[2] = {reinterpret_cast<double*>(smem_raw), reinterpret_cast<double*>(smem_raw) + 2 * PANEL};
  double* sB[2] = {reinterpret_cast<double*>(smem_raw) + PANEL, reinterpret_cast<double*>(smem_raw) + 3 * PANEL};
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ int64_t s_u;
  __shared__ int s_abort;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tr = tid >> 4, tc = tid & 15;
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    fence_mbar_init();
    s_abort = 0;
  }
  __syncthreads();
  uint32_t phase[2] = {0u, 0u};
  uint32_t inflight = 0;  // bit s: stage s has a copy that nobody waited for
  const int64_t nunits = batch.nunits / nq * NQ;  // the batch counts nq units per leaf

  for (;;) {
    if (tid == 0) s_u = (int64_t)atomicAdd(work, 1ull);
    __syncthreads();
    const int64_t u = s_u;
    if (u >= nunits || s_abort) break;
    const int64_t leaf = u / NQ;
    const int sub = (int)(u - leaf * NQ);
    const int r = plan_of(batch.ubegin, batch.nplans, leaf * nq);
    const PlanDev& pl = batch.plans[r];
    const int64_t li = leaf - batch.ubegin[r] / nq;  // leaf position in claiming order
    const int64_t g = pl.uorder ? pl.uorder[li] : li;
    const int64_t r0 = (int64_t)(sub / (BS / TILE)) * TILE, c0 = (int64_t)(sub % (BS / TILE)) * TILE;
    const int64_t q0 = pl.gstart[g], q1 = pl.gstart[g + 1];
    // step t: task q0 + t / NP, K-panel t % NP; issued by the 32 lanes of
    // warp 0 (lane 0 arms the barrier first)
    auto issue = [&](int64_t t, int s) {
      const int64_t q = q0 + t / NP;
      const int p = (int)(t % NP);
      const double* a = pl.poolA + pl.slotA[pl.ta[q]] * LEAF + r0 * BS + p * KP;
      const double* b = pl.poolB + pl.slotB[pl.tb[q]] * LEAF + (int64_t)p * KP * BS + c0;
      fence_proxy_async_smem();
      if (lane == 0) mbar_arrive_expect_tx(&bar[s], 2 * PANEL_BYTES);
      __syncwarp();
      if constexpr (NP == 1 && TILE == BS) {
        if (lane == 0) bulk_g2s(sA[s], a, PANEL_BYTES, &bar[s]);
      } else {
        for (int row = lane; row < TILE; row += 32)
          bulk_g2s(sA[s] + row * KP, a + (int64_t)row * BS, KP * sizeof(double), &bar[s]);
      }
      if constexpr (TILE == BS) {
        if (lane == 0) bulk_g2s(sB[s], b, PANEL_BYTES, &bar[s]);
      } else {
        for (int row = lane; row < KP; row += 32)
          bulk_g2s(sB[s] + row * TILE, b + (int64_t)row * BS, TILE * sizeof(double), &bar[s]);
      }
    };
    double acc[TM][TM];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TM; ++j) acc[i][j] = 0.0;
    const int64_t nsteps = (q1 - q0) * NP;
    if (warp == 0 && nsteps > 0) issue(0, 0);
    inflight |= 1u;
    for (int64_t t = 0; t < nsteps; ++t) {
      const int s = (int)(t & 1);
      if (t + 1 < nsteps) {
        if (warp == 0) issue(t + 1, s ^ 1);
        inflight |= 1u << (s ^ 1);
      }
      if (!mbar_wait_bounded(&bar[s], phase[s])) {
        atomicOr(err, DEV_ERR_TIMEOUT);
        s_abort = 1;
      } else {
        phase[s] ^= 1u;
        inflight &= ~(1u << s);
      }
      __syncthreads();
      if (s_abort) break;
      const double* As = sA[s];
      const double* Bs = sB[s];
#pragma unroll 4
      for (int kk = 0; kk < KP; ++kk) {
        double a[TM], b[TM];
#pragma unroll
        for (int i = 0; i < TM; ++i) a[i] = As[(tr + 16 * i) * KP + kk];
#pragma unroll
        for (int j = 0; j < TM; ++j) b[j] = Bs[kk * TILE + tc + 16 * j];
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TM; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
      }
      __syncthreads();
    }
    if (nsteps <= 0) inflight &= ~1u;
    if (s_abort) break;
    double* C = pl.cpool + g * LEAF + r0 * BS + c0;
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TM; ++j) C[(tr + 16 * i) * BS + tc + 16 * j] = acc[i][j];
  }
  // leave no bulk copy in flight into this CTA's shared memory
  if (tid == 0) {
    for (int s = 0; s < 2; ++s)
      if (inflight & (1u << s)) mbar_wait_bounded(&bar[s], phase[s]);
  }
  __syncthreads();
}

template <int BS, int TILE>
static void launch_tile(spamm_ctx ctx, const BatchDev& b) {
  constexpr int KP = 32;
  auto kern = gemm_fp64_kernel<BS, KP, TILE>;
  const size_t smem = 4 * (size_t)TILE * KP * sizeof(double);
  // looked up once per context (two kernels per leaf size)
  constexpr int id = (BS == 32 ? 0 : BS == 64 ? 2 : 4) + (TILE == (BS <= 64 ? BS : 64) ? 1 : 0);
  int& per_sm = ctx->fp64_ctas[BS == 256 ? id + 2 : id];
  if (per_sm == 0) {
    CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int n = 0;
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kGemmThreads, smem));
    per_sm = n < 1 ? 1 : n;
  }
  const int sms = ctx->gemm_sm_limit > 0 ? ctx->gemm_sm_limit : ctx->num_sms;
  const int nq = fp64_units_per_leaf(BS);
  const int64_t units = b.nunits / nq * ((BS / TILE) * (BS / TILE));
  int64_t grid = (int64_t)sms * per_sm;
  if (grid > units) grid = units;
  kern<<<(unsigned)grid, kGemmThreads, smem, ctx->stream>>>(b, nq, b.work, ctx->d_err);
  CK_LAUNCH("gemm_fp64_kernel");
}

// 64 x 64 tiles (whole 32 x 32 leaves) for at least kUnitsPerSm of them per SM, else
// quarters: with u equal units per SM the last ones leave SMs idle for about 1 / u of
// the time, and a tile of a quarter reads its operands twice as often from L2, which
// costs a per cent or two of the FP64 time (1271 leaves of 128 x 128, 33 tiles of 64 x 64
// per SM: 20.5 ms, 99.3 % of the pipe).
constexpr int64_t kUnitsPerSm = 24;
template <int BS>
static void launch_fp64(spamm_ctx ctx, const BatchDev& b) {
  constexpr int TILE = BS <= 64 ? BS : 64;
  const int sms = ctx->gemm_sm_limit > 0 ? ctx->gemm_sm_limit : ctx->num_sms;
  if (b.nunits >= kUnitsPerSm * sms)
    launch_tile<BS, TILE>(ctx, b);
  else
    launch_tile<BS, TILE / 2>(ctx, b);
}

int fp64_units_per_leaf(int bs) { return bs <= 64 ? 1 : (bs / 64) * (bs / 64); }

__global__ void unit_order_keys_kernel(const int64_t* __restrict__ gstart, int64_t ng, uint64_t* __restrict__ keys,
                                       int64_t* __restrict__ vals) {
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < ng; g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = gstart[g + 1] - gstart[g];
    keys[g] = (uint64_t)(kUnitKeyMax - (c < kUnitKeyMax ? c : kUnitKeyMax));
    vals[g] = g;
  }
}

BufP unit_order_longest(spamm_ctx ctx, const int64_t* start, int64_t n) {
  if (n <= 1) return BufP();
  BufP keys = alloc_n<uint64_t>(ctx, n), vals = alloc_n<int64_t>(ctx, n);
  int64_t grid = (n + 255) / 256;
  if (grid > 4 * (int64_t)ctx->num_sms) grid = 4 * (int64_t)ctx->num_sms;
  unit_order_keys_kernel<<<(unsigned)grid, 256, 0, ctx->stream>>>(start, n, P<uint64_t>(keys), P<int64_t>(vals));
  CK_LAUNCH("unit_order_keys_kernel");
  radix_sort_pairs(ctx, P<uint64_t>(keys), P<int64_t>(vals), n, kUnitKeyBits);
  return vals;
}

void gemm_fp64_batch(spamm_ctx ctx, int bs, const BatchDev& b) {
  if (b.nunits == 0) return;
  switch (bs) {
    case 32: launch_fp64<32>(ctx, b); break;
    case 64: launch_fp64<64>(ctx, b); break;
    case 128: launch_fp64<128>(ctx, b); break;
    case 256: launch_fp64<256>(ctx, b); break;
    default: fail(SPAMM_E_UNSUPPORTED, "FP64 leaf products are built for bs = 32, 64, 128 and 256");
  }
}

}  // namespace spamm
