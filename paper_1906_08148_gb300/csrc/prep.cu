// prep.cu -- the operand terms of the tensor-core forms: every (truncated)
// input leaf split into BF16 slices or per-leaf-scaled FP16 terms in the
// layout of tcforms.cuh, built once per multiply before the leaf products run.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "fbits.cuh"
#include "internal.cuh"
#include "ptx.cuh"
#include "slices.cuh"
#include "tcforms.cuh"

namespace spamm {

// Thread <-> element mapping shared by both kernels: one CTA of 512 threads
// per 64 x 64 tile of a leaf; a thread owns one 16-byte chunk of the K-major
// term tiles (8 consecutive k of one tile row), 8 FP64 elements.
// role 0 (A): tile row = leaf row t >> 3, k = leaf columns 8 (t & 7) ..
// role 1 (B): tile row = leaf column t & 63, k = leaf rows 8 (t >> 6) ..,
// so the lanes of a warp read consecutive doubles of each leaf row.
constexpr int kPrepThreads = 512;
struct ChunkMap {
  int row, c8;
  __device__ ChunkMap(int t, int role) {
    row = role == 0 ? t >> 3 : (t & 63);
    c8 = role == 0 ? (t & 7) : t >> 6;
  }
  // src: the tile's first element (GLOBAL: in global memory, else shared); ld: its row length
  template <bool GLOBAL>
  __device__ __forceinline__ void load(const unsigned long long* src, int ld, int role, unsigned long long (&v)[8]) const {
    if (role == 0) {
      // 8 consecutive doubles of one row: four 16-byte loads
      const ulonglong2* p = reinterpret_cast<const ulonglong2*>(src + row * ld + 8 * c8);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const ulonglong2 w = GLOBAL ? __ldg(p + e) : p[e];
        v[2 * e] = w.x;
        v[2 * e + 1] = w.y;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = GLOBAL ? __ldg(src + (8 * c8 + e) * ld + row) : src[(8 * c8 + e) * ld + row];
    }
  }
};

// Operand tiles of a leaf.  A 64 x 64 leaf is one tile; a 128 x 128 leaf is
// four, tile 2 r2 + kh holding rows 64 r2 .. of the leaf's row dimension for
// the operand (A: leaf rows; B: leaf columns) and k = 64 kh ..  (A: leaf
// columns; B: leaf rows), each split and scaled as a 64 x 64 leaf of its own,
// so the leaf-product kernel runs a 128-leaf product as two K-half steps
// over the four tiles of each operand.  Tile x of leaf m is at index
// m * tiles + x of the term and exponent arrays.
__device__ __forceinline__ const double* tile_src(const double* leaf, int bs, int role, int x) {
  if (bs == 64) return leaf;
  const int r2 = x >> 1, kh = x & 1;
  return role == 0 ? leaf + (int64_t)(64 * r2) * bs + 64 * kh : leaf + (int64_t)(64 * kh) * bs + 64 * r2;
}

// A CTA takes tiles blockIdx.x, blockIdx.x + gridDim.x, ...  A tile is measured, split
// and written with a barrier between, and while it was loaded into registers first
// the memory was idle half of the time.  STAGED (64 x 64 leaves: a tile is one run
// of memory): bulk copies bring the doubles into two buffers of shared memory, two
// tiles ahead.  The finished terms leave as one bulk copy.  Two CTAs per SM.
// Both operands, n = 65536 as 4 slices (32.8 GB moved) 7.8 -> 6.5 ms, n = 16384 as 3
// slices (4.2 GB) 0.87 -> 0.70.  The quarters of a 128 x 128 leaf are 64 runs of 512
// bytes each, for which the staged form is the slower one (n = 20000 FP16, 5.3 GB: 1.50
// ms, 1.17 with loads into registers).
// PAIR: both operands of a product share a launch, where it has few tiles per CTA
// (kPairTiles) and the latency of the first ones counts: 2 x 3536 tiles 84 -> 80 us, eight
// products with n = 1000 .. 5000 2.70 -> 2.67 ms.  With 2 x 37,624 tiles it is slower, 0.72 ms
// for 0.69 (both operands' tables are looked up for every tile).
struct PrepSide {
  const double* pool;
  const int64_t* slot;
  uint8_t* out;
  int32_t* expo;
  int64_t tiles;
};
struct PrepPair {
  PrepSide side[2];
  int role0;  // of side 0; side 1 (if it has tiles) is a B operand
};
constexpr uint32_t kTileBytes = 64 * 64 * sizeof(double);
template <bool PAIR>
struct TileStream {
  const PrepPair& P;
  int64_t total;  // tiles
  int bs;
  uint8_t* in;    // two tiles
  uint64_t* full;

  __device__ __forceinline__ bool second(int64_t m) const { return PAIR && m >= P.side[0].tiles; }
  __device__ __forceinline__ const double* source(int64_t m) const {
    const bool b = second(m);
    const double* pool = b ? P.side[1].pool : P.side[0].pool;
    const int64_t* slot = b ? P.side[1].slot : P.side[0].slot;
    if (b) m -= P.side[0].tiles;
    const int tiles = (bs / 64) * (bs / 64), shift = bs == 64 ? 0 : 2;
    const int64_t leaf = m >> shift;  // four tiles in a leaf of 128
    return tile_src(pool + __ldg(slot + leaf) * (int64_t)bs * bs, bs, b ? 1 : P.role0, (int)(m - leaf * tiles));
  }
  // STAGED, by one thread: tile m into buffer b (nothing past the last tile)
  __device__ __forceinline__ void fetch(int64_t m, int b) const {
    if (m >= total) return;
    const double* src = source(m);
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(&full[b], kTileBytes);
    bulk_g2s(in + (uint32_t)b * kTileBytes, src, kTileBytes, &full[b]);
  }
  // the last two fetches of a CTA that gave up have landed
  __device__ __forceinline__ void drain(int64_t m, uint32_t it) const {
    for (int i = 0; i < 2; ++i)
      if (m + (int64_t)i * gridDim.x < total) mbar_wait_bounded(&full[(it + i) & 1], ((it + i) >> 1) & 1u);
  }
};

// Form: measure(v) gives a thread's words for the line and tile maxima (the first
// combined by max, the second by or), shift the tile's scale exponent from them, split
// the thread's chunk of every term.
template <class Form, bool STAGED, bool PAIR>
__global__ void __launch_bounds__(kPrepThreads, STAGED || Form::kLines ? 2 : 3)
    prep_kernel(const __grid_constant__ PrepPair P, int bs, int* __restrict__ err) {
  constexpr uint32_t LEAF = Form::kLeaf;
  extern __shared__ __align__(128) uint8_t prep_smem[];
  uint8_t* stile = prep_smem + (STAGED ? 2 * kTileBytes : 0);  // the finished terms
  __shared__ __align__(8) uint64_t full[2];
  __shared__ uint32_t s_line[8][64];
  __shared__ uint2 s_warp[kPrepThreads / 32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const TileStream<PAIR> ts{P, P.side[0].tiles + (PAIR ? P.side[1].tiles : 0), bs, prep_smem, full};
  const ChunkMap cm0(t, P.role0);
  int64_t m = blockIdx.x;
  if (STAGED) {
    if (t == 0) {
      mbar_init(&full[0], 1);
      mbar_init(&full[1], 1);
      fence_mbar_init();
    }
    __syncthreads();
    if (t == 0) {
      ts.fetch(m, 0);
      ts.fetch(m + gridDim.x, 1);
    }
  }
  bool failed = false;
  uint32_t it = 0;
  for (; m < ts.total; m += gridDim.x, ++it) {
    const int b = (int)(it & 1);
    const bool side = ts.second(m);
    const int role = side ? 1 : P.role0;
    const ChunkMap cm = PAIR ? ChunkMap(t, role) : cm0;
    bool ok = true;
    unsigned long long v[8];
    if (STAGED) {
      ok = mbar_wait_bounded(&full[b], (it >> 1) & 1u);
      cm.load<false>(reinterpret_cast<const unsigned long long*>(prep_smem + (uint32_t)b * kTileBytes), 64, role, v);
    } else {
      cm.load<true>(reinterpret_cast<const unsigned long long*>(ts.source(m)), bs, role, v);
    }
    // the largest of this thread's line (A: row, B: column), then of the tile
    uint2 top = Form::measure(v);
    if (Form::kLines) {
      if (role == 0) {
        // a row's 8 chunks are held by 8 consecutive lanes
#pragma unroll
        for (int off = 1; off < 8; off <<= 1) top.x = max(top.x, __shfl_xor_sync(0xffffffffu, top.x, off));
      } else {
        // a column's 8 chunks are held by the threads t & 63 == column of 8 warp pairs
        s_line[t >> 6][t & 63] = top.x;
        __syncthreads();
#pragma unroll
        for (int h = 0; h < 8; ++h) top.x = max(top.x, s_line[h][t & 63]);
      }
    }
    const uint32_t line = top.x;
    const uint32_t wx = __reduce_max_sync(0xffffffffu, top.x), wy = __reduce_or_sync(0xffffffffu, top.y);
    if (lane == 0) s_warp[warp] = make_uint2(wx, wy);
    if (t == 0) bulk_wait_read();  // the last tile's terms have left stile
    failed = __syncthreads_or(!ok);
    if (failed) break;
    if (STAGED && t == 0) ts.fetch(m + 2 * (int64_t)gridDim.x, b);  // every thread holds its elements in registers
    const uint2 w = s_warp[lane & (kPrepThreads / 32 - 1)];
    const int f = Form::shift(__reduce_max_sync(0xffffffffu, w.x), __reduce_or_sync(0xffffffffu, w.y));
    const int64_t at = side ? m - P.side[0].tiles : m;
    if (t == 0) (side ? P.side[1].expo : P.side[0].expo)[at] = f;
    Form::split(v, (int)line, f, [&](int s, uint4 chunk) {
      *reinterpret_cast<uint4*>(stile + term_offset<Form::kParts>(Form::kTerms, s, cm.row, 8 * cm.c8)) = chunk;
    });
    fence_proxy_async_smem();
    __syncthreads();
    if (t == 0) bulk_s2g((side ? P.side[1].out : P.side[0].out) + at * (int64_t)LEAF, stile, LEAF);
  }
  if (t == 0) {
    bulk_wait_all();
    if (failed) {
      atomicOr(err, DEV_ERR_TIMEOUT);
      ts.drain(m, it);
    }
  }
}

// ------------------------------------------------------- BF16 slices (error-free split)
// Per tile: the largest biased exponent of every line (A: row, B: column) and
// of the tile, the tile's scale exponent f (stored in expo[m]), then every
// element's S digits (slices.cuh) as BF16 values d_s 2^(e - 8 - 9 s).
template <int PREC>
struct SliceForm {
  static constexpr int kTerms = FormCfg<PREC>::TERMS, kParts = FormCfg<PREC>::KPARTS;
  static constexpr uint32_t kLeaf = leaf_bytes<PREC>();
  static constexpr bool kLines = true;
  __device__ static __forceinline__ uint2 measure(const unsigned long long (&v)[8]) {
    int em = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) em = max(em, slice_biased_exp(v[e]));
    return make_uint2((uint32_t)em, 0u);
  }
  __device__ static __forceinline__ int shift(uint32_t emax, uint32_t) { return slice_leaf_shift((int)emax); }
  template <class Put>
  __device__ static __forceinline__ void split(const unsigned long long (&v)[8], int em, int f, Put put) {
    const int e = slice_line_exp(em, f);
    uint32_t term[kTerms][4];
    float unit[kTerms];
#pragma unroll
    for (int s = 0; s < kTerms; ++s) unit[s] = slice_unit(e - 8 - 9 * s);
#pragma unroll
    for (int q = 0; q < 8; q += 2) {
      int32_t d0[kTerms], d1[kTerms];
      slice_digits<kTerms>(v[q], em, d0);
      slice_digits<kTerms>(v[q + 1], em, d1);
#pragma unroll
      for (int s = 0; s < kTerms; ++s) term[s][q / 2] = slice_bf16_x2(d0[s], d1[s], unit[s]);
    }
#pragma unroll
    for (int s = 0; s < kTerms; ++s) put(s, make_uint4(term[s][0], term[s][1], term[s][2], term[s][3]));
  }
};

// ------------------------------------------------------------ FP16 terms
// Each element is rounded once to FP32 on its bits (fbits.cuh) with the
// per-tile scale 2^e folded in, max|a 2^e| in [2^14, 2^15), then split in
// FP32: h0 = f16(a 2^e), h1 = f16(a 2^e - h0) (the residual is exact in FP32).
// |x| of doubles orders like their bits without the sign, and the scale depends on the
// high word of the largest alone, but for an all-zero tile.
struct Fp16Form {
  static constexpr int PREC = SPAMM_PREC_FP16_SCALED;
  static constexpr int kTerms = FormCfg<PREC>::TERMS, kParts = FormCfg<PREC>::KPARTS;
  static constexpr uint32_t kLeaf = leaf_bytes<PREC>();
  static constexpr bool kLines = false;
  __device__ static __forceinline__ uint2 measure(const unsigned long long (&v)[8]) {
    uint32_t mh = 0, any = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      mh = max(mh, (uint32_t)(v[e] >> 32) & 0x7FFFFFFFu);
      any |= (uint32_t)v[e];
    }
    return make_uint2(mh, any);
  }
  __device__ static __forceinline__ int shift(uint32_t mh, uint32_t any) {
    return fp16_leaf_shift(((uint64_t)mh << 32) | (any != 0));
  }
  template <class Put>
  __device__ static __forceinline__ void split(const unsigned long long (&v)[8], int, int shift, Put put) {
    uint32_t term[kTerms][4];
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
      float2 a = make_float2(__uint_as_float(fbits_from_double_rn(v[e], shift)),
                             __uint_as_float(fbits_from_double_rn(v[e + 1], shift)));
#pragma unroll
      for (int s = 0; s < kTerms; ++s) {  // two at a time: one packed conversion each way
        const __half2 h = __float22half2_rn(a);
        term[s][e / 2] = *reinterpret_cast<const uint32_t*>(&h);
        const float2 g = __half22float2(h);
        a.x -= g.x;
        a.y -= g.y;
      }
    }
#pragma unroll
    for (int s = 0; s < kTerms; ++s) put(s, make_uint4(term[s][0], term[s][1], term[s][2], term[s][3]));
  }
};

static uint32_t form_leaf_bytes(spamm_prec prec) {
  switch (prec) {
    case SPAMM_PREC_BF16_SPLIT: return leaf_bytes<SPAMM_PREC_BF16_SPLIT>();
    case SPAMM_PREC_BF16_SPLIT4: return leaf_bytes<SPAMM_PREC_BF16_SPLIT4>();
    default: return leaf_bytes<SPAMM_PREC_FP16_SCALED>();
  }
}

constexpr int64_t kPairTiles = 32;
void prep_terms(spamm_ctx ctx, spamm_prec prec, const PrepReq* req, int k) {
  const int bs = req[0].M->bs;
  if (bs != 64 && bs != 128) fail(SPAMM_E_UNSUPPORTED, "tensor-core precision forms are built for bs = 64 and 128");
  const int64_t tiles0 = req[0].M->nleaves * tc_tiles_per_leaf(bs);
  if (k == 2 && tiles0 + req[1].M->nleaves * tc_tiles_per_leaf(bs) > kPairTiles * 2 * ctx->num_sms) {
    prep_terms(ctx, prec, req, 1);
    prep_terms(ctx, prec, req + 1, 1);
    return;
  }
  PrepPair pair{};
  int64_t ntiles = 0;
  for (int i = 0; i < k; ++i) {
    const PrepReq& r = req[i];
    const int64_t n = r.M->nleaves * tc_tiles_per_leaf(bs);
    *r.terms = alloc_n<uint8_t>(ctx, n * (int64_t)form_leaf_bytes(prec));
    *r.expo = alloc_n<int32_t>(ctx, n);
    pair.side[i] = {P<double>(r.M->pool), P<int64_t>(r.M->slot), P<uint8_t>(*r.terms), P<int32_t>(*r.expo), n};
    ntiles += n;
  }
  pair.role0 = req[0].role;
  if (ntiles == 0) return;
  // the blocks of a launch: staged, two fit an SM; from registers three in the FP16 form, for
  // which this was measured, and two in the BF16 forms, whose third block per SM waits (their
  // terms of 128-leaves, 2 x 8220 leaves: 1019 -> 846 us with 3 slices, 1203 -> 1032 with 4, against
  // 256 threads per tile)
  const int64_t cap = (int64_t)ctx->num_sms * (bs == 64 ? 2 : 3);
  const unsigned grid = (unsigned)(ntiles < cap ? ntiles : cap);
  const bool staged = bs == 64;
  const int smem = (int)((staged ? 2 * kTileBytes : 0) + form_leaf_bytes(prec));
  auto launch = [&](auto kern) {
    CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    kern<<<grid, kPrepThreads, smem, ctx->stream>>>(pair, bs, ctx->d_err);
    CK_LAUNCH("prep_kernel");
  };
  auto form = [&](auto f) {
    using Form = decltype(f);
    if (staged)
      k == 2 ? launch(prep_kernel<Form, true, true>) : launch(prep_kernel<Form, true, false>);
    else
      k == 2 ? launch(prep_kernel<Form, false, true>) : launch(prep_kernel<Form, false, false>);
  };
  if (prec == SPAMM_PREC_BF16_SPLIT)
    form(SliceForm<SPAMM_PREC_BF16_SPLIT>());
  else if (prec == SPAMM_PREC_BF16_SPLIT4)
    form(SliceForm<SPAMM_PREC_BF16_SPLIT4>());
  else
    form(Fp16Form());
}

}  // namespace spamm
