// prep.cu -- the operand terms of the tensor-core forms: every (truncated)
// input leaf split into BF16 slices or per-leaf-scaled FP16 terms in the
// layout of tcforms.cuh, built once per multiply before the leaf products run.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "fbits.cuh"
#include "internal.cuh"
#include "slices.cuh"
#include "tcforms.cuh"

namespace spamm {

// Thread <-> element mapping shared by both kernels: one CTA of 512 threads
// per 64 x 64 tile of a leaf; a thread owns one 16-byte chunk of the K-major
// term tiles (8 consecutive k of one tile row) and loads its 8 FP64 elements
// first.  A tile is loaded, measured (line and tile maxima), split and written with
// a barrier between, so other CTAs have to fill the gaps: one chunk per thread keeps
// the registers at 64, 1024 threads per SM, where two chunks in 256 threads (124
// registers, 512 threads) left the memory idle half of the time.  Both operands of the
// n = 16384 lattice as 3 slices (4.2 GB moved) 1.10 -> 0.87 ms, of n = 65536 as 4 slices
// (32.8 GB) 9.5 -> 7.8 ms, with the 32-bit digits of slices.cuh; FP16, whose packed
// conversions made up for its second barrier, unchanged.
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
  // src: the tile's first element; ld: the leaf's row length
  __device__ void load(const unsigned long long* src, int ld, int role, unsigned long long (&v)[8]) const {
    if (role == 0) {
      // 8 consecutive doubles of one row: four 16-byte loads
      const ulonglong2* p = reinterpret_cast<const ulonglong2*>(src + row * ld + 8 * c8);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const ulonglong2 w = __ldg(p + e);
        v[2 * e] = w.x;
        v[2 * e + 1] = w.y;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = __ldg(src + (8 * c8 + e) * ld + row);
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

// ------------------------------------------------------- BF16 slices (error-free split)
// Per leaf: the largest biased exponent of every line (A: row, B: column) and
// of the leaf, the leaf's scale exponent f (stored in expo[m]), then every
// element's S digits (slices.cuh) as BF16 values d_s 2^(e - 8 - 9 s).  The
// slices are assembled in shared memory and leave as one contiguous block.
template <int S, int KPARTS>
__global__ void __launch_bounds__(kPrepThreads, 2)
    prep_slices_kernel(const double* __restrict__ pool, const int64_t* __restrict__ slot, int64_t nleaves, int bs,
                       int role, uint8_t* __restrict__ out, int32_t* __restrict__ expo) {
  constexpr uint32_t LEAF = (uint32_t)S * kTerm;
  __shared__ uint4 stile[LEAF / 16];
  __shared__ int s_line[8][64];  // role 1: per-column maxima of each eighth of the leaf rows
  __shared__ int s_warp[kPrepThreads / 32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const ChunkMap cm(t, role);
  const int tiles = (bs / 64) * (bs / 64);
  for (int64_t m = blockIdx.x; m < nleaves * tiles; m += gridDim.x) {
    const int64_t leaf = m / tiles;
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(
        tile_src(pool + slot[leaf] * (int64_t)bs * bs, bs, role, (int)(m - leaf * tiles)));
    unsigned long long v[8];
    cm.load(src, bs, role, v);
    // largest biased exponent of this thread's line
    int em = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) em = max(em, slice_biased_exp(v[e]));
    if (role == 0) {
      // a row's 8 chunks are held by 8 consecutive lanes
#pragma unroll
      for (int off = 1; off < 8; off <<= 1) em = max(em, __shfl_xor_sync(0xffffffffu, em, off));
    } else {
      // a column's 8 chunks are held by the threads t & 63 == column of 8 warp pairs
      s_line[t >> 6][t & 63] = em;
      __syncthreads();
#pragma unroll
      for (int h = 0; h < 8; ++h) em = max(em, s_line[h][t & 63]);
    }
    const int lm = __reduce_max_sync(0xffffffffu, em);
    if (lane == 0) s_warp[warp] = lm;
    __syncthreads();
    const int leaf_max = __reduce_max_sync(0xffffffffu, s_warp[lane & (kPrepThreads / 32 - 1)]);
    const int f = slice_leaf_shift(leaf_max);
    if (t == 0) expo[m] = f;
    const int e = slice_line_exp(em, f);
    float unit[S];
#pragma unroll
    for (int s = 0; s < S; ++s) unit[s] = slice_unit(e - 8 - 9 * s);
    uint32_t term[S][4];
#pragma unroll
    for (int q = 0; q < 8; q += 2) {
      int32_t d0[S], d1[S];
      slice_digits<S>(v[q], em, d0);
      slice_digits<S>(v[q + 1], em, d1);
#pragma unroll
      for (int s = 0; s < S; ++s) term[s][q / 2] = slice_bf16_x2(d0[s], d1[s], unit[s]);
    }
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const uint32_t off = term_offset<KPARTS>(S, s, cm.row, 8 * cm.c8);
      stile[off >> 4] = make_uint4(term[s][0], term[s][1], term[s][2], term[s][3]);
    }
    __syncthreads();
    // the leaf's slices leave in order: consecutive threads, consecutive 16-byte chunks
    uint4* d4 = reinterpret_cast<uint4*>(out + m * (int64_t)LEAF);
#pragma unroll
    for (int i = 0; i < (int)(LEAF / 16) / kPrepThreads; ++i) d4[t + i * kPrepThreads] = stile[t + i * kPrepThreads];
    __syncthreads();  // stile, s_line and s_warp are reused by the next leaf
  }
}

// ------------------------------------------------------------ FP16 terms
// Each element is rounded once to FP32 on its bits (fbits.cuh) with the
// per-leaf scale 2^e folded in, max|a 2^e| in [2^14, 2^15), then split in
// FP32: h0 = f16(a 2^e), h1 = f16(a 2^e - h0) (the residual is exact in FP32).
__global__ void __launch_bounds__(kPrepThreads, 2)
    prep_fp16_kernel(const double* __restrict__ pool, const int64_t* __restrict__ slot, int64_t nleaves, int bs, int role,
                     uint8_t* __restrict__ out, int32_t* __restrict__ expo) {
  constexpr int TERMS = FormCfg<SPAMM_PREC_FP16_SCALED>::TERMS;
  constexpr uint32_t LEAF = leaf_bytes<SPAMM_PREC_FP16_SCALED>();
  __shared__ uint2 smax[kPrepThreads / 32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const ChunkMap cm(t, role);
  const int tiles = (bs / 64) * (bs / 64);
  for (int64_t m = blockIdx.x; m < nleaves * tiles; m += gridDim.x) {
    const int64_t leaf = m / tiles;
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(
        tile_src(pool + slot[leaf] * (int64_t)bs * bs, bs, role, (int)(m - leaf * tiles)));
    unsigned long long v[8];
    cm.load(src, bs, role, v);
    // largest |a| of the tile: |x| of doubles orders like their bits without the sign,
    // and the scale depends on the high word of the largest alone, but for an all-zero tile
    uint32_t mh = 0, any = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      mh = max(mh, (uint32_t)(v[e] >> 32) & 0x7FFFFFFFu);
      any |= (uint32_t)v[e];
    }
    mh = __reduce_max_sync(0xffffffffu, mh);
    any = __any_sync(0xffffffffu, any != 0);
    if (lane == 0) smax[warp] = make_uint2(mh, any);
    __syncthreads();
    const uint2 w = smax[lane & (kPrepThreads / 32 - 1)];
    mh = __reduce_max_sync(0xffffffffu, w.x);
    any = __any_sync(0xffffffffu, w.y != 0);
    const unsigned long long mx = ((unsigned long long)mh << 32) | any;
    const int shift = fp16_leaf_shift(mx);
    if (t == 0) expo[m] = shift;
    uint8_t* dst = out + m * (int64_t)LEAF;
    uint32_t term[TERMS][4];
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
      float2 a = make_float2(__uint_as_float(fbits_from_double_rn(v[e], shift)),
                             __uint_as_float(fbits_from_double_rn(v[e + 1], shift)));
#pragma unroll
      for (int s = 0; s < TERMS; ++s) {  // two at a time: one packed conversion each way
        const __half2 h = __float22half2_rn(a);
        term[s][e / 2] = *reinterpret_cast<const uint32_t*>(&h);
        const float2 g = __half22float2(h);
        a.x -= g.x;
        a.y -= g.y;
      }
    }
#pragma unroll
    for (int s = 0; s < TERMS; ++s)
      *reinterpret_cast<uint4*>(dst + term_offset<FormCfg<SPAMM_PREC_FP16_SCALED>::KPARTS>(TERMS, s, cm.row, 8 * cm.c8)) =
          make_uint4(term[s][0], term[s][1], term[s][2], term[s][3]);
    __syncthreads();  // smax is reused by the next leaf
  }
}

static uint32_t form_leaf_bytes(spamm_prec prec) {
  switch (prec) {
    case SPAMM_PREC_BF16_SPLIT: return leaf_bytes<SPAMM_PREC_BF16_SPLIT>();
    case SPAMM_PREC_BF16_SPLIT4: return leaf_bytes<SPAMM_PREC_BF16_SPLIT4>();
    default: return leaf_bytes<SPAMM_PREC_FP16_SCALED>();
  }
}

void prep_terms(spamm_mat M, spamm_prec prec, int role, BufP* terms, BufP* expo, spamm_ctx on) {
  spamm_ctx ctx = on ? on : M->ctx;
  const int bs = M->bs;
  if (bs != 64 && bs != 128) fail(SPAMM_E_UNSUPPORTED, "tensor-core precision forms are built for bs = 64 and 128");
  const int64_t ntiles = M->nleaves * tc_tiles_per_leaf(bs), cap = (int64_t)ctx->num_sms * 8;
  const unsigned grid = (unsigned)(ntiles < cap ? (ntiles > 0 ? ntiles : 1) : cap);
  *terms = alloc_n<uint8_t>(ctx, ntiles * (int64_t)form_leaf_bytes(prec));
  *expo = alloc_n<int32_t>(ctx, ntiles);
  if (M->nleaves == 0) return;
  const double* pool = P<double>(M->pool);
  const int64_t* slot = P<int64_t>(M->slot);
  if (prec == SPAMM_PREC_BF16_SPLIT) {
    prep_slices_kernel<3, FormCfg<SPAMM_PREC_BF16_SPLIT>::KPARTS><<<grid, kPrepThreads, 0, ctx->stream>>>(pool, slot, M->nleaves, bs, role,
                                                                P<uint8_t>(*terms), P<int32_t>(*expo));
    CK_LAUNCH("prep_slices_kernel<3>");
  } else if (prec == SPAMM_PREC_BF16_SPLIT4) {
    prep_slices_kernel<4, FormCfg<SPAMM_PREC_BF16_SPLIT4>::KPARTS><<<grid, kPrepThreads, 0, ctx->stream>>>(pool, slot, M->nleaves, bs, role,
                                                               P<uint8_t>(*terms), P<int32_t>(*expo));
    CK_LAUNCH("prep_slices_kernel<4>");
  } else {
    prep_fp16_kernel<<<grid, kPrepThreads, 0, ctx->stream>>>(pool, slot, M->nleaves, bs, role, P<uint8_t>(*terms),
                                                    P<int32_t>(*expo));
    CK_LAUNCH("prep_fp16_kernel");
  }
}

}  // namespace spamm
