// store.cu -- the device quadtree store: leaf norms (kernel a), parent norms,
// input truncation, builders from dense / blocks / COO / generator, exports
// and the error walk.
//
// Layout in HBM: a matrix is a payload pool of bs*bs row-major FP64 leaves
// plus, for every quadtree level t = 0..L, the nodes of that level sorted by
// the Morton code of their (row, col) position, their squared Frobenius norms
// and (t < L) an int4 of child node indices (-1 = null child).  Leaf m's
// payload is at pool + slot[m]*bs*bs, so truncated views share the pool.
#include <cstdio>

#include "../../synth/decaygen.h"
#include "internal.cuh"
#include "leafpass.cuh"

namespace spamm {

constexpr int kThreads = 256;

void fill_iota_i64(spamm_ctx ctx, int64_t* p, int64_t n);
void and_u8(spamm_ctx ctx, uint8_t* a, const uint8_t* b, int64_t n);

static unsigned grid_for(spamm_ctx ctx, int64_t items, int per_block, int max_per_sm = 32) {
  int64_t g = (items + per_block - 1) / per_block;
  int64_t cap = (int64_t)ctx->num_sms * max_per_sm;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (unsigned)g;
}

// ------------------------------------------------------------------------
// Kernel (a): squared Frobenius norm of each leaf (Section 2, Section 4.2:
// every matrix stores its squared norm).  One warp per leaf; lane l reads
// the 16-byte pairs l, l+32, ... (coalesced 512-byte rows), squares are
// accumulated with explicit FMAs in that fixed order and the 32 partial sums
// are combined by a butterfly, so every build path gives identical bits.
// The FMA is the only FP64 instruction per element: this part issues two FP64
// operations per clock per SM, so the non-zero and finiteness checks work on
// the bit patterns in the integer pipe (any bit besides the sign set: non-zero;
// exponent field all ones: Inf or NaN).  U pairs per lane are read before the
// first is used (bs^2 / 2 is a multiple of 512 pairs for every leaf size, so U
// is at most 16): a lane that reads one pair at a time waits for memory 64 times
// in a 64 x 64 leaf.
template <int U, class Get>
__device__ __forceinline__ void warp_leaf_sumsq(Get get, int bs, int lane, double* s_out, bool* nz_out, bool* bad_out) {
  const int pairs = bs * bs / 2;
  double s = 0.0;
  uint32_t bits = 0, emax = 0;
  for (int i = lane; i < pairs; i += 32 * U) {
    double2 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = get(i + 32 * u);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      s = __fma_rn(v[u].x, v[u].x, s);
      s = __fma_rn(v[u].y, v[u].y, s);
      const uint32_t hx = (uint32_t)__double2hiint(v[u].x), hy = (uint32_t)__double2hiint(v[u].y);
      bits |= (uint32_t)__double2loint(v[u].x) | (uint32_t)__double2loint(v[u].y) | ((hx | hy) & 0x7fffffffu);
      emax = max(emax, max(hx & 0x7ff00000u, hy & 0x7ff00000u));
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  *s_out = s;
  *nz_out = __any_sync(0xffffffffu, bits != 0);
  *bad_out = __any_sync(0xffffffffu, emax == 0x7ff00000u);
}

// Block b takes leaves [8 b, 8 b + 8), one per warp (larger grids stride by whole
// blocks): with 64 leaves per block a few thousand leaves kept only a third of
// the SMs busy.
constexpr int64_t kNormLeavesPerBlock = 8;
__global__ void leaf_sqnorm_kernel(const double* __restrict__ pool, const int64_t* __restrict__ slot, int64_t m,
                                   int bs, double* __restrict__ sq, uint8_t* __restrict__ nonzero, int check_finite,
                                   int* err) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwb = blockDim.x >> 5;
  const int64_t e = (int64_t)bs * bs;
  for (int64_t q = (int64_t)blockIdx.x * kNormLeavesPerBlock + warp; q < m; q += (int64_t)gridDim.x * nwb) {
    const double2* src = reinterpret_cast<const double2*>(pool + (slot ? slot[q] : q) * e);
    double s;
    bool nz, bad;
    warp_leaf_sumsq<8>([&](int i) { return __ldg(src + i); }, bs, lane, &s, &nz, &bad);
    if (lane == 0) {
      sq[q] = s;
      if (nonzero) nonzero[q] = nz;
      if (bad && check_finite) atomicOr(err, DEV_ERR_NONFINITE);
    }
  }
}

void leaf_sqnorms(spamm_ctx ctx, const double* pool, const int64_t* slot, int64_t nleaves, int bs, double* sq,
                  uint8_t* nonzero, int check_finite) {
  if (nleaves <= 0) return;
  const int64_t nblk = (nleaves + kNormLeavesPerBlock - 1) / kNormLeavesPerBlock;
  leaf_sqnorm_kernel<<<(unsigned)(nblk < (1ll << 30) ? nblk : (1ll << 30)), kThreads, 0, ctx->stream>>>(
      pool, slot, nleaves, bs, sq, nonzero, check_finite, ctx->d_err);
  CK_LAUNCH("leaf_sqnorm_kernel");
}

// Kernel (a) on the outputs of a batch of FP64 products, and their payload slots: one
// launch for all of them, bound by the FP64 pipe.  A leaf's bs^2 / 32 additions per lane
// follow one another at 64 cycles each, which takes 1, 4, 17 or 68 us for leaves of 32, 64,
// 128 or 256, however few there are (a launch per output: eight products of one 256-leaf
// each 1264 us, in one launch 407).  So a lane's next eight pairs are on their way while
// it adds the eight before (every leaf has a multiple of 64 x 8 pairs), and a block is one
// warp, which gives each its own quarter of a pipe: 40 leaves of 256 95 us, 140 with eight
// warps per block; 60,000 leaves of 32 156 us, 158 with eight.
__global__ void __launch_bounds__(32) out_sqnorm_kernel(const __grid_constant__ OutBatch out, int bs) {
  constexpr int U = 8;
  const int lane = threadIdx.x;
  const int pairs = bs * bs / 2;
  for (int64_t u = blockIdx.x; u < out.total; u += gridDim.x) {
    const int r = out.n > 1 ? plan_of(out.first, out.n, u) : 0;
    const OutLeaves C = out.n > 1 ? out.tab[r] : out.only;
    const int64_t q = out.n > 1 ? u - out.first[r] : u;
    const double2* src = reinterpret_cast<const double2*>(C.pool + q * ((int64_t)bs * bs)) + lane;
    double2 a[U], b[U];
    double s = 0.0;
    auto read = [&](double2(&v)[U], int i) {
#pragma unroll
      for (int k = 0; k < U; ++k) v[k] = __ldg(src + i + 32 * k);
    };
    auto add = [&](const double2(&v)[U]) {
#pragma unroll
      for (int k = 0; k < U; ++k) {
        s = __fma_rn(v[k].x, v[k].x, s);
        s = __fma_rn(v[k].y, v[k].y, s);
      }
    };
    read(a, 0);
    for (int i = 0; i < pairs; i += 64 * U) {
      read(b, i + 32 * U);
      add(a);
      if (i + 64 * U < pairs) read(a, i + 64 * U);
      add(b);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) {
      C.sq[q] = s;
      C.slot[q] = q;
    }
  }
}

void out_sqnorms(spamm_ctx ctx, const OutBatch& out, int bs) {
  if (out.total <= 0) return;
  out_sqnorm_kernel<<<(unsigned)(out.total < (1ll << 30) ? out.total : (1ll << 30)), 32, 0, ctx->stream>>>(out, bs);
  CK_LAUNCH("out_sqnorm_kernel");
}

spamm_mat new_mat(spamm_ctx ctx, int64_t n, int bs) {
  spamm_mat m = new spamm_mat_s();
  m->ctx = ctx;
  m->n = n;
  m->bs = bs;
  m->L = levels_for(n, bs);
  m->lv.resize(m->L + 1);
  return m;
}

void set_leaves_compacted(spamm_mat m, int64_t ncand, const uint32_t* code, const double* sq, const int64_t* slot,
                          const uint8_t* keep) {
  if (ncand <= 0) {
    m->nleaves = 0;
    return;
  }
  TreeReq r{m, ncand, code, sq, slot, keep, 0.0};
  tree_from_candidates(m->ctx, &r, 1, true);
}

void alloc_norms(spamm_mat m) {
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const int64_t n = m->lv[m->L].count;
  size_t bytes = up(n * sizeof(int64_t));
  for (const Level& lv : m->lv) bytes += up(lv.count * sizeof(double));
  BufP arena = alloc_bytes(m->ctx, bytes);
  size_t at = 0;
  for (Level& lv : m->lv) {
    lv.sq = sub_buf(arena, at, lv.count * sizeof(double));
    at += up(lv.count * sizeof(double));
  }
  m->slot = sub_buf(arena, at, n * sizeof(int64_t));
}

// ----------------------------------------------------------- truncation
// Block rule: drop leaf iff sqrt(s) < tau (the pool is shared, no copy).
__global__ void block_keep_kernel(const double* __restrict__ sq, int64_t n, double tau, uint8_t* __restrict__ keep) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
    keep[q] = !(sqrt(sq[q]) < tau);
}

// A view of `in` without leaves of its own yet.
static spamm_mat view_of(spamm_ctx ctx, spamm_mat in) {
  spamm_mat out = new_mat(ctx, in->n, in->bs);
  out->symmetric = in->symmetric;
  out->pool = in->pool;
  return out;
}
static TreeReq block_request(spamm_mat out, spamm_mat in, double tau) {
  return {out, in->nleaves, P<uint32_t>(in->lv[in->L].code), P<double>(in->lv[in->L].sq), P<int64_t>(in->slot), nullptr,
          tau};
}

spamm_mat truncate_block(spamm_mat in, double tau, spamm_ctx on) {
  spamm_ctx ctx = on ? on : in->ctx;
  std::unique_ptr<spamm_mat_s> out(view_of(ctx, in));
  if (in->nleaves > 0) {
    TreeReq r = block_request(out.get(), in, tau);
    tree_from_candidates(ctx, &r, 1, true);
  }
  return out.release();
}

void truncate_pair(spamm_ctx ctx, spamm_mat A, spamm_mat B, double tau, spamm_mat* At, spamm_mat* Bt) {
  TreeReq r[2];
  int k = 0;
  std::unique_ptr<spamm_mat_s> a(view_of(ctx, A)), b(A == B ? nullptr : view_of(ctx, B));
  if (A->nleaves > 0) r[k++] = block_request(a.get(), A, tau);
  if (b && B->nleaves > 0) r[k++] = block_request(b.get(), B, tau);
  if (k) tree_from_candidates(ctx, r, k, false);
  *At = a.release();
  *Bt = b ? b.release() : *At;
}

// Error-controlled rule: drop the smallest leaves (ascending squared norm,
// ties in Morton order) as long as the sum of their squared norms, added in
// that order, stays <= tau^2, so ||A - A~||_F <= tau.  The squared norms are
// non-negative doubles, so their bit patterns sort like their values.
//
// Only a leaf whose own squared norm is within the budget can be dropped (a running
// sum is at least its last term), so the others are left out of the sort and of the
// sums: the candidates come first in the sorted order, and the running sums over them
// are the same numbers without what follows.
constexpr int kSelectPer = 4;
constexpr int64_t kSelectTile = kThreads * kSelectPer;

// Candidates per tile; with `tiles` scanned (place = true) their keys and indexes, in
// leaf order.
__global__ void __launch_bounds__(kThreads)
    select_small_kernel(const double* __restrict__ sq, int64_t n, double budget, uint64_t* __restrict__ tiles, bool place,
                        uint64_t* __restrict__ keys, int64_t* __restrict__ idx) {
  __shared__ unsigned ws[kThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t q0 = (int64_t)blockIdx.x * kSelectTile + (int64_t)threadIdx.x * kSelectPer;
  double v[kSelectPer];
  unsigned c = 0;
#pragma unroll
  for (int i = 0; i < kSelectPer; ++i) {
    v[i] = q0 + i < n ? sq[q0 + i] : budget + 1.0;
    c += (q0 + i < n) && v[i] <= budget;
  }
  unsigned x = c;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) ws[warp] = x;
  __syncthreads();
  unsigned before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) {
    if (w < warp) before += ws[w];
    all += ws[w];
  }
  if (!place) {
    if (threadIdx.x == 0) tiles[blockIdx.x] = all;
    return;
  }
  int64_t p = (int64_t)tiles[blockIdx.x] + before + x - c;
#pragma unroll
  for (int i = 0; i < kSelectPer; ++i)
    if (q0 + i < n && v[i] <= budget) {
      keys[p] = (uint64_t)__double_as_longlong(v[i]);
      idx[p++] = q0 + i;
    }
}

// Number of running sums within the budget.
__global__ void within_budget_kernel(const double* __restrict__ csum, int64_t n, double budget,
                                     unsigned long long* __restrict__ count) {
  unsigned long long c = 0;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
    c += csum[q] <= budget ? 1u : 0u;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(count, c);
}

// The first *ndrop of the sorted candidates are dropped (a prefix, even if
// rounding made the running sums non-monotone by an ulp).
__global__ void drop_prefix_kernel(const int64_t* __restrict__ idx, int64_t n, const uint64_t* __restrict__ ndrop,
                                   uint8_t* __restrict__ keep) {
  const int64_t k = min((int64_t)*ndrop, n);
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < k; q += (int64_t)gridDim.x * blockDim.x)
    keep[idx[q]] = 0;
}

spamm_mat truncate_error_controlled(spamm_mat in, double tau, spamm_ctx on) {
  spamm_ctx ctx = on ? on : in->ctx;
  std::unique_ptr<spamm_mat_s> out(view_of(ctx, in));
  const int64_t n = in->nleaves;
  BufP keep = alloc_n<uint8_t>(ctx, n);
  if (n > 0) {
    const double budget = tau * tau;
    const double* sq = P<double>(in->lv[in->L].sq);
    CK(cudaMemsetAsync(P<uint8_t>(keep), 1, n, ctx->stream));
    const int64_t ntiles = (n + kSelectTile - 1) / kSelectTile;
    BufP tiles = alloc_n<uint64_t>(ctx, ntiles + 1);
    select_small_kernel<<<(unsigned)ntiles, kThreads, 0, ctx->stream>>>(sq, n, budget, P<uint64_t>(tiles), false, nullptr,
                                                                        nullptr);
    CK_LAUNCH("select_small_kernel");
    scan_exclusive_u64(ctx, P<uint64_t>(tiles), P<uint64_t>(tiles), ntiles, P<uint64_t>(tiles) + ntiles);
    const int64_t c = (int64_t)read_scalar<uint64_t>(ctx, P<uint64_t>(tiles) + ntiles);
    if (c > 0) {
      BufP keys = alloc_n<uint64_t>(ctx, c), idx = alloc_n<int64_t>(ctx, c), csum = alloc_n<double>(ctx, c);
      BufP ndrop = alloc_n<uint64_t>(ctx, 1);
      CK(cudaMemsetAsync(P<uint64_t>(ndrop), 0, sizeof(uint64_t), ctx->stream));
      select_small_kernel<<<(unsigned)ntiles, kThreads, 0, ctx->stream>>>(sq, n, budget, P<uint64_t>(tiles), true,
                                                                          P<uint64_t>(keys), P<int64_t>(idx));
      CK_LAUNCH("select_small_kernel");
      const unsigned g = grid_for(ctx, c, kThreads);
      radix_sort_pairs(ctx, P<uint64_t>(keys), P<int64_t>(idx), c, 64);  // stable: ties keep Morton order
      scan_inclusive_f64(ctx, P<double>(keys), P<double>(csum), c);  // the sorted keys are the squared norms' bits
      within_budget_kernel<<<g, kThreads, 0, ctx->stream>>>(P<double>(csum), c, budget, P<unsigned long long>(ndrop));
      CK_LAUNCH("within_budget_kernel");
      drop_prefix_kernel<<<g, kThreads, 0, ctx->stream>>>(P<int64_t>(idx), c, P<uint64_t>(ndrop), P<uint8_t>(keep));
      CK_LAUNCH("drop_prefix_kernel");
    }
  }
  set_leaves_compacted(out.get(), n, P<uint32_t>(in->lv[in->L].code), P<double>(in->lv[in->L].sq), P<int64_t>(in->slot),
                       P<uint8_t>(keep));
  return out.release();
}

// Element rule (Theorem 1): a -> 0 iff |a| < tau, into a fresh pool.
spamm_mat truncate_element(spamm_mat in, double tau) {
  spamm_ctx ctx = in->ctx;
  const int64_t n = in->nleaves, e = (int64_t)in->bs * in->bs;
  std::unique_ptr<spamm_mat_s> out(new_mat(ctx, in->n, in->bs));
  out->symmetric = in->symmetric;
  out->pool = alloc_n<double>(ctx, n * e);
  BufP sq = alloc_n<double>(ctx, n), nz = alloc_n<uint8_t>(ctx, n);
  if (n > 0) {
    // tau may be -0.0, which the pass, comparing bit patterns, must not see
    const double least = tau > 0.0 ? tau : 0.0;
    leaf_pass(ctx, CopyOp{P<double>(in->pool), P<int64_t>(in->slot), least, nullptr}, n, in->bs, P<double>(out->pool),
              P<double>(sq), P<uint8_t>(nz), 0);
  }
  set_leaves_compacted(out.get(), n, P<uint32_t>(in->lv[in->L].code), P<double>(sq), nullptr, P<uint8_t>(nz));
  return out.release();
}

// --------------------------------------------------------------- builders
__global__ void block_codes_kernel(const int32_t* __restrict__ bi, const int32_t* __restrict__ bj, int64_t n,
                                   int64_t nb, uint64_t* __restrict__ keys, int64_t* __restrict__ vals, int* err) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    int32_t r = bi[q], c = bj[q];
    if (r < 0 || c < 0 || r >= nb || c >= nb) {
      atomicOr(err, DEV_ERR_RANGE);
      r = 0;
      c = 0;
    }
    keys[q] = morton2((uint32_t)r, (uint32_t)c);
    vals[q] = q;
  }
}

__global__ void gather_sorted_kernel(int64_t n, const uint64_t* __restrict__ keys, const int64_t* __restrict__ vals,
                                     const double* __restrict__ sq_by_input, const uint8_t* __restrict__ nz_by_input,
                                     double tau, int block_rule, uint32_t* __restrict__ code, double* __restrict__ sq,
                                     int64_t* __restrict__ slot, uint8_t* __restrict__ keep, int* err) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    int64_t v = vals[q];
    code[q] = (uint32_t)keys[q];
    sq[q] = sq_by_input[v];
    slot[q] = v;
    bool k = nz_by_input[v] != 0;
    if (block_rule && tau > 0.0 && sqrt(sq_by_input[v]) < tau) k = false;
    keep[q] = k;
    if (q > 0 && keys[q] == keys[q - 1]) atomicOr(err, DEV_ERR_DUPLICATE);
  }
}

__global__ void zero_below_kernel(double* __restrict__ a, int64_t n, double tau) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
    if (fabs(a[q]) < tau) a[q] = 0.0;
}

// Leaves given as `nblocks` payloads on the device in input order: at `payload`, to be
// copied into the pool, or (null) in the pool already.
static spamm_mat finish_from_pool(spamm_ctx ctx, int64_t n, int bs, BufP pool, const double* payload, int64_t nblocks,
                                  const int32_t* d_bi, const int32_t* d_bj, double tau, spamm_trunc_rule rule) {
  std::unique_ptr<spamm_mat_s> m(new_mat(ctx, n, bs));
  m->pool = pool;
  const int64_t e = (int64_t)bs * bs;
  const bool element = rule == SPAMM_TRUNC_ELEMENT && tau > 0.0;
  if (element && nblocks > 0 && !payload) {
    zero_below_kernel<<<grid_for(ctx, nblocks * e, kThreads), kThreads, 0, ctx->stream>>>(P<double>(pool),
                                                                                         nblocks * e, tau);
    CK_LAUNCH("zero_below_kernel");
  }
  BufP sq = alloc_n<double>(ctx, nblocks), nz = alloc_n<uint8_t>(ctx, nblocks);
  BufP keys = alloc_n<uint64_t>(ctx, nblocks), vals = alloc_n<int64_t>(ctx, nblocks);
  BufP code = alloc_n<uint32_t>(ctx, nblocks), ssq = alloc_n<double>(ctx, nblocks);
  BufP slot = alloc_n<int64_t>(ctx, nblocks), keep = alloc_n<uint8_t>(ctx, nblocks);
  if (nblocks > 0) {
    if (payload)
      leaf_pass(ctx, CopyOp{payload, nullptr, element ? tau : 0.0, nullptr}, nblocks, bs, P<double>(pool), P<double>(sq),
                P<uint8_t>(nz), 1);
    else
      leaf_sqnorms(ctx, P<double>(pool), nullptr, nblocks, bs, P<double>(sq), P<uint8_t>(nz), 1);
    const int64_t nb = (n + bs - 1) / bs;
    block_codes_kernel<<<grid_for(ctx, nblocks, kThreads), kThreads, 0, ctx->stream>>>(
        d_bi, d_bj, nblocks, nb, P<uint64_t>(keys), P<int64_t>(vals), ctx->d_err);
    CK_LAUNCH("block_codes_kernel");
    radix_sort_pairs(ctx, P<uint64_t>(keys), P<int64_t>(vals), nblocks, 2 * m->L);
    gather_sorted_kernel<<<grid_for(ctx, nblocks, kThreads), kThreads, 0, ctx->stream>>>(
        nblocks, P<uint64_t>(keys), P<int64_t>(vals), P<double>(sq), P<uint8_t>(nz), tau,
        rule == SPAMM_TRUNC_BLOCK_FROB, P<uint32_t>(code), P<double>(ssq), P<int64_t>(slot), P<uint8_t>(keep),
        ctx->d_err);
    CK_LAUNCH("gather_sorted_kernel");
    sync_and_check(ctx);
  }
  set_leaves_compacted(m.get(), nblocks, P<uint32_t>(code), P<double>(ssq), P<int64_t>(slot), P<uint8_t>(keep));
  return m.release();
}

spamm_mat build_from_blocks(spamm_ctx ctx, int64_t n, int bs, int64_t nblocks, const int32_t* bi, const int32_t* bj,
                            const double* payload, int on_device, double tau, spamm_trunc_rule rule) {
  const int64_t e = (int64_t)bs * bs;
  BufP pool = alloc_n<double>(ctx, nblocks * e);
  // coordinates on the device are read where they are; from an address between 32-bit
  // words they are copied first, like those of the host
  auto words = [](const int32_t* p) { return (reinterpret_cast<uintptr_t>(p) & 3) == 0; };
  const bool place_i = !on_device || !words(bi), place_j = !on_device || !words(bj);
  BufP dbi, dbj;
  if (place_i) dbi = alloc_n<int32_t>(ctx, nblocks);
  if (place_j) dbj = alloc_n<int32_t>(ctx, nblocks);
  // leaves on the device are copied and their norms taken in one pass (which reads
  // 16-byte pairs; a payload that starts between them is copied first)
  const bool pass = on_device && (reinterpret_cast<uintptr_t>(payload) & 15) == 0;
  cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  if (nblocks > 0) {
    if (!pass) CK(cudaMemcpyAsync(P<double>(pool), payload, nblocks * e * sizeof(double), kind, ctx->stream));
    if (place_i) CK(cudaMemcpyAsync(P<int32_t>(dbi), bi, nblocks * sizeof(int32_t), kind, ctx->stream));
    if (place_j) CK(cudaMemcpyAsync(P<int32_t>(dbj), bj, nblocks * sizeof(int32_t), kind, ctx->stream));
  }
  return finish_from_pool(ctx, n, bs, pool, pass ? payload : nullptr, nblocks, place_i ? P<int32_t>(dbi) : bi,
                          place_j ? P<int32_t>(dbj) : bj, tau, rule);
}

// Candidate leaves in Morton order over the 2^L x 2^L grid, those inside
// the ceil(n/bs) x ceil(n/bs) block range only.  Warp per candidate.
template <class Elem>
__global__ void candidate_stats_kernel(Elem elem, int64_t ncand, int bs, int64_t nb, double tau, int rule,
                                       double* __restrict__ sq, uint8_t* __restrict__ keep, int* err) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < ncand; q += nw) {
    const uint32_t r = code_row((uint32_t)q), c = code_col((uint32_t)q);
    if (r >= nb || c >= nb || elem.skip(r, c, tau, rule)) {
      if (lane == 0) {
        keep[q] = 0;
        sq[q] = 0.0;
      }
      continue;
    }
    double s;
    bool nz, bad;
    warp_leaf_sumsq<1>(
        [&](int i) {
          int e0 = 2 * i;
          double x = elem(r, c, e0 / bs, e0 % bs), y = elem(r, c, e0 / bs, e0 % bs + 1);
          if (rule == SPAMM_TRUNC_ELEMENT) {
            if (fabs(x) < tau) x = 0.0;
            if (fabs(y) < tau) y = 0.0;
          }
          return make_double2(x, y);
        },
        bs, lane, &s, &nz, &bad);
    if (lane == 0) {
      bool k = nz;
      if (rule == SPAMM_TRUNC_BLOCK_FROB && tau > 0.0 && sqrt(s) < tau) k = false;
      keep[q] = k;
      sq[q] = s;
      if (bad) atomicOr(err, DEV_ERR_NONFINITE);
    }
  }
}

template <class Elem>
__global__ void candidate_fill_kernel(Elem elem, int64_t nleaves, const uint32_t* __restrict__ code, int bs,
                                      double tau, int rule, double* __restrict__ pool) {
  const int64_t e = (int64_t)bs * bs;
  for (int64_t q = blockIdx.x; q < nleaves; q += gridDim.x) {
    const uint32_t r = code_row(code[q]), c = code_col(code[q]);
    for (int64_t i = threadIdx.x; i < e; i += blockDim.x) {
      double x = elem(r, c, (int)(i / bs), (int)(i % bs));
      if (rule == SPAMM_TRUNC_ELEMENT && fabs(x) < tau) x = 0.0;
      pool[q * e + i] = x;
    }
  }
}

struct DenseElem {
  const double* a;
  int64_t lda, n;
  int bs;
  __device__ double operator()(uint32_t r, uint32_t c, int i, int j) const {
    int64_t gi = (int64_t)r * bs + i, gj = (int64_t)c * bs + j;
    return (gi < n && gj < n) ? a[gi * lda + gj] : 0.0;
  }
  __device__ bool skip(uint32_t, uint32_t, double, int) const { return false; }
};

struct GenElem {
  synth_params p;
  int bs;
  __device__ double operator()(uint32_t r, uint32_t c, int i, int j) const {
    return synth_element(&p, (int64_t)r * bs + i, (int64_t)c * bs + j);
  }
  // A leaf whose bound says every element is below the cutoff is null; under
  // the block rule a leaf whose norm bound bs * max|a| is below tau is dropped.
  __device__ bool skip(uint32_t r, uint32_t c, double tau, int rule) const {
    double b = synth_leaf_bound(&p, bs, r, c);
    if (b < p.cutoff) return true;
    if (rule == SPAMM_TRUNC_ELEMENT && b < tau) return true;
    if (rule == SPAMM_TRUNC_BLOCK_FROB && tau > 0.0 && b * bs < tau) return true;
    return false;
  }
};

template <class Elem>
static std::unique_ptr<spamm_mat_s> build_from_elements(spamm_ctx ctx, int64_t n, int bs, Elem elem, double tau, spamm_trunc_rule rule) {
  std::unique_ptr<spamm_mat_s> m(new_mat(ctx, n, bs));
  const int64_t nb = (n + bs - 1) / bs;
  const int64_t ncand = (int64_t)1 << (2 * m->L);
  BufP sq = alloc_n<double>(ctx, ncand), keep = alloc_n<uint8_t>(ctx, ncand);
  candidate_stats_kernel<<<grid_for(ctx, ncand, kThreads / 32), kThreads, 0, ctx->stream>>>(
      elem, ncand, bs, nb, tau, (int)rule, P<double>(sq), P<uint8_t>(keep), ctx->d_err);
  CK_LAUNCH("candidate_stats_kernel");
  sync_and_check(ctx);
  // the candidates' codes are their indices 0 .. 4^L - 1
  set_leaves_compacted(m.get(), ncand, nullptr, P<double>(sq), nullptr, P<uint8_t>(keep));
  // payload for the kept leaves, slot = leaf index
  const int64_t e = (int64_t)bs * bs;
  m->pool = alloc_n<double>(ctx, m->nleaves * e);
  if (m->nleaves > 0) {
    candidate_fill_kernel<<<grid_for(ctx, m->nleaves, 1, 64), kThreads, 0, ctx->stream>>>(
        elem, m->nleaves, P<uint32_t>(m->lv[m->L].code), bs, tau, (int)rule, P<double>(m->pool));
    CK_LAUNCH("candidate_fill_kernel");
    fill_iota_i64(ctx, P<int64_t>(m->slot), m->nleaves);
  }
  return m;
}

__global__ void iota_i64_kernel(int64_t* p, int64_t n) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
    p[q] = q;
}
void fill_iota_i64(spamm_ctx ctx, int64_t* p, int64_t n) {
  if (n <= 0) return;
  iota_i64_kernel<<<grid_for(ctx, n, kThreads), kThreads, 0, ctx->stream>>>(p, n);
  CK_LAUNCH("iota_i64_kernel");
}

spamm_mat build_from_dense(spamm_ctx ctx, int64_t n, const double* a, int64_t lda, int on_device, int bs, double tau,
                           spamm_trunc_rule rule) {
  BufP tmp;
  const double* da = a;
  int64_t dlda = lda;
  if (!on_device) {
    tmp = alloc_n<double>(ctx, n * n);
    CK(cudaMemcpy2DAsync(P<double>(tmp), n * sizeof(double), a, lda * sizeof(double), n * sizeof(double), n,
                         cudaMemcpyHostToDevice, ctx->stream));
    da = P<double>(tmp);
    dlda = n;
  }
  DenseElem el{da, dlda, n, bs};
  std::unique_ptr<spamm_mat_s> m = build_from_elements(ctx, n, bs, el, tau, rule);
  sync_and_check(ctx);  // the temporary copy must outlive the fill
  return m.release();
}

spamm_mat build_generated(spamm_ctx ctx, const spamm_gen_params* gp, int bs, double tau, spamm_trunc_rule rule) {
  GenElem el;
  el.p.n = gp->n;
  el.p.kind = gp->kind;
  el.p.law = gp->law;
  el.p.alpha = gp->alpha;
  el.p.c = gp->c;
  el.p.cutoff = gp->cutoff;
  el.p.seed = gp->seed;
  el.bs = bs;
  std::unique_ptr<spamm_mat_s> m = build_from_elements(ctx, gp->n, bs, el, tau, rule);
  m->symmetric = 1;  // u_ij and the decay law are symmetric in (i, j)
  return m.release();
}

// COO: sort (leaf code, in-leaf offset) keys stably, sum runs of equal keys
// in input order, scatter into zeroed leaves.
__global__ void coo_keys_kernel(const int64_t* __restrict__ row, const int64_t* __restrict__ col,
                                const double* __restrict__ val, int64_t nnz, int64_t n, int bs, int lbs,
                                uint64_t* __restrict__ keys, int64_t* __restrict__ vals, int* err) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nnz; q += (int64_t)gridDim.x * blockDim.x) {
    int64_t r = row[q], c = col[q];
    if (r < 0 || c < 0 || r >= n || c >= n) {
      atomicOr(err, DEV_ERR_RANGE);
      r = 0;
      c = 0;
    }
    if (!isfinite(val[q])) atomicOr(err, DEV_ERR_NONFINITE);
    uint64_t leaf = morton2((uint32_t)(r / bs), (uint32_t)(c / bs));
    uint64_t off = (uint64_t)((r % bs) * bs + (c % bs));
    keys[q] = (leaf << (2 * lbs)) | off;
    vals[q] = q;
  }
}

__global__ void coo_leaf_flags_kernel(const uint64_t* __restrict__ keys, int64_t nnz, int lbs,
                                      uint64_t* __restrict__ flags) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nnz; q += (int64_t)gridDim.x * blockDim.x)
    flags[q] = (q == 0 || (keys[q] >> (2 * lbs)) != (keys[q - 1] >> (2 * lbs))) ? 1u : 0u;
}

__global__ void coo_scatter_kernel(const uint64_t* __restrict__ keys, const int64_t* __restrict__ vals,
                                   const double* __restrict__ val, int64_t nnz, int lbs,
                                   const uint64_t* __restrict__ flags, const uint64_t* __restrict__ excl,
                                   double* __restrict__ pool, uint32_t* __restrict__ code) {
  const int64_t e = (int64_t)1 << (2 * lbs);
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nnz; q += (int64_t)gridDim.x * blockDim.x) {
    if (q > 0 && keys[q] == keys[q - 1]) continue;  // not the head of its run
    int64_t leaf = (int64_t)(excl[q] + flags[q]) - 1;
    if (flags[q]) code[leaf] = (uint32_t)(keys[q] >> (2 * lbs));
    double s = 0.0;
    for (int64_t p = q; p < nnz && keys[p] == keys[q]; ++p) s += val[vals[p]];
    pool[leaf * e + (int64_t)(keys[q] & (uint64_t)(e - 1))] = s;
  }
}

spamm_mat build_from_coo(spamm_ctx ctx, int64_t n, int64_t nnz, const int64_t* row, const int64_t* col,
                         const double* val, int on_device, int bs, double tau, spamm_trunc_rule rule) {
  std::unique_ptr<spamm_mat_s> m(new_mat(ctx, n, bs));
  int lbs = 0;
  while ((1 << lbs) < bs) ++lbs;
  const int64_t e = (int64_t)bs * bs;
  BufP drow, dcol, dval;
  const int64_t *r = row, *c = col;
  const double* v = val;
  if (!on_device && nnz > 0) {
    drow = alloc_n<int64_t>(ctx, nnz);
    dcol = alloc_n<int64_t>(ctx, nnz);
    dval = alloc_n<double>(ctx, nnz);
    CK(cudaMemcpyAsync(P<int64_t>(drow), row, nnz * 8, cudaMemcpyHostToDevice, ctx->stream));
    CK(cudaMemcpyAsync(P<int64_t>(dcol), col, nnz * 8, cudaMemcpyHostToDevice, ctx->stream));
    CK(cudaMemcpyAsync(P<double>(dval), val, nnz * 8, cudaMemcpyHostToDevice, ctx->stream));
    r = P<int64_t>(drow);
    c = P<int64_t>(dcol);
    v = P<double>(dval);
  }
  if (nnz == 0) {
    set_leaves_compacted(m.get(), 0, nullptr, nullptr, nullptr, nullptr);
    return m.release();
  }
  BufP keys = alloc_n<uint64_t>(ctx, nnz), vals = alloc_n<int64_t>(ctx, nnz);
  coo_keys_kernel<<<grid_for(ctx, nnz, kThreads), kThreads, 0, ctx->stream>>>(
      r, c, v, nnz, n, bs, lbs, P<uint64_t>(keys), P<int64_t>(vals), ctx->d_err);
  CK_LAUNCH("coo_keys_kernel");
  sync_and_check(ctx);
  radix_sort_pairs(ctx, P<uint64_t>(keys), P<int64_t>(vals), nnz, 2 * m->L + 2 * lbs);
  BufP flags = alloc_n<uint64_t>(ctx, nnz), excl = alloc_n<uint64_t>(ctx, nnz), tot = alloc_n<uint64_t>(ctx, 1);
  coo_leaf_flags_kernel<<<grid_for(ctx, nnz, kThreads), kThreads, 0, ctx->stream>>>(P<uint64_t>(keys), nnz, lbs,
                                                                                   P<uint64_t>(flags));
  CK_LAUNCH("coo_leaf_flags_kernel");
  scan_exclusive_u64(ctx, P<uint64_t>(flags), P<uint64_t>(excl), nnz, P<uint64_t>(tot));
  const int64_t nl = (int64_t)read_scalar<uint64_t>(ctx, P<uint64_t>(tot));
  BufP pool = alloc_n<double>(ctx, nl * e), code = alloc_n<uint32_t>(ctx, nl);
  CK(cudaMemsetAsync(P<double>(pool), 0, nl * e * sizeof(double), ctx->stream));
  coo_scatter_kernel<<<grid_for(ctx, nnz, kThreads), kThreads, 0, ctx->stream>>>(
      P<uint64_t>(keys), P<int64_t>(vals), v, nnz, lbs, P<uint64_t>(flags), P<uint64_t>(excl), P<double>(pool),
      P<uint32_t>(code));
  CK_LAUNCH("coo_scatter_kernel");
  if (rule == SPAMM_TRUNC_ELEMENT && tau > 0.0) {
    zero_below_kernel<<<grid_for(ctx, nl * e, kThreads), kThreads, 0, ctx->stream>>>(P<double>(pool), nl * e, tau);
    CK_LAUNCH("zero_below_kernel");
  }
  BufP sq = alloc_n<double>(ctx, nl), nz = alloc_n<uint8_t>(ctx, nl);
  leaf_sqnorms(ctx, P<double>(pool), nullptr, nl, bs, P<double>(sq), P<uint8_t>(nz), 0);
  if (rule == SPAMM_TRUNC_BLOCK_FROB && tau > 0.0) {
    BufP keep2 = alloc_n<uint8_t>(ctx, nl);
    block_keep_kernel<<<grid_for(ctx, nl, kThreads), kThreads, 0, ctx->stream>>>(P<double>(sq), nl, tau,
                                                                                P<uint8_t>(keep2));
    CK_LAUNCH("block_keep_kernel");
    and_u8(ctx, P<uint8_t>(nz), P<uint8_t>(keep2), nl);
  }
  m->pool = pool;
  set_leaves_compacted(m.get(), nl, P<uint32_t>(code), P<double>(sq), nullptr, P<uint8_t>(nz));
  return m.release();
}

__global__ void and_u8_kernel(uint8_t* a, const uint8_t* b, int64_t n) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
    a[q] = a[q] && b[q];
}
void and_u8(spamm_ctx ctx, uint8_t* a, const uint8_t* b, int64_t n) {
  if (n <= 0) return;
  and_u8_kernel<<<grid_for(ctx, n, kThreads), kThreads, 0, ctx->stream>>>(a, b, n);
  CK_LAUNCH("and_u8_kernel");
}

// ---------------------------------------------------------------- exports
__global__ void to_dense_kernel(const double* __restrict__ pool, const int64_t* __restrict__ slot,
                                const uint32_t* __restrict__ code, int64_t nleaves, int bs, int64_t n,
                                double* __restrict__ out, int64_t ld) {
  const int64_t e = (int64_t)bs * bs;
  for (int64_t q = blockIdx.x; q < nleaves; q += gridDim.x) {
    const int64_t r0 = (int64_t)code_row(code[q]) * bs, c0 = (int64_t)code_col(code[q]) * bs;
    const double* src = pool + slot[q] * e;
    for (int64_t i = threadIdx.x; i < e; i += blockDim.x) {
      int64_t r = r0 + i / bs, c = c0 + i % bs;
      if (r < n && c < n) out[r * ld + c] = src[i];
    }
  }
}

void export_dense(spamm_mat m, double* out, int64_t ld, int on_device) {
  spamm_ctx ctx = m->ctx;
  BufP tmp;
  double* dst = out;
  int64_t dld = ld;
  if (!on_device) {
    tmp = alloc_n<double>(ctx, m->n * m->n);
    dst = P<double>(tmp);
    dld = m->n;
  }
  CK(cudaMemset2DAsync(dst, dld * sizeof(double), 0, m->n * sizeof(double), m->n, ctx->stream));
  if (m->nleaves > 0) {
    to_dense_kernel<<<grid_for(ctx, m->nleaves, 1, 64), kThreads, 0, ctx->stream>>>(
        P<double>(m->pool), P<int64_t>(m->slot), P<uint32_t>(m->lv[m->L].code), m->nleaves, m->bs, m->n, dst, dld);
    CK_LAUNCH("to_dense_kernel");
  }
  if (!on_device)
    CK(cudaMemcpy2DAsync(out, ld * sizeof(double), dst, dld * sizeof(double), m->n * sizeof(double), m->n,
                         cudaMemcpyDeviceToHost, ctx->stream));
  sync_and_check(ctx);
}

// The squared norms go along with the leaves: a copy of their own is some 5 us of launch
// and gap (100 leaves of 32 x 32: 208 -> 206 us with the product before it).
__global__ void to_blocks_kernel(const double* __restrict__ pool, const int64_t* __restrict__ slot,
                                 const uint32_t* __restrict__ code, const double* __restrict__ lsq, int64_t nleaves,
                                 int bs, int32_t* bi, int32_t* bj, double* __restrict__ payload, double* sq) {
  const int64_t e = (int64_t)bs * bs;
  for (int64_t q = blockIdx.x; q < nleaves; q += gridDim.x) {
    if (threadIdx.x == 0) {
      if (bi) bi[q] = (int32_t)code_row(code[q]);
      if (bj) bj[q] = (int32_t)code_col(code[q]);
      if (sq) sq[q] = lsq[q];
    }
    if (payload) {
      const double2* src = reinterpret_cast<const double2*>(pool + slot[q] * e);
      double2* dst = reinterpret_cast<double2*>(payload + q * e);
      for (int64_t i = threadIdx.x; i < e / 2; i += blockDim.x) dst[i] = src[i];
    }
  }
}

void export_blocks(spamm_mat m, int32_t* bi, int32_t* bj, double* payload, double* sq, int on_device) {
  spamm_ctx ctx = m->ctx;
  const int64_t nl = m->nleaves, e = (int64_t)m->bs * m->bs;
  if (nl == 0) return;
  BufP tbi, tbj, tpay;
  int32_t *dbi = bi, *dbj = bj;
  double* dpay = payload;
  if (!on_device) {
    if (bi) dbi = P<int32_t>(tbi = alloc_n<int32_t>(ctx, nl));
    if (bj) dbj = P<int32_t>(tbj = alloc_n<int32_t>(ctx, nl));
    // a product's leaves lie in order: to the host straight from its pool (15,300 leaves,
    // 0.5 GB: a pass of 0.15 ms beside 2.6 ms on the link, and a buffer of that size)
    if (payload) dpay = m->packed ? nullptr : P<double>(tpay = alloc_n<double>(ctx, nl * e));
  }
  const bool along = on_device && (reinterpret_cast<uintptr_t>(sq) & 7) == 0;
  to_blocks_kernel<<<grid_for(ctx, nl, 1, 64), kThreads, 0, ctx->stream>>>(
      P<double>(m->pool), P<int64_t>(m->slot), P<uint32_t>(m->lv[m->L].code), P<double>(m->lv[m->L].sq), nl, m->bs, dbi, dbj,
      dpay, along ? sq : nullptr);
  CK_LAUNCH("to_blocks_kernel");
  cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  if (!on_device) {
    if (bi) CK(cudaMemcpyAsync(bi, dbi, nl * sizeof(int32_t), kind, ctx->stream));
    if (bj) CK(cudaMemcpyAsync(bj, dbj, nl * sizeof(int32_t), kind, ctx->stream));
    if (payload)
      CK(cudaMemcpyAsync(payload, dpay ? dpay : P<double>(m->pool), nl * e * sizeof(double), kind, ctx->stream));
  }
  if (sq && !along) CK(cudaMemcpyAsync(sq, P<double>(m->lv[m->L].sq), nl * sizeof(double), kind, ctx->stream));
  sync_and_check(ctx);
}

__global__ void gather_leaves_kernel(const double* __restrict__ pool, const int64_t* __restrict__ slot,
                                     const uint32_t* __restrict__ code, int64_t nleaves, int bs, int64_t nq,
                                     const int32_t* __restrict__ bi, const int32_t* __restrict__ bj,
                                     double* __restrict__ out, int32_t* __restrict__ found);

void gather_leaves(spamm_mat m, int64_t nq, const int32_t* bi, const int32_t* bj, double* out, int32_t* found,
                   int on_device) {
  spamm_ctx ctx = m->ctx;
  if (nq <= 0) return;
  const int64_t e = (int64_t)m->bs * m->bs;
  BufP tbi, tbj, tout, tfound;
  const int32_t *dbi = bi, *dbj = bj;
  double* dout = out;
  int32_t* dfound = found;
  if (!on_device) {
    tbi = alloc_n<int32_t>(ctx, nq);
    tbj = alloc_n<int32_t>(ctx, nq);
    tout = alloc_n<double>(ctx, nq * e);
    tfound = alloc_n<int32_t>(ctx, nq);
    CK(cudaMemcpyAsync(P<int32_t>(tbi), bi, nq * sizeof(int32_t), cudaMemcpyHostToDevice, ctx->stream));
    CK(cudaMemcpyAsync(P<int32_t>(tbj), bj, nq * sizeof(int32_t), cudaMemcpyHostToDevice, ctx->stream));
    dbi = P<int32_t>(tbi);
    dbj = P<int32_t>(tbj);
    dout = P<double>(tout);
    dfound = P<int32_t>(tfound);
  }
  gather_leaves_kernel<<<grid_for(ctx, nq, 1, 64), kThreads, 0, ctx->stream>>>(
      P<double>(m->pool), P<int64_t>(m->slot), P<uint32_t>(m->lv[m->L].code), m->nleaves, m->bs, nq, dbi, dbj, dout,
      dfound);
  CK_LAUNCH("gather_leaves_kernel");
  if (!on_device) {
    CK(cudaMemcpyAsync(out, dout, nq * e * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    if (found) CK(cudaMemcpyAsync(found, dfound, nq * sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
  }
  sync_and_check(ctx);
}

// ------------------------------------------------------- error ||X - Y||_F
__device__ __forceinline__ int64_t find_code(const uint32_t* __restrict__ codes, int64_t n, uint32_t key) {
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (codes[mid] < key)
      lo = mid + 1;
    else
      hi = mid;
  }
  return (lo < n && codes[lo] == key) ? lo : -1;
}

__global__ void error_x_kernel(const double* __restrict__ xpool, const int64_t* __restrict__ xslot,
                               const uint32_t* __restrict__ xcode, const double* __restrict__ xsq, int64_t nx,
                               const double* __restrict__ ypool, const int64_t* __restrict__ yslot,
                               const uint32_t* __restrict__ ycode, int64_t ny, int bs, double* __restrict__ part) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t e = (int64_t)bs * bs;
  for (int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < nx; q += nw) {
    int64_t p = find_code(ycode, ny, xcode[q]);
    if (p < 0) {
      if (lane == 0) part[q] = xsq[q];
      continue;
    }
    const double2* xs = reinterpret_cast<const double2*>(xpool + xslot[q] * e);
    const double2* ys = reinterpret_cast<const double2*>(ypool + yslot[p] * e);
    double s;
    bool nz, bad;
    warp_leaf_sumsq<4>(
        [&](int i) {
          double2 a = __ldg(xs + i), b = __ldg(ys + i);
          return make_double2(a.x - b.x, a.y - b.y);
        },
        bs, lane, &s, &nz, &bad);
    if (lane == 0) part[q] = s;
  }
}

__global__ void error_y_kernel(const uint32_t* __restrict__ xcode, int64_t nx, const uint32_t* __restrict__ ycode,
                               const double* __restrict__ ysq, int64_t ny, double* __restrict__ part) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < ny; q += (int64_t)gridDim.x * blockDim.x)
    part[q] = find_code(xcode, nx, ycode[q]) < 0 ? ysq[q] : 0.0;
}

// Deterministic sum: fixed tiles of kSumTile elements reduced by a fixed tree, then the
// tiles' sums the same way by the block that is last to finish, which leaves the result
// in the host's memory: one launch, and the caller's wait is the only one (an error of
// two matrices waited three times: a purification step 2.57 -> 2.52 ms with both).
constexpr int64_t kSumTile = 4096;
template <class Load>
__device__ __forceinline__ double tile_sum(Load load, int64_t n) {
  __shared__ double sh[kThreads];
  double s = 0.0;
  for (int i = 0; i < kSumTile / kThreads; ++i) {
    const int64_t q = threadIdx.x + (int64_t)i * kThreads;
    if (q < n) s += load(q);
  }
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  const double all = sh[0];
  __syncthreads();
  return all;
}
__global__ void __launch_bounds__(kThreads)
    sum_kernel(const double* __restrict__ in, int64_t n, double* __restrict__ tiles, unsigned* __restrict__ ticket,
               double* __restrict__ result) {
  __shared__ bool s_last;
  const int64_t base = (int64_t)blockIdx.x * kSumTile;
  const double s = tile_sum([&](int64_t q) { return in[base + q]; }, n - base);
  if (gridDim.x == 1) {
    if (threadIdx.x == 0) *result = s;
    return;
  }
  if (threadIdx.x == 0) {
    tiles[blockIdx.x] = s;
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const double all = tile_sum([&](int64_t q) { return __ldcg(tiles + q); }, gridDim.x);
  if (threadIdx.x == 0) {
    *result = all;
    *ticket = 0;
  }
}
// More tiles than one block adds up.
__global__ void __launch_bounds__(kThreads)
    sum_tiles_kernel(const double* __restrict__ in, int64_t n, double* __restrict__ out) {
  const int64_t base = (int64_t)blockIdx.x * kSumTile;
  const double s = tile_sum([&](int64_t q) { return in[base + q]; }, n - base);
  if (threadIdx.x == 0) out[blockIdx.x] = s;
}

void device_sum_async(spamm_ctx ctx, const double* in, int64_t n, double* host) {
  if (n <= 0) {
    *host = 0.0;
    return;
  }
  BufP cur;
  while (n > kSumTile * kSumTile) {
    const int64_t nb = (n + kSumTile - 1) / kSumTile;
    BufP out = alloc_n<double>(ctx, nb);
    sum_tiles_kernel<<<(unsigned)nb, kThreads, 0, ctx->stream>>>(in, n, P<double>(out));
    CK_LAUNCH("sum_tiles_kernel");
    cur = out;
    in = P<double>(cur);
    n = nb;
  }
  const int64_t nb = (n + kSumTile - 1) / kSumTile;
  BufP tiles = alloc_n<double>(ctx, nb);
  sum_kernel<<<(unsigned)nb, kThreads, 0, ctx->stream>>>(in, n, P<double>(tiles),
                                                         reinterpret_cast<unsigned*>(ctx->d_scratch + 11), host);
  CK_LAUNCH("sum_kernel");
}

__global__ void gather_leaves_kernel(const double* __restrict__ pool, const int64_t* __restrict__ slot,
                                     const uint32_t* __restrict__ code, int64_t nleaves, int bs, int64_t nq,
                                     const int32_t* __restrict__ bi, const int32_t* __restrict__ bj,
                                     double* __restrict__ out, int32_t* __restrict__ found) {
  const int64_t e = (int64_t)bs * bs;
  const int64_t side = (int64_t)1 << 16;
  for (int64_t q = blockIdx.x; q < nq; q += gridDim.x) {
    const int32_t r = bi[q], c = bj[q];
    int64_t p = -1;
    if (r >= 0 && c >= 0 && r < side && c < side) p = find_code(code, nleaves, morton2((uint32_t)r, (uint32_t)c));
    if (threadIdx.x == 0 && found) found[q] = p >= 0;
    for (int64_t i = threadIdx.x; i < e; i += blockDim.x) out[q * e + i] = p >= 0 ? pool[slot[p] * e + i] : 0.0;
  }
}

double error_fro(spamm_mat X, spamm_mat Y) {
  spamm_ctx ctx = X->ctx;
  const int64_t nx = X->nleaves, ny = Y->nleaves;
  BufP px = alloc_n<double>(ctx, nx), py = alloc_n<double>(ctx, ny);
  double* sums = static_cast<double*>(ctx->h_pinned);
  if (nx > 0) {
    error_x_kernel<<<grid_for(ctx, nx, kThreads / 32), kThreads, 0, ctx->stream>>>(
        P<double>(X->pool), P<int64_t>(X->slot), P<uint32_t>(X->lv[X->L].code), P<double>(X->lv[X->L].sq), nx,
        P<double>(Y->pool), P<int64_t>(Y->slot), P<uint32_t>(Y->lv[Y->L].code), ny, X->bs, P<double>(px));
    CK_LAUNCH("error_x_kernel");
  }
  device_sum_async(ctx, P<double>(px), nx, sums);
  if (ny > 0) {
    error_y_kernel<<<grid_for(ctx, ny, kThreads), kThreads, 0, ctx->stream>>>(
        P<uint32_t>(X->lv[X->L].code), nx, P<uint32_t>(Y->lv[Y->L].code), P<double>(Y->lv[Y->L].sq), ny,
        P<double>(py));
    CK_LAUNCH("error_y_kernel");
  }
  device_sum_async(ctx, P<double>(py), ny, sums + 1);
  sync_and_check(ctx);
  return sqrt(sums[0] + sums[1]);
}

}  // namespace spamm
