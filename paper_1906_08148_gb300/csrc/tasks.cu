// tasks.cu -- kernel (b): the SpAMM task-list builder.
//
// Algorithm 1 descends both quadtrees together: a pair (A_IK, B_KJ) that was
// entered on level t spawns the eight child pairs (A_ik, B_kj), i in {2I,
// 2I+1}, k in {2K, 2K+1}, j in {2J, 2J+1}; a child pair is entered iff both
// children are non-null and ||A_ik|| ||B_kj|| >= tau (Truncmul: no test).  The
// test is carried down to leaf pairs (Section 4.4) and the whole output
// structure is known before any leaf product runs, as the batched "in
// advance" multiplication of Section 4.4 does.
//
// Representation on level t: "groups" are the output nodes (I, J) that have
// at least one entered pair, in Morton order, each owning a contiguous run of
// pairs (a = node index in A, b = node index in B) ordered by K ascending.
// One level step:
//   count  (warp per group) evaluate the 8 children of every pair, store an 8-bit
//          kept mask per pair and per child output node c = 2ci + cj the number
//          of kept pairs, packed as (count | nonempty << 36); the sums of
//          each tile of groups, and by the last block the level's totals.
//   write  (block per tile) offsets from the tiles before and a prefix sum over
//          the tile, then (warp per group) every lane takes one pair, per child
//          group two warp ballots (k-child 0 and 1) place the kept pairs; within
//          a child group pairs stay in parent order with k = 2K, 2K+1, so the
//          children are again sorted by k.
// The first steps (at most four, as long as a leaf step remains: up to 512
// pairs each) run in one launch of one block that keeps the pairs in shared
// memory; the records of every level's nodes are made by one launch before.  So
// the list of a 4096-row lattice with 64-leaves, output structure included, takes seven
// launches and 0.10 ms instead of 54 and 0.33.
// Because a parent's squared norm is a floating-point sum of non-negative
// children, the test is monotone down the tree and the pruned descent keeps
// exactly the leaf pairs that pass the leaf-level test.
//
// For the tensor-core forms with 64 x 64 leaves the leaf step also lists the
// steps of every quad (the four children of one group): child k-index ck of a
// pair is a step if any of the four children keeps it, and pairs are in k
// order, so the same ballots place the steps; nothing has to be merged by k.
#include "internal.cuh"
#include "screen.cuh"

namespace spamm {

constexpr int kWarpsPerBlock = 8;
constexpr uint64_t kCountMask = (1ull << 36) - 1;

__device__ __forceinline__ int comp4(const int4& v, int i) {
  return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w));
}

__device__ __forceinline__ double comp4d(const double4& v, int i) {
  return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w));
}

// Per node of a level, one 16-byte record: the index of its first child on
// the next level (the children of a node are consecutive there: every level
// is in Morton order) and the four children's 24-bit norm keys (screen.cuh;
// kNullKey where a child is null), so the descent reads one 16-byte load per
// node of a pair.  The norms themselves (-1 where null) go to a second array
// that only the pairs the screen leaves undecided read.  One launch covers
// both operands' levels (A's nodes first); a node whose children are not
// consecutive sets the range error (a broken quadtree).
struct __align__(16) NodeRec {
  uint32_t base;
  uint32_t w[3];  // keys k0..k3, 24 bits each, k0 in the low bits of w[0]
};

__device__ __forceinline__ uint32_t rec_key(const NodeRec& r, int c) {
  switch (c) {
    case 0: return r.w[0] & 0xFFFFFFu;
    case 1: return (r.w[0] >> 24) | ((r.w[1] & 0xFFFFu) << 8);
    case 2: return (r.w[1] >> 16) | ((r.w[2] & 0xFFu) << 16);
    default: return r.w[2] >> 8;
  }
}

// Next-level indices of the four children (-1 where null).
__device__ __forceinline__ int4 rec_children(const NodeRec& r) {
  unsigned pres = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) pres |= (unsigned)(rec_key(r, i) != kNullKey) << i;
  const int b = (int)r.base;
  return make_int4(pres & 1u ? b : -1, pres & 2u ? b + __popc(pres & 1u) : -1, pres & 4u ? b + __popc(pres & 3u) : -1,
                   pres & 8u ? b + __popc(pres & 7u) : -1);
}

struct RecLevel {
  const int4* child;
  const double* csq;  // the next level's squared norms
  const uint64_t* n;  // nodes of this level
  NodeRec* rec;
  double4* norm;
};
struct RecTable {
  RecLevel lv[2 * SPAMM_MAX_LEVELS];  // A's levels, then B's (if B is not A)
};

// Records of every level of both operands: block row y takes table entry y.  Clears the
// `words` words that the steps count in.
__global__ void __launch_bounds__(256)
    node_rec_kernel(const __grid_constant__ RecTable T, unsigned* __restrict__ clear, int words, int* err) {
  if (blockIdx.x == 0 && blockIdx.y == 0)
    for (int i = threadIdx.x; i < words; i += blockDim.x) clear[i] = 0;
  const RecLevel& R = T.lv[blockIdx.y];
  const int64_t n = (int64_t)*R.n;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    const int4 c = R.child[q];
    const double* sq = R.csq;
    const double4 v = make_double4(c.x >= 0 ? sqrt(sq[c.x]) : -1.0, c.y >= 0 ? sqrt(sq[c.y]) : -1.0,
                                   c.z >= 0 ? sqrt(sq[c.z]) : -1.0, c.w >= 0 ? sqrt(sq[c.w]) : -1.0);
    const int ch[4] = {c.x, c.y, c.z, c.w};
    uint32_t k[4];
    int base = -1, rank = 0;
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (ch[i] < 0) {
        k[i] = kNullKey;
        continue;
      }
      if (base < 0) base = ch[i];
      ok &= ch[i] == base + rank;
      ++rank;
      k[i] = pack_norm(comp4d(v, i));
    }
    if (!ok) atomicOr(err, DEV_ERR_RANGE);
    NodeRec rec;
    rec.base = (uint32_t)(base < 0 ? 0 : base);
    rec.w[0] = k[0] | (k[1] << 24);
    rec.w[1] = (k[1] >> 8) | (k[2] << 16);
    rec.w[2] = (k[2] >> 16) | (k[3] << 8);
    R.rec[q] = rec;
    R.norm[q] = v;
  }
}

// The FP64 decision p >= tau (and the borderline count at the leaf level).
__device__ __forceinline__ bool exact_keep(double na, double nb, double tau, bool leaf, long long* border) {
  const double prod = __dmul_rn(na, nb);
  const long long pb = __double_as_longlong(prod), tb = __double_as_longlong(tau);
  const long long dist = pb > tb ? pb - tb : tb - pb;
  if (leaf && dist <= (1ll << 14) && fabs(prod - tau) <= 1e-12 * tau) ++*border;
  return pb >= tb;  // prod >= tau for prod, tau >= 0
}

// mask bit (2*c + ck) for child group c = 2*ci + cj and child k-index ck;
// na / nb: the children's norms of the pair's A and B nodes.  The product is
// the FP64 round-to-nearest product of the two norms; the comparisons use its
// bits (non-negative doubles order like their bit patterns), because this part
// issues FP64 instructions at two per clock per SM.  The borderline test
// |prod - tau| <= 1e-12 tau is evaluated in FP64 only for products within
// 2^14 units in the last place of tau (1e-12 relative is about 4500 of them).
__device__ __forceinline__ unsigned child_mask(const NodeRec& ra, const NodeRec& rb, const double4* na,
                                               const double4* nb, const TauScreen& sc, double tau, int test,
                                               bool leaf, long long* cand, long long* border) {
  uint32_t ka[4], kb[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    ka[i] = rec_key(ra, i);
    kb[i] = rec_key(rb, i);
  }
  unsigned m = 0;
#pragma unroll
  for (int ci = 0; ci < 2; ++ci)
#pragma unroll
    for (int cj = 0; cj < 2; ++cj)
#pragma unroll
      for (int ck = 0; ck < 2; ++ck) {
        const int ia = 2 * ci + ck, ib = 2 * ck + cj;
        if (ka[ia] == kNullKey || kb[ib] == kNullKey) continue;
        ++*cand;
        bool keep = true;
        if (test) {
          const int d = screen_decide(ka[ia], kb[ib], sc);
          keep = d >= 0 ? d == 1 : exact_keep(comp4d(*na, ia), comp4d(*nb, ib), tau, leaf, border);
        }
        if (keep) m |= 1u << (2 * (2 * ci + cj) + ck);
      }
  return m;
}

// Sizes and statistics of one level, on the device.  pairs, groups: entered on this
// level; cand, border: child pairs formed and borderline cases when it was made;
// steps: quad steps (of the leaf level's quads, in the entry of the leaf level), half:
// those of them whose kept pairs lie in one column of the quad.
struct LevelInfo {
  unsigned long long pairs, groups, cand, border, steps, half;
};

// One level step's view.
struct StepDev {
  const LevelInfo* in;  // this level
  LevelInfo* out;       // the next
  const int64_t* gstart;
  const uint32_t* gcode;
  const int32_t *ta, *tb;
  const NodeRec *recA, *recB;
  const double4 *normA, *normB;
  uint8_t* mask;
  uint64_t* packed;      // 4 per group
  uint64_t* tiles;       // per tile of groups: sum of packed
  uint32_t* tile_steps;  // leaf step: quad steps
  unsigned* ticket;      // blocks that have counted
  // leaf step: the sizes of all levels and the operands' node counts for the host
  const uint64_t* info;  // the LevelInfo entries as words
  const uint64_t *countA, *countB;
  uint64_t* host;        // pinned memory: levels (LevelInfo + 2 words)
  int levels;
  int32_t *ta2, *tb2;    // outputs
  uint32_t* gcode2;
  int64_t* gstart2;
  int32_t* quad;         // leaf step: the four children of each group
};

// Groups per tile: eight (one per warp of a block) while there are few tiles, so that
// a level of a thousand groups still spreads over the SMs (16 blocks and 28 us with 64
// groups per tile, n = 4096 lattice), else 64, as every tile adds up the tiles before it.
constexpr int kFewGroups = 8, kManyGroups = 64;
static int tile_groups(int64_t groups) { return groups <= (1 << 14) ? kFewGroups : kManyGroups; }

// Number of quad steps in a pair's mask: its two child k-indices, each a step if
// any of the four child groups keeps it.
__device__ __forceinline__ unsigned mask_steps(unsigned m) { return ((m & 0x55u) != 0) + ((m & 0xAAu) != 0); }
// Those of them whose kept child groups lie in one column (children 0, 2 or 1, 3).
__device__ __forceinline__ unsigned mask_half_steps(unsigned m) {
  return (((m & 0x11u) != 0) != ((m & 0x44u) != 0)) + (((m & 0x22u) != 0) != ((m & 0x88u) != 0));
}

template <bool LEAF>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
    task_count_kernel(const __grid_constant__ StepDev S, int tg, TauScreen sc, double tau, int test) {
  __shared__ unsigned long long s_tile, s_cand, s_border, s_half;
  __shared__ unsigned s_steps, s_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t G = (int64_t)S.in->groups;
  const int64_t ntiles = (G + tg - 1) / tg;
  long long cand = 0, border = 0;
  unsigned half = 0;
  if (threadIdx.x == 0) s_cand = s_border = s_half = 0;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    if (threadIdx.x == 0) {
      s_tile = 0;
      s_steps = 0;
    }
    __syncthreads();
    uint64_t sum = 0;
    unsigned steps = 0;
    for (int64_t g = tile * tg + warp; g < min(G, (tile + 1) * tg); g += kWarpsPerBlock) {
      const int64_t q0 = S.gstart[g], q1 = S.gstart[g + 1];
      uint64_t cnt01 = 0, cnt23 = 0;  // kept pairs of the four children, two per word
      for (int64_t q = q0 + lane; q < q1; q += 32) {
        const int32_t ia = S.ta[q], ib = S.tb[q];
        const unsigned m = child_mask(S.recA[ia], S.recB[ib], S.normA + ia, S.normB + ib, sc, tau, test, LEAF, &cand,
                                      &border);
        S.mask[q] = (uint8_t)m;
        cnt01 += (uint64_t)__popc(m & 3u) | ((uint64_t)__popc((m >> 2) & 3u) << 32);
        cnt23 += (uint64_t)__popc((m >> 4) & 3u) | ((uint64_t)__popc((m >> 6) & 3u) << 32);
        if (LEAF) {
          steps += mask_steps(m);
          half += mask_half_steps(m);
        }
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        cnt01 += __shfl_xor_sync(0xffffffffu, cnt01, off);
        cnt23 += __shfl_xor_sync(0xffffffffu, cnt23, off);
      }
      if (lane < 4) {
        const uint64_t c = ((lane < 2 ? cnt01 : cnt23) >> (32 * (lane & 1))) & 0xffffffffu;
        const uint64_t p = c | ((uint64_t)(c > 0) << 36);
        S.packed[4 * g + lane] = p;
        sum += p;
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      sum += __shfl_xor_sync(0xffffffffu, sum, off);
      if (LEAF) steps += __shfl_xor_sync(0xffffffffu, steps, off);
    }
    if (lane == 0) {
      atomicAdd(&s_tile, (unsigned long long)sum);
      if (LEAF) atomicAdd(&s_steps, steps);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      S.tiles[tile] = s_tile;
      if (LEAF) S.tile_steps[tile] = s_steps;
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    cand += __shfl_xor_sync(0xffffffffu, cand, off);
    border += __shfl_xor_sync(0xffffffffu, border, off);
    if (LEAF) half += __shfl_xor_sync(0xffffffffu, half, off);
  }
  __syncthreads();
  if (lane == 0) {
    if (cand) atomicAdd(&s_cand, (unsigned long long)cand);
    if (border) atomicAdd(&s_border, (unsigned long long)border);
    if (half) atomicAdd(&s_half, (unsigned long long)half);
  }
  __syncthreads();
  // one atomic per block; the block that is last to finish adds up the tiles
  if (threadIdx.x == 0) {
    if (s_cand) atomicAdd(&S.out->cand, s_cand);
    if (s_border) atomicAdd(&S.out->border, s_border);
    if (s_half) atomicAdd(&S.out->half, s_half);
    __threadfence();
    s_last = atomicAdd(S.ticket, 1u) == gridDim.x - 1;
    s_tile = 0;
    s_cand = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  unsigned long long sum = 0, steps = 0;
  for (int64_t i = threadIdx.x; i < ntiles; i += blockDim.x) {
    sum += __ldcg(S.tiles + i);
    if (LEAF) steps += __ldcg(S.tile_steps + i);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    sum += __shfl_xor_sync(0xffffffffu, sum, off);
    steps += __shfl_xor_sync(0xffffffffu, steps, off);
  }
  if (lane == 0) {
    atomicAdd(&s_tile, sum);
    atomicAdd(&s_cand, steps);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    S.out->pairs = s_tile & kCountMask;
    S.out->groups = s_tile >> 36;
    S.out->steps = s_cand;
  }
  if (!LEAF) return;
  // straight to the host's memory: three copies would take 3 us each
  __syncthreads();
  const int words = S.levels * (int)(sizeof(LevelInfo) / sizeof(uint64_t));
  for (int i = threadIdx.x; i < words + 2 * S.levels; i += blockDim.x)
    S.host[i] = i < words               ? __ldcg(S.info + i)
                : i < words + S.levels ? S.countA[i - words]
                                       : S.countB[i - words - S.levels];
}

// What the quad steps need beside the pairs (leaf step of the tensor-core forms).
struct StepsDev {
  QuadStep* steps;        // null: no quad steps
  int64_t* qstart;        // per group, and the total
  const int32_t *expA, *expB, *bmap;
};

// Prefix sum over the block's 256 threads (exclusive); *total the sum.
__device__ __forceinline__ uint64_t block_prefix_u64(uint64_t v, uint64_t* total) {
  __shared__ uint64_t ws[kWarpsPerBlock];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint64_t x = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) ws[warp] = x;
  __syncthreads();
  uint64_t before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kWarpsPerBlock; ++w) {
    if (w < warp) before += ws[w];
    all += ws[w];
  }
  __syncthreads();
  *total = all;
  return before + x - v;
}

template <bool LEAF>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
    task_write_kernel(const __grid_constant__ StepDev S, int tg, const __grid_constant__ StepsDev Q) {
  static_assert(kManyGroups * 4 == kWarpsPerBlock * 32, "at most one child group of a tile per thread");
  __shared__ uint64_t s_off[kManyGroups * 4];
  __shared__ unsigned long long s_base, s_sbase;
  __shared__ unsigned s_step[kManyGroups];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t G = (int64_t)S.in->groups;
  const int64_t ntiles = (G + tg - 1) / tg;
  const bool want_steps = LEAF && Q.steps != nullptr;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    S.gstart2[S.out->groups] = (int64_t)S.out->pairs;
    if (want_steps) Q.qstart[G] = (int64_t)S.out->steps;
  }
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    if (threadIdx.x == 0) s_base = s_sbase = 0;
    __syncthreads();
    unsigned long long v = 0, w = 0;
    for (int64_t i = threadIdx.x; i < tile; i += blockDim.x) {
      v += S.tiles[i];
      if (want_steps) w += S.tile_steps[i];
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      v += __shfl_xor_sync(0xffffffffu, v, off);
      w += __shfl_xor_sync(0xffffffffu, w, off);
    }
    if (lane == 0) {
      if (v) atomicAdd(&s_base, v);
      if (w) atomicAdd(&s_sbase, w);
    }
    const int64_t g0 = tile * tg;
    const int64_t ge = min(G, g0 + tg);
    if (want_steps) {  // steps of each group of the tile
      for (int64_t g = g0 + warp; g < ge; g += kWarpsPerBlock) {
        unsigned n = 0;
        for (int64_t q = S.gstart[g] + lane; q < S.gstart[g + 1]; q += 32) n += mask_steps(S.mask[q]);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) n += __shfl_xor_sync(0xffffffffu, n, off);
        if (lane == 0) s_step[g - g0] = n;
      }
    }
    __syncthreads();
    // offset (low 36 bits) and index among the non-empty ones of every child group
    const int64_t gt = g0 + (threadIdx.x >> 2);
    const uint64_t p = gt < ge ? S.packed[4 * g0 + threadIdx.x] : 0;
    uint64_t total;
    const uint64_t off = s_base + block_prefix_u64(p, &total);
    s_off[threadIdx.x] = off;
    if (gt < ge) {
      const int64_t gid = (int64_t)(off >> 36);
      const bool present = (p & kCountMask) != 0;
      if (present) {
        S.gcode2[gid] = 4u * S.gcode[gt] + (threadIdx.x & 3u);
        S.gstart2[gid] = (int64_t)(off & kCountMask);
      }
      if (LEAF) S.quad[4 * gt + (threadIdx.x & 3)] = present ? (int32_t)gid : -1;
    }
    if (want_steps) {
      const uint64_t mine = threadIdx.x < ge - g0 ? s_step[threadIdx.x] : 0;
      const uint64_t so = s_sbase + block_prefix_u64(mine, &total);
      if (threadIdx.x < ge - g0) Q.qstart[g0 + threadIdx.x] = (int64_t)so;
    }
    __syncthreads();  // s_off and this block's qstart entries
    for (int64_t g = g0 + warp; g < ge; g += kWarpsPerBlock) {
      const int64_t q0 = S.gstart[g], q1 = S.gstart[g + 1];
      int64_t base[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) base[c] = (int64_t)(s_off[4 * (g - g0) + c] & kCountMask);
      int64_t sbase = want_steps ? Q.qstart[g] : 0;
      for (int64_t qb = q0; qb < q1; qb += 32) {
        const int64_t q = qb + lane;
        const unsigned m = q < q1 ? S.mask[q] : 0u;
        int4 ca = make_int4(-1, -1, -1, -1), cb = ca;
        if (m) {
          ca = rec_children(S.recA[S.ta[q]]);
          cb = rec_children(S.recB[S.tb[q]]);
        }
        const unsigned lt = (1u << lane) - 1u;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const unsigned bits = (m >> (2 * c)) & 3u;
          // warp ballots compact the kept children: a lane's entries follow
          // every kept child of the lanes before it (k-child 0, then 1)
          const unsigned b0 = __ballot_sync(0xffffffffu, bits & 1u), b1 = __ballot_sync(0xffffffffu, bits & 2u);
          int64_t pos = base[c] + __popc(b0 & lt) + __popc(b1 & lt);
          const int ci = c >> 1, cj = c & 1;
          if (bits & 1u) {
            S.ta2[pos] = comp4(ca, 2 * ci + 0);
            S.tb2[pos] = comp4(cb, 0 + cj);
            ++pos;
          }
          if (bits & 2u) {
            S.ta2[pos] = comp4(ca, 2 * ci + 1);
            S.tb2[pos] = comp4(cb, 2 + cj);
          }
          base[c] += __popc(b0) + __popc(b1);
        }
        if (want_steps) {
          const unsigned b0 = __ballot_sync(0xffffffffu, m & 0x55u), b1 = __ballot_sync(0xffffffffu, m & 0xAAu);
          int64_t pos = sbase + __popc(b0 & lt) + __popc(b1 & lt);
          sbase += __popc(b0) + __popc(b1);
#pragma unroll
          for (int ck = 0; ck < 2; ++ck) {
            const unsigned has = (m >> ck) & 0x55u;  // bit 2 c: child c keeps k-child ck
            if (!has) continue;
            // children 0/1 share the A leaf of row half 0, 2/3 that of half 1; 0/2 and 1/3 share B leaves
            QuadStep st;
            st.a[0] = has & 0x05u ? comp4(ca, ck) : -1;
            st.a[1] = has & 0x50u ? comp4(ca, 2 + ck) : -1;
            st.b[0] = has & 0x11u ? comp4(cb, 2 * ck) : -1;
            st.b[1] = has & 0x44u ? comp4(cb, 2 * ck + 1) : -1;
            if (Q.bmap) {
              if (st.b[0] >= 0) st.b[0] = Q.bmap[st.b[0]];
              if (st.b[1] >= 0) st.b[1] = Q.bmap[st.b[1]];
            }
            // 2^-(eA + eB) as a product of two normal powers of two (|e| <= 120)
            float fa[2], fb[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              fa[h] = st.a[h] >= 0 ? __int_as_float((127 - Q.expA[st.a[h]]) << 23) : 0.f;
              fb[h] = st.b[h] >= 0 ? __int_as_float((127 - Q.expB[st.b[h]]) << 23) : 0.f;
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) st.scale[c] = has & (1u << (2 * c)) ? fa[c >> 1] * fb[c & 1] : 0.f;
            Q.steps[pos++] = st;
          }
        }
      }
    }
    __syncthreads();  // the shared words are reused by the next tile
  }
}

// The first `steps` level steps (at most four: 8^3 pairs, 4^3 groups at the last)
// by one block, from the root pair; the last one's pairs and groups go to memory.  (A
// fifth step of up to 4096 pairs takes one SM 25 us, two tiled launches 15.)  One block
// lives on latency: the node records of all its levels are fetched at once, one warp
// takes the prefix of a step, and 32 warps share the groups.  Four steps 13 us
// (15.2 with a record's fetch in every step, a prefix over the block and 16 warps).
constexpr int kTopSteps = 4;
constexpr int kTopThreads = 1024;
constexpr int kTopPairs = 512, kTopGroups = 64;
constexpr int kTopNodes = 1 + 4 + 16 + 64;  // on the levels the steps start from
__device__ __forceinline__ int top_node(int t) { return ((1 << 2 * t) - 1) / 3; }  // level t's first of them
struct TopDev {
  const uint64_t *countA, *countB;  // nodes per level
  const NodeRec *recA[kTopSteps], *recB[kTopSteps];
  const double4 *normA[kTopSteps], *normB[kTopSteps];
  LevelInfo* lv;  // level t's entry at lv[t]
  int32_t *ta, *tb;
  uint32_t* gcode;
  int64_t* gstart;
};
struct TopShared {
  int32_t ta[2][kTopPairs], tb[2][kTopPairs];
  uint8_t mask[kTopPairs];
  NodeRec recA[kTopNodes], recB[kTopNodes];
  uint32_t cnt[4 * kTopGroups], off[4 * kTopGroups];  // off: prefix of cnt | (cnt > 0) << 20
  uint32_t gcode[2][kTopGroups];
  uint32_t gstart[2][kTopGroups + 1];
  uint32_t total;
  unsigned cand, border;
};

__global__ void __launch_bounds__(kTopThreads)
    task_top_kernel(const __grid_constant__ TopDev T, int steps, TauScreen sc, double tau, int test) {
  __shared__ TopShared s;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int Q = *T.countA > 0 && *T.countB > 0 ? 1 : 0, G = Q;  // the root pair is entered
  {
    const int i = (int)threadIdx.x & 127;
    const int t = i < 1 ? 0 : i < 5 ? 1 : i < 21 ? 2 : 3, m = i - top_node(t);
    if (i < kTopNodes && t < steps) {
      if (threadIdx.x < 128) {
        if (m < (int64_t)T.countA[t]) s.recA[i] = T.recA[t][m];
      } else if (threadIdx.x < 256) {
        if (m < (int64_t)T.countB[t]) s.recB[i] = T.recB[t][m];
      }
    }
  }
  if (threadIdx.x == 0) {
    s.ta[0][0] = s.tb[0][0] = 0;
    s.gcode[0][0] = 0;
    s.gstart[0][0] = 0;
    s.gstart[0][1] = 1;
    T.lv[0].pairs = T.lv[0].groups = (unsigned long long)Q;
  }
  for (int t = 0; t < steps; ++t) {
    const int cur = t & 1, nxt = cur ^ 1;
    const bool out = t + 1 == steps;
    const NodeRec *recA = s.recA + top_node(t), *recB = s.recB + top_node(t);
    if (threadIdx.x == 0) s.cand = s.border = 0;
    __syncthreads();
    // the children of every pair
    long long cand = 0, border = 0;
    for (int q = threadIdx.x; q < Q; q += kTopThreads) {
      const int32_t ia = s.ta[cur][q], ib = s.tb[cur][q];
      s.mask[q] = (uint8_t)child_mask(recA[ia], recB[ib], T.normA[t] + ia, T.normB[t] + ib, sc, tau, test,
                                      false, &cand, &border);
    }
    cand += __shfl_xor_sync(0xffffffffu, cand, 16);
    cand += __shfl_xor_sync(0xffffffffu, cand, 8);
    cand += __shfl_xor_sync(0xffffffffu, cand, 4);
    cand += __shfl_xor_sync(0xffffffffu, cand, 2);
    cand += __shfl_xor_sync(0xffffffffu, cand, 1);
    if (lane == 0 && cand) atomicAdd(&s.cand, (unsigned)cand);
    __syncthreads();
    // kept pairs of every child group
    for (int g = warp; g < G; g += kTopThreads / 32) {
      unsigned c01 = 0, c23 = 0;
      for (int q = (int)s.gstart[cur][g] + lane; q < (int)s.gstart[cur][g + 1]; q += 32) {
        const unsigned m = s.mask[q];
        c01 += (unsigned)__popc(m & 3u) | ((unsigned)__popc((m >> 2) & 3u) << 16);
        c23 += (unsigned)__popc((m >> 4) & 3u) | ((unsigned)__popc((m >> 6) & 3u) << 16);
      }
      c01 = __reduce_add_sync(0xffffffffu, c01);
      c23 = __reduce_add_sync(0xffffffffu, c23);
      if (lane < 4) s.cnt[4 * g + lane] = ((lane < 2 ? c01 : c23) >> (16 * (lane & 1))) & 0xffffu;
    }
    __syncthreads();
    // offsets (low 20 bits) and indexes among the non-empty ones
    if (warp == 0) {
      constexpr int kPer = 4 * kTopGroups / 32;
      uint32_t v[kPer], sum = 0;
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        const int i = kPer * lane + k;
        const uint32_t c = i < 4 * G ? s.cnt[i] : 0;
        v[k] = sum;
        sum += c | ((uint32_t)(c > 0) << 20);
      }
      uint32_t x = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
#pragma unroll
      for (int k = 0; k < kPer; ++k) s.off[kPer * lane + k] = x - sum + v[k];
      if (lane == 31) s.total = x;
    }
    __syncthreads();
    const uint32_t total = s.total;
    const int Q2 = (int)(total & 0xfffffu), G2 = (int)(total >> 20);
    const int i = threadIdx.x;
    if (i < 4 * G) {
      const uint32_t off = s.off[i];
      if (s.cnt[i]) {
        const uint32_t gid = off >> 20, code = 4u * s.gcode[cur][i >> 2] + (uint32_t)(i & 3);
        if (out) {
          T.gcode[gid] = code;
          T.gstart[gid] = (int64_t)(off & 0xfffffu);
        } else {
          s.gcode[nxt][gid] = code;
          s.gstart[nxt][gid] = off & 0xfffffu;
        }
      }
    }
    if (threadIdx.x == 0) {
      if (out)
        T.gstart[G2] = Q2;
      else
        s.gstart[nxt][G2] = (uint32_t)Q2;
      LevelInfo& lv = T.lv[t + 1];
      lv.pairs = (unsigned long long)Q2;
      lv.groups = (unsigned long long)G2;
      lv.cand = s.cand;
    }
    int32_t* ta2 = out ? T.ta : s.ta[nxt];
    int32_t* tb2 = out ? T.tb : s.tb[nxt];
    for (int g = warp; g < G; g += kTopThreads / 32) {
      int base[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) base[k] = (int)(s.off[4 * g + k] & 0xfffffu);
      const int q1 = (int)s.gstart[cur][g + 1];
      for (int qb = (int)s.gstart[cur][g]; qb < q1; qb += 32) {
        const int q = qb + lane;
        const unsigned m = q < q1 ? s.mask[q] : 0u;
        int4 ca = make_int4(-1, -1, -1, -1), cb = ca;
        if (m) {
          ca = rec_children(recA[s.ta[cur][q]]);
          cb = rec_children(recB[s.tb[cur][q]]);
        }
        const unsigned lt = (1u << lane) - 1u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const unsigned bits = (m >> (2 * k)) & 3u;
          const unsigned b0 = __ballot_sync(0xffffffffu, bits & 1u), b1 = __ballot_sync(0xffffffffu, bits & 2u);
          int pos = base[k] + __popc(b0 & lt) + __popc(b1 & lt);
          const int ci = k >> 1, cj = k & 1;
          if (bits & 1u) {
            ta2[pos] = comp4(ca, 2 * ci + 0);
            tb2[pos] = comp4(cb, 0 + cj);
            ++pos;
          }
          if (bits & 2u) {
            ta2[pos] = comp4(ca, 2 * ci + 1);
            tb2[pos] = comp4(cb, 2 + cj);
          }
          base[k] += __popc(b0) + __popc(b1);
        }
      }
    }
    Q = Q2;
    G = G2;
  }
}

// A single leaf on each side: the root pair is the only leaf pair and takes the leaf
// test.  One output leaf, one quad holding only child 0.
__global__ void root_test_kernel(const uint64_t* nA, const double* sqA, const uint64_t* nB, const double* sqB, double tau,
                                 int test, LevelInfo* lv) {
  if (threadIdx.x != 0) return;
  const bool both = *nA > 0 && *nB > 0;
  const double prod = both ? __dmul_rn(sqrt(sqA[0]), sqrt(sqB[0])) : 0.0;
  const bool keep = both && (!test || prod >= tau);
  lv[0].pairs = lv[0].groups = lv[0].steps = lv[0].half = keep ? 1 : 0;
  lv[0].border = both && test && fabs(prod - tau) <= 1e-12 * tau ? 1 : 0;
}
__global__ void root_list_kernel(uint32_t* gcode, int64_t* gstart, int32_t* ta, int32_t* tb, int32_t* quads, StepsDev Q) {
  if (threadIdx.x != 0) return;
  gcode[0] = 0;
  gstart[0] = 0;
  gstart[1] = 1;
  ta[0] = tb[0] = 0;
  for (int c = 0; c < 4; ++c) quads[c] = c == 0 ? 0 : -1;
  if (Q.steps) {
    QuadStep st;
    st.a[0] = 0;
    st.b[0] = Q.bmap ? Q.bmap[0] : 0;
    st.a[1] = st.b[1] = -1;
    st.scale[0] = __int_as_float((127 - Q.expA[0]) << 23) * __int_as_float((127 - Q.expB[st.b[0]]) << 23);
    st.scale[1] = st.scale[2] = st.scale[3] = 0.f;
    Q.steps[0] = st;
    Q.qstart[0] = 0;
    Q.qstart[1] = 1;
  }
}

static unsigned warps_grid(spamm_ctx ctx, int64_t items) {
  int64_t g = (items + kWarpsPerBlock - 1) / kWarpsPerBlock;
  int64_t cap = (int64_t)ctx->num_sms * 16;
  if (g > cap) g = cap;
  return (unsigned)(g < 1 ? 1 : g);
}
static unsigned tiles_grid(spamm_ctx ctx, int64_t groups, int tg) {
  const int64_t g = (groups + tg - 1) / tg, cap = (int64_t)ctx->num_sms * 64;
  return (unsigned)(g < 1 ? 1 : (g > cap ? cap : g));
}

// Upper bounds on the next level's sizes below which the host does not wait
// for the exact counts (buffers are allocated at the bound instead).  The
// leaf level always waits: its arrays are the plan's task list, kept for the
// leaf products.
constexpr int64_t kPairsNoSync = 1ll << 22;
constexpr int64_t kGroupsNoSync = 1ll << 20;

// What task_begin leaves for task_finish.
struct TaskBuild {
  spamm_mat A = nullptr, B = nullptr;
  StepDev leaf{};         // the leaf step, counted
  int tg = kManyGroups;   // its groups per tile
  std::vector<BufP> keep; // its buffers
  LevelInfo* lv = nullptr;
};

std::shared_ptr<TaskBuild> task_begin(spamm_mat A, spamm_mat B, double tau, int test_norms, spamm_ctx ctx, TaskList* T) {
  auto tb = std::make_shared<TaskBuild>();
  tb->A = A;
  tb->B = B;
  const int L = A->L;
  uint64_t* host = static_cast<uint64_t*>(ctx->h_pinned);
  auto finish_counts = [&](LevelInfo* dlv, bool written) {
    // the level sizes and both operands' node counts, one wait (written: by the leaf step's kernel)
    LevelInfo* hl = reinterpret_cast<LevelInfo*>(host);
    uint64_t* ha = reinterpret_cast<uint64_t*>(hl + (L + 1));
    uint64_t* hb = ha + (L + 1);
    static_assert((SPAMM_MAX_LEVELS) * (sizeof(LevelInfo) + 2 * sizeof(uint64_t)) <= 4096, "fits the pinned page");
    if (dlv && !written)
      CK(cudaMemcpyAsync(hl, dlv, (L + 1) * sizeof(LevelInfo), cudaMemcpyDeviceToHost, ctx->stream));
    const bool pa = A->pending, pb = B != A && B->pending;
    if (pa && !written) tree_counts_async(ctx, A, ha);
    if (pb && !written) tree_counts_async(ctx, B, hb);
    if (dlv || pa || pb) CK(cudaStreamSynchronize(ctx->stream));
    if (pa) tree_set_counts(A, ha);
    if (pb) tree_set_counts(B, hb);
    if (!dlv) return;
    for (int t = L > 0 ? 1 : 0; t <= L; ++t) {
      if (L > 0) {
        T->n_candidates[t] = (int64_t)hl[t].cand;
        T->n_kept_level[t] = (int64_t)hl[t].pairs;
      }
    }
    T->n_borderline = (int64_t)hl[L].border;
    T->ngroups = (int64_t)hl[L].groups;
    T->ntasks = (int64_t)hl[L].pairs;
    T->nquads = L > 0 ? (int64_t)hl[L - 1].groups : T->ngroups;
    T->nsteps = (int64_t)hl[L].steps;
    T->nhalf = (int64_t)hl[L].half;
  };
  if (!A->dcount || !B->dcount) {  // an operand without leaves
    finish_counts(nullptr, false);
    return tb;
  }
  const int nlev = L + 1;
  BufP info = alloc_bytes(ctx, nlev * (sizeof(LevelInfo) + sizeof(unsigned)));
  LevelInfo* lv = static_cast<LevelInfo*>(info->p);
  unsigned* tickets = reinterpret_cast<unsigned*>(lv + nlev);
  tb->keep.push_back(info);
  tb->lv = lv;
  const size_t clear = nlev * (sizeof(LevelInfo) + sizeof(unsigned));
  if (L == 0) {
    CK(cudaMemsetAsync(lv, 0, clear, ctx->stream));
    root_test_kernel<<<1, 32, 0, ctx->stream>>>(P<uint64_t>(A->dcount), P<double>(A->lv[0].sq), P<uint64_t>(B->dcount),
                                                P<double>(B->lv[0].sq), tau, test_norms, lv);
    CK_LAUNCH("root_test_kernel");
    finish_counts(lv, false);
    return tb;
  }
  const TauScreen screen = make_screen(tau);
  // records of every level of both operands
  RecTable tab;
  NodeRec *recA[SPAMM_MAX_LEVELS], *recB[SPAMM_MAX_LEVELS];
  double4 *normA[SPAMM_MAX_LEVELS], *normB[SPAMM_MAX_LEVELS];
  {
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    size_t bytes = 0;
    int64_t most = 1;
    for (spamm_mat m : {A, B})
      for (int t = 0; t < L && (m == A || B != A); ++t) {
        bytes += up(m->lv[t].count * sizeof(NodeRec)) + up(m->lv[t].count * sizeof(double4));
        most = m->lv[t].count > most ? m->lv[t].count : most;
      }
    BufP recs = alloc_bytes(ctx, bytes);
    tb->keep.push_back(recs);
    uint8_t* p = static_cast<uint8_t*>(recs->p);
    int rows = 0;
    for (int side = 0; side < (B == A ? 1 : 2); ++side) {
      spamm_mat m = side ? B : A;
      for (int t = 0; t < L; ++t) {
        (side ? recB : recA)[t] = reinterpret_cast<NodeRec*>(p);
        p += up(m->lv[t].count * sizeof(NodeRec));
        (side ? normB : normA)[t] = reinterpret_cast<double4*>(p);
        p += up(m->lv[t].count * sizeof(double4));
        tab.lv[rows++] = {P<int4>(m->lv[t].child), P<double>(m->lv[t + 1].sq), P<uint64_t>(m->dcount) + t,
                          (side ? recB : recA)[t], (side ? normB : normA)[t]};
      }
    }
    if (B == A)
      for (int t = 0; t < L; ++t) {
        recB[t] = recA[t];
        normB[t] = normA[t];
      }
    int64_t g = (most + 255) / 256;
    const int64_t cap = (int64_t)ctx->num_sms * 8;
    if (g > cap) g = cap;
    node_rec_kernel<<<dim3((unsigned)g, (unsigned)rows), 256, 0, ctx->stream>>>(tab, reinterpret_cast<unsigned*>(lv),
                                                                                  (int)(clear / sizeof(unsigned)), ctx->d_err);
    CK_LAUNCH("node_rec_kernel");
  }
  // the first steps in one block
  const int top = L - 1 < kTopSteps ? L - 1 : kTopSteps;
  int64_t Q = 1, G = 1;  // capacities of the current level
  for (int t = 0; t < top; ++t) {
    Q *= 8;
    G *= 4;
  }
  BufP ta = alloc_n<int32_t>(ctx, 2 * Q), gc = alloc_bytes(ctx, (G + 1) * sizeof(int64_t) + G * sizeof(uint32_t));
  int32_t *dta = P<int32_t>(ta), *dtb = dta + Q;
  int64_t* dgs = static_cast<int64_t*>(gc->p);
  uint32_t* dgc = reinterpret_cast<uint32_t*>(dgs + G + 1);
  if (top == 0) {  // only the leaf step: the root pair itself
    CK(cudaMemsetAsync(dta, 0, 2 * sizeof(int32_t), ctx->stream));
  }
  {
    TopDev T0{};
    T0.countA = P<uint64_t>(A->dcount);
    T0.countB = P<uint64_t>(B->dcount);
    for (int t = 0; t < top; ++t) {
      T0.recA[t] = recA[t];
      T0.recB[t] = recB[t];
      T0.normA[t] = normA[t];
      T0.normB[t] = normB[t];
    }
    T0.lv = lv;
    T0.ta = dta;
    T0.tb = dtb;
    T0.gcode = dgc;
    T0.gstart = dgs;
    task_top_kernel<<<1, kTopThreads, 0, ctx->stream>>>(T0, top, screen, tau, test_norms);
    CK_LAUNCH("task_top_kernel");
    if (top == 0) {
      const int64_t h[2] = {0, 1};
      CK(cudaMemcpyAsync(dgs, h, sizeof h, cudaMemcpyHostToDevice, ctx->stream));
      CK(cudaMemsetAsync(dgc, 0, sizeof(uint32_t), ctx->stream));
    }
  }
  for (int t = top; t < L; ++t) {
    const bool leaf = t + 1 == L;
    const int tg = tile_groups(G);
    const int64_t ntiles = (G + tg - 1) / tg;
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t mb = up(Q), pb = up(4 * G * sizeof(uint64_t)), tbts = up(ntiles * sizeof(uint64_t));
    BufP work = alloc_bytes(ctx, mb + pb + tbts + ntiles * sizeof(uint32_t));
    uint8_t* w = static_cast<uint8_t*>(work->p);
    StepDev S{};
    S.in = lv + t;
    S.out = lv + t + 1;
    S.gstart = dgs;
    S.gcode = dgc;
    S.ta = dta;
    S.tb = dtb;
    S.recA = recA[t];
    S.recB = recB[t];
    S.normA = normA[t];
    S.normB = normB[t];
    S.mask = w;
    S.packed = reinterpret_cast<uint64_t*>(w + mb);
    S.tiles = reinterpret_cast<uint64_t*>(w + mb + pb);
    S.tile_steps = reinterpret_cast<uint32_t*>(w + mb + pb + tbts);
    S.ticket = tickets + t;
    S.info = reinterpret_cast<const uint64_t*>(lv);
    S.countA = P<uint64_t>(A->dcount);
    S.countB = P<uint64_t>(B->dcount);
    S.host = host;
    S.levels = nlev;
    if (leaf)
      task_count_kernel<true><<<tiles_grid(ctx, G, tg), kWarpsPerBlock * 32, 0, ctx->stream>>>(S, tg, screen, tau,
                                                                                              test_norms);
    else
      task_count_kernel<false><<<tiles_grid(ctx, G, tg), kWarpsPerBlock * 32, 0, ctx->stream>>>(S, tg, screen, tau,
                                                                                               test_norms);
    CK_LAUNCH("task_count_kernel");
    if (leaf) {
      tb->leaf = S;
      tb->tg = tg;
      tb->keep.push_back(ta);
      tb->keep.push_back(gc);
      tb->keep.push_back(work);
      finish_counts(lv, true);
      break;
    }
    // capacities of the next level: exact after a wait, else the bounds 8 Q and 4 G
    int64_t Q2 = 8 * Q, G2 = 4 * G;
    if (Q2 > kPairsNoSync || G2 > kGroupsNoSync) {
      CK(cudaMemcpyAsync(host, lv + t + 1, sizeof(LevelInfo), cudaMemcpyDeviceToHost, ctx->stream));
      CK(cudaStreamSynchronize(ctx->stream));
      Q2 = (int64_t)reinterpret_cast<LevelInfo*>(host)->pairs;
      G2 = (int64_t)reinterpret_cast<LevelInfo*>(host)->groups;
    }
    BufP ta2 = alloc_n<int32_t>(ctx, 2 * Q2), gc2 = alloc_bytes(ctx, (G2 + 1) * sizeof(int64_t) + G2 * sizeof(uint32_t));
    S.ta2 = P<int32_t>(ta2);
    S.tb2 = S.ta2 + Q2;
    S.gstart2 = static_cast<int64_t*>(gc2->p);
    S.gcode2 = reinterpret_cast<uint32_t*>(S.gstart2 + G2 + 1);
    task_write_kernel<false><<<tiles_grid(ctx, G, tg), kWarpsPerBlock * 32, 0, ctx->stream>>>(S, tg, StepsDev{});
    CK_LAUNCH("task_write_kernel");
    ta = ta2;
    gc = gc2;
    dta = S.ta2;
    dtb = S.tb2;
    dgs = S.gstart2;
    dgc = S.gcode2;
    Q = Q2;
    G = G2;
  }
  return tb;
}

void task_finish(spamm_ctx ctx, TaskBuild* tb, TaskList* T, const StepExps* exps, BufP* qstart, BufP* qsteps) {
  T->gstart = alloc_n<int64_t>(ctx, T->ngroups + 1);
  const int64_t nq = T->ngroups > 0 ? T->nquads : 0;
  StepsDev Q{};
  if (exps) {
    *qstart = alloc_n<int64_t>(ctx, nq + 1);
    *qsteps = alloc_n<QuadStep>(ctx, T->nsteps);
    if (T->ngroups == 0) CK(cudaMemsetAsync(P<int64_t>(*qstart), 0, sizeof(int64_t), ctx->stream));
    Q.steps = P<QuadStep>(*qsteps);
    Q.qstart = P<int64_t>(*qstart);
    Q.expA = exps->expA;
    Q.expB = exps->expB;
    Q.bmap = exps->bmap;
  }
  if (T->ngroups == 0) {
    T->nquads = 0;
    CK(cudaMemsetAsync(P<int64_t>(T->gstart), 0, sizeof(int64_t), ctx->stream));
    return;
  }
  T->gcode = alloc_n<uint32_t>(ctx, T->ngroups);
  T->ta = alloc_n<int32_t>(ctx, T->ntasks);
  T->tb = alloc_n<int32_t>(ctx, T->ntasks);
  T->quads = alloc_n<int32_t>(ctx, 4 * T->nquads);
  if (tb->A->L == 0) {
    root_list_kernel<<<1, 32, 0, ctx->stream>>>(P<uint32_t>(T->gcode), P<int64_t>(T->gstart), P<int32_t>(T->ta),
                                                P<int32_t>(T->tb), P<int32_t>(T->quads), Q);
    CK_LAUNCH("root_list_kernel");
    return;
  }
  StepDev S = tb->leaf;
  S.ta2 = P<int32_t>(T->ta);
  S.tb2 = P<int32_t>(T->tb);
  S.gcode2 = P<uint32_t>(T->gcode);
  S.gstart2 = P<int64_t>(T->gstart);
  S.quad = P<int32_t>(T->quads);
  task_write_kernel<true><<<tiles_grid(ctx, T->nquads, tb->tg), kWarpsPerBlock * 32, 0, ctx->stream>>>(S, tb->tg, Q);
  CK_LAUNCH("task_write_kernel");
}

// (i, k, j) of every task, for the parity hook.
__global__ void tasks_to_ikj_kernel(int64_t G, const int64_t* __restrict__ gstart, const uint32_t* __restrict__ gcode,
                                    const int32_t* __restrict__ ta, const uint32_t* __restrict__ codeA,
                                    int32_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < G; g += nw) {
    const int32_t i = (int32_t)code_row(gcode[g]), j = (int32_t)code_col(gcode[g]);
    for (int64_t q = gstart[g] + lane; q < gstart[g + 1]; q += 32) {
      out[3 * q + 0] = i;
      out[3 * q + 1] = (int32_t)code_col(codeA[ta[q]]);
      out[3 * q + 2] = j;
    }
  }
}

void tasks_to_ikj(spamm_ctx ctx, spamm_mat A, const TaskList& T, int32_t* d_out) {
  if (T.ngroups == 0) return;
  tasks_to_ikj_kernel<<<warps_grid(ctx, T.ngroups), kWarpsPerBlock * 32, 0, ctx->stream>>>(
      T.ngroups, P<int64_t>(T.gstart), P<uint32_t>(T.gcode), P<int32_t>(T.ta), P<uint32_t>(A->lv[A->L].code), d_out);
  CK_LAUNCH("tasks_to_ikj_kernel");
}

}  // namespace spamm
