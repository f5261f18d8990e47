// tree.cu -- quadtree structure: the leaf set kept from sorted candidates
// (truncation, builders), the levels above it and their squared norms.
//
// Every level is in Morton order: the kept leaves are a compaction of the
// candidates, and the parents of a level are its runs of equal code >> 2, a parent's
// children being consecutive nodes.  The squared norms follow over the parents (an
// FP64 addition keeps a quarter SM's pipe for 64 cycles whether one lane needs it or 32).
//
// Two forms.  Up to kTopNodes items one block of 1024 threads takes a whole tree in
// one launch, all levels' structure in one pass: truncating both operands of a 4096-row
// lattice (some 4000 leaves of 64 x 64 each, seven levels) is 12.5 us of kernel, where
// five launches per level took 360; up to kBoundNodes the block takes one piece of that
// size after the other.  Larger levels take two launches each, a count per tile of 1024 and the placing, where
// every tile adds up the counts before it, until the level is small enough for the rest;
// there the thread that sees the first child of a run also sees the others (at most
// three nodes further on), so it writes the parent's code and child links at once.
// Node counts stay on the device; the host reads them once.
#include <cmath>
#include <cstring>

#include "internal.cuh"

namespace spamm {

namespace {

constexpr int kTopThreads = 1024;
constexpr int64_t kTopNodes = 4096;
constexpr int64_t kBoundNodes = 32768;  // one block's; up to here the leaf level is allocated for every candidate
constexpr int kTileThreads = 256;
constexpr int kTilePer = 4;
constexpr int64_t kTile = kTileThreads * kTilePer;
// Up to this many tiles every tile adds up the counts before it itself (at most
// four loads per thread); more are scanned first.
constexpr int64_t kTilesSummed = 1024;

// One tree to build.  rule 0: level t0 is there (count[t0] nodes); 1: leaf q is kept iff
// keep[q]; 2: iff !(sq[q] < smin); 3: the leaf level is there (n nodes).  Levels t0 - 1 .. 0
// are built.
struct TreeDev {
  int64_t n = 0;                   // candidates
  const uint32_t* code = nullptr;  // null: candidate q has code q
  const double* sq = nullptr;
  const int64_t* slot = nullptr;   // null: candidate q has slot q
  const uint8_t* keep = nullptr;
  double smin = 0.0;
  int rule = 0;
  int L = 0, t0 = 0;
  uint64_t* count = nullptr;  // nodes per level
  uint64_t* host = nullptr;   // the same in pinned memory, for the host (null: not wanted)
  uint32_t* ocode[SPAMM_MAX_LEVELS] = {};
  double* osq[SPAMM_MAX_LEVELS] = {};  // null: no norms
  int4* ochild[SPAMM_MAX_LEVELS] = {};
  int64_t* oslot = nullptr;
};
struct TreePair {
  TreeDev t[2];
};

// !(sq < smin) for squared norms (no negative values: they order like their bits, NaN
// last), without an FP64 comparison.
__device__ __forceinline__ bool kept_norm(double sq, double smin) {
  return (uint64_t)__double_as_longlong(sq) >= (uint64_t)__double_as_longlong(smin);
}
__device__ __forceinline__ bool kept(const TreeDev& T, int64_t q) {
  return T.rule == 1 ? T.keep[q] != 0 : kept_norm(T.sq[q], T.smin);
}
__device__ __forceinline__ void place_leaf(const TreeDev& T, int64_t q, int64_t p) {
  T.ocode[T.L][p] = T.code ? T.code[q] : (uint32_t)q;
  T.osq[T.L][p] = T.sq[q];
  T.oslot[p] = T.slot ? T.slot[q] : q;
}
// Node q of a level of n nodes starts a parent.
__device__ __forceinline__ bool first_child(const uint32_t* code, int64_t q) {
  return q == 0 || (code[q] >> 2) != (code[q - 1] >> 2);
}
// Parent p (on level t - 1) whose first child is node q of level t (n nodes).
__device__ __forceinline__ void place_parent(const TreeDev& T, int t, int64_t n, int64_t q, int64_t p) {
  const uint32_t* code = T.ocode[t];
  const uint32_t up = code[q] >> 2;
  int ch[4] = {-1, -1, -1, -1};
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (q + i < n) {
      const uint32_t c = code[q + i];
      if ((c >> 2) == up) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if ((c & 3u) == (uint32_t)k) ch[k] = (int)(q + i);
      }
    }
  T.ocode[t - 1][p] = up;
  T.ochild[t - 1][p] = make_int4(ch[0], ch[1], ch[2], ch[3]);
}
// ||A^t||_F^2 = sum of the children's squared norms, added in the fixed order
// (0,0), (0,1), (1,0), (1,1) (Section 2).
__device__ __forceinline__ double child_sum(const int4& ch, const double* csq) {
  double s = ch.x >= 0 ? csq[ch.x] : 0.0;
  if (ch.y >= 0) s += csq[ch.y];
  if (ch.z >= 0) s += csq[ch.z];
  if (ch.w >= 0) s += csq[ch.w];
  return s;
}

// Parents p0 .. p1 - 1 of level t - 1, by the block.
__device__ __forceinline__ void sum_parents(const TreeDev& T, int t, int64_t p0, int64_t p1) {
  double* out = T.osq[t - 1];
  if (!out) return;
  for (int64_t p = p0 + threadIdx.x; p < p1; p += blockDim.x) out[p] = child_sum(T.ochild[t - 1][p], T.osq[t]);
}

// Exclusive prefix of v over the block's threads, the sum in *total.
template <int THREADS>
__device__ __forceinline__ uint32_t block_prefix(uint32_t v, uint32_t* total) {
  __shared__ uint32_t ws[THREADS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) ws[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < THREADS / 32 ? ws[lane] : 0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, w, off);
      if (lane >= off) w += y;
    }
    if (lane < THREADS / 32) ws[lane] = w;
  }
  __syncthreads();
  const uint32_t before = warp ? ws[warp - 1] : 0;
  *total = ws[THREADS / 32 - 1];
  __syncthreads();
  return before + x - v;
}

// The structure above level t0 in one pass over its nodes.  Node i starts a node on
// every level from first_level on, so its position on level t is the number of nodes up
// to i with first_level <= t: one ballot per 32 nodes and level, and a prefix over the
// warps' counts, for all levels at once.
__device__ __forceinline__ int first_level(uint32_t code, uint32_t prev, int64_t i, int t0) {
  return i == 0 ? 0 : t0 - (31 - __clz((int)((code ^ prev) | 1u))) / 2;
}
// What node i (code; first_level s) writes on the levels below t0, whose child links
// are empty (-1): its own and its ancestors' places in the links, its ancestors' codes.
// before(t): nodes of level t that start in earlier groups of 32.  Called by whole
// warps, lanes without a node with s = kNoNode; no level below the first on which no
// lane starts a node has anything to write (of 32 leaves of a filled tree three levels).
constexpr int kNoNode = 255;
template <class Before>
__device__ __forceinline__ void place_levels(const TreeDev& T, int i, uint32_t code, int s, Before before) {
  const unsigned upto = 0xFFFFFFFFu >> (31 - (threadIdx.x & 31));  // this lane and those before
  int below = i;  // the node's position one level further down
  for (int t = T.t0 - 1; t >= 0; --t) {
    const unsigned b = __ballot_sync(0xffffffffu, s <= t);
    const int p = before(t) + __popc(b & upto) - 1;
    if (s <= t + 1) {
      reinterpret_cast<int*>(T.ochild[t] + p)[code & 3u] = below;
      code >>= 2;
      below = p;
      if (s <= t) T.ocode[t][p] = code;
    }
    if (b == 0) break;
  }
}
// Squared norms of the levels `top` .. 0 (count[t] <= kTopNodes nodes) by one block, from
// those of level top + 1: level by level through `s` in place (a parent's position is
// never above its children's).  Four levels' links are on their way ahead, each in
// registers of its own (a copy would wait for its load).  A level of few nodes takes
// some 950 cycles, nearly all of them its three dependent FP64 additions.
template <class Child, class Sq>
__device__ __forceinline__ void block_norms(int top, const int* count, Child child, Sq sq, double* s) {
  constexpr int kAhead = 4, kPer = (int)kTopNodes / kTopThreads;
  const int tid = threadIdx.x;
  int4 ch[kAhead];
  auto links = [&](int t) { return t >= 0 && tid < count[t] ? child(t)[tid] : make_int4(-1, -1, -1, -1); };
#pragma unroll
  for (int j = 0; j < kAhead; ++j) ch[j] = links(top - j);
  const double* csq = sq(top + 1);
  for (int t0 = top; t0 >= 0; t0 -= kAhead)
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      const int t = t0 - j;
      if (t < 0) break;
      const int nt = count[t];
      double v[kPer];
#pragma unroll
      for (int k = 0; k < kPer; ++k)
        if (tid + k * kTopThreads < nt) v[k] = child_sum(k == 0 ? ch[j] : child(t)[tid + k * kTopThreads], csq);
      ch[j] = links(t - kAhead);
      if (t < top) __syncthreads();  // every child's norm has been read
      double* out = sq(t);
#pragma unroll
      for (int k = 0; k < kPer; ++k)
        if (tid + k * kTopThreads < nt) out[tid + k * kTopThreads] = s[tid + k * kTopThreads] = v[k];
      __syncthreads();
      csq = s;
    }
}

// Exclusive prefixes of the rows v[r][0 .. kGroups) of shared memory, warp r row r < rows;
// the rows' sums in total[r].
constexpr int kGroups = (int)kTopNodes / 32;
__device__ __forceinline__ void group_prefixes(uint32_t (*v)[kGroups], int rows, int* total) {
  constexpr int kPer = kGroups / 32;
  const int lane = threadIdx.x & 31, r = threadIdx.x >> 5;
  if (r >= rows) return;
  uint32_t e[kPer], sum = 0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    e[k] = sum;
    sum += v[r][kPer * lane + k];
  }
  uint32_t x = sum;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
#pragma unroll
  for (int k = 0; k < kPer; ++k) v[r][kPer * lane + k] = x - sum + e[k];
  if (lane == 31) total[r] = (int)x;
}

// One block per tree: the leaves (rules 1, 2), then the levels t0 - 1 .. 0, kTopNodes
// nodes at a time.  A block lives on latency: every thread's loads of a phase are in
// flight together, and groups of 32 nodes keep a warp's accesses together.  All levels'
// structure in one pass, instead of a flag, prefix and placing pass per level:
// truncating both 4,088-leaf operands of a 4096-row lattice 20.8 -> 12.5 us.  Up to
// kBoundNodes the block takes one piece after the other: the tree of 12,000 leaves from
// triplets one launch instead of eleven (the whole building 570 -> 534 us).  (A cluster of
// eight blocks takes 522, but waits for eight free multiprocessors next to one another,
// which a persistent launch on another stream may not leave.)
__global__ void __launch_bounds__(kTopThreads) tree_top_kernel(const __grid_constant__ TreePair P) {
  constexpr int kWarps = kTopThreads / 32, kPer = kGroups / kWarps;  // groups per warp
  __shared__ union {
    uint32_t code[kTopNodes];
    double sq[kTopNodes];
  } s_node;
  __shared__ uint32_t s_before[SPAMM_MAX_LEVELS][kGroups];
  __shared__ int s_add[SPAMM_MAX_LEVELS], s_n[SPAMM_MAX_LEVELS];
  const TreeDev& T = P.t[blockIdx.x];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, t0 = T.t0;
  const unsigned earlier = (1u << lane) - 1u;
  int n = 0;
  if (T.rule == 1 || T.rule == 2) {
    const int cand = (int)T.n;
    for (int node0 = 0; node0 < cand; node0 += (int)kTopNodes) {
      double sq[kPer] = {};
      int64_t slot[kPer];
      uint32_t code[kPer];
      unsigned keep[kPer];
      auto each = [&](auto f) {
#pragma unroll
        for (int k = 0; k < kPer; ++k) f(k, node0 + 32 * (warp + k * kWarps) + lane);
      };
      each([&](int k, int q) {
        slot[k] = q;
        code[k] = (uint32_t)q;
        keep[k] = 1;
        if (q < cand) sq[k] = T.sq[q];
      });
      if (T.code) each([&](int k, int q) { if (q < cand) code[k] = T.code[q]; });
      if (T.slot) each([&](int k, int q) { if (q < cand) slot[k] = T.slot[q]; });
      if (T.rule == 1) each([&](int k, int q) { if (q < cand) keep[k] = T.keep[q]; });
      if (T.rule == 2) each([&](int k, int) { keep[k] = kept_norm(sq[k], T.smin); });
      each([&](int k, int q) { keep[k] = q < cand && keep[k]; });
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        keep[k] = __ballot_sync(0xffffffffu, keep[k] != 0);
        if (lane == 0) s_before[0][warp + k * kWarps] = (uint32_t)__popc(keep[k]);
      }
      __syncthreads();
      group_prefixes(s_before, 1, s_add);
      __syncthreads();
#pragma unroll
      for (int k = 0; k < kPer; ++k)
        if (keep[k] >> lane & 1u) {
          const int p = n + (int)s_before[0][warp + k * kWarps] + __popc(keep[k] & earlier);
          T.ocode[T.L][p] = code[k];
          T.osq[T.L][p] = sq[k];
          T.oslot[p] = slot[k];
        }
      n += s_add[0];
      __syncthreads();
    }
    if (tid == 0) T.count[T.L] = (uint64_t)n;
  } else {
    n = T.rule == 3 && t0 == T.L ? (int)T.n : (int)T.count[t0];
    if (T.rule == 3 && tid == 0) T.count[T.L] = (uint64_t)T.n;
  }
  if (tid < t0) s_n[tid] = 0;
  __syncthreads();
  uint32_t last = 0;  // the code before the piece
  for (int node0 = 0; node0 < n; node0 += (int)kTopNodes) {
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int i = tid + k * kTopThreads;
      if (node0 + i < n) s_node.code[i] = T.ocode[t0][node0 + i];
    }
    __syncthreads();
    uint32_t code[kPer];
    int first[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int g = warp + k * kWarps, i = 32 * g + lane;
      const bool in = node0 + i < n;
      code[k] = in ? s_node.code[i] : 0;
      first[k] = in ? first_level(code[k], i > 0 ? s_node.code[i - 1] : last, node0 + i, t0) : kNoNode;
      uint32_t c = 0;  // lane t: the group's nodes of level t
      for (int t = t0 - 1; t >= 0; --t) {
        const unsigned b = __ballot_sync(0xffffffffu, first[k] <= t);
        if (b == 0) break;
        if (lane == t) c = (uint32_t)__popc(b);
      }
      if (lane < t0) s_before[lane][g] = c;
    }
    last = s_node.code[kTopNodes - 1];  // of a whole piece, if another follows
    __syncthreads();
    group_prefixes(s_before, t0, s_add);
    __syncthreads();
    for (int t = 0; t < t0; ++t)
      for (int p = tid; p < s_add[t]; p += kTopThreads) T.ochild[t][s_n[t] + p] = make_int4(-1, -1, -1, -1);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int g = warp + k * kWarps;
      place_levels(T, node0 + 32 * g + lane, code[k], first[k], [&](int t) { return s_n[t] + (int)s_before[t][g]; });
    }
    __syncthreads();
    if (tid < t0) s_n[tid] += s_add[tid];
    __syncthreads();
  }
  if (tid < t0) T.count[tid] = (uint64_t)s_n[tid];
  if (T.host && tid <= T.L) T.host[tid] = tid < t0 ? (uint64_t)s_n[tid] : T.count[tid];
  if (t0 == 0 || !T.osq[t0 - 1]) return;
  int top = t0 - 1;
  for (; top >= 0 && s_n[top] > kTopNodes; --top) {
    sum_parents(T, top + 1, 0, s_n[top]);
    __syncthreads();
  }
  block_norms(top, s_n, [&](int t) { return T.ochild[t]; }, [&](int t) { return T.osq[t]; }, s_node.sq);
}

// The tiled form of one step: t = L + 1 the candidates' compaction, else the
// parents of level t (whose node count is on the device).
__device__ __forceinline__ unsigned tile_flags(const TreeDev& T, int t, int64_t n, int64_t q0) {
  unsigned f = 0;
#pragma unroll
  for (int i = 0; i < kTilePer; ++i)
    if (q0 + i < n && (t > T.L ? kept(T, q0 + i) : first_child(T.ocode[t], q0 + i))) f |= 1u << i;
  return f;
}

__global__ void __launch_bounds__(kTileThreads)
    tile_count_kernel(const __grid_constant__ TreeDev T, int t, uint64_t* __restrict__ tiles) {
  const int64_t n = t > T.L || (t == T.L && T.rule == 3) ? T.n : (int64_t)T.count[t];
  const unsigned f = tile_flags(T, t, n, (int64_t)blockIdx.x * kTile + (int64_t)threadIdx.x * kTilePer);
  uint32_t total;
  block_prefix<kTileThreads>((uint32_t)__popc(f), &total);
  if (threadIdx.x == 0) tiles[blockIdx.x] = total;
}

// Sum of tiles[0 .. upto) by the whole block.
__device__ __forceinline__ int64_t tiles_before(const uint64_t* __restrict__ tiles, int64_t upto) {
  __shared__ unsigned long long s_sum;
  if (threadIdx.x == 0) s_sum = 0;
  __syncthreads();
  unsigned long long v = 0;
  for (int64_t i = threadIdx.x; i < upto; i += blockDim.x) v += tiles[i];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(&s_sum, v);
  __syncthreads();
  return (int64_t)s_sum;
}

__global__ void tile_total_kernel(const uint64_t* __restrict__ tiles, int64_t ntiles, uint64_t* __restrict__ out) {
  const int64_t s = tiles_before(tiles, ntiles);
  if (threadIdx.x == 0) *out = (uint64_t)s;
}

__global__ void __launch_bounds__(kTileThreads)
    tile_place_kernel(const __grid_constant__ TreeDev T, int t, const uint64_t* __restrict__ tiles, int64_t ntiles) {
  const int64_t n = t > T.L || (t == T.L && T.rule == 3) ? T.n : (int64_t)T.count[t];
  const int64_t q0 = (int64_t)blockIdx.x * kTile + (int64_t)threadIdx.x * kTilePer;
  const int64_t base = ntiles > kTilesSummed ? (int64_t)tiles[blockIdx.x] : tiles_before(tiles, blockIdx.x);
  const unsigned f = tile_flags(T, t, n, q0);
  uint32_t total;
  int64_t p = base + block_prefix<kTileThreads>((uint32_t)__popc(f), &total);
#pragma unroll
  for (int i = 0; i < kTilePer; ++i)
    if (f >> i & 1u) {
      if (t > T.L)
        place_leaf(T, q0 + i, p++);
      else
        place_parent(T, t, n, q0 + i, p++);
    }
  if (t <= T.L) {
    __syncthreads();
    sum_parents(T, t, base, base + total);
  }
  if (blockIdx.x == ntiles - 1 && threadIdx.x == 0) T.count[t - 1] = (uint64_t)(base + total);
}

// Smallest squared norm a leaf may have without being dropped: the least double s
// with sqrt(s) >= tau (the rounded square root is monotone, so the block rule's
// test !(sqrt(s) < tau) equals !(s < smin), without a square root per leaf).
double least_kept(double tau) {
  uint64_t lo = 0, hi = 0x7FF0000000000000ull;  // sqrt(inf) >= tau
  while (lo < hi) {
    const uint64_t mid = lo + (hi - lo) / 2;
    double s;
    memcpy(&s, &mid, sizeof s);
    if (std::sqrt(s) >= tau)
      hi = mid;
    else
      lo = mid + 1;
  }
  double s;
  memcpy(&s, &lo, sizeof s);
  return s;
}

int64_t level_cap(int64_t nleaves, int t) {
  const int64_t grid = (int64_t)1 << (2 * t);
  return nleaves < grid ? nleaves : grid;
}

// Storage of the levels t < L (codes, child links, norms unless `structure`),
// and of the leaf level and slots if `leaves`, for at most n leaves, in one block.
void alloc_levels(spamm_ctx ctx, spamm_mat m, int64_t n, bool leaves, bool structure) {
  const int L = m->L;
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  size_t bytes = up((L + 1) * sizeof(uint64_t));
  for (int t = 0; t < L; ++t) {
    const int64_t c = level_cap(n, t);
    bytes += up(c * sizeof(uint32_t)) + up(c * sizeof(int4)) + (structure ? 0 : up(c * sizeof(double)));
  }
  if (leaves) bytes += up(n * sizeof(uint32_t)) + up(n * sizeof(double)) + up(n * sizeof(int64_t));
  BufP arena = alloc_bytes(ctx, bytes);
  size_t at = 0;
  auto take = [&](size_t b) {
    BufP v = sub_buf(arena, at, b);
    at += up(b);
    return v;
  };
  m->dcount = take((L + 1) * sizeof(uint64_t));
  for (int t = 0; t < L; ++t) {
    const int64_t c = level_cap(n, t);
    m->lv[t].count = c;
    m->lv[t].code = take(c * sizeof(uint32_t));
    m->lv[t].child = take(c * sizeof(int4));
    m->lv[t].sq = structure ? BufP() : take(c * sizeof(double));
  }
  if (leaves) {
    m->lv[L].count = n;
    m->lv[L].code = take(n * sizeof(uint32_t));
    m->lv[L].sq = take(n * sizeof(double));
    m->slot = take(n * sizeof(int64_t));
  }
}

void point_at(TreeDev* T, spamm_mat m) {
  T->L = m->L;
  T->count = P<uint64_t>(m->dcount);
  for (int t = 0; t <= m->L; ++t) {
    T->ocode[t] = P<uint32_t>(m->lv[t].code);
    T->osq[t] = P<double>(m->lv[t].sq);
    T->ochild[t] = t < m->L ? P<int4>(m->lv[t].child) : nullptr;
  }
  T->oslot = P<int64_t>(m->slot);
}

// One step in tiles over at most n items.
void tiled_step(spamm_ctx ctx, const TreeDev& T, int t, int64_t n, uint64_t* tiles) {
  const int64_t ntiles = (n + kTile - 1) / kTile;
  if (t <= T.L) {  // the candidates' tiles were counted before the leaf level was allocated
    tile_count_kernel<<<(unsigned)ntiles, kTileThreads, 0, ctx->stream>>>(T, t, tiles);
    CK_LAUNCH("tile_count_kernel");
    if (ntiles > kTilesSummed) scan_exclusive_u64(ctx, tiles, tiles, ntiles, nullptr);
  }
  tile_place_kernel<<<(unsigned)ntiles, kTileThreads, 0, ctx->stream>>>(T, t, tiles, ntiles);
  CK_LAUNCH("tile_place_kernel");
}

// The levels above the leaves (at most n), large ones in tiles; T.t0 is left at the
// level that tree_top_kernel starts from.
void tiled_levels(spamm_ctx ctx, TreeDev* T, int64_t n) {
  int t = T->L;
  int64_t cap = n;
  if (cap > kBoundNodes) {
    BufP tiles = alloc_n<uint64_t>(ctx, (cap + kTile - 1) / kTile);
    for (; t >= 1 && cap > kBoundNodes; --t, cap = level_cap(n, t)) tiled_step(ctx, *T, t, cap, P<uint64_t>(tiles));
  }
  T->t0 = t;
}

}  // namespace

void tree_from_candidates(spamm_ctx ctx, TreeReq* req, int k, bool resolve) {
  if (k > 2) fail(SPAMM_E_CUDA, "at most two trees are built at once");
  TreePair pair;
  BufP tiles[2];
  bool wide[2] = {false, false};
  uint64_t* host = static_cast<uint64_t*>(ctx->h_pinned);
  for (int i = 0; i < k; ++i) {
    TreeReq& r = req[i];
    TreeDev& T = pair.t[i];
    T.n = r.n;
    T.code = r.code;
    T.sq = r.sq;
    T.slot = r.slot;
    T.keep = r.keep;
    T.rule = r.keep ? 1 : 2;
    T.smin = r.keep ? 0.0 : least_kept(r.tau);
    T.L = r.m->L;
    T.t0 = T.L;
    wide[i] = r.n > kBoundNodes;
    if (!wide[i]) {
      alloc_levels(ctx, r.m, r.n, true, false);
      point_at(&T, r.m);
      continue;
    }
    // of many candidates the exact leaf count first: the leaf level may be much smaller
    const int64_t ntiles = (r.n + kTile - 1) / kTile;
    tiles[i] = alloc_n<uint64_t>(ctx, ntiles);
    tile_count_kernel<<<(unsigned)ntiles, kTileThreads, 0, ctx->stream>>>(T, T.L + 1, P<uint64_t>(tiles[i]));
    CK_LAUNCH("tile_count_kernel");
    BufP total = alloc_n<uint64_t>(ctx, 1);
    if (ntiles > kTilesSummed) {
      scan_exclusive_u64(ctx, P<uint64_t>(tiles[i]), P<uint64_t>(tiles[i]), ntiles, P<uint64_t>(total));
    } else {
      tile_total_kernel<<<1, 1024, 0, ctx->stream>>>(P<uint64_t>(tiles[i]), ntiles, P<uint64_t>(total));
      CK_LAUNCH("tile_total_kernel");
    }
    CK(cudaMemcpyAsync(host + i, P<uint64_t>(total), sizeof(uint64_t), cudaMemcpyDeviceToHost, ctx->stream));
  }
  if (wide[0] || wide[1]) CK(cudaStreamSynchronize(ctx->stream));
  for (int i = 0; i < k; ++i) {
    if (!wide[i]) continue;
    TreeDev& T = pair.t[i];
    const int64_t n = (int64_t)host[i];
    alloc_levels(ctx, req[i].m, n, true, false);
    point_at(&T, req[i].m);
    tiled_step(ctx, T, T.L + 1, T.n, P<uint64_t>(tiles[i]));
    T.rule = 0;  // tree_top_kernel starts above the leaves
    tiled_levels(ctx, &T, n);
  }
  if (resolve)
    for (int i = 0; i < k; ++i) pair.t[i].host = host + i * SPAMM_MAX_LEVELS;
  tree_top_kernel<<<k, kTopThreads, 0, ctx->stream>>>(pair);
  CK_LAUNCH("tree_top_kernel");
  for (int i = 0; i < k; ++i) req[i].m->pending = true;
  if (!resolve) return;
  CK(cudaStreamSynchronize(ctx->stream));
  for (int i = 0; i < k; ++i) tree_set_counts(req[i].m, host + i * SPAMM_MAX_LEVELS);
}

void tree_skeleton(spamm_ctx ctx, spamm_mat m, uint64_t* host) {
  const int64_t n = m->lv[m->L].count;
  alloc_levels(ctx, m, n, false, true);
  TreePair pair;
  TreeDev& T = pair.t[0];
  point_at(&T, m);
  T.n = n;
  T.rule = 3;
  T.host = host;
  tiled_levels(ctx, &T, n);
  tree_top_kernel<<<1, kTopThreads, 0, ctx->stream>>>(pair);
  CK_LAUNCH("tree_top_kernel");
  m->pending = true;
}

void tree_counts_async(spamm_ctx ctx, spamm_mat m, uint64_t* host) {
  CK(cudaMemcpyAsync(host, P<uint64_t>(m->dcount), (m->L + 1) * sizeof(uint64_t), cudaMemcpyDeviceToHost, ctx->stream));
}

void tree_set_counts(spamm_mat m, const uint64_t* host) {
  for (int t = 0; t <= m->L; ++t) {
    m->lv[t].count = (int64_t)host[t];
    if (host[t] == 0) {
      m->lv[t].code.reset();
      m->lv[t].child.reset();
      if (t < m->L) m->lv[t].sq.reset();
    }
  }
  m->nleaves = (int64_t)host[m->L];
  m->pending = false;
}

// ------------------------------------------------------ norms of given trees
// The parents' squared norms of an output whose structure was built at plan
// time, from its leaves' norms up, for every tree of a batch: levels of more than
// kTopNodes nodes one launch each (all trees), the rest by one block per tree in
// one launch.  The additions are child_sum's, in its order.
struct NormTree {
  int64_t L;
  const uint64_t* count;  // nodes per level, on the device
  const int4* child[SPAMM_MAX_LEVELS];
  double* sq[SPAMM_MAX_LEVELS];
};

__device__ __forceinline__ void node_norm(const NormTree& T, int t, int64_t p) {
  const int4 ch = T.child[t][p];
  T.sq[t][p] = child_sum(ch, T.sq[t + 1]);
}

// Height h above the leaves of every tree that has more than kTopNodes nodes there.
__global__ void norms_wide_kernel(const NormTree* __restrict__ tab, int ntrees, int h) {
  for (int r = blockIdx.y; r < ntrees; r += gridDim.y) {
    const NormTree& T = tab[r];
    const int t = (int)T.L - h;
    const int64_t n = t >= 0 && T.count ? (int64_t)T.count[t] : 0;
    if (n <= kTopNodes) continue;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x)
      node_norm(T, t, p);
  }
}

__global__ void __launch_bounds__(kTopThreads) norms_top_kernel(const NormTree* __restrict__ tab) {
  __shared__ double s_sq[kTopNodes];
  __shared__ const int4* s_child[SPAMM_MAX_LEVELS];
  __shared__ double* s_out[SPAMM_MAX_LEVELS];
  __shared__ int s_n[SPAMM_MAX_LEVELS];
  const NormTree& T = tab[blockIdx.x];
  const int t = threadIdx.x;
  if (!T.count) return;  // no leaves
  if (t <= T.L) {
    s_child[t] = T.child[t];
    s_out[t] = T.sq[t];
    s_n[t] = (int)T.count[t];
  }
  __syncthreads();
  int top = (int)T.L - 1;
  while (top >= 0 && s_n[top] > kTopNodes) --top;
  if (top >= 0) block_norms(top, s_n, [&](int l) { return s_child[l]; }, [&](int l) { return s_out[l]; }, s_sq);
}

size_t norm_table_bytes(size_t ntrees) { return ntrees * sizeof(NormTree); }

void norm_tables(const std::vector<spamm_mat>& ms, void* host, const void* device, NormBatch* nb) {
  NormTree* tab = static_cast<NormTree*>(host);
  nb->tab = device;
  nb->ntrees = (int)ms.size();
  nb->wide = 0;
  nb->widest = 0;
  for (size_t r = 0; r < ms.size(); ++r) {
    spamm_mat m = ms[r];
    NormTree& T = tab[r];
    memset(&T, 0, sizeof T);
    T.L = m->L;
    T.count = P<uint64_t>(m->dcount);
    for (int t = 0; t <= m->L; ++t) {
      T.child[t] = t < m->L ? P<int4>(m->lv[t].child) : nullptr;
      T.sq[t] = P<double>(m->lv[t].sq);
      if (t < m->L && m->lv[t].count > kTopNodes) {  // exact, or an upper bound
        nb->wide = nb->wide > m->L - t ? nb->wide : m->L - t;
        nb->widest = nb->widest > m->lv[t].count ? nb->widest : m->lv[t].count;
      }
    }
  }
}

void propagate_norms(spamm_ctx ctx, const NormBatch& nb) {
  const NormTree* tab = static_cast<const NormTree*>(nb.tab);
  if (nb.ntrees == 0) return;
  int64_t g = (nb.widest + 255) / 256;
  const int64_t cap = (int64_t)ctx->num_sms * 8;
  if (g > cap) g = cap;
  for (int h = 1; h <= nb.wide; ++h) {
    norms_wide_kernel<<<dim3((unsigned)g, (unsigned)(nb.ntrees < 1024 ? nb.ntrees : 1024)), 256, 0, ctx->stream>>>(
        tab, nb.ntrees, h);
    CK_LAUNCH("norms_wide_kernel");
  }
  norms_top_kernel<<<(unsigned)nb.ntrees, kTopThreads, 0, ctx->stream>>>(tab);
  CK_LAUNCH("norms_top_kernel");
}

}  // namespace spamm
