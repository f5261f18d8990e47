// prims.cu -- errors, device memory, prefix sums and radix sort.
#include <cstdio>
#include <cstring>

#include "internal.cuh"

namespace spamm {

thread_local unsigned long long g_kernel_launches = 0;  // per host thread: a context is used by one thread

void fail(spamm_status st, const std::string& msg) { throw Error{st, msg}; }

void check_cuda(cudaError_t e, const char* what, const char* file, int line) {
  if (e == cudaSuccess) return;
  char buf[512];
  snprintf(buf, sizeof(buf), "%s failed: %s (%s:%d)", what, cudaGetErrorString(e), file, line);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    fail(SPAMM_E_OOM, buf);
  }
  fail(SPAMM_E_CUDA, buf);
}

Buf::~Buf() {
  if (!p || owner) return;
  if (ctx->ufree)
    ctx->ufree(p, ctx->user);
  else
    cudaFreeAsync(p, ctx->stream);
}

BufP alloc_bytes(spamm_ctx ctx, size_t bytes) {
  auto b = std::make_shared<Buf>();
  b->ctx = ctx;
  b->bytes = bytes;
  if (bytes == 0) return b;
  size_t rounded = (bytes + 255) & ~(size_t)255;
  if (ctx->ualloc) {
    b->p = ctx->ualloc(rounded, ctx->user);
    if (!b->p) fail(SPAMM_E_OOM, "allocator returned NULL for " + std::to_string(rounded) + " bytes");
  } else {
    cudaError_t e = cudaMallocAsync(&b->p, rounded, ctx->stream);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (e == cudaErrorMemoryAllocation && cudaStreamIsCapturing(ctx->stream, &cap) == cudaSuccess &&
        cap == cudaStreamCaptureStatusNone) {
      // the pool keeps freed blocks; hand them back to the device and try once more
      cudaGetLastError();
      cudaMemPool_t pool;
      if (cudaStreamSynchronize(ctx->stream) == cudaSuccess &&
          cudaDeviceGetDefaultMemPool(&pool, ctx->device) == cudaSuccess &&
          cudaMemPoolTrimTo(pool, 0) == cudaSuccess)
        e = cudaMallocAsync(&b->p, rounded, ctx->stream);
    }
    if (e != cudaSuccess) {
      b->p = nullptr;
      cudaGetLastError();
      fail(e == cudaErrorMemoryAllocation ? SPAMM_E_OOM : SPAMM_E_CUDA,
           "device allocation of " + std::to_string(rounded) + " bytes failed: " + cudaGetErrorString(e));
    }
  }
  return b;
}

BufP sub_buf(const BufP& whole, size_t at, size_t bytes) {
  auto b = std::make_shared<Buf>();
  b->ctx = whole->ctx;
  b->owner = whole;
  b->bytes = bytes;
  b->p = bytes ? static_cast<uint8_t*>(whole->p) + at : nullptr;
  return b;
}

template <class T>
T read_scalar(spamm_ctx ctx, const T* d) {
  CK(cudaMemcpyAsync(ctx->h_pinned, d, sizeof(T), cudaMemcpyDeviceToHost, ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));
  T v;
  memcpy(&v, ctx->h_pinned, sizeof(T));
  return v;
}
template uint64_t read_scalar<uint64_t>(spamm_ctx, const uint64_t*);
template int64_t read_scalar<int64_t>(spamm_ctx, const int64_t*);
template double read_scalar<double>(spamm_ctx, const double*);
template int read_scalar<int>(spamm_ctx, const int*);

void clear_device_error(spamm_ctx ctx) { CK(cudaMemsetAsync(ctx->d_err, 0, sizeof(int), ctx->stream)); }

// One wait for the work and the error word (read into the last word of the pinned page).
void sync_and_check(spamm_ctx ctx) {
  int* word = reinterpret_cast<int*>(static_cast<uint8_t*>(ctx->h_pinned) + 4096) - 1;
  CK(cudaMemcpyAsync(word, ctx->d_err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));
  CK(cudaGetLastError());
  const int err = *word;
  if (!err) return;
  clear_device_error(ctx);
  if (err & DEV_ERR_TIMEOUT) fail(SPAMM_E_TIMEOUT, "a bounded device-side wait ran out");
  if (err & DEV_ERR_NONFINITE) fail(SPAMM_E_NONFINITE, "input contains Inf or NaN");
  if (err & DEV_ERR_DUPLICATE) fail(SPAMM_E_INVALID_ARG, "repeated leaf coordinate");
  fail(SPAMM_E_INVALID_ARG, "index out of range");
}

// ------------------------------------------------------------ prefix sums
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

// Exclusive scan across the 256 threads of a block; *total = block sum.
// T = uint64_t (exact) or double (fixed tiling, so the rounding is the same
// on every run).
template <class T>
__device__ __forceinline__ T block_exclusive_scan(T v, T* total) {
  __shared__ T warp_tot[kScanThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T x = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    T y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) warp_tot[warp] = x;
  __syncthreads();
  T before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kScanThreads / 32; ++w) {
    T t = warp_tot[w];
    if (w < warp) before += t;
    all += t;
  }
  __syncthreads();
  *total = all;
  const T prev = __shfl_up_sync(0xffffffffu, x, 1);  // the previous lane's inclusive sum
  return lane == 0 ? before : before + prev;
}

template <class T>
__global__ void scan_reduce_kernel(const T* __restrict__ in, int64_t n, T* __restrict__ bsum) {
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  T s = 0;
  for (int i = threadIdx.x; i < kScanTile; i += kScanThreads) {
    int64_t q = base + i;
    if (q < n) s += in[q];
  }
  T total;
  block_exclusive_scan(s, &total);
  if (threadIdx.x == 0) bsum[blockIdx.x] = total;
}

template <class T>
__global__ void scan_blocksums_kernel(T* bsum, int64_t nblocks, T* d_total) {
  T carry = 0;
  for (int64_t base = 0; base < nblocks; base += kScanThreads) {
    int64_t q = base + threadIdx.x;
    T v = q < nblocks ? bsum[q] : 0;
    T total;
    T ex = block_exclusive_scan(v, &total);
    if (q < nblocks) bsum[q] = carry + ex;
    carry += total;
  }
  if (threadIdx.x == 0 && d_total) *d_total = carry;
}

// inclusive = false: out[q] = sum of in[0 .. q-1]; true: sum of in[0 .. q]
template <class T>
__global__ void scan_down_kernel(const T* __restrict__ in, T* __restrict__ out, int64_t n, const T* __restrict__ bsum,
                                 bool inclusive) {
  __shared__ T tile[kScanTile];
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  for (int i = threadIdx.x; i < kScanTile; i += kScanThreads) {
    int64_t q = base + i;
    tile[i] = q < n ? in[q] : 0;
  }
  __syncthreads();
  T loc[kScanItems];
  T s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    loc[i] = s;
    s += tile[threadIdx.x * kScanItems + i];
  }
  T total;
  T ex = block_exclusive_scan(s, &total) + bsum[blockIdx.x];
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    const T mine = tile[threadIdx.x * kScanItems + i];
    tile[threadIdx.x * kScanItems + i] = inclusive ? (ex + loc[i]) + mine : ex + loc[i];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kScanTile; i += kScanThreads) {
    int64_t q = base + i;
    if (q < n) out[q] = tile[i];
  }
}

// n <= kScanTile: the whole scan in one block, one launch.
template <class T>
__global__ void scan_one_tile_kernel(const T* __restrict__ in, T* __restrict__ out, int64_t n, T* d_total,
                                     bool inclusive) {
  __shared__ T tile[kScanTile];
  for (int i = threadIdx.x; i < kScanTile; i += kScanThreads) tile[i] = i < n ? in[i] : 0;
  __syncthreads();
  T loc[kScanItems];
  T s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    loc[i] = s;
    s += tile[threadIdx.x * kScanItems + i];
  }
  T total;
  const T ex = block_exclusive_scan(s, &total);
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    const T mine = tile[threadIdx.x * kScanItems + i];
    tile[threadIdx.x * kScanItems + i] = inclusive ? (ex + loc[i]) + mine : ex + loc[i];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kScanTile; i += kScanThreads)
    if (i < n) out[i] = tile[i];
  if (threadIdx.x == 0 && d_total) *d_total = total;
}

template <class T>
static void scan_any(spamm_ctx ctx, const T* in, T* out, int64_t n, T* d_total, bool inclusive) {
  if (n <= 0) {
    if (d_total) CK(cudaMemsetAsync(d_total, 0, sizeof(T), ctx->stream));
    return;
  }
  if (n <= kScanTile) {
    scan_one_tile_kernel<T><<<1, kScanThreads, 0, ctx->stream>>>(in, out, n, d_total, inclusive);
    CK_LAUNCH("scan_one_tile_kernel");
    return;
  }
  const int64_t nblocks = (n + kScanTile - 1) / kScanTile;
  BufP bs = alloc_n<T>(ctx, nblocks);
  scan_reduce_kernel<T><<<(unsigned)nblocks, kScanThreads, 0, ctx->stream>>>(in, n, P<T>(bs));
  CK_LAUNCH("scan_reduce_kernel");
  scan_blocksums_kernel<T><<<1, kScanThreads, 0, ctx->stream>>>(P<T>(bs), nblocks, d_total);
  CK_LAUNCH("scan_blocksums_kernel");
  scan_down_kernel<T><<<(unsigned)nblocks, kScanThreads, 0, ctx->stream>>>(in, out, n, P<T>(bs), inclusive);
  CK_LAUNCH("scan_down_kernel");
}

void scan_exclusive_u64(spamm_ctx ctx, const uint64_t* in, uint64_t* out, int64_t n, uint64_t* d_total) {
  scan_any<uint64_t>(ctx, in, out, n, d_total, false);
}

void scan_inclusive_f64(spamm_ctx ctx, const double* in, double* out, int64_t n) {
  scan_any<double>(ctx, in, out, n, nullptr, true);
}

// ------------------------------------------------------------- radix sort
// Stable LSD sort of (key, value) pairs by 8-bit digits.  Items are ranked in
// rounds of 32 by a warp: the lanes that share a digit (match) take consecutive
// places after the warp's earlier ones, counted per warp and digit in shared
// memory; the warps of a block own consecutive runs of items, so a prefix over
// warps, tiles and digits gives every item its place.  Up to kSortSmall items one
// block takes all passes in one launch; more take three launches a pass (some 19 us at
// that size): digit counts per tile, their prefix per digit, placing.  A purification,
// whose error-controlled truncation sorts some 10^4 norms by 64 bits, 2.76 -> 2.69 ms.
// 2,000,000 pairs by 32 bits: 0.23 ms where eight 4-bit passes, each a scan over all
// blocks and digits, took 0.85.
constexpr int kDigits = 256;
constexpr int kSortThreads = 256;
constexpr int kSortRounds = 8;                        // rounds of 32 items per warp
constexpr int kSortTile = kSortThreads * kSortRounds;  // items per block
constexpr int kSmallThreads = 1024;
constexpr int kSmallRounds = 16;
constexpr int64_t kSortSmall = kSmallThreads * kSmallRounds;

// Ranks the warp's items (digit d[r] of round r, valid where bit r of `in`) within its
// counters cnt[256], which it leaves at the warp's digit counts.
__device__ __forceinline__ void warp_rank(const uint32_t (&d)[kSortRounds], uint32_t in, uint32_t* cnt,
                                          uint32_t (&rank)[kSortRounds]) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r) {
    const bool on = in >> r & 1u;
    const unsigned act = __ballot_sync(0xffffffffu, on);
    if (on) {
      const unsigned same = __match_any_sync(act, d[r]);
      const uint32_t before = cnt[d[r]];
      __syncwarp(act);
      if ((same & lt) == 0) cnt[d[r]] = before + (uint32_t)__popc(same);
      __syncwarp(act);
      rank[r] = before + (uint32_t)__popc(same & lt);
    }
    __syncwarp();
  }
}

__global__ void __launch_bounds__(kSortThreads)
    radix_hist_kernel(const uint64_t* __restrict__ keys, int64_t n, int shift, uint64_t* __restrict__ hist,
                      int64_t ntiles) {
  __shared__ uint32_t cnt[kSortThreads / 32][kDigits];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kDigits * (kSortThreads / 32); i += kSortThreads) (&cnt[0][0])[i] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kSortTile + warp * (32 * kSortRounds) + lane;
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r) {
    const int64_t q = base + 32 * r;
    const unsigned act = __ballot_sync(0xffffffffu, q < n);
    if (q < n) {
      const uint32_t d = (uint32_t)(keys[q] >> shift) & (kDigits - 1);
      const unsigned same = __match_any_sync(act, d);
      if ((same & ((1u << lane) - 1u)) == 0) cnt[warp][d] += (uint32_t)__popc(same);
    }
    __syncwarp();
  }
  __syncthreads();
  uint64_t s = 0;
  for (int w = 0; w < kSortThreads / 32; ++w) s += cnt[w][threadIdx.x];
  hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = s;
}

// Block d: digit d's counts of all tiles to their exclusive prefix, the total to total[d].
__global__ void __launch_bounds__(kScanThreads)
    radix_digit_scan_kernel(uint64_t* __restrict__ hist, int64_t ntiles, uint64_t* __restrict__ total) {
  uint64_t* h = hist + (int64_t)blockIdx.x * ntiles;
  uint64_t carry = 0;
  for (int64_t b = 0; b < ntiles; b += kScanThreads) {
    const int64_t q = b + threadIdx.x;
    const uint64_t v = q < ntiles ? h[q] : 0;
    uint64_t all;
    const uint64_t ex = block_exclusive_scan(v, &all);
    if (q < ntiles) h[q] = carry + ex;
    carry += all;
  }
  if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

__global__ void __launch_bounds__(kSortThreads)
    radix_scatter_kernel(const uint64_t* __restrict__ kin, const int64_t* __restrict__ vin, uint64_t* __restrict__ kout,
                         int64_t* __restrict__ vout, int64_t n, int shift, const uint64_t* __restrict__ hist,
                         const uint64_t* __restrict__ total, int64_t ntiles) {
  static_assert(kSortThreads == kDigits && kScanThreads == kSortThreads, "one thread per digit");
  __shared__ uint32_t cnt[kSortThreads / 32][kDigits];
  __shared__ uint64_t place[kDigits];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kDigits * (kSortThreads / 32); i += kSortThreads) (&cnt[0][0])[i] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kSortTile + warp * (32 * kSortRounds) + lane;
  uint64_t key[kSortRounds];
  uint32_t d[kSortRounds], rank[kSortRounds], in = 0;
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r) {
    const int64_t q = base + 32 * r;
    key[r] = q < n ? kin[q] : 0;
    in |= (uint32_t)(q < n) << r;
    d[r] = (uint32_t)(key[r] >> shift) & (kDigits - 1);
  }
  warp_rank(d, in, cnt[warp], rank);
  uint64_t all;
  const uint64_t first = block_exclusive_scan(total[threadIdx.x], &all);  // items of smaller digits
  __syncthreads();
  place[threadIdx.x] = first + hist[(int64_t)threadIdx.x * ntiles + blockIdx.x];
  uint32_t s = 0;
  for (int w = 0; w < kSortThreads / 32; ++w) {
    const uint32_t c = cnt[w][threadIdx.x];
    cnt[w][threadIdx.x] = s;
    s += c;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r)
    if (in >> r & 1u) {
      const uint64_t p = place[d[r]] + cnt[warp][d[r]] + rank[r];
      kout[p] = key[r];
      vout[p] = vin[base + 32 * r];
    }
}

// All passes of a sort of at most 1024 ROUNDS pairs by one block; the result is in (ka, va)
// if the number of passes is even, else in (kb, vb).
template <int ROUNDS>
__global__ void __launch_bounds__(kSmallThreads)
    radix_small_kernel(uint64_t* ka, int64_t* va, uint64_t* kb, int64_t* vb, int n, int bits) {
  extern __shared__ uint32_t small_cnt[];  // [32][256], then 256 digit bases
  __shared__ uint32_t wsum[kDigits / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  uint32_t* mine = small_cnt + warp * kDigits;
  uint32_t* place = small_cnt + 32 * kDigits;
  const int per = (n + kSmallThreads - 1) / kSmallThreads;  // rounds per warp
  const int base = warp * 32 * per + lane;
  for (int shift = 0; shift < bits; shift += 8) {
    for (int i = lane; i < kDigits; i += 32) mine[i] = 0;
    __syncwarp();
    uint64_t key[ROUNDS];
    uint32_t at[ROUNDS];  // digit << 16 | rank among the warp's items of that digit
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) key[r] = r < per && base + 32 * r < n ? ka[base + 32 * r] : 0;
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
      if (r >= per) break;
      const bool on = base + 32 * r < n;
      const unsigned act = __ballot_sync(0xffffffffu, on);
      if (on) {
        const uint32_t d = (uint32_t)(key[r] >> shift) & (kDigits - 1);
        const unsigned same = __match_any_sync(act, d);
        const uint32_t before = mine[d];
        __syncwarp(act);
        if ((same & lt) == 0) mine[d] = before + (uint32_t)__popc(same);
        __syncwarp(act);
        at[r] = d << 16 | (before + (uint32_t)__popc(same & lt));
      }
      __syncwarp();
    }
    __syncthreads();
    // thread t < 256: digit t over the warps, then over the digits
    uint32_t s = 0, x = 0;
    if (threadIdx.x < kDigits) {
#pragma unroll 8
      for (int w = 0; w < kSmallThreads / 32; ++w) {
        const uint32_t c = small_cnt[w * kDigits + threadIdx.x];
        small_cnt[w * kDigits + threadIdx.x] = s;
        s += c;
      }
      x = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (lane == 31) wsum[warp] = x;
    }
    __syncthreads();
    if (threadIdx.x < kDigits) {
      uint32_t before = 0;
      for (int w = 0; w < warp; ++w) before += wsum[w];
      place[threadIdx.x] = before + x - s;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r)
      if (r < per && base + 32 * r < n) {
        const uint32_t d = at[r] >> 16, p = place[d] + mine[d] + (at[r] & 0xffffu);
        kb[p] = key[r];
        vb[p] = va[base + 32 * r];
      }
    __syncthreads();
    uint64_t* k = ka;
    ka = kb;
    kb = k;
    int64_t* v = va;
    va = vb;
    vb = v;
  }
}

template <int ROUNDS>
static void radix_small(spamm_ctx ctx, uint64_t* ka, int64_t* va, uint64_t* kb, int64_t* vb, int n, int bits) {
  const int smem = (int)sizeof(uint32_t) * kDigits * (kSmallThreads / 32 + 1);
  radix_small_kernel<ROUNDS><<<1, kSmallThreads, smem, ctx->stream>>>(ka, va, kb, vb, n, bits);
  CK_LAUNCH("radix_small_kernel");
}

void radix_sort_pairs(spamm_ctx ctx, uint64_t* keys, int64_t* vals, int64_t n, int bits) {
  if (n <= 1 || bits <= 0) return;
  BufP k2 = alloc_n<uint64_t>(ctx, n), v2 = alloc_n<int64_t>(ctx, n);
  uint64_t *ka = keys, *kb = P<uint64_t>(k2);
  int64_t *va = vals, *vb = P<int64_t>(v2);
  const int passes = (bits + 7) / 8;
  if (n <= kSortSmall) {
    if (n <= kSmallThreads * 4)
      radix_small<4>(ctx, ka, va, kb, vb, (int)n, bits);
    else
      radix_small<kSmallRounds>(ctx, ka, va, kb, vb, (int)n, bits);
    if (passes & 1) ka = kb, va = vb;
  } else {
    const int64_t ntiles = (n + kSortTile - 1) / kSortTile;
    BufP hist = alloc_n<uint64_t>(ctx, (ntiles + 1) * kDigits);
    uint64_t* total = P<uint64_t>(hist) + ntiles * kDigits;
    for (int p = 0; p < passes; ++p) {
      radix_hist_kernel<<<(unsigned)ntiles, kSortThreads, 0, ctx->stream>>>(ka, n, 8 * p, P<uint64_t>(hist), ntiles);
      CK_LAUNCH("radix_hist_kernel");
      radix_digit_scan_kernel<<<kDigits, kScanThreads, 0, ctx->stream>>>(P<uint64_t>(hist), ntiles, total);
      CK_LAUNCH("radix_digit_scan_kernel");
      radix_scatter_kernel<<<(unsigned)ntiles, kSortThreads, 0, ctx->stream>>>(ka, va, kb, vb, n, 8 * p,
                                                                              P<uint64_t>(hist), total, ntiles);
      CK_LAUNCH("radix_scatter_kernel");
      std::swap(ka, kb);
      std::swap(va, vb);
    }
  }
  if (ka != keys) {
    CK(cudaMemcpyAsync(keys, ka, n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, ctx->stream));
    CK(cudaMemcpyAsync(vals, va, n * sizeof(int64_t), cudaMemcpyDeviceToDevice, ctx->stream));
  }
}

}  // namespace spamm
