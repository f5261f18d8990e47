// leafpass.cuh -- one pass that makes leaves and takes their norms: copies into a
// pool, the element rule of the input truncation and alpha X + beta Y.  One warp
// per leaf in kernel (a)'s order (lane l takes the 16-byte pairs l, l + 32, ..., one
// FMA per element, a butterfly over the lanes), so the stored norms are kernel
// (a)'s on the finished leaves, bit for bit, without reading them back.  Bound by
// HBM for a copy (16 B moved per element, one FP64 instruction at two per clock and
// SM): 62,000 leaves of 64 x 64 (4.06 GB moved) in 0.63 ms, where a device copy and
// kernel (a) took 0.60 + 0.44.
#pragma once
#include "internal.cuh"

namespace spamm {

constexpr int kPassThreads = 256;
constexpr int kPassAhead = 4;  // pairs a lane reads before it uses the first

// Op: begin(q) points at leaf q's sources, read(i) loads pair i, value(raw) makes it;
// overflowed() (after the leaf) reports a value the rounded operations would have
// made infinite.
template <class Op>
__global__ void __launch_bounds__(kPassThreads)
    leaf_pass_kernel(Op proto, int64_t m, int bs, double* __restrict__ out, double* __restrict__ sq,
                     uint8_t* __restrict__ nonzero, int check_finite, int* err) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int nwb = kPassThreads / 32;
  const int pairs = bs * bs / 2;
  for (int64_t q = (int64_t)blockIdx.x * nwb + warp; q < m; q += (int64_t)gridDim.x * nwb) {
    Op op = proto;
    op.begin(q, (int64_t)bs * bs);
    double2* dst = reinterpret_cast<double2*>(out + q * ((int64_t)bs * bs));
    double s = 0.0;
    uint32_t bits = 0, emax = 0;
    for (int i = lane; i < pairs; i += 32 * kPassAhead) {
      typename Op::Raw raw[kPassAhead];
#pragma unroll
      for (int u = 0; u < kPassAhead; ++u) raw[u] = op.read(i + 32 * u);
#pragma unroll
      for (int u = 0; u < kPassAhead; ++u) {
        const double2 v = op.value(raw[u]);
        dst[i + 32 * u] = v;
        s = __fma_rn(v.x, v.x, s);
        s = __fma_rn(v.y, v.y, s);
        const uint32_t hx = (uint32_t)__double2hiint(v.x), hy = (uint32_t)__double2hiint(v.y);
        bits |= (uint32_t)__double2loint(v.x) | (uint32_t)__double2loint(v.y) | ((hx | hy) & 0x7fffffffu);
        emax = max(emax, max(hx & 0x7ff00000u, hy & 0x7ff00000u));
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    const bool nz = __any_sync(0xffffffffu, bits != 0);
    const bool bad = __any_sync(0xffffffffu, emax == 0x7ff00000u || op.overflowed());
    if (lane == 0) {
      sq[q] = s;
      nonzero[q] = nz;
      if (bad && check_finite) atomicOr(err, DEV_ERR_NONFINITE);
    }
  }
}

// Leaf q from src + slot[q] (q without slots), elements below tau zeroed (tau = +0:
// none, and not -0, whose pattern lies above all; |a| < tau on the two words of the bit patterns, which order like the
// magnitudes: compared as one 64-bit word the compiler takes the FP64 pipe for it,
// which made the pass 1.6 times as long).
struct CopyOp {
  const double* src;
  const int64_t* slot;
  double tau;
  const double2* p;
  using Raw = double2;
  __device__ __forceinline__ void begin(int64_t q, int64_t e) {
    p = reinterpret_cast<const double2*>(src + (slot ? slot[q] : q) * e);
  }
  __device__ __forceinline__ double2 read(int i) const { return __ldg(p + i); }
  __device__ __forceinline__ double keep(double v) const {
    const uint32_t h = (uint32_t)__double2hiint(v) & 0x7fffffffu, l = (uint32_t)__double2loint(v);
    const uint32_t th = (uint32_t)__double2hiint(tau), tl = (uint32_t)__double2loint(tau);
    const bool drop = h < th || (h == th && l < tl);
    return __hiloint2double(drop ? 0 : __double2hiint(v), drop ? 0 : (int)l);
  }
  __device__ __forceinline__ double2 value(const double2& v) const { return make_double2(keep(v.x), keep(v.y)); }
  __device__ __forceinline__ bool overflowed() const { return false; }
};

template <class Op>
void leaf_pass(spamm_ctx ctx, const Op& op, int64_t m, int bs, double* out, double* sq, uint8_t* nonzero,
               int check_finite) {
  if (m <= 0) return;
  const int64_t nblk = (m + kPassThreads / 32 - 1) / (kPassThreads / 32);
  leaf_pass_kernel<Op><<<(unsigned)(nblk < (1ll << 30) ? nblk : (1ll << 30)), kPassThreads, 0, ctx->stream>>>(
      op, m, bs, out, sq, nonzero, check_finite, ctx->d_err);
  CK_LAUNCH("leaf_pass_kernel");
}

}  // namespace spamm
