// select_device.cuh -- the per-expert selection of Algorithm 1 (steps 3 and
// 5-6) and the Eq. (2) centering (arXiv 2609.28053, Sec. 2 and App. C), as
// device functions shared by the selection kernels (select.cu) and the fine
// histogram pass, which selects in its blocks in the one-call step
// (hist.cu).
#pragma once

#include "eqb_device.cuh"

namespace eqb {

// The first of 256 bins whose inclusive prefix count reaches `target`, lane j
// of the warp holding the counts of bins 8j..8j+7: every lane gets the bin
// (-1: the target is below 1 or above the total) and `rest` = target minus
// the counts below that bin.  I is wide enough for the total count.
template <class I>
__device__ __forceinline__ int warp_pick(const I (&cnt)[8], I target, int lane, I& rest) {
  I incl = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) incl += cnt[j];
  I cum = -incl;  // becomes the count below this lane's bins
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const I o = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += o;
  }
  cum += incl;
  const unsigned hit = __ballot_sync(kFull, cum < target && target <= incl);
  int bin = lane * 8;
  I below = cum;
#pragma unroll
  for (int j = 0; j < 7; ++j) {  // the target lies in this lane's bins: not past the last
    cum += cnt[j];
    const bool past = cum < target;
    bin += past ? 1 : 0;
    below = past ? cum : below;
  }
  if (hit == 0u || target < 1) return -1;
  const int src = __ffs(hit) - 1;
  rest = __shfl_sync(kFull, target - below, src);
  return __shfl_sync(kFull, bin, src);
}

// bf16 pattern of the quantile with high key byte u_e and low byte v (a zero
// is returned as +0; v < 0, an unreachable rank, as NaN).
__device__ __forceinline__ uint32_t quantile_bits(uint32_t u_e, int v) {
  if (v < 0) return 0x7fc0u;
  const uint32_t q = kappa16_inv((u_e << 8) | static_cast<uint32_t>(v));
  return q == 0x8000u ? 0u : q;
}

// Exponent range of a non-zero bf16 pattern: [ulp exponent, leading-bit exponent].
__device__ __forceinline__ void bf16_exp_range(uint32_t x, int& lo, int& hi) {
  const int ex = (x >> 7) & 0xff;
  const uint32_t man = x & 0x7f;
  if (ex != 0) { lo = ex - 127 - 7; hi = ex - 127; }
  else { lo = -133; hi = -134 + (32 - __clz(man)); }  // subnormal
}

// b_next = q_hat - mean(q_hat), mean = (sum in ascending e, fp64) / E.
// If every non-zero q_hat lies within a window where all partial sums of up
// to E terms are exact in fp64 (leading-bit exponent - ulp exponent + 1 +
// ceil(log2 E) <= 52), any summation order gives the exact sum, so a warp
// tree reduction reproduces the sequential sum bit for bit.  Otherwise one
// thread sums in ascending order.
// Threads [0, nthreads) of the block compute b_next from q_hat (they share
// the final subtraction; warp 0 forms the mean); sync() is their barrier.
// q_hat is read through L2 (it may have been written earlier in the same
// kernel, by other blocks).
template <class Sync>
__device__ __forceinline__ void block_bias_update(const uint16_t* q_hat, int E, float* __restrict__ b_next,
                                                  int nthreads, Sync sync) {
  __shared__ double mean;
  auto q_at = [&](int e) -> uint32_t { return __ldcg(q_hat + e); };
  const uint32_t mine = threadIdx.x < E ? q_at(threadIdx.x) : 0u;  // in flight beside warp 0's

  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    double part = 0.0;
    int lo = 1 << 20, hi = -(1 << 20);
    for (int e0 = lane; e0 < E; e0 += 256) {
      uint32_t x[8];  // eight loads in flight; +0 past E changes neither the sum nor its range
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = e0 + 32 * k < E ? q_at(e0 + 32 * k) : 0u;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if ((x[k] & 0x7fffu) != 0u) {
          int l, h;
          bf16_exp_range(x[k], l, h);
          lo = min(lo, l);
          hi = max(hi, h);
        }
        part = __dadd_rn(part, (double)bf16_bits_to_f32(x[k]));
      }
    }
    lo = __reduce_min_sync(kFull, lo);
    hi = __reduce_max_sync(kFull, hi);
    double sum;
    const int lg = 32 - __clz(E - 1);  // ceil(log2 E)
    if (hi - lo + 1 + lg <= 52 || hi < lo) {
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) part = __dadd_rn(part, __shfl_xor_sync(kFull, part, d));
      sum = part;
    } else {
      sum = 0.0;
      if (lane == 0)
        for (int e = 0; e < E; ++e) sum = __dadd_rn(sum, (double)bf16_bits_to_f32(q_at(e)));
    }
    if (lane == 0) mean = __ddiv_rn(sum, (double)E);
  }
  sync();
  if (threadIdx.x < E) b_next[threadIdx.x] = __double2float_rn(__dsub_rn((double)bf16_bits_to_f32(mine), mean));
  for (int e = threadIdx.x + nthreads; e < E; e += nthreads)
    b_next[e] = __double2float_rn(__dsub_rn((double)bf16_bits_to_f32(q_at(e)), mean));
}

}  // namespace eqb
