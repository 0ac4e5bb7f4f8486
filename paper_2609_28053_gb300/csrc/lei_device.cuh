// lei_device.cuh -- the coefficients of Eq. (norm) (arXiv 2609.28053, Sec. 4)
// for one microbatch, formed by one block: shared by the LEI kernels (lei.cu)
// and by the blocks of the coarse histogram pass that form the step's
// coefficient table (hist.cu).
#pragma once

#include <limits.h>

#include "eqb_device.cuh"

namespace eqb {

// Eq. (norm) coefficients eta * sigma * rho_e of one microbatch with n tokens
// and loads f (one row of [M,E]), computed by a whole block of NT threads
// into out[0..E) (shared or global memory) and visible to the block on return.
// fp64 runs at two lanes a clock per SM here, so each expert takes one
// multiply-add and one multiply in fp64 at the end and nothing before:
// max |rho| lies at the largest or the smallest load (rho grows with the
// load, rounding included), which integer reductions find.
template <int NT>
__device__ __forceinline__ void block_lei_coef(const int32_t* __restrict__ f, int64_t n, int E, int K, float eta, float c,
                               float* out) {
  __shared__ int2 red[NT / 32];  // least and largest load of each warp's experts
  __shared__ double scal[2];     // 1 / fbar, eta sigma
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // this thread's experts: threadIdx.x + k * NT
  constexpr int kPer = (kMaxE + NT - 1) / NT;
  int load[kPer];
  int lo = INT_MAX, hi = INT_MIN;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int e = threadIdx.x + k * NT;
    load[k] = e < E ? __ldg(f + e) : 0;
    if (e < E) {
      lo = min(lo, load[k]);
      hi = max(hi, load[k]);
    }
  }
  lo = __reduce_min_sync(kFull, lo);
  hi = __reduce_max_sync(kFull, hi);
  __syncthreads();  // a previous call has finished reading red, scal and out
  if (lane == 0) red[wid] = make_int2(lo, hi);
  __syncthreads();
  if (wid == 0) {
    const double inv_fbar = n > 0 ? (double)E / ((double)K * (double)n) : 0.0;
    const int2 r = red[lane < NT / 32 ? lane : 0];
    const int least = __reduce_min_sync(kFull, r.x), most = __reduce_max_sync(kFull, r.y);
    const double rmax = inv_fbar > 0.0 ? fmax(fabs((double)least * inv_fbar - 1.0), fabs((double)most * inv_fbar - 1.0))
                                       : 0.0;
    // sigma = tanh(xi) / xi in fp32: its relative error (a few ulp of fp32)
    // stays far inside the LEI tolerance, and it spares the serial fp64
    // division and tanh of this warp
    float sigma = 1.0f;
    if (c > 0.0f) {
      const float xi = __fdiv_rn(static_cast<float>(rmax), c);
      sigma = (xi == 0.0f) ? 1.0f : __fdiv_rn(tanhf(xi), xi);
    }
    if (lane == 0) {
      scal[0] = inv_fbar;
      scal[1] = (double)eta * (double)sigma;
    }
  }
  __syncthreads();
  const double inv_fbar = scal[0], es = scal[1];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int e = threadIdx.x + k * NT;
    if (e < E) out[e] = __double2float_rn(es * (inv_fbar > 0.0 ? (double)load[k] * inv_fbar - 1.0 : 0.0));
  }
  __syncthreads();
}

// The same coefficients by one warp (bit for bit: the same operations per
// expert, and exact reductions), for blocks that form several rows at once.
__device__ __forceinline__ void warp_lei_coef(const int32_t* __restrict__ f, int64_t n, int E, int K, float eta,
                                              float c, float* out, int lane) {
  int lo = INT_MAX, hi = INT_MIN;
#pragma unroll 8
  for (int e = lane; e < E; e += 32) {
    const int v = __ldg(f + e);
    lo = min(lo, v);
    hi = max(hi, v);
  }
  lo = __reduce_min_sync(kFull, lo);
  hi = __reduce_max_sync(kFull, hi);
  const double inv_fbar = n > 0 ? (double)E / ((double)K * (double)n) : 0.0;
  const double rmax =
      inv_fbar > 0.0 ? fmax(fabs((double)lo * inv_fbar - 1.0), fabs((double)hi * inv_fbar - 1.0)) : 0.0;
  float sigma = 1.0f;
  if (c > 0.0f) {
    const float xi = __fdiv_rn(static_cast<float>(rmax), c);
    sigma = (xi == 0.0f) ? 1.0f : __fdiv_rn(tanhf(xi), xi);
  }
  const double es = (double)eta * (double)sigma;
#pragma unroll 4
  for (int e = lane; e < E; e += 32)
    out[e] = __double2float_rn(es * (inv_fbar > 0.0 ? (double)__ldg(f + e) * inv_fbar - 1.0 : 0.0));
}

}  // namespace eqb
