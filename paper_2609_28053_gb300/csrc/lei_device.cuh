// lei_device.cuh -- the coefficients of Eq. (norm) (arXiv 2609.28053, Sec. 4)
// for one microbatch, formed by one block: shared by the LEI kernels (lei.cu)
// and by the blocks of the coarse histogram pass that form the step's
// coefficient table (hist.cu).
#pragma once

#include "eqb_device.cuh"

namespace eqb {

// Eq. (norm) coefficients eta * sigma * rho_e of one microbatch with n tokens
// and loads f (one row of [M,E]), computed by a whole block of NT threads
// into out[0..E) (shared or global memory) and visible to the block
// on return.  fp64 throughput is low on this part, so each thread does only
// a multiply-add and a multiply per expert; the reciprocal of the target
// load and tanh are formed once.
template <int NT>
__device__ __forceinline__ void block_lei_coef(const int32_t* __restrict__ f, int64_t n, int E, int K, float eta, float c,
                               float* out) {
  __shared__ double red[NT / 32];
  __shared__ double scal[2];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();  // a previous call has finished reading scal and out
  if (threadIdx.x == 0) scal[0] = n > 0 ? (double)E / ((double)K * (double)n) : 0.0;  // 1 / fbar
  __syncthreads();
  const double inv_fbar = scal[0];
  // each thread holds the rho of experts threadIdx.x + k * NT
  constexpr int kPer = (kMaxE + NT - 1) / NT;
  double rho[kPer];
  double amax = 0.0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int e = threadIdx.x + k * NT;
    rho[k] = (e < E && inv_fbar > 0.0) ? (double)__ldg(f + e) * inv_fbar - 1.0 : 0.0;
    amax = fmax(amax, fabs(rho[k]));
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) amax = fmax(amax, __shfl_xor_sync(kFull, amax, d));
  if (lane == 0) red[wid] = amax;
  __syncthreads();
  if (wid == 0) {
    double rmax = lane < NT / 32 ? red[lane] : 0.0;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) rmax = fmax(rmax, __shfl_xor_sync(kFull, rmax, d));
    // sigma = tanh(xi) / xi in fp32: its relative error (a few ulp of fp32)
    // stays far inside the LEI tolerance, and it spares the serial fp64
    // division and tanh of this warp
    float sigma = 1.0f;
    if (c > 0.0f) {
      const float xi = __fdiv_rn(static_cast<float>(rmax), c);
      sigma = (xi == 0.0f) ? 1.0f : __fdiv_rn(tanhf(xi), xi);
    }
    if (lane == 0) scal[1] = (double)eta * (double)sigma;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int e = threadIdx.x + k * NT;
    if (e < E) out[e] = __double2float_rn(scal[1] * rho[k]);
  }
  __syncthreads();
}

}  // namespace eqb
