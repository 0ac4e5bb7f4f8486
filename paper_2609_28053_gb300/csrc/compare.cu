// compare.cu -- the two estimates of the global quantile that Sec. 2 of
// arXiv 2609.28053 contrasts with EQB, on the GPU:
//   rank-averaged QB       every data-parallel shard selects its own K/E
//                          quantile of the margins (exactly, with the same
//                          two radix passes as EQB, run over all shards at
//                          once with one histogram per shard), the shards'
//                          quantiles are averaged and centered as in Eq. (2);
//   fixed-resolution bins  256 equal-width bins of the margins summed over
//                          all tokens; the estimate is the upper edge of the
//                          first bin whose cumulative count reaches r,
//                          centered as in Eq. (2).
// Both finish with one small kernel that forms the fp64 estimates, sums them
// in ascending expert order for the mean and writes b_e = fp32(x_e - mean).
#include <cuda_runtime.h>
#include <stdint.h>

#include "eqb.h"
#include "eqb_device.cuh"

namespace eqb {

namespace {

// b_e = fp32(x_e - mean(x)), mean summed sequentially in ascending e.
__device__ void center_store(double* x, int E, float* b) {
  __shared__ double mean;
  __syncthreads();
  if (threadIdx.x == 0) {
    double acc = 0.0;
    for (int e = 0; e < E; e += 8) {  // E is a multiple of 8: eight reads ahead of the chain of sums
      double v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = x[e + k];
#pragma unroll
      for (int k = 0; k < 8; ++k) acc += v[k];
    }
    mean = acc / (double)E;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < E; e += blockDim.x) b[e] = __double2float_rn(x[e] - mean);
}

// Average of the non-empty shards' quantiles (bf16 [P,E]) per expert,
// summed over the shards in ascending order, then centered.
__global__ void __launch_bounds__(256) shard_average_kernel(const uint16_t* q, const int64_t* off, int P, int E,
                                                            float* b) {
  __shared__ double x[kMaxE];
  griddep_wait();
  for (int e = threadIdx.x; e < E; e += blockDim.x) {
    double acc = 0.0;
    int cnt = 0;
    for (int p0 = 0; p0 < P; p0 += 8) {  // eight shards' loads in flight
      uint32_t v[8];
      bool some[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int p = min(p0 + k, P - 1);
        v[k] = q[(int64_t)p * E + e];
        some[k] = p0 + k < P && off[p + 1] > off[p];
      }
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (some[k]) {
          acc += (double)bf16_bits_to_f32(v[k]);
          ++cnt;
        }
    }
    x[e] = acc / (double)cnt;
  }
  center_store(x, E, b);
}

// The first kernel of a comparison: zeros n16 16-byte words of its histograms
// and, up to kParamShards shards, writes the shard offsets, which come as an
// argument (in place of two memsets and a copy from pageable memory, none of
// which overlap anything).
constexpr int kParamShards = 128;
struct ShardOffsets {
  int64_t v[kParamShards + 1];
};
__global__ void __launch_bounds__(256) setup_kernel(uint4* w, int64_t n16, int64_t* off, int n,
                                                    const __grid_constant__ ShardOffsets so) {
  griddep_wait();
  griddep_launch();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += stride)
    w[i] = make_uint4(0u, 0u, 0u, 0u);
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < n; i += blockDim.x) off[i] = so.v[i];
}
int launch_setup(void* w, size_t bytes, int64_t* off, const int64_t* off_host, int n, cudaStream_t s) {
  ShardOffsets so;
  for (int i = 0; i < n; ++i) so.v[i] = off_host[i];
  const int64_t n16 = static_cast<int64_t>(bytes / 16);
  const int64_t grid = (n16 + 1023) / 1024;
  return launch_dependent(setup_kernel, dim3((unsigned)(grid < 608 ? grid : 608)), dim3(256), 0, s,
                          static_cast<uint4*>(w), n16, off, n, so) == cudaSuccess
             ? kOk
             : kErrCuda;
}

// Scratch of the rank average: per-shard histograms H and L [P,E,256],
// u [P,E], rho [P,E] int32 and the shard offsets [P+1] int64.
struct ShardWs {
  int32_t *H, *L;
  uint8_t* u;
  int32_t* rho;
  int64_t* off;
};
size_t carve_shards(void* base, int E, int P, ShardWs* w) {
  size_t o = 0;
  auto take = [&](size_t n) {
    uint8_t* p = base ? static_cast<uint8_t*>(base) + o : nullptr;
    o = (o + n + 255) / 256 * 256;
    return p;
  };
  const size_t PE = (size_t)P * (size_t)E;
  w->H = reinterpret_cast<int32_t*>(take(PE * 256 * 4));
  w->L = reinterpret_cast<int32_t*>(take(PE * 256 * 4));
  w->u = take(PE);
  w->rho = reinterpret_cast<int32_t*>(take(PE * 4));
  w->off = reinterpret_cast<int64_t*>(take(((size_t)P + 1) * 8));
  return o;
}

// Upper edge lo + (u_e + 1) w of the selected bin, then centered.
__global__ void __launch_bounds__(256) bin_edge_kernel(const uint8_t* u, int E, float lo, float w, float* b,
                                                       double* est) {
  __shared__ double x[kMaxE];
  griddep_wait();
  for (int e = threadIdx.x; e < E; e += blockDim.x) {
    x[e] = (double)lo + (double)(u[e] + 1) * (double)w;
    if (est) est[e] = x[e];
  }
  center_store(x, E, b);
}

inline eqb_status st(int rc) { return static_cast<eqb_status>(rc); }
inline bool aligned(const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

eqb_status check_common(const eqb_bf16* z, const float* tau, int64_t T, int32_t E, int32_t K, float* b_out,
                        void* workspace, int32_t* err_flag) {
  if (T < 1 || E < 2 || K < 1 || K >= E) return EQB_ERR_INVALID_ARG;
  if (E > kMaxE || (E % 8) != 0) return EQB_ERR_UNSUPPORTED;
  if (T > (int64_t(1) << 31) - (int64_t(1) << 24)) return EQB_ERR_UNSUPPORTED;
  if (!z || !tau || !b_out || !workspace) return EQB_ERR_INVALID_ARG;
  if (!aligned(z, 16) || !aligned(tau, 4) || !aligned(b_out, 4) || !aligned(workspace, 256) ||
      !aligned(err_flag, 4))
    return EQB_ERR_INVALID_ARG;
  return EQB_OK;
}

}  // namespace

}  // namespace eqb

extern "C" {

size_t eqb_rank_averaged_workspace_bytes(int32_t E, int32_t P) {
  if (E < 1 || P < 1) return 0;
  eqb::ShardWs w;
  return eqb::carve_shards(nullptr, E, P, &w);
}

eqb_status eqb_rank_averaged_bias(const eqb_bf16* z, const float* tau, int64_t T, int32_t E, int32_t K,
                                  const int64_t* shard_offsets_host, int32_t P, eqb_bf16* q_shards,
                                  float* b_out, void* workspace, size_t workspace_bytes, int32_t* err_flag,
                                  void* stream) {
  eqb_status rs = eqb::check_common(z, tau, T, E, K, b_out, workspace, err_flag);
  if (rs != EQB_OK) return rs;
  if (P < 1 || P > 65535 || !shard_offsets_host || !q_shards || !eqb::aligned(q_shards, 2))
    return EQB_ERR_INVALID_ARG;
  if (shard_offsets_host[0] != 0 || shard_offsets_host[P] != T) return EQB_ERR_INVALID_ARG;
  for (int p = 0; p < P; ++p)
    if (shard_offsets_host[p + 1] < shard_offsets_host[p]) return EQB_ERR_INVALID_ARG;
  eqb::ShardWs w;
  if (eqb::carve_shards(workspace, E, P, &w) > workspace_bytes) return EQB_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  // H and L are adjacent (each a multiple of 256 bytes)
  const size_t hb = 2 * (size_t)P * (size_t)E * 256 * 4;
  const int n = P <= eqb::kParamShards ? P + 1 : 0;
  if (n == 0 && cudaMemcpyAsync(w.off, shard_offsets_host, ((size_t)P + 1) * 8, cudaMemcpyHostToDevice, s) !=
                    cudaSuccess)
    return EQB_ERR_CUDA;
  if (int rc = eqb::launch_setup(w.H, hb, w.off, shard_offsets_host, n, s)) return eqb::st(rc);
  // Both radix passes over all tokens at once, each shard counted into its
  // own histogram, then one selection per (shard, expert).
  eqb::HistArgs h1{z, tau, T, E, nullptr, w.H, err_flag};
  h1.shard_off = w.off;
  h1.P = P;
  if (int rc = eqb::launch_hist(h1, 1, s)) return eqb::st(rc);
  if (int rc = eqb::launch_select_sharded(w.H, E, 1, w.off, P, K, w.u, w.rho, nullptr, err_flag, s))
    return eqb::st(rc);
  eqb::HistArgs h2{z, tau, T, E, w.u, w.L, nullptr};
  h2.shard_off = w.off;
  h2.P = P;
  if (int rc = eqb::launch_hist(h2, 2, s)) return eqb::st(rc);
  if (int rc = eqb::launch_select_sharded(w.L, E, 2, w.off, P, K, w.u, w.rho, q_shards, err_flag, s))
    return eqb::st(rc);
  return eqb::launch_dependent(eqb::shard_average_kernel, dim3(1), dim3(256), 0, s,
                               static_cast<const uint16_t*>(q_shards), static_cast<const int64_t*>(w.off), (int)P,
                               (int)E, b_out) == cudaSuccess
             ? EQB_OK
             : EQB_ERR_CUDA;
}

eqb_status eqb_fixed_hist_bias(const eqb_bf16* z, const float* tau, int64_t T, int32_t E, int32_t K, float lo,
                               float width, float* b_out, double* estimate, void* workspace,
                               size_t workspace_bytes, int32_t* err_flag, void* stream) {
  eqb_status rs = eqb::check_common(z, tau, T, E, K, b_out, workspace, err_flag);
  if (rs != EQB_OK) return rs;
  if (!(width > 0.0f) || width == INFINITY || !(lo == lo) || lo == INFINITY || lo == -INFINITY)
    return EQB_ERR_INVALID_ARG;
  if (!eqb::aligned(estimate, 8)) return EQB_ERR_INVALID_ARG;
  eqb::StepWorkspace w;
  if (eqb::carve_workspace(workspace, E, &w) > workspace_bytes) return EQB_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (int rc = eqb::launch_setup(w.H, (size_t)E * 1024, nullptr, nullptr, 0, s)) return eqb::st(rc);
  eqb::HistArgs h{z, tau, T, E, nullptr, w.H, err_flag};
  h.lo = lo;
  h.inv_w = 1.0f / width;
  if (int rc = eqb::launch_hist(h, 3, s)) return eqb::st(rc);
  const int64_t r = eqb_target_rank(T, E, K);
  if (int rc = eqb::launch_select(w.H, E, 3, r, w.u, w.rho, nullptr, err_flag, s)) return eqb::st(rc);
  return eqb::launch_dependent(eqb::bin_edge_kernel, dim3(1), dim3(256), 0, s, static_cast<const uint8_t*>(w.u),
                               (int)E, lo, width, b_out, estimate) == cudaSuccess
             ? EQB_OK
             : EQB_ERR_CUDA;
}

}  // extern "C"
