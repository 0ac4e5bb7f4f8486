// lei.cu -- Load-Error Injection (arXiv 2609.28053, Sec. 4, Eq. (LEI) and
// Eq. (norm)).
//
// For microbatch l with n_l tokens and loads f_{l,e}:
//   rho_e = f_{l,e} / (K n_l / E) - 1,
//   sigma = tanh(xi) / xi with xi = max_e |rho_e| / c   (c > 0; 1 at xi = 0),
//   sigma = 1                                            (c <= 0, unnormalised),
//   grad_s[t, e] += eta * sigma * rho_e   for every t of the microbatch, every e.
//
// The path is a pure HBM stream (read and write grad_s once), so each CTA
// takes a contiguous token range, computes the E coefficients of each
// microbatch it meets (fp64, the threads striding over the experts, a block
// max for xi) into shared memory as fp32, and then streams its range with
// 16-byte loads and stores using evict-first cache hints.
//
// For the one-call step the coefficients are also formed once per microbatch
// into an [M,E] table (lei_coef_kernel, or blocks of the coarse histogram
// pass), from which the fine pass streams the injection beside its own work
// (hist.cu).
#include "lei_device.cuh"

namespace eqb {

namespace {

constexpr int kLeiThreads = 256;
constexpr int kLeiUnroll = 4;

__global__ void __launch_bounds__(kLeiThreads) lei_kernel(LeiArgs a, int64_t tokens_per_cta) {
  __shared__ __align__(16) float coef[kMaxE];
  griddep_wait();
  const int E = a.E, E4 = a.E >> 2;
  const int64_t tb = (int64_t)blockIdx.x * tokens_per_cta;
  const int64_t te = min(tb + tokens_per_cta, a.T);
  if (tb >= te) return;
  float4* g4 = reinterpret_cast<float4*>(a.g);
  const float4* c4 = reinterpret_cast<const float4*>(coef);

  int64_t t = tb;
  while (t < te) {
    const int l = microbatch_of(a.off, a.M, t + a.tbase);
    const int64_t lo = __ldg(a.off + l) - a.tbase, hi = __ldg(a.off + l + 1) - a.tbase;
    // Malformed offsets (off[M] < T) must not stall the loop: tokens past
    // the last boundary are treated as the last microbatch's.
    const int64_t seg_end = (hi > t) ? min(te, hi) : te;
    block_lei_coef<kLeiThreads>(a.loads + (int64_t)l * E, hi - lo, E, a.K, a.eta, a.c, coef);

    // ---- stream grad_s[t .. seg_end) in float4 units
    const int64_t i0 = t * E4, i1 = seg_end * E4;
    const int S = blockDim.x;
    const int dcol = S % E4;
    int col = threadIdx.x % E4;
    int64_t i = i0 + threadIdx.x;
    for (; i + (int64_t)(kLeiUnroll - 1) * S < i1; i += (int64_t)kLeiUnroll * S) {
      float4 v[kLeiUnroll];
      int cc[kLeiUnroll];
#pragma unroll
      for (int u = 0; u < kLeiUnroll; ++u) {
        v[u] = __ldcs(g4 + i + (int64_t)u * S);
        cc[u] = col;
        col += dcol;
        if (col >= E4) col -= E4;
      }
#pragma unroll
      for (int u = 0; u < kLeiUnroll; ++u) {
        const float4 cf = c4[cc[u]];
        v[u].x = __fadd_rn(v[u].x, cf.x);
        v[u].y = __fadd_rn(v[u].y, cf.y);
        v[u].z = __fadd_rn(v[u].z, cf.z);
        v[u].w = __fadd_rn(v[u].w, cf.w);
        __stcs(g4 + i + (int64_t)u * S, v[u]);
      }
    }
    for (; i < i1; i += S) {
      float4 v = __ldcs(g4 + i);
      const float4 cf = c4[col];
      v.x = __fadd_rn(v.x, cf.x);
      v.y = __fadd_rn(v.y, cf.y);
      v.z = __fadd_rn(v.z, cf.z);
      v.w = __fadd_rn(v.w, cf.w);
      __stcs(g4 + i, v);
      col += dcol;
      if (col >= E4) col -= E4;
    }
    t = seg_end;
  }
}

// One block per microbatch: row l of the [M,E] coefficient table.
__global__ void __launch_bounds__(kLeiThreads) lei_coef_kernel(LeiArgs a, float* coef) {
  griddep_wait();
  griddep_launch();
  const int l = blockIdx.x;
  const int64_t n = __ldg(a.off + l + 1) - __ldg(a.off + l);
  block_lei_coef<kLeiThreads>(a.loads + (int64_t)l * a.E, n, a.E, a.K, a.eta, a.c, coef + (int64_t)l * a.E);
}

}  // namespace

int launch_lei_coef(const LeiArgs& a, float* coef, cudaStream_t s) {
  if (a.M < 1) return kErrInvalidArg;
  return launch_dependent(lei_coef_kernel, dim3((unsigned)a.M), dim3(kLeiThreads), 0, s, a, coef) ==
                 cudaSuccess
             ? kOk
             : kErrCuda;
}

int launch_lei(const LeiArgs& a, cudaStream_t s) {
  DeviceInfo di;
  if (int rc = device_info(&di)) return rc;
  int64_t grid = (int64_t)di.sm_count * 8;
  // At least 256 tokens per CTA, so that the per-microbatch prologue stays
  // small, but no fewer CTAs than SMs while they have 16 tokens.
  int64_t least = a.T / di.sm_count;
  least = least < 16 ? 16 : least > 256 ? 256 : least;
  const int64_t max_grid = (a.T + least - 1) / least;
  if (grid > max_grid) grid = max_grid;
  if (grid < 1) grid = 1;
  const int64_t tpc = (a.T + grid - 1) / grid;
  return launch_dependent(lei_kernel, dim3((unsigned)grid), dim3(kLeiThreads), 0, s, a, tpc) == cudaSuccess
             ? kOk
             : kErrCuda;
}

}  // namespace eqb
