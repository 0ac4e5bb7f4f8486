// eqb_internal.h -- launch-side declarations shared by the .cu files of
// libeqb.so (not part of the public ABI; see include/eqb.h for that).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace eqb {

// Status codes mirrored from eqb.h for device code.
enum : int {
  kOk = 0,
  kErrInvalidArg = 1,
  kErrUnsupported = 2,
  kErrCuda = 3,
  kErrNonfinite = 4,
  kErrRank = 5,
};

constexpr int kMaxDevices = 64;

struct DeviceInfo {
  int dev;             // its number, below kMaxDevices
  int sm_count;
  int max_smem_optin;  // bytes of dynamic shared memory a block may opt into
};

// Cached per-device attributes (queried once per device).
int device_info(DeviceInfo* out);

// Load-Error Injection streamed by a histogram pass beside its own work:
// grad_s[t, e] += coef[mb(t), e] for the tokens [t0, t1), from the [M,E]
// coefficient table of launch_lei_coef.  Token numbers are absolute.
struct LeiStream {
  float* g = nullptr;  // nullptr: no injection
  const float* coef = nullptr;
  const int64_t* off = nullptr;
  int M = 0;
  int64_t t0 = 0, t1 = 0;
  int warps = 0;  // of a block that only stream (set at the launch)
};

struct RouteArgs {
  const uint16_t* z;
  const float* b;
  int64_t T;
  int E, K;
  const int64_t* off;  // microbatch boundaries, absolute token numbers
  int M;
  int64_t tbase;       // absolute number of token 0 of this call
  int32_t* idx;
  float* tau;
  int32_t* loads;
  int32_t* err;
};

// Largest expert count of the routing, EQB, LEI, GShard and MaxVio paths
// (per-expert state of the per-microbatch kernels lives in shared memory).
constexpr int kMaxE = 1024;

// Most microbatches of MaxVio (a double each in shared memory).
constexpr int kMaxMicrobatches = 16384;

// Most expert tiles a histogram pass is cut into.
constexpr int kMaxHistTiles = 31;

struct HistArgs {
  const uint16_t* z;
  const float* tau;
  int64_t T;
  int E;
  const uint8_t* u;  // pass 2 only
  int32_t* hist;
  int32_t* err;
  float lo = 0.f, inv_w = 0.f;  // pass 3 (equal-width bins) only
  // Optional token shards (device int64 [P+1]): shard p's counts go to
  // hist + p*E*256, and pass 2 takes shard p's selected bins from u + p*E.
  const int64_t* shard_off = nullptr;
  int P = 0;
  // Algorithm 1's selections inside pass 2 (the one-call step; no shards):
  // with `coarse` (pass 1's [E,256] counts) every block selects u, rho of its
  // experts at rank r itself (one of them also into sel_u, sel_rho).  With
  // `done` (zero before the pass), done[i] counts the blocks of expert tile i
  // that finished, the tile's last one selects its q_hat, done[kMaxHistTiles]
  // counts the tiles selected, and the last one forms b_next (Eq. 2).  Selection flags go to sel_err.
  const int32_t* coarse = nullptr;
  int32_t* done = nullptr;
  int32_t r = 0;
  uint8_t* sel_u = nullptr;
  int32_t* sel_rho = nullptr;
  uint16_t* q_hat = nullptr;
  float* b_next = nullptr;
  int32_t* sel_err = nullptr;
};

struct LeiArgs {
  float* g;
  const int32_t* loads;
  const int64_t* off;  // microbatch boundaries, absolute token numbers
  int M;
  int64_t tbase;       // absolute number of token 0 of this call
  int64_t T;
  int E, K;
  float eta, c;
};

struct GshardArgs {
  float* g;
  const uint16_t* z;
  const int32_t* loads;
  const int64_t* off;
  int M;
  int64_t T;
  int E, K;
  float alpha;
};

// Capacity (floats) of the step's LEI coefficient table: the fused step
// (injection streamed by the histogram passes) runs when M * E fits.
constexpr int64_t kLeiCoefCap = 65536;

// The step's scratch, carved from one caller-provided buffer (256-byte
// aligned pieces): the two [E,256] histograms and the fine pass's block
// counters (adjacent, cleared together before every step), u, rho, q_hat and
// the [M,E] LEI coefficient table.
struct StepWorkspace {
  int32_t* H;
  int32_t* L;
  int32_t* done;  // kMaxHistTiles + 1 counters
  uint8_t* u;
  int32_t* rho;
  uint16_t* q;
  float* coef;
};
constexpr size_t kDoneBytes = (kMaxHistTiles + 1) * 4;
constexpr size_t carve_round(size_t n) { return (n + 255) / 256 * 256; }
constexpr size_t step_workspace_bytes(int E) {
  return 2 * carve_round(static_cast<size_t>(E) * 1024) + carve_round(kDoneBytes) +
         carve_round(static_cast<size_t>(E)) + carve_round(4 * static_cast<size_t>(E)) +
         carve_round(2 * static_cast<size_t>(E)) + carve_round(4 * static_cast<size_t>(kLeiCoefCap));
}
// Carves `base` (or, with base == nullptr, only measures); returns the bytes
// used, step_workspace_bytes(E) by construction.
size_t carve_workspace(void* base, int E, StepWorkspace* w);
// Zeros the workspace's histograms and counters and the loads [n]: the first
// kernel of a step.
int launch_clear(const StepWorkspace& w, int E, int32_t* loads, int64_t n, cudaStream_t s);

int launch_route(const RouteArgs& a, cudaStream_t s);
// The routing kernels of compile-time row widths (K + 1 <= 16): E <= 128 and
// E <= 640.
int launch_route_narrow(const RouteArgs& a, cudaStream_t s);
int launch_route_wide(const RouteArgs& a, cudaStream_t s);
// One warp per token (any E, K + 1 <= 32).
int launch_route_warp(const RouteArgs& a, cudaStream_t s);
// Routing and the coarse histogram (hist, [E,256] +=) in one pass over z
// (route_hist.cu; E = 128 or 256, K + 1 <= 16).
bool route_hist_supported(int E, int K);
int launch_route_hist(const RouteArgs& a, int32_t* hist, cudaStream_t s);
int launch_hist(const HistArgs& a, int pass, cudaStream_t s);
// Pass 1 with a few of its blocks forming the [M,E] LEI coefficient table of
// `la` (the step: the loads are complete, the fine pass injects).
int launch_hist_coef(const HistArgs& a, const LeiArgs& la, float* coef, cudaStream_t s);
// A histogram pass (1 or 2) with the injection `ls` streamed beside it.
int launch_hist_lei(const HistArgs& a, int pass, const LeiStream& ls, cudaStream_t s);
int launch_select(const int32_t* hist, int E, int pass, int64_t r, uint8_t* u, int32_t* rho,
                  uint16_t* q_hat, int32_t* err, cudaStream_t s);
// One selection per token shard (device int64 [P+1]): shard p reads
// hist + p*E*256 and writes u, rho, q_hat + p*E at its own rank
// ceil(n_p K / E); an empty shard gets u = rho = 0 and q_hat = +0.
int launch_select_sharded(const int32_t* hist, int E, int pass, const int64_t* shard_off, int P, int K,
                          uint8_t* u, int32_t* rho, uint16_t* q_hat, int32_t* err, cudaStream_t s);
int launch_bias_update(const uint16_t* q_hat, int E, float* b_next, cudaStream_t s);
int launch_lei(const LeiArgs& a, cudaStream_t s);
// The [M,E] fp32 table of Eq. (norm) coefficients, row l for microbatch l
// (bit-identical to the coefficients launch_lei forms).
int launch_lei_coef(const LeiArgs& a, float* coef, cudaStream_t s);
// z = bf16(x W^T).  With `split`, few tokens take the split kernel below.
int launch_router_gemm(const uint16_t* x, const uint16_t* W, int64_t T, int d, int E, uint16_t* z,
                       int32_t* err, bool split, cudaStream_t s);
// Few tokens (router_split.cu): a cluster of n blocks shares each 128-token
// tile, every block a part of the columns of x; router_splits says how many
// pay (1: the persistent kernel).  With ro.b the tokens are routed too.
struct SplitRoute {
  const float* b = nullptr;
  int K = 0;
  const int64_t* off = nullptr;
  int M = 0;
  int32_t* idx = nullptr;
  float* tau = nullptr;
  int32_t* loads = nullptr;
};
int router_splits(int64_t T, int d, int E, int sm_count);
// Many experts, columns and tokens (router_pair.cu; E a multiple of 32, at
// most 256): pairs of SMs.
int launch_router_pair(const uint16_t* x, const uint16_t* W, int64_t T, int d, int E, uint16_t* z, int32_t* err,
                       cudaStream_t s);
int launch_router_split(const uint16_t* x, const uint16_t* W, int64_t T, int d, int E, int n, uint16_t* z,
                        const SplitRoute& ro, int32_t* err, cudaStream_t s);
int launch_gshard(const GshardArgs& a, cudaStream_t s);
int launch_maxvio(const int32_t* loads, const int64_t* off, int M, int E, int K, double* out, double* per_mb,
                  cudaStream_t s);
// The router projection routing each token from its accumulators (E = 64 or
// 128, K <= 8); with hist (nullable) also the coarse histogram ([E,256] +=),
// counted in the epilogue when no block routes more than 65,535 tokens, else
// by the coarse pass over z after it.  `split` as for launch_router_gemm.
int launch_router_route(const uint16_t* x, const uint16_t* W, int64_t T, int d, int E, int K, const float* b,
                        const int64_t* off, int M, uint16_t* z, int32_t* idx, float* tau, int32_t* loads,
                        int32_t* hist, int32_t* err, bool split, cudaStream_t s);

}  // namespace eqb
