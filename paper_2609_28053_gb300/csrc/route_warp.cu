// route_warp.cu -- top-K routing, cutoff tau_t and per-microbatch loads
// (Sec. 2, Eq. 1 and the QB paragraph of arXiv 2609.28053) with one warp per
// token: for batches too small to fill the machine with 32-token tiles, where
// a tile's serial work is what a call takes, and for rows too wide for tiles
// in shared memory.
//
// Lanes read the row straight into registers, the next token's while this one
// is routed.  The steps are those of warp_route (route_warp.cuh) for runs of
// eight experts, written out: as a call of such a function they compile to a
// schedule that takes 2% longer at K = 2, 10% at 8 and 14% at 12 (T = 300,000, E
// = 1024, K = 8 274 us against 250).  What is mended here is mended there.
#include "route_warp.cuh"

namespace eqb {

namespace {

constexpr int kWarps = 8;  // per block
// Blocks that an SM holds, by registers (48, 62 and 110 a thread).
template <int CPL>
constexpr int kResident = CPL == 1 ? 5 : CPL == 2 ? 4 : 2;

// CPL chunks per lane: rows of up to 256 * CPL experts.
template <int CPL>
__global__ void __launch_bounds__(32 * kWarps, kResident<CPL>)
    route_warp_kernel(RouteArgs a, int tokens_per_block, int count_shared) {
  constexpr int N = 8 * CPL;
  __shared__ __align__(16) float bs[256 * CPL];
  __shared__ int cnt[256 * CPL];  // the block's loads of one microbatch (count_shared)
  __shared__ uint2 cand[kWarps][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int E = a.E, K = a.K, nch = E >> 3;

  const int64_t tb = min((int64_t)blockIdx.x * tokens_per_block, a.T);
  const int64_t te = min(tb + tokens_per_block, a.T);
  griddep_wait();
  auto load_row = [&](int64_t t, uint4 (&w)[CPL]) {
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
      const int c = lane + 32 * k;
      w[k] = t < te && c < nch ? __ldg(reinterpret_cast<const uint4*>(a.z + t * E) + c)
                               : make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u);
    }
  };
  uint4 w[CPL];
  load_row(tb + wid, w);
  for (int e = threadIdx.x; e < 256 * CPL; e += blockDim.x) {
    const float v = e < E ? a.b[e] : 0.f;
    bs[e] = v;
    cnt[e] = 0;
    if (!isfinite(v)) raise_flag(a.err, kErrNonfinite);
  }
  __syncthreads();

  int mb = 0;
  int64_t mb_lo = 1, mb_hi = 0;  // token range of mb (none yet)
  int64_t t = tb + wid;          // this warp's next token
  for (int64_t s0 = tb; s0 < te;) {
    // one segment: the whole range, or its part in one microbatch
    int64_t s1 = te;
    if (count_shared) {
      mb = warp_microbatch_of(a.off, a.M, s0 + a.tbase, lane);
      const int64_t hi = __ldg(a.off + mb + 1) - a.tbase;
      if (hi > s0 && hi < s1) s1 = hi;
    }
    for (; t < s1; t += kWarps) {
      // ---- scores, lane maximum
      float s[N];
      float lmax = -INFINITY;
#pragma unroll
      for (int k = 0; k < CPL; ++k) {
        const float4 b0 = reinterpret_cast<const float4*>(bs)[2 * (lane + 32 * k)];
        const float4 b1 = reinterpret_cast<const float4*>(bs)[2 * (lane + 32 * k) + 1];
        s[8 * k + 0] = bf16_lo(w[k].x) + b0.x;
        s[8 * k + 1] = bf16_hi(w[k].x) + b0.y;
        s[8 * k + 2] = bf16_lo(w[k].y) + b0.z;
        s[8 * k + 3] = bf16_hi(w[k].y) + b0.w;
        s[8 * k + 4] = bf16_lo(w[k].z) + b1.x;
        s[8 * k + 5] = bf16_hi(w[k].z) + b1.y;
        s[8 * k + 6] = bf16_lo(w[k].w) + b1.z;
        s[8 * k + 7] = bf16_hi(w[k].w) + b1.w;
#pragma unroll
        for (int i = 0; i < 8; ++i) lmax = fmax_nan(lmax, s[8 * k + i]);
      }
      load_row(t + kWarps, w);
      if (lmax != lmax) raise_flag(a.err, kErrNonfinite);

      // ---- bound: the (K+1)st largest lane maximum
      uint32_t key = score_key(lmax), theta = 0u;
      for (int r = 0; r <= K; ++r) {
        theta = __reduce_max_sync(kFull, key);
        if (key == theta) key = 0u;
      }

      // ---- the experts at or above it (a NaN counts as above)
      uint32_t m = 0u;
      const uint32_t tu = theta ^ ((theta & 0x80000000u) ? 0x80000000u : 0xffffffffu);
      const float th = theta == 0u ? -INFINITY : __uint_as_float(tu);
#pragma unroll
      for (int i = 0; i < N; ++i) m |= (!(s[i] < th) ? 1u : 0u) << i;
      // experts past E are -inf: only in when everything is
      const int total = __reduce_add_sync(kFull, __popc(m));

      int my_e = 0;          // entry `rank` of the list
      float my_s = -INFINITY;
      int rank = 32;
      if (total <= 32) {
        int base = 0;
        unsigned more = __ballot_sync(kFull, m != 0u);
        while (more) {
          const int i = __ffs(m) - 1;
          float si = s[0];
#pragma unroll
          for (int q = 1; q < N; ++q) si = i == q ? s[q] : si;
          if (m != 0u) {
            const int e = 8 * (lane + 32 * (i >> 3)) + (i & 7);
            cand[wid][base + __popc(more & ((1u << lane) - 1u))] =
                make_uint2(__float_as_uint(si != si ? INFINITY : si), e);
          }
          base += __popc(more);
          m &= m - 1u;
          more = __ballot_sync(kFull, m != 0u);
        }
        __syncwarp();
        if (lane < total) {
          const uint2 mine = cand[wid][lane];
          my_s = __uint_as_float(mine.x);
          my_e = static_cast<int>(mine.y);
          rank = 0;
          for (int q = 0; q < total; ++q) {
            const uint2 o = cand[wid][q];
            const float os = __uint_as_float(o.x);
            rank += os > my_s || (os == my_s && static_cast<int>(o.y) < my_e) ? 1 : 0;
          }
        }
        __syncwarp();  // every lane has read the list
      } else {
        uint32_t gone = 0u;  // this lane's experts already listed
        for (int r = 0; r <= K; ++r) {
          float best = -INFINITY;
          int bi = -1;
#pragma unroll
          for (int i = 0; i < N; ++i) {
            const bool in = !(gone >> i & 1u) && 8 * (lane + 32 * (i >> 3)) < E;
            if (in && (bi < 0 || s[i] > best)) {
              best = s[i];
              bi = i;
            }
          }
          const uint32_t bk = bi < 0 ? 0u : score_key(best);
          const uint32_t top = __reduce_max_sync(kFull, bk);
          const unsigned be = bi < 0 ? 0xffffu : 8u * (lane + 32 * (bi >> 3)) + (bi & 7);
          const unsigned win = __reduce_min_sync(kFull, bk == top ? be : 0xffffu);
          const bool mine = bi >= 0 && be == win;
          if (mine) gone |= 1u << bi;
          const float ws = __shfl_sync(kFull, best, __ffs(__ballot_sync(kFull, mine)) - 1);
          if (lane == r) {
            my_e = static_cast<int>(win);
            my_s = ws;
            rank = r;
          }
        }
      }

      // ---- outputs
      if (rank == K) {
        a.tau[t] = my_s;
        if (!isfinite(my_s)) raise_flag(a.err, kErrNonfinite);
      }
      if (rank < K) {
        if (a.idx) a.idx[t * K + rank] = my_e;
        if (count_shared) atomicAdd(cnt + my_e, 1);
      }
      if (a.loads && !count_shared) {
        const int64_t at = t + a.tbase;
        if (!(at >= mb_lo && at < mb_hi)) {
          mb = warp_microbatch_of(a.off, a.M, at, lane);
          mb_lo = __ldg(a.off + mb);
          mb_hi = __ldg(a.off + mb + 1);
        }
        if (rank < K) atomicAdd(a.loads + (int64_t)mb * E + my_e, 1);
      }
    }
    if (count_shared) {
      __syncthreads();
      for (int e = threadIdx.x; e < E; e += blockDim.x) {
        const int v = cnt[e];
        cnt[e] = 0;
        if (v) atomicAdd(a.loads + (int64_t)mb * E + e, v);
      }
      __syncthreads();
    }
    s0 = s1;
  }
}

template <int CPL>
int launch_warp_t(const RouteArgs& a, cudaStream_t s) {
  DeviceInfo di;
  if (int rc = device_info(&di)) return rc;
  auto kern = route_warp_kernel<CPL>;
  static std::atomic<int> known[kMaxDevices];
  const int per_sm = resident_blocks(kern, 32 * kWarps, 0, di.dev, known);
  if (per_sm < 1) return kErrCuda;
  const int64_t most = (int64_t)di.sm_count * per_sm;
  int64_t tpb = (a.T + most - 1) / most;
  tpb = (tpb + kWarps - 1) / kWarps * kWarps;
  const int64_t grid = (a.T + tpb - 1) / tpb;
  // Loads in shared memory where a block has many tokens, or where many tokens
  // share a counter: the few lanes of a token add to scattered words of a few
  // lines, a block's flush to whole lines.  K = 8, us, each token's adds /
  // flushed: T = 4,096, M = 1 (avg. load 256, 128, 64 at E = 128, 256, 512) 10.7
  // / 5.3, 11.9 / 7.0 and 8.3 / 6.5; M = 3 8.3 / 5.3, 7.9 / 5.1 and, at 21, 5.7 /
  // 6.3; M = 16 and more the same or the former.
  const int count_shared = a.loads && (tpb > 256 || a.T * a.K > 40 * (int64_t)a.M * a.E) ? 1 : 0;
  return launch_dependent(kern, dim3((unsigned)grid), dim3(32 * kWarps), 0, s, a, (int)tpb, count_shared) ==
                 cudaSuccess
             ? kOk
             : kErrCuda;
}

}  // namespace

int launch_route_warp(const RouteArgs& a, cudaStream_t s) {
  if (a.K + 1 > 32) return kErrUnsupported;
  if (a.E <= 256) return launch_warp_t<1>(a, s);
  if (a.E <= 512) return launch_warp_t<2>(a, s);
  if (a.E <= 1024) return launch_warp_t<4>(a, s);
  return kErrUnsupported;
}

}  // namespace eqb
