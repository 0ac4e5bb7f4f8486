// route_warp.cuh -- one token routed by one warp (Sec. 2, Eq. 1 and the QB
// paragraph of arXiv 2609.28053): warp_route for the split router projection
// (router_split.cu), and the score key and microbatch search that it shares
// with route_warp.cu, which writes the same steps out for wider rows.
//
// Every lane holds the exact scores s_e = fp32(z_e) + b_e of its share of the
// row, four experts in a run.  The (K+1)st largest of the 32 lane maxima, found
// by K + 1 warp reductions (lanes with equal maxima leave together, which only
// lowers it), is <= tau_t, so the scores >= it hold the top K + 1; about K + 3
// of them do.  They are collected in shared memory, one per lane, each lane
// counts the ones that come before its own (higher score, ties to the lower
// index), and the lane of rank r holds entry r.  A NaN (flagged) is listed as
// +inf, so that the ranks stay a permutation and every output of the token is
// written, with experts in range.  More than 32 of them (many equal scores, or
// fewer than K + 1 lanes with a share) are selected one by one over the whole
// row instead.
#pragma once

#include "eqb_device.cuh"

namespace eqb {

// Order-preserving key of a score; -0 and +0 get the same key (they are equal
// scores).
__device__ __forceinline__ uint32_t score_key(float s) {
  const uint32_t u = __float_as_uint(__fadd_rn(s, 0.0f));
  return u ^ ((u & 0x80000000u) ? 0xffffffffu : 0x80000000u);
}

// Microbatch of token t, as microbatch_of, by a whole warp: each round of
// loads probes 32 boundaries and leaves a 32nd of the microbatches (at most
// three rounds for 8,192 of them).
__device__ __forceinline__ int warp_microbatch_of(const int64_t* __restrict__ off, int M, int64_t t, int lane) {
  int l = 0, n = M;  // the token's is one of [l, l + n)
  while (n > 1) {
    const int step = (n + 30) >> 5;
    const int j = l + step * (lane + 1);
    const int below = __popc(__ballot_sync(kFull, j < l + n && __ldg(off + j) <= t));
    l += below * step;
    n = min(step, n - below * step);
  }
  return l;
}

// One token routed by a whole warp.  s[] are the lane's exact scores, of the
// experts 4 lane .. 4 lane + 3, -inf past E (a multiple of 4), lmax their maximum
// (NaN if there is one); cand 32 entries of the warp's own.  The lane of rank r
// <= K gets entry r of the list: r, the expert my_e and its score my_s (the lane
// of rank K holds the cutoff); the other lanes a rank above K.
__device__ __forceinline__ int warp_route(const float (&s)[4], float lmax, int E, int K, uint2* cand, int lane,
                                          int32_t* err, int& my_e, float& my_s) {
  constexpr int N = 4;
  if (lmax != lmax) raise_flag(err, kErrNonfinite);

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

  my_e = 0;
  my_s = -INFINITY;
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
        const int e = 4 * lane + i;
        cand[base + __popc(more & ((1u << lane) - 1u))] = make_uint2(__float_as_uint(si != si ? INFINITY : si), e);
      }
      base += __popc(more);
      m &= m - 1u;
      more = __ballot_sync(kFull, m != 0u);
    }
    __syncwarp();
    if (lane < total) {
      const uint2 mine = cand[lane];
      my_s = __uint_as_float(mine.x);
      my_e = static_cast<int>(mine.y);
      rank = 0;
      for (int q = 0; q < total; ++q) {
        const uint2 o = cand[q];
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
        const bool in = !(gone >> i & 1u) && 4 * lane < E;
        if (in && (bi < 0 || s[i] > best)) {
          best = s[i];
          bi = i;
        }
      }
      const uint32_t bk = bi < 0 ? 0u : score_key(best);
      const uint32_t top = __reduce_max_sync(kFull, bk);
      const unsigned be = bi < 0 ? 0xffffu : static_cast<unsigned>(4 * lane + bi);
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
  return rank;
}

}  // namespace eqb
