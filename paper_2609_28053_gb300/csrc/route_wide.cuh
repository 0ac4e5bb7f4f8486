// route_wide.cuh -- the per-token part of routing by tiles (Sec. 2, Eq. 1
// and the QB paragraph of arXiv 2609.28053), shared by the routing kernels
// (route_wide.cu, route_narrow.cu) and the routing + coarse-histogram kernel
// (route_hist.cu).
//
// One thread owns one token whose row of z sits in shared memory (rows of a
// 32-token tile padded to a stride of 4 (mod 8) words, so the 32 lanes reading
// the same 16-byte chunk of their own rows hit distinct banks).  The row
// width E is a compile-time multiple of 32, so every loop over the row
// unrolls; a narrower row is padded to it with z = -inf, which is never
// selected:
//   A. packed bf16x2 maxima of L_e = bf16(z_e + RD(b_e)) over the row's words
//      congruent mod 16: 32 groups, 16 of even and 16 of odd experts.  One
//      bf16x2 max/min network sorts both halves at once, and the KP1-th
//      largest group maximum is min_{i<KP1} max(A[i], B[KP1-1-i]) for the two
//      sorted lists A, B.  KP1 >= K+1 groups each hold an element with L at
//      or above it, so one bf16 step below it is <= tau_t and bounds every
//      expert that can be selected; two steps below it is the filter
//      threshold.  (Groups of E/32 experts leave 9.7, 10.1, 10.3 and 10.5
//      candidates of 64, 128, 256 and 512 for K + 1 = 9; more groups cost
//      more in the network than the fewer candidates save.)
//   B. masks of U_e = bf16(z_e + RU(b_e)) >= threshold, 32 experts to a word,
//      every one of the experts with s_e >= tau_t among them, with the set of
//      non-zero words.
//   C. the listed experts, in ascending index, are inserted into a sorted
//      (K+1)-list by their exact fp32 score s_e = fp32(z_e) + b_e; a new
//      element goes after equal scores, so ties keep the lower index first.
#pragma once

#include "eqb_device.cuh"

namespace eqb {

// Polls of at most ~1 us each before a bulk-copy wait gives up: about a second.
constexpr uint32_t kRouteWaitLimit = 1u << 20;

// One contiguous global -> shared copy by the bulk-copy engine.
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
__device__ __forceinline__ uint32_t lds_u16(const void* p) {
  return *reinterpret_cast<const uint16_t*>(p);
}

__host__ __device__ constexpr int wide_row_stride(int E) { return 4 * (E / 2 + ((4 - E / 2) & 7)); }

template <int E>
struct WideLayout {
  static constexpr int NCH = E / 8;              // 16-byte chunks per row
  static constexpr int RS = wide_row_stride(E);  // staged row stride, bytes
  static constexpr int TILE = 32 * RS;
  static constexpr int ENT = 32 * (NCH / 4) * 4;  // chunk masks, four per word, per lane
  static constexpr int WL = 4 * E;               // load counters
  static constexpr int WARP = (TILE + ENT + WL + 8 + 15) & ~15;  // + the mbarrier
  static constexpr int HEAD = 4 * E + 2 * (2 * E);               // b, RD(b), RU(b)
};

// The block's copy of the bias (0 for the experts [real, E) of a padded row):
// b as fp32, and RD(b), RU(b) as packed bf16
// pairs (the bounds of phases A and B).  A non-finite b raises the flag.
template <int E>
__device__ __forceinline__ void load_bias_tables(const float* __restrict__ b, int real, float* bs, uint32_t* bdn,
                                                 uint32_t* bup, int32_t* err) {
  for (int e = threadIdx.x; e < E; e += blockDim.x) {
    const float v = e < real ? b[e] : 0.f;
    bs[e] = v;
    if (!isfinite(v)) raise_flag(err, kErrNonfinite);
  }
  for (int q = threadIdx.x; q < E / 2; q += blockDim.x) {
    const float b0 = 2 * q < real ? b[2 * q] : 0.f, b1 = 2 * q < real ? b[2 * q + 1] : 0.f;
    bdn[q] = bf16_round_down(b0) | (bf16_round_down(b1) << 16);
    bup[q] = bf16_round_up(b0) | (bf16_round_up(b1) << 16);
  }
}

// x >> n, 0 for n >= 32.
__device__ __forceinline__ uint32_t shr_clamp(uint32_t x, int n) {
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
  return r;
}

// Phases A-C for the token whose row starts at rowp: on return v[0..KP1)
// holds the top-(K+1) scores in descending order (ties: lower index first)
// and id[] their experts, so tau_t = v[K].  mw is the warp's mask-word area
// ([NCH/4][32 lanes] words).  Every lane of the warp must call it (phase C
// is a warp-wide loop); `valid` only gates the non-finite check.
template <int E, int KP1>
__device__ __forceinline__ void route_row(const uint8_t* rowp, const float* bs, const uint4* bdn4, const uint4* bup4,
                                          uint32_t* mw, int lane, bool valid, int32_t* err, float (&v)[KP1],
                                          int (&id)[KP1]) {
  constexpr int NCH = E / 8;

  // ---- A: maxima of L over the words congruent mod 16, both halves
  uint32_t cm[16];
#pragma unroll
  for (int c = 0; c < NCH; ++c) {
    // From E = 256 on the unrolled loads do not fit in registers if all are
    // hoisted (at E = 256 the 168 registers of a 12-warp block spilled):
    // let at most sixteen chunks be in flight.
    if (NCH > 16 && c > 0 && (c & 15) == 0) asm volatile("" ::: "memory");
    const uint4 w = lds128(rowp + 16 * c), bd = bdn4[c];
    const uint32_t q[4] = {hadd2_bf16(w.x, bd.x), hadd2_bf16(w.y, bd.y), hadd2_bf16(w.z, bd.z),
                           hadd2_bf16(w.w, bd.w)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int g = (c & 3) * 4 + i;
      cm[g] = c < 4 ? q[i] : hmax2_nan_bf16(cm[g], q[i]);
    }
  }
  uint32_t anynan = cm[0];
#pragma unroll
  for (int c = 1; c < 16; ++c) anynan = hmax2_nan_bf16(anynan, cm[c]);
  if (valid && ((anynan & 0x7fffu) > 0x7f80u || (anynan >> 16 & 0x7fffu) > 0x7f80u)) raise_flag(err, kErrNonfinite);
  sort_desc_bf16x2<16>(cm);
  float theta = INFINITY;
#pragma unroll
  for (int i = 0; i < KP1; ++i) {
    const int j = KP1 - 1 - i;
    const float x = bf16_lo(cm[i]), y = bf16_hi(cm[j]);  // KP1 <= 16
    theta = fminf(theta, fmaxf(x, y));
  }
  // Near zero, flushing of subnormal bf16 sums could move L by up to
  // 2^-126; lowering theta below that range keeps the bound safe.
  if (fabsf(theta) < 0x1p-124f) theta = -0x1p-124f;
  // Filter threshold: one bf16 step below theta is enough.  KP1 experts have
  // L_e >= theta, and L_e = RN_bf16(z + RD(b)) <= RN_bf16(s_e) (RN is monotone,
  // RD(b) <= b, s_e the exact sum), so their exact sums are >= theta - half a
  // bf16 step and their fp32 scores >= pred(theta): tau >= pred(theta).  An
  // expert with fp32 score >= tau has an exact sum within half an fp32 step
  // of it or above, so U_e = RN_bf16(z + RU(b)) >= RN_bf16(s_e) >= pred(theta).
  // Two steps keep one step of margin (near zero theta was moved below the
  // range where subnormal flushing could matter).
  const uint32_t thf = bf16_steps_down(__float_as_uint(theta) >> 16, 2u);
  const uint32_t thf2 = thf | (thf << 16);

  // ---- B: per-chunk masks of U >= threshold, four to a word (bit 31 -
  // 8u - j of word k is expert 32k + 8u + j: the first expert is the highest
  // bit, one count of leading zeros away), and the set of non-zero words.
  // Up to 64 experts the words stay in registers, else in shared memory.
  uint32_t hits = 0u;
  uint32_t m = 0u, m1 = 0u;  // the current mask word; E <= 64: the words themselves
#pragma unroll
  for (int k = 0; k < NCH / 4; ++k) {
    uint32_t word = 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int c = 4 * k + u;
      const uint4 w = lds128(rowp + 16 * c);
      const uint4 bu = bup4[c];
      const uint32_t r0 = hge2_bf16(hadd2_bf16(w.x, bu.x), thf2);
      const uint32_t r1 = hge2_bf16(hadd2_bf16(w.y, bu.y), thf2);
      const uint32_t r2 = hge2_bf16(hadd2_bf16(w.z, bu.z), thf2);
      const uint32_t r3 = hge2_bf16(hadd2_bf16(w.w, bu.w), thf2);
      // element 2q -> bit 7 - 2q (low half of r_q), element 2q+1 -> bit 22 - 2q
      const uint32_t y = (r0 & 0x00400080u) | (r1 & 0x00100020u) | (r2 & 0x00040008u) | (r3 & 0x00010002u);
      word |= ((y | (y >> 16)) & 0xffu) << (24 - 8 * u);
    }
    if (E <= 64) {
      if (k == 0) m = word;
      else m1 = word;
    } else {
      mw[(k << 5) | lane] = word;
      hits |= (word != 0u ? 0x80000000u : 0u) >> k;
    }
  }

  // a lane past the end of the batch has no candidates (its row is zeros or
  // left over, often all equal: the warp would walk every expert of it)
  if (!valid) hits = m = m1 = 0u;

  // ---- C: exact top-(K+1) of the experts with a hit, in ascending index,
  // one per lane per step, taken from the mask words 32 experts at a time;
  // the next candidate's z and b are read one step ahead.  Refills are
  // branch-free, and a lane that is done inserts -inf, which leaves its
  // list unchanged.
#pragma unroll
  for (int j = 0; j < KP1; ++j) { v[j] = -INFINITY; id[j] = 0; }
  int wb = 0;  // first expert of the current mask word
  auto fetch = [&]() -> int {
    if constexpr (E <= 64) {
      if constexpr (E > 32) {
        const bool need = m == 0u;
        m = need ? m1 : m;
        wb = need ? 32 : wb;
        m1 = need ? 0u : m1;
      }
      const int p = __clz(m);
      const int e = m != 0u ? wb + p : -1;
      m &= shr_clamp(0x7fffffffu, p);
      return e;
    }
    const bool need = m == 0u && hits != 0u;
    const int k = __clz(hits);  // 32 when there is none
    const uint32_t word = mw[((need ? k : 0) << 5) | lane];
    m = need ? word : m;
    wb = need ? k << 5 : wb;
    hits = need ? hits ^ shr_clamp(0x80000000u, k) : hits;
    const int p = __clz(m);
    const int e = m != 0u ? wb + p : -1;
    m &= shr_clamp(0x7fffffffu, p);  // experts before p are already gone
    return e;
  };
  int e0 = fetch();
  uint32_t z0 = lds_u16(rowp + 2 * max(e0, 0));
  float b0 = bs[max(e0, 0)];
  while (__any_sync(kFull, e0 >= 0)) {
    const int e1 = fetch();
    const uint32_t z1 = lds_u16(rowp + 2 * max(e1, 0));
    const float b1 = bs[max(e1, 0)];
    insert_sorted<KP1>(v, id, e0 >= 0 ? bf16_bits_to_f32(z0) + b0 : -INFINITY, e0);
    e0 = e1;
    z0 = z1;
    b0 = b1;
  }
  // after a NaN score (flagged) a finished lane's -1 can enter the list: the
  // loads are counted by these numbers
#pragma unroll
  for (int j = 0; j < KP1; ++j) id[j] = max(id[j], 0);
}

// tau_t = v[K] of the sorted list (K < KP1 chosen at run time).
template <int KP1>
__device__ __forceinline__ float list_tau(const float (&v)[KP1], int K) {
  float tau_t = v[0];
#pragma unroll
  for (int j = 1; j < KP1; ++j) tau_t = (j == K) ? v[j] : tau_t;
  return tau_t;
}

// Per-warp load counters (E ints in shared memory) of the warp's current
// microbatch, flushed when it changes; every warp owns a contiguous range of
// tiles, so flushes are rare.  A tile inside the current microbatch skips the
// lookup.
struct TileLoads {
  int* wl;
  int cur = -1;
  int64_t lo = 0, hi = 0;  // token range of cur

  __device__ __forceinline__ void flush(const RouteArgs& a, int lane) {
    __syncwarp();
    if (cur >= 0) {
      for (int e = lane; e < a.E; e += 32) {
        const int v = wl[e];
        if (v) atomicAdd(a.loads + (int64_t)cur * a.E + e, v);
        wl[e] = 0;
      }
    }
    __syncwarp();
  }

  // Counts the top-K experts id[0..K) of this lane's token t (if valid) of
  // the tile starting at t0.  Called by all lanes.
  template <int KP1>
  __device__ __forceinline__ void count(const RouteArgs& a, int64_t t0, bool valid, const int (&id)[KP1], int lane) {
    const int K = a.K;
    const int64_t t_last = min(t0 + 31, a.T - 1) + a.tbase;
    int l = cur;
    if (!(t0 + a.tbase >= lo && t_last < hi)) {
      // the tile leaves the current microbatch: per-lane lookup
      l = valid ? microbatch_of(a.off, a.M, t0 + lane + a.tbase) : -1;
      const int l0 = __shfl_sync(kFull, l, 0);
      if (l0 != cur) {
        flush(a, lane);
        cur = l0;
        lo = __ldg(a.off + l0);
        hi = __ldg(a.off + l0 + 1);
      }
    }
    if (!valid) return;
    if (l == cur) {
#pragma unroll
      for (int j = 0; j < KP1; ++j)
        if (j < K) atomicAdd(wl + id[j], 1);
    } else {
#pragma unroll
      for (int j = 0; j < KP1; ++j)
        if (j < K) atomicAdd(a.loads + (int64_t)l * a.E + id[j], 1);
    }
  }
};

// tau and the top-K list of token t.
template <int KP1>
__device__ __forceinline__ void store_route(const RouteArgs& a, int64_t t, const float (&v)[KP1],
                                            const int (&id)[KP1]) {
  const float tau_t = list_tau<KP1>(v, a.K);
  a.tau[t] = tau_t;
  if (!isfinite(tau_t)) raise_flag(a.err, kErrNonfinite);
  if (a.idx) {
    int32_t* out = a.idx + t * a.K;
#pragma unroll
    for (int j = 0; j < KP1; ++j)
      if (j < a.K) out[j] = id[j];
  }
}

// Columns [a.E, E) of `rows` staged rows set to -inf by a warp (copies of a
// row never reach them).
template <int E>
__device__ __forceinline__ void pad_rows(uint8_t* rows, int n, int stride, int real, int lane) {
  for (int c = real / 8; c < E / 8; ++c)
    for (int r = lane; r < n; r += 32)
      *reinterpret_cast<uint4*>(rows + r * stride + 16 * c) =
          make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u);
}

}  // namespace eqb
