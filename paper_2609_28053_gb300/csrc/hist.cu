// hist.cu -- Algorithm 1's two margin-histogram passes (arXiv 2609.28053,
// Sec. 3 and App. C, steps 1 and 4).
//
// Both passes recompute every routing margin m = bf16_rne(tau_t - fp32(z))
// from z and tau instead of reading a stored margin array (Sec. 3: the second
// pass rescans the local margins).  Keys are kappa(m) (negative patterns
// complemented, others with the sign bit set).  Pass 1 counts the high byte of
// every key; pass 2 counts the low byte of the keys whose high byte is u_e.
// Pass 3 is the fixed-resolution histogram that Sec. 2 compares against:
// 256 equal bins, j = floor((m - lo) * inv_w) clamped to [0, 255].
//
// Work per element is kept to a handful of instructions by working on packed
// pairs: one 32-bit word of z holds two experts, their two fp32 differences
// are one packed f32x2 subtraction, rounded with one cvt.rn.bf16x2, and one
// PRMT (sign replicate) plus one LOP3 give both internal keys (kappa ^ 0x8000, so the stored high byte is the
// true one ^ 0x80 and is translated back at the flush).
//
// Bins: a CTA owns a tile of up to 128 experts (cut_hist) and keeps their
// 256 bins as 16-bit counters, two experts per 32-bit word: the experts of
// one z word share a word, the even one in the low half, so the increment is
// a constant.  512 bytes per expert: 64 KiB for 128 experts.  Thread i owns
// chunk i mod nct (8 experts) of token slot i / nct, so a warp reads
// contiguous pieces of rows whatever the expert count; chunk c's rows start
// c words past a 1 KiB boundary so equal bins of different chunks fall in
// different banks.  Where a warp holds several tokens of a tile, the tile can
// have as many copies of its bins (added at the flush).  A counter gains at
// most one per token, so the CTA flushes (adds its non-zero counters into
// the global int32 [E,256] histogram) at least every 65,535 tokens; the
// flush is also how token partitions are summed in device memory.
// Each lane keeps eight 16-byte loads in flight (eight tokens per round),
// which covers the DRAM latency without L2 prefetches.
//
// Fused with Load-Error Injection (the one-call step): the passes are bound
// by issue, not by DRAM, while LEI (Sec. 4) is a pure DRAM stream that needs
// only the loads.  A fused block gives a quarter of its warps to streaming
// grad_s[t, e] += coef[mb(t), e] over its slice of a token range from the
// start, the other warps count, and each counting warp joins the stream when
// its counting is done; the stream is cut into chunks of about 8 KiB of
// grad_s handed out by a shared counter, so no warp idles while the block
// has work.  Each pass carries half of the step's tokens, which turns both
// passes into DRAM-bound ones.
#include "select_device.cuh"

namespace eqb {

namespace {

constexpr int kUnroll = 8;  // 16-byte loads in flight per lane (64 registers at 1024 threads)
constexpr int64_t kFlushTokens = 65535;
// The injection share of a fused block (see above): chunks of about 8 KiB of
// grad_s from this block's slice of [ls.t0, ls.t1), taken through the shared
// counter *next.  Every element gets one fp32 addition (round to nearest) of
// its microbatch's coefficient, as in lei.cu.
__device__ __forceinline__ void stream_lei(const LeiStream& ls, int E, int* next) {
  int64_t q0, q1;
  lei_block_slice(ls.t0, ls.t1, (int64_t)blockIdx.y * gridDim.x + blockIdx.x, (int64_t)gridDim.x * gridDim.y, &q0,
                  &q1);
  int64_t mlo = 1, mhi = 0;  // token range of microbatch ml (none yet)
  int ml = 0;
  while (lei_warp_next_chunk(ls, E, q0, q1, next, mlo, mhi, ml)) {
  }
}

// Algorithm 1's selection for the experts [ea, eb) of a tile by nw warps
// (warp wid, lane), one warp per expert, the counts of two experts in flight:
// pick(e, i, bin, rest) receives, in every lane, expert e's first bin whose
// prefix count reaches target(i), i = e - ea, and the rank left in it (bin
// -1: unreachable).  The counts were added by other blocks' atomics and are
// read from L2.  FIRST: counts in the bins of non-finite margins are flagged.
template <bool FIRST, class Target, class Pick>
__device__ __forceinline__ void select_tile(const int32_t* hist, int ea, int eb, int nw, int wid, int lane,
                                            int32_t* err, Target target, Pick pick) {
  constexpr int B = 2;
#pragma unroll 1
  for (int e0 = ea + wid; e0 < eb; e0 += nw * B) {
    int4 ca[B], cb[B];
#pragma unroll
    for (int k = 0; k < B; ++k) {
      const int e = min(e0 + k * nw, eb - 1);
      const int4* h = reinterpret_cast<const int4*>(hist + (int64_t)e * 256 + lane * 8);
      ca[k] = __ldcg(h);
      cb[k] = __ldcg(h + 1);
    }
#pragma unroll
    for (int k = 0; k < B; ++k) {
      const int e = e0 + k * nw;
      if (e >= eb) break;
      const int32_t cnt[8] = {ca[k].x, ca[k].y, ca[k].z, ca[k].w, cb[k].x, cb[k].y, cb[k].z, cb[k].w};
      if (FIRST && ((lane == 0 && cnt[0] != 0) || (lane == 31 && cnt[7] != 0))) raise_flag(err, kErrNonfinite);
      int32_t rest = 0;
      const int bin = warp_pick<int32_t>(cnt, target(e - ea), lane, rest);
      if (bin < 0 && lane == 0) raise_flag(err, kErrRank);
      pick(e, e - ea, bin, rest);
    }
  }
}

// First word of pair row `row` of a block's bins (see above).
__device__ __forceinline__ int row_word(int row) { return row * 256 + (row >> 2); }
// Words of the bins of nct chunks, a multiple of four.
__host__ __device__ constexpr int bin_words(int nct) { return (nct * 1024 + nct + 3) & ~3; }
// Widest tile of a block, in 8-expert chunks.
constexpr int kMaxTileChunks = 16;
static_assert(kMaxE / 64 <= kMaxHistTiles, "tiles of 8 chunks or more");

template <int PASS, bool LEI>
__global__ void __launch_bounds__(1024) hist_kernel(HistArgs a, int tile_chunks, int copies,
                                                    int64_t tokens_per_cta, LeiStream ls) {
  extern __shared__ __align__(16) uint32_t bins[];
  __shared__ int lei_next;  // next injection chunk of this block (fused only)
  __shared__ uint8_t su[PASS == 2 ? kMaxTileChunks * 8 : 1];    // the tile's u and rho (the one-call step)
  __shared__ int32_t srho[PASS == 2 ? kMaxTileChunks * 8 : 1];
  const int E = a.E;
  const int e0 = blockIdx.x * tile_chunks * 8;
  const int nct = min(tile_chunks, (E - e0) >> 3);  // chunks of this tile (the last may be narrower)
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nw = LEI ? (blockDim.x >> 5) - (blockDim.x >> 7) : (blockDim.x >> 5);  // counting warps
  const int nt = nw * 32;
  const int slots = nt / nct;                        // tokens per round of the block
  const int tok = static_cast<int>(threadIdx.x) / nct;  // token slot (>= slots: no counting)
  const int c = static_cast<int>(threadIdx.x) - tok * nct;  // 8-expert chunk of the tile owned by this thread
  // Barrier of the counting warps (all warps unless fused).
  auto sync_counting = [&]() {
    if (LEI) asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory");
    else __syncthreads();
  };

  const int ncp = PASS == 2 ? 1 : copies;
  for (int i = threadIdx.x; i < bin_words(nct * ncp) / 4; i += blockDim.x)
    reinterpret_cast<uint4*>(bins)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (LEI && threadIdx.x == 0) lei_next = 0;
  // Shared address of this thread's first pair row; pair p adds p * 1 KiB.
  const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(bins)) +
                        4u * static_cast<uint32_t>(row_word(4 * (ncp > 1 ? c + tok % ncp * nct : c)));
  uint32_t sel[4] = {0, 0, 0, 0};
  // internal high bytes (u ^ 0x80) of the selected bins, placed where the
  // internal keys carry them: bits 8-15 (even expert) and 24-31 (odd).
  auto load_sel = [&](const uint8_t* ub) {
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const uint32_t ue = ub[c * 8 + 2 * p] ^ 0x80u;
      const uint32_t uo = ub[c * 8 + 2 * p + 1] ^ 0x80u;
      sel[p] = (ue << 8) | (uo << 24);
    }
  };
  griddep_wait();  // the bins were zeroed above; global reads start here
  if (PASS == 2 && !a.shard_off && !a.coarse) load_sel(a.u + e0);
  __syncthreads();
  if (LEI && wid >= nw) {
    stream_lei(ls, E, &lei_next);
    return;
  }
  if (PASS == 2 && a.coarse) {
    // Algorithm 1 step 3: every block selects u, rho for its own tile
    select_tile<true>(a.coarse, e0, e0 + nct * 8, nw, wid, lane, a.sel_err,
                      [&](int) { return a.r; },
                      [&](int, int i, int bin, int32_t rest) {
                        if (lane == 0) {
                          su[i] = static_cast<uint8_t>(bin < 0 ? 255 : bin);
                          srho[i] = rest;
                        }
                      });
    sync_counting();
    load_sel(su);
  }

  // Token indices fit in 32 bits (T < 2^31 is checked on the host).
  const int tb = static_cast<int>(min((int64_t)blockIdx.y * tokens_per_cta, a.T));
  const int te = static_cast<int>(min((int64_t)tb + tokens_per_cta, a.T));
  const int step = slots;
  const size_t zstride = static_cast<size_t>(step) * E;
  const uint16_t* zlane = a.z + e0 + c * 8;

  auto process = [&](const uint4& w4, float tv) {
    const uint32_t zw[4] = {w4.x, w4.y, w4.z, w4.w};
    const uint64_t tt = f32x2_splat(tv);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const uint32_t m = margins_bf16x2(tt, zw[p]);
      const uint32_t k = kappa2_internal(m);
      const uint32_t row = base + 1024u * p;
      if (PASS == 1) {
        const uint32_t he = prmt(k, 0u, 0x4441u), ho = k >> 24;  // internal high bytes
        const bool same = he == ho;
        red_shared_add(row + 4u * he, same ? 0x10001u : 1u);
        if (!same) red_shared_add(row + 4u * ho, 0x10000u);
      } else if (PASS == 3) {
        // equal-width bins: j = floor((m - lo) * inv_w), clamped to [0, 255]
        const uint32_t he = static_cast<uint32_t>(min(max(__float2int_rd(__fmul_rn(__fsub_rn(bf16_lo(m), a.lo), a.inv_w)), 0), 255));
        const uint32_t ho = static_cast<uint32_t>(min(max(__float2int_rd(__fmul_rn(__fsub_rn(bf16_hi(m), a.lo), a.inv_w)), 0), 255));
        const bool same = he == ho;
        red_shared_add(row + 4u * he, same ? 0x10001u : 1u);
        if (!same) red_shared_add(row + 4u * ho, 0x10000u);
      } else {
        const uint32_t d = (k ^ sel[p]) & 0xff00ff00u;
        if ((d & 0x0000ff00u) == 0u) red_shared_add(row + 4u * (k & 0xffu), 1u);
        if ((d & 0xff000000u) == 0u) red_shared_add(row + 4u * prmt(k, 0u, 0x4442u), 0x10000u);
      }
    }
  };

  for (int cb = tb; cb < te;) {
    int ce = static_cast<int>(min((int64_t)cb + kFlushTokens, (int64_t)te));
    int64_t hbase = 0;  // this chunk's histogram (shards: one per shard)
    if (a.shard_off) {
      const int sp = microbatch_of(a.shard_off, a.P, cb);
      const int64_t send = __ldg(a.shard_off + sp + 1);
      if (send > cb && send < ce) ce = static_cast<int>(send);  // chunks end at shard boundaries
      hbase = (int64_t)sp * E * 256;
      if (PASS == 2) load_sel(a.u + (int64_t)sp * E + e0);
    }
    int t = tok < slots ? cb + tok : ce;
    const uint16_t* zp = zlane + static_cast<size_t>(t) * E;
    // full rounds of kUnroll tokens per thread, no guards
    for (; t + (kUnroll - 1) * step < ce; t += kUnroll * step, zp += kUnroll * zstride) {
      uint4 w[kUnroll];
      float tt[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        w[u] = __ldcs(reinterpret_cast<const uint4*>(zp + u * zstride));
        tt[u] = __ldg(a.tau + t + u * step);
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) process(w[u], tt[u]);
    }
    // the rest, two tokens in flight (a block of few tokens has only these)
    for (; t < ce; t += 2 * step, zp += 2 * zstride) {
      const bool two = t + step < ce;
      const uint4 w0 = __ldcs(reinterpret_cast<const uint4*>(zp));
      const float t0 = __ldg(a.tau + t);
      const uint4 w1 = two ? __ldcs(reinterpret_cast<const uint4*>(zp + zstride)) : make_uint4(0u, 0u, 0u, 0u);
      const float t1 = two ? __ldg(a.tau + t + step) : 0.f;
      process(w0, t0);
      if (two) process(w1, t1);
    }
    sync_counting();
    // Flush: add every non-zero 16-bit counter to the global histogram.
    for (int i = threadIdx.x; i < nct * 1024; i += nt) {
      const int row = i >> 8, slot = i & 255;
      const int wi = row_word(row) + slot;
      uint32_t v = bins[wi];
      if (v) bins[wi] = 0u;
      for (int k = 1; k < ncp; ++k) {  // the copies' halves add up to at most the tokens counted
        const int wk = row_word(row + 4 * k * nct) + slot;
        const uint32_t vk = bins[wk];
        if (vk) bins[wk] = 0u;
        v += vk;
      }
      if (v) {
        const int bin = (PASS == 1) ? (slot ^ 0x80) : slot;  // pass 1 stores internal keys
        const int ee = e0 + 2 * row;
        if (v & 0xffffu) atomicAdd(a.hist + hbase + (int64_t)ee * 256 + bin, static_cast<int>(v & 0xffffu));
        if (v >> 16) atomicAdd(a.hist + hbase + (int64_t)(ee + 1) * 256 + bin, static_cast<int>(v >> 16));
        if (PASS == 1 && (bin == 0 || bin == 255)) raise_flag(a.err, kErrNonfinite);
      }
    }
    sync_counting();
    cb = ce;
  }
  if (PASS == 2 && a.done) {
    // Algorithm 1 steps 5-6 in the last block of this expert tile to get
    // here, for the tile's experts, and Eq. (2) in the last tile to have
    // selected.  After a barrier (every write of this block issued), one
    // thread's fence releases the block's writes before its count; the last
    // block's fence after its count orders the other blocks' writes before
    // its reads.
    __shared__ int last;
    auto count_last = [&](int32_t* counter, int n) {
      if (threadIdx.x == 0) {
        __threadfence();
        const bool l = atomicAdd(counter, 1) == n - 1;
        if (l) __threadfence();
        last = l;
      }
      sync_counting();
      return last != 0;
    };
    if (count_last(a.done + blockIdx.x, gridDim.y)) {
      select_tile<false>(a.hist, e0, e0 + nct * 8, nw, wid, lane, a.sel_err,
                         [&](int i) { return srho[i]; },
                         [&](int e, int i, int bin, int32_t) {
                           if (lane == 0) a.q_hat[e] = static_cast<uint16_t>(quantile_bits(su[i], bin));
                         });
      sync_counting();  // this tile's q_hat are written, and `last` was read
      if (count_last(a.done + kMaxHistTiles, gridDim.x)) block_bias_update(a.q_hat, E, a.b_next, nt, sync_counting);
    }
  }
  if (LEI) stream_lei(ls, E, &lei_next);
}

// How a pass is cut into blocks: expert tiles of `chunks` 8-expert chunks
// times token ranges of `tpc` tokens, about one block per SM, each with
// `copies` copies of its tile's bins.
struct HistCut {
  int tiles, chunks, copies, ranges;
  int64_t tpc;
};

// A block's fixed cost (zeroing, flushing and selecting over its tile's bins)
// grows with the tile; what narrow tiles cost is lanes of a warp that count
// the same experts and meet in popular bins.  Measured on pass 1 / pass 2 /
// the step without LEI, us, for tiles of 8, 16 and 32 chunks: T = 30,873,
// E = 256 (6,500 chunks of z per SM) 9.2 / 6.3 / 40, 9.5 / 7.0 / 45 and
// 12.0 / 8.2 / 74 (one 32-chunk tile on 2,048-token blocks before: 33.5 /
// 27.1 / 93); T = 147,456 (31,000) 27 / 15 / 81, 21 / 16 / 76 and 22 / 17 /
// 89; T = 1,048,576, E = 384 143 / 134 / 462 for 16, 162 / 136 / 487 for 24.
// From 7,000 chunks per SM on, copies that give the 32 lanes of a warp bins
// of their own pay for their zeroing: T = 1,000,000, E = 64 31 us against
// 45 (pass 1), T = 60,000, E = 160 10.3 against 12.1; T = 65,536, E = 64
// (3,400) 7.5 against 6.8.  Pass 2 counts few elements and takes one copy.
HistCut cut_hist(int64_t T, int E, int pass, int sm_count) {
  const int nch = E >> 3;
  const int64_t per_sm = T * nch / sm_count;  // chunks of z to count per SM
  const int want = per_sm < 10000 ? 8 : 16;
  HistCut h;
  h.tiles = (nch + want - 1) / want;
  h.chunks = (nch + h.tiles - 1) / h.tiles;
  h.tiles = (nch + h.chunks - 1) / h.chunks;
  h.copies = pass != 2 && per_sm >= 7000 ? 32 / h.chunks : 1;
  int64_t ranges = sm_count / h.tiles;
  const int64_t most = (T * h.chunks + 1023) / 1024;  // a chunk for every thread
  if (ranges > most) ranges = most;
  if (ranges < 1) ranges = 1;
  h.tpc = (T + ranges - 1) / ranges;
  h.ranges = static_cast<int>((T + h.tpc - 1) / h.tpc);
  return h;
}

template <int PASS, bool LEI>
int launch_hist_pass(const HistArgs& a, const LeiStream& ls, cudaStream_t s) {
  DeviceInfo di;
  if (int rc = device_info(&di)) return rc;
  const HistCut h = cut_hist(a.T, a.E, PASS, di.sm_count);
  const int smem = bin_words(h.chunks * h.copies) * 4;
  auto kern = hist_kernel<PASS, LEI>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
    return kErrCuda;
  dim3 grid((unsigned)h.tiles, (unsigned)h.ranges);
  return launch_dependent(kern, grid, dim3(1024), smem, s, a, h.chunks, h.copies, h.tpc, ls) == cudaSuccess ? kOk
                                                                                                      : kErrCuda;
}

}  // namespace

int launch_hist(const HistArgs& a, int pass, cudaStream_t s) {
  const LeiStream none;
  if (pass == 3) return launch_hist_pass<3, false>(a, none, s);
  return pass == 1 ? launch_hist_pass<1, false>(a, none, s) : launch_hist_pass<2, false>(a, none, s);
}

int launch_hist_lei(const HistArgs& a, int pass, const LeiStream& ls, cudaStream_t s) {
  if (!ls.g || !ls.coef || !ls.off || ls.M < 1 || ls.t0 < 0 || ls.t1 < ls.t0) return kErrInvalidArg;
  return pass == 1 ? launch_hist_pass<1, true>(a, ls, s) : launch_hist_pass<2, true>(a, ls, s);
}

}  // namespace eqb
