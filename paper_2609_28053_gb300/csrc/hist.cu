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
// contiguous pieces of rows whatever the expert count.
// Two layouts.  Banked (BANK, from 5,000 chunks of z per SM on, passes 1 and
// 3): 32 columns, a lane's by its chunk and, where the warp holds several tokens
// of the tile, copy, the bank of every word of a column the same: word (bin * 4
// + pair) * 32 + column.  Where the tile's chunks divide 32 every lane of a warp
// has a column of its own, so no two lanes of an increment meet.  Otherwise
// (tiles of 5, 7, 11 or 13 chunks) there are fewer columns than lanes and up to
// 32 - nct * copies lanes share one, the same word at times: the increments have
// to be atomic.  What bounds these passes otherwise is the banks in which random
// bins meet: 2.8 to 3.7 clocks an increment of a warp, against 1.4 or less.
// T = 2,097,152, E = 256 202 -> 160 us (the copy rate), T = 524,288, E = 128
// 34 -> 26, T = 147,456, E = 256 21 -> 16.6; pass 3 260 -> 192 and 49 -> 40 (a
// comparison).  It takes 128 KiB to zero and flush whatever the tile: small
// batches, and pass 2, which counts few elements, use rows of 256 bins, chunk
// c's c words past a 1 KiB boundary so equal bins of different chunks fall in
// different banks.
// A counter gains at most one per token, so the CTA flushes (adds its non-zero counters into
// the global int32 [E,256] histogram) at least every 65,535 tokens; the
// flush is also how token partitions are summed in device memory.
// Each thread keeps several 16-byte loads in flight (kUnroll tokens per
// round), which covers the DRAM latency without L2 prefetches.
//
// Fused with Load-Error Injection (the one-call step): counting takes issue
// slots beside DRAM, while LEI (Sec. 4) is a pure DRAM stream that needs only
// the loads.  A fused block gives some of its warps to streaming
// grad_s[t, e] += coef[mb(t), e] over its slice of a token range from the
// start, the other warps count, and each counting warp joins the stream when
// its counting is done; the stream is cut into chunks of about 8 KiB of
// grad_s handed out by a shared counter, so no warp idles while the block
// has work.  The step's fine pass carries all of the tokens, and a few blocks
// of its coarse pass form the coefficients.
#include "lei_device.cuh"
#include "select_device.cuh"

namespace eqb {

namespace {

// 16-byte loads in flight per thread (64 registers at 1024 threads).  Pass 1
// (before its banked bins) / pass 2 alone at T = 2,097,152, E = 256: 187 / 171 us with six, 185 / 185
// with seven, 194 / 184 with eight, 221 / 181 with four.  Beside the injection
// eight (the step at T = 1,048,576, E = 512 1229 us, 1241 with six); ptxas then
// spills 32 bytes in the fine pass, which runs at 99% of the copy rate with them.
template <bool LEI>
constexpr int kUnroll = LEI ? 8 : 6;
constexpr int64_t kFlushTokens = 65535;

// The LEI coefficient table formed by blocks of pass 1 (none: blocks == 0).
struct CoefRows {
  LeiArgs a = {};
  float* coef = nullptr;
  int blocks = 0;
};

// The injection share of a fused block (see above): chunks of about 8 KiB of
// grad_s from this block's slice of [ls.t0, ls.t1), taken through the shared
// counter *next.  Every element gets one fp32 addition (round to nearest) of
// its microbatch's coefficient, as in lei.cu.
__device__ __forceinline__ void stream_lei(const LeiStream& ls, int E, int* next) {
  int64_t q0, q1;
  lei_block_slice(ls.t0, ls.t1, blockIdx.x, gridDim.x, &q0, &q1);
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
// The banked bins: (slot * 4 + pair) * 32 + column.
constexpr int kBankWords = 256 * 4 * 32;
// Widest tile of a block, in 8-expert chunks.
constexpr int kMaxTileChunks = 16;
static_assert(kMaxE / 64 <= kMaxHistTiles, "tiles of 8 chunks or more");

// Where a thread stands in the pass's cut (cut_hist): read from the special
// registers at every construction, never carried over from an earlier one.
struct HistPlace {
  int tid, lane, wid;
  int tile, range;  // expert tile and token range of the block
  int e0, nct;      // the tile's first expert and its chunks (the last tile may be narrower)
  int nw, nt;       // counting warps and threads (the last lei_warps of a fused block stream LEI)
  __device__ __forceinline__ HistPlace(int tiles, int tile_chunks, int E, int lei_warps) {
    int cta, n;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
    asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(cta));
    asm volatile("mov.u32 %0, %%ntid.x;" : "=r"(n));
    lane = tid & 31;
    wid = tid >> 5;
    tile = cta % tiles;
    range = cta / tiles;
    e0 = tile * tile_chunks * 8;
    nct = min(tile_chunks, (E - e0) >> 3);
    nw = (n >> 5) - lei_warps;
    nt = nw * 32;
  }
};

template <int PASS, bool LEI, bool BANK>
__global__ void __launch_bounds__(1024) hist_kernel(HistArgs a, int tiles, int tile_chunks, int copies,
                                                    int64_t tokens_per_cta, LeiStream ls, CoefRows cr) {
  constexpr int U = kUnroll<LEI>;
  extern __shared__ __align__(16) uint32_t bins[];
  __shared__ int lei_next;  // next injection chunk of this block (fused only)
  __shared__ uint8_t su[PASS == 2 ? kMaxTileChunks * 8 : 1];    // the tile's u and rho (the one-call step)
  __shared__ int32_t srho[PASS == 2 ? kMaxTileChunks * 8 : 1];
  const int E = a.E;
  if (PASS == 1 && !LEI && blockIdx.x >= gridDim.x - cr.blocks) {
    // the last cr.blocks blocks form the coefficient table meanwhile
    griddep_wait();
    // a warp per row, the rows dealt out to the blocks first
    const int first = (threadIdx.x >> 5) * cr.blocks + blockIdx.x - (gridDim.x - cr.blocks);
    for (int l = first; l < cr.a.M; l += (blockDim.x >> 5) * cr.blocks) {
      const int64_t n = __ldg(cr.a.off + l + 1) - __ldg(cr.a.off + l);
      warp_lei_coef(cr.a.loads + (int64_t)l * E, n, E, cr.a.K, cr.a.eta, cr.a.c, cr.coef + (int64_t)l * E,
                    threadIdx.x & 31);
    }
    return;
  }
  const HistPlace pl(tiles, tile_chunks, E, LEI ? ls.warps : 0);
  const int tok = pl.tid / pl.nct;           // token slot (>= slots: no counting)
  const int c = pl.tid - tok * pl.nct;       // 8-expert chunk of the tile owned by this thread
  // Barrier of the counting warps (all warps unless fused).
  auto sync_counting = [&]() {
    if (LEI) asm volatile("bar.sync 1, %0;" ::"r"(pl.nt) : "memory");
    else __syncthreads();
  };

  for (int i = threadIdx.x; i < (BANK ? kBankWords : bin_words(pl.nct)) / 4; i += blockDim.x)
    reinterpret_cast<uint4*>(bins)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (LEI && threadIdx.x == 0) lei_next = 0;
  // Shared address of this thread's bin 0 of its first pair; pair p adds
  // p * kPairBytes, bin j j << kBinShift.
  constexpr uint32_t kPairBytes = BANK ? 128u : 1024u;
  constexpr int kBinShift = BANK ? 9 : 2;
  const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(bins)) +
                        4u * static_cast<uint32_t>(BANK ? c + tok % copies * pl.nct : row_word(4 * c));
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
  if (PASS == 2 && !a.shard_off && !a.coarse) load_sel(a.u + pl.e0);
  __syncthreads();
  if (LEI && pl.wid >= pl.nw) {
    stream_lei(ls, E, &lei_next);
    return;
  }
  if (PASS == 2 && a.coarse) {
    // Algorithm 1 step 3: every block selects u, rho for its own tile
    select_tile<true>(a.coarse, pl.e0, pl.e0 + pl.nct * 8, pl.nw, pl.wid, pl.lane, a.sel_err,
                      [&](int) { return a.r; },
                      [&](int e, int i, int bin, int32_t rest) {
                        if (pl.lane == 0) {
                          su[i] = static_cast<uint8_t>(bin < 0 ? 255 : bin);
                          srho[i] = rest;
                          if (pl.range == 0) {
                            a.sel_u[e] = su[i];
                            a.sel_rho[e] = rest;
                          }
                        }
                      });
    sync_counting();
    load_sel(su);
  }

  // Token indices fit in 32 bits (T < 2^31 is checked on the host).
  const int tb = static_cast<int>(min((int64_t)pl.range * tokens_per_cta, a.T));
  const int te = static_cast<int>(min((int64_t)tb + tokens_per_cta, a.T));
  const int step = pl.nt / pl.nct;  // token slots: tokens per round of the block
  const uint32_t zstep = static_cast<uint32_t>(step) * static_cast<uint32_t>(E) * 2u;  // bytes of z per round

  auto process = [&](const uint4& w4, float tv) {
    const uint32_t zw[4] = {w4.x, w4.y, w4.z, w4.w};
    const uint64_t tt = f32x2_splat(tv);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const uint32_t m = margins_bf16x2(tt, zw[p]);
      const uint32_t k = kappa2_internal(m);
      const uint32_t row = base + kPairBytes * p;
      if (PASS == 1) {
        const uint32_t he = prmt(k, 0u, 0x4441u), ho = k >> 24;  // internal high bytes
        if (BANK) {
          red_shared_add(row + (he << kBinShift), 1u);
          red_shared_add(row + (ho << kBinShift), 0x10000u);
        } else {
          const bool same = he == ho;
          red_shared_add(row + (he << kBinShift), same ? 0x10001u : 1u);
          if (!same) red_shared_add(row + (ho << kBinShift), 0x10000u);
        }
      } else if (PASS == 3) {
        // equal-width bins: j = floor((m - lo) * inv_w), clamped to [0, 255]
        const uint32_t he = static_cast<uint32_t>(min(max(__float2int_rd(__fmul_rn(__fsub_rn(bf16_lo(m), a.lo), a.inv_w)), 0), 255));
        const uint32_t ho = static_cast<uint32_t>(min(max(__float2int_rd(__fmul_rn(__fsub_rn(bf16_hi(m), a.lo), a.inv_w)), 0), 255));
        if (BANK) {
          red_shared_add(row + (he << kBinShift), 1u);
          red_shared_add(row + (ho << kBinShift), 0x10000u);
        } else {
          const bool same = he == ho;
          red_shared_add(row + (he << kBinShift), same ? 0x10001u : 1u);
          if (!same) red_shared_add(row + (ho << kBinShift), 0x10000u);
        }
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
      if (PASS == 2) load_sel(a.u + (int64_t)sp * E + pl.e0);
    }
    int t = tok < step ? cb + tok : ce;
    const char* zp = reinterpret_cast<const char*>(a.z + static_cast<size_t>(t) * E + pl.e0 + c * 8);
    // full rounds of U tokens per thread, no guards
    for (; t + (U - 1) * step < ce; t += U * step, zp += U * zstep) {
      uint4 w[U];
      float tt[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        w[u] = __ldcs(reinterpret_cast<const uint4*>(zp + u * zstep));
        tt[u] = __ldg(a.tau + t + u * step);
      }
      asm volatile("" ::: "memory");  // every load is issued before the first count
#pragma unroll
      for (int u = 0; u < U; ++u) process(w[u], tt[u]);
    }
    // the rest, two tokens in flight (a block of few tokens has only these)
    for (; t < ce; t += 2 * step, zp += 2 * zstep) {
      const bool two = t + step < ce;
      const uint4 w0 = __ldcs(reinterpret_cast<const uint4*>(zp));
      const float t0 = __ldg(a.tau + t);
      const uint4 w1 = two ? __ldcs(reinterpret_cast<const uint4*>(zp + zstep)) : make_uint4(0u, 0u, 0u, 0u);
      const float t1 = two ? __ldg(a.tau + t + step) : 0.f;
      process(w0, t0);
      if (two) process(w1, t1);
    }
    // from here on the thread's place is formed anew, so that the counting
    // loop does not hold it in registers
    const HistPlace fl(tiles, tile_chunks, E, LEI ? ls.warps : 0);
    sync_counting();
    // Flush: add every non-zero 16-bit counter to the global histogram.
    auto add = [&](uint32_t v, int row, int slot) {
      const int bin = (PASS == 1) ? (slot ^ 0x80) : slot;  // pass 1 stores internal keys
      const int ee = fl.e0 + 2 * row;
      if (v & 0xffffu) atomicAdd(a.hist + hbase + (int64_t)ee * 256 + bin, static_cast<int>(v & 0xffffu));
      if (v >> 16) atomicAdd(a.hist + hbase + (int64_t)(ee + 1) * 256 + bin, static_cast<int>(v >> 16));
      if (PASS == 1 && (bin == 0 || bin == 255)) raise_flag(a.err, kErrNonfinite);
    };
    if constexpr (BANK) {
      // A warp takes 32 slots of one pair: read with a lane per column, turned
      // in place (element (slot, column) to row `column`), read back with a lane
      // per slot, so that neither the reads meet in a bank nor the global
      // additions of a warp scatter.
#pragma unroll 1
      for (int blk = fl.wid; blk < 32; blk += fl.nw) {
        uint32_t* const w = bins + (blk >> 2) * 4096 + (blk & 3) * 32;  // 32 rows, 128 words apart
        uint32_t v[32], some = 0;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          v[j] = w[j * 128 + fl.lane];
          some |= v[j];
        }
        if (!__any_sync(kFull, some != 0u)) continue;  // (every lane has read)
#pragma unroll
        for (int j = 0; j < 32; ++j) w[fl.lane * 128 + ((j + fl.lane) & 31)] = v[j];
        __syncwarp();
        for (int ch = 0; ch < fl.nct; ++ch) {
          uint32_t sum = 0;  // the copies' halves add up to at most the tokens counted
          for (int r = ch; r < fl.nct * copies; r += fl.nct) sum += w[r * 128 + ((fl.lane + r) & 31)];
          if (sum) add(sum, 4 * ch + (blk & 3), (blk >> 2) * 32 + fl.lane);
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 32; ++j) w[j * 128 + fl.lane] = 0u;
      }
    } else {
      for (int i = fl.tid; i < fl.nct * 1024; i += fl.nt) {
        const int row = i >> 8, slot = i & 255;
        const int wi = row_word(row) + slot;
        const uint32_t v = bins[wi];
        if (v) {
          bins[wi] = 0u;
          add(v, row, slot);
        }
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
    const HistPlace fl(tiles, tile_chunks, E, LEI ? ls.warps : 0);
    auto count_last = [&](int32_t* counter, int n) {
      if (fl.tid == 0) {
        __threadfence();
        const bool l = atomicAdd(counter, 1) == n - 1;
        if (l) __threadfence();
        last = l;
      }
      sync_counting();
      return last != 0;
    };
    if (count_last(a.done + fl.tile, (int)gridDim.x / tiles)) {
      select_tile<false>(a.hist, fl.e0, fl.e0 + fl.nct * 8, fl.nw, fl.wid, fl.lane, a.sel_err,
                         [&](int i) { return srho[i]; },
                         [&](int e, int i, int bin, int32_t) {
                           if (fl.lane == 0) a.q_hat[e] = static_cast<uint16_t>(quantile_bits(su[i], bin));
                         });
      sync_counting();  // this tile's q_hat are written, and `last` was read
      if (count_last(a.done + kMaxHistTiles, tiles)) block_bias_update(a.q_hat, E, a.b_next, fl.nt, sync_counting);
    }
  }
  if (LEI) stream_lei(ls, E, &lei_next);
}

// How a pass is cut into blocks: expert tiles of `chunks` 8-expert chunks
// times token ranges of `tpc` tokens, about one block per SM, with `copies`
// columns for each chunk of the banked layout (1: rows of bins), `threads` to a
// block.  `counted`: the tiles have counters (HistArgs::done).
struct HistCut {
  int tiles, chunks, copies, ranges, threads;
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
// From 5,000 chunks per SM on the banked layout, `copies` columns a chunk,
// pays for its zeroing and flush: the step at T = 30,873, E = 256 36.5 -> 35.6
// us, T = 40,000, E = 96 (3,200) 29.5 against 29.9 with it.  Tiles of 32
// chunks with it: pass 1 at T = 147,456, E = 256 18.3 us against 16.6, T =
// 524,288 48.5 against 45.7, T = 2,097,152 159.9 against 159.7.  Pass 2 counts
// few elements, so that its lanes rarely meet: rows of bins, and narrower
// tiles, whose selections take one round of the block's warps and whose
// flushes (nearly every low byte occurs) add fewer counters to the global
// histogram.  The step with tiles of 4, 8 and 16
// chunks: T = 30,873, E = 256 35 / 37 / 42 us, T = 65,536, E = 64 31 / 35 /
// 35, T = 524,288, E = 128 185 / 187 / 190, E = 256 321 / 321 / 325, T =
// 1,048,576, E = 512 1220 / 1219 / 1211.
// The smallest batches take one or two chunks a tile and 512 threads (half of
// them stream LEI as half of 1,024 do): little else than the fixed cost is left.
// Pass 1 / pass 2 alone, us, 8 and 4 chunks with 1,024 threads / now (33
// one-chunk tiles before the cut by size): T = 100, E = 264 4.45 / 2.6 (2.45)
// and 4.95 / 3.3 (2.90); T = 1,000 4.75 / 4.2 (4.1) and 5.42 / 4.06 (3.80); T =
// 60,000, E = 24 5.93 / 4.43 (4.86) in pass 2, T = 20,000, E = 200 7.14 / 6.29
// (6.11).  Pass 2 with LEI: T = 1,000, E = 8 6.3 / 5.5 (5.7), E = 256 5.9 / 5.1.
// The step: T = 4,096, E = 8 16.8 / 15.3, E = 128 22.8 / 21.2.
// Shards of a few hundred tokens are flushed one by one, which wide tiles do in
// fewer rounds: the rank average of 1,000 shards, T = 524,288, in tiles of 4 / 16
// chunks in pass 2: E = 128 556 / 517, E = 256 986 / 910.
HistCut cut_hist(int64_t T, int E, int pass, bool lei, bool counted, int shards, int blocks) {
  const int nch = E >> 3;
  const int64_t per_sm = T * nch / blocks;  // chunks of z to count per SM
  int want = T <= 512 ? 1 : per_sm <= (lei ? 512 : 1000) ? 2 : per_sm < 10000 ? 8 : 16;
  if (pass == 2) {
    want = per_sm < (lei ? 4000 : 5000) ? 2 : per_sm < 64000 ? 4 : per_sm < 200000 ? 8 : 16;
    if (shards > 1) {
      if (T / shards < 600) want = 16;
    } else if (per_sm < 2000 ? !lei || T <= 512 : per_sm < 10000 && nch <= 5) {
      want = 1;
    }
    if (counted && want * kMaxHistTiles < nch) want = (nch + kMaxHistTiles - 1) / kMaxHistTiles;
  }
  HistCut h;
  h.tiles = (nch + want - 1) / want;
  h.chunks = (nch + h.tiles - 1) / h.tiles;
  h.tiles = (nch + h.chunks - 1) / h.chunks;
  h.threads = per_sm <= 512 && h.chunks <= 2 ? 512 : 1024;
  h.copies = pass != 2 && per_sm >= 5000 ? 32 / h.chunks : 1;
  int64_t ranges = blocks / h.tiles;
  const int64_t most = (T * h.chunks + h.threads - 1) / h.threads;  // a chunk for every thread
  if (ranges > most) ranges = most;
  if (ranges < 1) ranges = 1;
  h.tpc = (T + ranges - 1) / ranges;
  h.ranges = static_cast<int>((T + h.tpc - 1) / h.tpc);
  return h;
}

// SMs that form the coefficient table.  A warp takes 2-3 us a row and a row
// some 500 clocks of its SM's fp64 pipe, so that many microbatches need more
// SMs: a short pass gives them 16 and one for every 16 rows, a long one four
// and one for every 32, at most 64.  The step, us, with 4 / 16 / 32 / 64: T =
// 16,384, E = 64, M = 16 23.3 (16), M = 256 38.9 / 25.3 / 24.2 / 24.3, M = 1,024 93 /
// 39.7 / 30.7 / 26.2; T = 147,456, E = 256, M = 64 100.5 / 101.6 / 102.6 / 106.4;
// T = 524,288, E = 128, M = 32 175.0 / 176.6 / 178.6, M = 512 203.6 / 180.4 / 182.6
// / 188.8; T = 1,000,003, E = 16, M = 4,096 317 / 137 / 106 / 91 (122 with the
// table in a kernel of its own).
int coef_blocks(int64_t T, int E, int M, int sm_count) {
  const bool brief = T * (E >> 3) / sm_count < 10000;
  int n = brief ? M / 16 : M / 32;
  const int least = brief ? 16 : 4;
  n = n < least ? least : n > 64 ? 64 : n;
  return M < n ? M : n;
}

template <int PASS, bool LEI>
int launch_hist_pass(const HistArgs& a, LeiStream ls, CoefRows cr, cudaStream_t s) {
  DeviceInfo di;
  if (int rc = device_info(&di)) return rc;
  cr.blocks = cr.coef ? coef_blocks(a.T, a.E, cr.a.M, di.sm_count) : 0;
  const HistCut h = cut_hist(a.T, a.E, PASS, LEI, a.done != nullptr, a.shard_off ? a.P : 1, di.sm_count - cr.blocks);
  if (LEI) ls.warps = ls.warps * h.threads / 1024;
  const int smem = (h.copies > 1 ? kBankWords : bin_words(h.chunks)) * 4;
  auto kern = hist_kernel<PASS, LEI, false>;
  int most = bin_words(kMaxTileChunks) * 4;
  if constexpr (PASS != 2)
    if (h.copies > 1) {
      kern = hist_kernel<PASS, LEI, true>;
      most = kBankWords * 4;
    }
  if (!allow_smem(kern, most)) return kErrCuda;
  return launch_dependent(kern, dim3((unsigned)(h.tiles * h.ranges + cr.blocks)), dim3(h.threads), smem, s, a, h.tiles,
                          h.chunks, h.copies, h.tpc, ls, cr) == cudaSuccess
             ? kOk
             : kErrCuda;
}

}  // namespace

int launch_hist(const HistArgs& a, int pass, cudaStream_t s) {
  const LeiStream none;
  if (pass == 3) return launch_hist_pass<3, false>(a, none, CoefRows(), s);
  return pass == 1 ? launch_hist_pass<1, false>(a, none, CoefRows(), s)
                   : launch_hist_pass<2, false>(a, none, CoefRows(), s);
}

int launch_hist_coef(const HistArgs& a, const LeiArgs& la, float* coef, cudaStream_t s) {
  if (la.M < 1 || !coef) return kErrInvalidArg;
  return launch_hist_pass<1, false>(a, LeiStream(), CoefRows{la, coef, 0}, s);
}

int launch_hist_lei(const HistArgs& a, int pass, const LeiStream& lei, cudaStream_t s) {
  LeiStream ls = lei;
  // of 32 (half of them of 16): the passes are DRAM-bound, and the more warps stream from the start
  // the sooner they are, until counting is what takes longest.  A pass that
  // carries every token, 14 / 16 / 18 / 20: T = 65,536, E = 64 30.9 / 31.1 /
  // 33.9 / 32.7 us a step, T = 200,003, E = 96 72.2 / 71.5 / 71.9 / 71.7, T =
  // 524,288, E = 256 311.6 / 311.2 / 310.3 / 308.9, T = 2,097,152 1168.7 /
  // 1166.8 / 1166.1 / 1165.9; half of them each, 8 / 12 / 14 / 16: T =
  // 2,097,152, E = 256 1198 / 1180 / 1175 / 1191.
  ls.warps = ls.t1 - ls.t0 < a.T ? 14 : a.T * a.E > int64_t(1) << 26 ? 20 : 16;
  if (!ls.g || !ls.coef || !ls.off || ls.M < 1 || ls.t0 < 0 || ls.t1 < ls.t0) return kErrInvalidArg;
  return pass == 1 ? launch_hist_pass<1, true>(a, ls, CoefRows(), s) : launch_hist_pass<2, true>(a, ls, CoefRows(), s);
}

}  // namespace eqb
