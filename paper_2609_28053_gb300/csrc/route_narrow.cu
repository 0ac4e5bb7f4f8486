// route_narrow.cu -- top-K routing, cutoff tau_t and per-microbatch loads
// (Sec. 2, Eq. 1 and the QB paragraph of arXiv 2609.28053) for rows of up to
// 128 experts with K + 1 <= 16.
//
// As route_wide.cu: one thread owns one token, a warp a tile of 32, the
// per-token work is route_row() at a compile-time row width of 32, 64, 96 or
// 128 experts (narrower rows padded with -inf).  Narrow rows are too short
// for a bulk copy each, so the warp brings the next tile, one contiguous
// piece of z, into the other of two buffers with 16-byte asynchronous copies
// (consecutive lanes take consecutive chunks) while it routes this one.
// Blocks of four warps, as many to an SM as registers and shared memory hold.
// Bound by the ALU pipe (79% busy at E = 64): T = 1,000,000, E = 64, K = 8
// takes 60 us, T = 200,003, E = 96, K = 6 16, T = 2,000,000, E = 8, K = 2 42;
// 108, 26 and 105 with the runtime-width kernel that it replaced, which staged
// rows with a copy loop per row, sorted 16 groups in fp32, listed chunks
// behind branches and searched the microbatch of every token.
#include "route_wide.cuh"

namespace eqb {

namespace {

constexpr int kNarrowWarps = 4;

template <int E>
struct NarrowLayout {
  using W = WideLayout<E>;
  static constexpr int WARP = 2 * W::TILE + W::ENT + W::WL;
  static constexpr int SMEM = W::HEAD + kNarrowWarps * WARP;
};

// EXACT: the row has E experts.
template <int E, int KP1, bool EXACT>
__global__ void __launch_bounds__(32 * kNarrowWarps) route_narrow_kernel(RouteArgs a, int64_t tiles_per_warp) {
  using L = NarrowLayout<E>;
  using W = WideLayout<E>;
  extern __shared__ __align__(16) uint8_t smem[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int real = EXACT ? E : a.E;
  const int nch = real >> 3;

  float* bs = reinterpret_cast<float*>(smem);
  uint32_t* bdn = reinterpret_cast<uint32_t*>(smem + 4 * E);  // RD(b) packed pairs
  uint32_t* bup = bdn + E / 2;                                 // RU(b) packed pairs
  uint8_t* tiles = smem + W::HEAD + wid * L::WARP;
  uint32_t* mw = reinterpret_cast<uint32_t*>(tiles + 2 * W::TILE);  // [E/32][32 lanes]
  TileLoads loads{reinterpret_cast<int*>(tiles + 2 * W::TILE + W::ENT)};

  if (!EXACT) pad_rows<E>(tiles, 64, W::RS, real, lane);
  for (int e = lane; e < E; e += 32) loads.wl[e] = 0;
  griddep_wait();

  const int64_t ntiles = (a.T + 31) >> 5;
  const int64_t gw = (int64_t)blockIdx.x * kNarrowWarps + wid;
  const int64_t tb = min(gw * tiles_per_warp, ntiles);
  const int64_t te = min(tb + tiles_per_warp, ntiles);
  const uint4* bdn4 = reinterpret_cast<const uint4*>(bdn);
  const uint4* bup4 = reinterpret_cast<const uint4*>(bup);

  // Chunk lane, lane + 32, ... of the tile's 32 * nch; rows past T are
  // zero-filled (their results are never stored).
  const int row0 = lane / nch, col0 = lane - row0 * nch;
  const int drow = 32 / nch, dcol = 32 - drow * nch;
  auto load_tile = [&](int64_t tl, int buf) {
    const int64_t t0 = tl << 5;
    const int rows = static_cast<int>(min((int64_t)32, a.T - t0));
    const uint16_t* src = a.z + t0 * real + lane * 8;
    uint8_t* dst = tiles + buf * W::TILE;
    int row = row0, col = col0;
    for (int k = 0; k < nch; ++k, src += 256) {
      const bool ok = row < rows;
      cp_async16(dst + row * W::RS + col * 16, ok ? src : a.z, ok ? 16 : 0);
      row += drow;
      col += dcol;
      if (col >= nch) {
        col -= nch;
        ++row;
      }
    }
    cp_async_commit();
  };

  if (tb < te) load_tile(tb, 0);
  load_bias_tables<E>(a.b, real, bs, bdn, bup, a.err);
  __syncthreads();
  int buf = 0;
  for (int64_t tl = tb; tl < te; ++tl, buf ^= 1) {
    if (tl + 1 < te) {
      load_tile(tl + 1, buf ^ 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncwarp();
    const int64_t t = (tl << 5) + lane;
    const bool valid = t < a.T;
    float v[KP1];
    int id[KP1];
    route_row<E, KP1>(tiles + buf * W::TILE + lane * W::RS, bs, bdn4, bup4, mw, lane, valid, a.err, v, id);
    if (valid) store_route<KP1>(a, t, v, id);
    if (a.loads) loads.count<KP1>(a, tl << 5, valid, id, lane);
    __syncwarp();  // every lane is done with the buffer and the mask words
  }
  if (a.loads) loads.flush(a, lane);
}

template <int E, int KP1, bool EXACT>
int launch_narrow_t(const RouteArgs& a, cudaStream_t s) {
  DeviceInfo di;
  if (int rc = device_info(&di)) return rc;
  auto kern = route_narrow_kernel<E, KP1, EXACT>;
  constexpr int smem = NarrowLayout<E>::SMEM;
  if (!allow_smem(kern, smem)) return kErrCuda;
  // by registers (72 to 98 a thread) or by shared memory
  static std::atomic<int> known[kMaxDevices];
  const int per_sm = resident_blocks(kern, 32 * kNarrowWarps, smem, di.dev, known);
  if (per_sm < 1) return kErrCuda;
  const int64_t ntiles = (a.T + 31) / 32;
  int64_t grid = (int64_t)di.sm_count * per_sm;
  const int64_t max_grid = (ntiles + kNarrowWarps - 1) / kNarrowWarps;
  if (grid > max_grid) grid = max_grid;
  const int64_t tpw = (ntiles + grid * kNarrowWarps - 1) / (grid * kNarrowWarps);
  return launch_dependent(kern, dim3((unsigned)grid), dim3(32 * kNarrowWarps), smem, s, a, tpw) == cudaSuccess
             ? kOk
             : kErrCuda;
}

template <int E, bool EXACT>
int launch_narrow_e(const RouteArgs& a, cudaStream_t s) {
  const int kp1 = a.K + 1;
  if (kp1 <= 3) return launch_narrow_t<E, 3, EXACT>(a, s);
  if (kp1 <= 5) return launch_narrow_t<E, 5, EXACT>(a, s);
  if (kp1 <= 7) return launch_narrow_t<E, 7, EXACT>(a, s);
  if (kp1 <= 9) return launch_narrow_t<E, 9, EXACT>(a, s);
  return launch_narrow_t<E, 16, EXACT>(a, s);
}

}  // namespace

int launch_route_narrow(const RouteArgs& a, cudaStream_t s) {
  if (a.K + 1 > 16) return kErrUnsupported;
  if (a.E == 64) return launch_narrow_e<64, true>(a, s);
  if (a.E == 128) return launch_narrow_e<128, true>(a, s);
  if (a.E <= 32) return launch_narrow_e<32, false>(a, s);
  if (a.E <= 64) return launch_narrow_e<64, false>(a, s);
  if (a.E <= 96) return launch_narrow_e<96, false>(a, s);
  if (a.E <= 128) return launch_narrow_e<128, false>(a, s);
  return kErrUnsupported;
}

}  // namespace eqb
