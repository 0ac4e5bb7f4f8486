// route_wide.cu -- top-K routing, cutoff tau_t and per-microbatch loads
// (Sec. 2, Eq. 1 and the QB paragraph of arXiv 2609.28053) for rows of 136 to
// 640 experts with K + 1 <= 16, at a compile-time row width of 160, 192, 224,
// 256, 320, 384, 512 or 640 experts (narrower rows padded with -inf).
//
// One thread owns one token; a warp owns a tile of 32 consecutive tokens,
// which each lane brings into shared memory with one bulk copy of its row
// (completion on a per-warp mbarrier) while the next tile is prefetched into
// L2.  Rows are padded to a stride of 4 (mod 8) words so the 32 lanes reading
// the same 16-byte chunk of their own rows hit distinct banks.  The per-token
// work (bound from packed group maxima, candidate masks, exact insertion of
// the candidates) is route_row() in route_wide.cuh.  It is bound by the ALU
// pipe and by the latency of its dependent instructions (12 warps an SM at
// E = 256): T = 2,097,152, E = 256, K = 8 takes 211 us (169 at the copy
// peak), T = 1,000,000, E = 264 152 us (219 with the runtime-width kernel it
// replaced there), E = 160 91 (139).  Four warps at E = 640: T = 131,072, E =
// 520 52 us (95; a warp per token 115).
#include "route_wide.cuh"

namespace eqb {

namespace {

// Warps per block: as many as shared memory holds (12 at E = 256), at most 16.
template <int E>
constexpr int wide_max_warps() {
  return (232448 - WideLayout<E>::HEAD) / WideLayout<E>::WARP < 16
             ? (232448 - WideLayout<E>::HEAD) / WideLayout<E>::WARP
             : 16;
}

// EXACT: the row has E experts, so that the copies' addresses and sizes are
// constants too (T = 2,097,152, E = 256, K = 8 214 us, 224 without).
template <int E, int KP1, bool EXACT>
__global__ void __launch_bounds__(32 * wide_max_warps<E>(), 1)
    route_wide_kernel(RouteArgs a, int64_t tiles_per_warp) {
  using L = WideLayout<E>;
  const int real = EXACT ? E : a.E;
  extern __shared__ __align__(16) uint8_t smem[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5;

  float* bs = reinterpret_cast<float*>(smem);
  uint32_t* bdn = reinterpret_cast<uint32_t*>(smem + 4 * E);  // RD(b) packed pairs
  uint32_t* bup = bdn + E / 2;                                 // RU(b) packed pairs
  uint8_t* wreg = smem + L::HEAD + wid * L::WARP;
  uint8_t* tile = wreg;
  uint32_t* mw = reinterpret_cast<uint32_t*>(wreg + L::TILE);  // [NCH/4][32 lanes]
  TileLoads loads{reinterpret_cast<int*>(wreg + L::TILE + L::ENT)};
  const uint32_t bar = saddr(wreg + L::TILE + L::ENT + L::WL);

  if (!EXACT) pad_rows<E>(tile, 32, L::RS, real, lane);
  for (int e = lane; e < E; e += 32) loads.wl[e] = 0;
  if (lane == 0) {
    bar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  griddep_wait();
  load_bias_tables<E>(a.b, real, bs, bdn, bup, a.err);
  __syncthreads();

  const int64_t ntiles = (a.T + 31) >> 5;
  const int64_t gw = (int64_t)blockIdx.x * nw + wid;
  const int64_t tb = gw * tiles_per_warp;
  const int64_t te = min(tb + tiles_per_warp, ntiles);
  if (tb >= te) return;
  const uint4* bdn4 = reinterpret_cast<const uint4*>(bdn);
  const uint4* bup4 = reinterpret_cast<const uint4*>(bup);
  const uint8_t* rowp = tile + lane * L::RS;

  // Lane r copies row r of the tile (rows past T are left as they are: their
  // results are never stored).
  auto load_tile = [&](int64_t tl) {
    const int64_t t0 = tl << 5;
    const int rows = static_cast<int>(min((int64_t)32, a.T - t0));
    if (lane == 0) bar_expect_tx(bar, static_cast<uint32_t>(rows * real * 2));
    __syncwarp();
    if (lane < rows) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bulk_copy(saddr(tile + lane * L::RS), a.z + (t0 + lane) * real, real * 2, bar);
    }
  };
  auto prefetch = [&](int64_t tl) {
    if (lane == 0 && tl < te) {
      const int64_t t0 = tl << 5;
      const uint32_t bytes = static_cast<uint32_t>(min((int64_t)32, a.T - t0) * real * 2);
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a.z + t0 * real), "r"(bytes) : "memory");
    }
  };

  uint32_t phase = 0;
  load_tile(tb);
  prefetch(tb + 1);
  for (int64_t tl = tb; tl < te; ++tl) {
    if (!__all_sync(kFull, bar_wait_bounded(bar, phase, kRouteWaitLimit))) {
      // The copy did not complete in time: report it, give the copies in
      // flight one more bounded wait, and stop.
      raise_flag(a.err, kErrCuda);
      bar_wait_bounded(bar, phase, kRouteWaitLimit);
      return;
    }
    phase ^= 1u;

    const int64_t t = (tl << 5) + lane;
    const bool valid = t < a.T;

    float v[KP1];
    int id[KP1];
    route_row<E, KP1>(rowp, bs, bdn4, bup4, mw, lane, valid, a.err, v, id);
    __syncwarp();  // every lane is done with the tile

    if (tl + 1 < te) {
      load_tile(tl + 1);
      prefetch(tl + 2);
    }
    if (valid) store_route<KP1>(a, t, v, id);
    if (a.loads) loads.count<KP1>(a, tl << 5, valid, id, lane);
  }
  if (a.loads) loads.flush(a, lane);
}

template <int E, int KP1, bool EXACT>
int launch_wide_t(const RouteArgs& a, cudaStream_t s) {
  using L = WideLayout<E>;
  DeviceInfo di;
  if (int rc = device_info(&di)) return rc;
  constexpr int nw_max = wide_max_warps<E>();
  const int64_t ntiles = (a.T + 31) / 32;
  // few tiles: as few warps a block as leave none idle, over all SMs
  int64_t nw = (ntiles + di.sm_count - 1) / di.sm_count;
  if (nw > nw_max) nw = nw_max;
  const int smem = L::HEAD + static_cast<int>(nw) * L::WARP;
  if (smem > di.max_smem_optin) return kErrUnsupported;
  int64_t grid = di.sm_count;
  const int64_t max_grid = (ntiles + nw - 1) / nw;
  if (grid > max_grid) grid = max_grid;
  const int64_t tpw = (ntiles + grid * nw - 1) / (grid * nw);
  auto kern = route_wide_kernel<E, KP1, EXACT>;
  if (!allow_smem(kern, L::HEAD + nw_max * L::WARP)) return kErrCuda;
  return launch_dependent(kern, dim3((unsigned)grid), dim3((unsigned)nw * 32), smem, s, a, tpw) == cudaSuccess
             ? kOk
             : kErrCuda;
}

template <int E>
int launch_wide_e(const RouteArgs& a, cudaStream_t s) {
  const int kp1 = a.K + 1;
  if (kp1 <= 3) return launch_wide_t<E, 3, true>(a, s);
  if (kp1 <= 5) return launch_wide_t<E, 5, true>(a, s);
  if (kp1 <= 7) return launch_wide_t<E, 7, true>(a, s);
  if (kp1 <= 9) return launch_wide_t<E, 9, true>(a, s);
  return launch_wide_t<E, 16, true>(a, s);
}

// A row of fewer than E experts.
template <int E>
int launch_wide_padded(const RouteArgs& a, cudaStream_t s) {
  const int kp1 = a.K + 1;
  if (kp1 <= 5) return launch_wide_t<E, 5, false>(a, s);
  if (kp1 <= 9) return launch_wide_t<E, 9, false>(a, s);
  return launch_wide_t<E, 16, false>(a, s);
}

}  // namespace

int launch_route_wide(const RouteArgs& a, cudaStream_t s) {
  if (a.K + 1 > 16) return kErrUnsupported;
  if (a.E == 256) return launch_wide_e<256>(a, s);
  if (a.E == 384) return launch_wide_e<384>(a, s);
  if (a.E == 512) return launch_wide_e<512>(a, s);
  if (a.E <= 160) return launch_wide_padded<160>(a, s);
  if (a.E <= 192) return launch_wide_padded<192>(a, s);
  if (a.E <= 224) return launch_wide_padded<224>(a, s);
  if (a.E <= 256) return launch_wide_padded<256>(a, s);
  if (a.E <= 320) return launch_wide_padded<320>(a, s);
  if (a.E <= 384) return launch_wide_padded<384>(a, s);
  if (a.E <= 512) return launch_wide_padded<512>(a, s);
  if (a.E <= 640) return launch_wide_padded<640>(a, s);
  return kErrUnsupported;
}

}  // namespace eqb
