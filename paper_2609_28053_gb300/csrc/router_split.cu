// router_split.cu -- router logits z_t = W_r x_t (arXiv 2609.28053, Sec. 2,
// Eq. 1) for few tokens, with routing: the projection of decoding batches.
//
// The persistent kernel (router_gemm.cu) gives a 128-token tile to one SM,
// which then reads the whole of W_r and the tile's rows of x by itself (2 MB
// at d = 4096, E = 128: 25 us, the SM's own bandwidth).  Here a cluster of n
// blocks shares the tile: block r multiplies its part of the columns (TMA
// ring, tcgen05.mma into tensor memory as there), parks its fp32 partial
// [128, E] in its own shared memory, and after a cluster barrier reduces
// every n-th row over the blocks' partials, in block order, through
// distributed shared memory: a warp per token, each load a 512-byte run of
// another block's row (16-byte pieces 32 bytes apart took twice as long),
// rounded to bf16 and stored as z, and routed from the same registers
// (warp_route, route_warp.cuh).  A block counts the loads of the microbatch
// that its tile starts in in shared memory and adds them as whole lines: T =
// 4,224, d = 1,024, E = 64, M = 4 with the coarse pass 14.0 us, 20.5 with each
// token's eight scattered adds to global memory (15.6 unsplit).
//
// Each partial sum is shorter than the whole: 329, 672 and 1,226 of 1e6 logits
// round to another bf16 value than the 64-bit sums do in eight, four and two
// parts (d = 4,096, E = 128), 2,295 in one sum.
//
// Every mbarrier wait is bounded and every thread reaches both cluster
// barriers, whether or not a wait ran out; after one that did, the tile loads
// in flight are waited for (bounded again) before the block returns.
#include "route_warp.cuh"
#include "tcgen05.cuh"

namespace eqb {

namespace {

constexpr int kThreads = 512;  // warp 0 TMA, warp 1 MMA, warps 4..7 read the accumulator; all reduce

struct SplitArgs {
  uint16_t* z;
  int T, d, N, S;  // N experts, S stages
  int32_t* err;
  SplitRoute ro;
};

// 16 bytes of block `rank`'s shared memory at this block's address `addr`.
__device__ __forceinline__ float4 ld_dsmem(uint32_t addr, uint32_t rank) {
  uint32_t ra;
  float4 v;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(ra)
               : "memory");
  return v;
}

// Four columns of a row summed over the cluster's NB partials in block order,
// as bf16 pairs; every load is in flight before the first use.
template <int NB>
__device__ __forceinline__ uint2 sum_columns(uint32_t at) {
  float4 p[NB];
#pragma unroll
  for (int k = 0; k < NB; ++k) p[k] = ld_dsmem(at, k);
  float4 s = p[0];
#pragma unroll
  for (int k = 1; k < NB; ++k) {
    s.x += p[k].x;
    s.y += p[k].y;
    s.z += p[k].z;
    s.w += p[k].w;
  }
  return make_uint2(pack_bf16x2_rn(s.x, s.y), pack_bf16x2_rn(s.z, s.w));
}

// NB blocks to a cluster.
template <int NB>
__global__ void __launch_bounds__(kThreads, 1)
    router_split_kernel(const __grid_constant__ CUtensorMap tmx, const __grid_constant__ CUtensorMap tmw,
                        SplitArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(16) float bs[128];
  __shared__ uint2 cand[kThreads / 32][32];
  __shared__ __align__(8) uint64_t bars[2 * 8 + 1];  // full, empty, accumulator done
  __shared__ uint32_t tmem_holder;
  __shared__ int cnt[128];       // loads of the tile's first microbatch
  __shared__ int tile_mb;        // which it is,
  __shared__ int64_t tile_mb_hi; // and where it ends
  __shared__ int abort_word, issued;  // issued: the producer's loads, for the drain after an abort
  volatile int* abort_flag = &abort_word;
  const int T = a.T, N = a.N, S = a.S;
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;  // 1 KiB alignment for the swizzle atoms
  const uint32_t a_bytes = kBM * kBK * 2;
  const uint32_t stage_bytes = a_bytes + static_cast<uint32_t>(N) * kBK * 2;
  auto full = [&](int s) { return smem_u32(bars + s); };
  auto empty = [&](int s) { return smem_u32(bars + 8 + s); };
  const uint32_t accf = smem_u32(bars + 16);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int tile = static_cast<int>(blockIdx.x) / NB;
  const int KB = a.d / kBK;
  const int kb0 = static_cast<int>(rank) * KB / NB, kb1 = (static_cast<int>(rank) + 1) * KB / NB;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full(s), 1);
      mbar_init(empty(s), 1);
    }
    mbar_init(accf, 1);
    abort_word = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_holder)),
                 "r"(256u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_holder;
  griddep_wait();

  if (warp == 0) {
    if (lane == 0) {
      int stage = 0, kb = kb0;
      uint32_t phase = 0;
      for (; kb < kb1; ++kb) {
        if (!mbar_wait(empty(stage), phase ^ 1u, abort_flag)) break;
        const uint32_t dst = base + static_cast<uint32_t>(stage) * stage_bytes;
        mbar_expect_tx(full(stage), stage_bytes);
        tma_load_2d(dst, &tmx, full(stage), kb * kBK, tile * kBM);
        tma_load_2d(dst + a_bytes, &tmw, full(stage), kb * kBK, 0);
        if (++stage == S) { stage = 0; phase ^= 1u; }
      }
      issued = kb - kb0;
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = umma_idesc_bf16(kBM, N);
      int stage = 0;
      uint32_t phase = 0;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!mbar_wait(full(stage), phase, abort_flag)) break;
        tc_fence_after();
        const uint32_t sa = base + static_cast<uint32_t>(stage) * stage_bytes;
        const uint64_t ad = sw128_desc(sa), bd = sw128_desc(sa + a_bytes);
#pragma unroll
        for (int kk = 0; kk < kBK / 16; ++kk)  // K = 16 per MMA: +32 bytes in the atom
          umma_bf16(tmem, ad + 2u * kk, bd + 2u * kk, idesc, (kb != kb0 || kk != 0) ? 1u : 0u);
        umma_commit(empty(stage));
        if (++stage == S) { stage = 0; phase ^= 1u; }
      }
      umma_commit(accf);  // after a wait that ran out too: the MMAs issued are drained
    }
  } else if (a.ro.b) {
    for (int e = threadIdx.x - 64; e < N; e += kThreads - 64) {
      const float bv = a.ro.b[e];
      bs[e] = bv;
      if (!isfinite(bv)) raise_flag(a.err, kErrNonfinite);
      cnt[e] = 0;
    }
    if (a.ro.loads && warp == 2) {
      const int l = warp_microbatch_of(a.ro.off, a.ro.M, (int64_t)tile * kBM, lane);
      if (lane == 0) {
        tile_mb = l;
        tile_mb_hi = __ldg(a.ro.off + l + 1);
      }
    }
  }
  __syncwarp();

  // The accumulator into shared memory, over the stages (every MMA that reads
  // them is done, and with it every TMA load): row stride N + 4 floats, so the
  // lanes' 16-byte stores meet no bank twice.
  const bool done = mbar_wait(accf, 0u, abort_flag);
  const uint32_t pstride = 4u * static_cast<uint32_t>(N + 4);
  float* part = reinterpret_cast<float*>(smem_raw + (base - raw));
  __syncthreads();  // no role is still using the stages
  if (warp >= 4 && warp < 8 && __all_sync(kFull, done)) {
    tc_fence_after();
    const int q = warp & 3;  // TMEM lane quarter accessible to this warp
    for (int c = 0; c < N; c += 32) {
      uint32_t r[32];
      tmem_ld32(tmem + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(c), r);
      uint4* dst = reinterpret_cast<uint4*>(part + (q * 32 + lane) * (N + 4) + c);
#pragma unroll
      for (int v = 0; v < 8; ++v)
        if (c + 4 * v < N) dst[v] = make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
    }
    tc_fence_before();
  }
  cluster_sync();  // every block's partial is in its shared memory

  // Rows rank, rank + NB, ... of the tile, a warp per row.
  constexpr int R = kBM / NB;
  int mb = 0;
  int64_t mb_lo = 1, mb_hi = 0;  // token range of mb (none yet)
  for (int i = warp; i < R; i += kThreads / 32) {
    const int row = static_cast<int>(rank) + NB * i;
    const int64_t t = (int64_t)tile * kBM + row;
    if (t >= T) break;
    // Lane l sums columns 4l..4l+3 and, past 128 experts, 128 + 4l.. : whole
    // 512-byte runs of the other blocks' rows.
    uint2 lo = make_uint2(0u, 0u), hi = lo;
    const uint32_t at = base + static_cast<uint32_t>(row) * pstride + 16u * lane;
    if (4 * lane < N) lo = sum_columns<NB>(at);
    if (128 + 4 * lane < N) hi = sum_columns<NB>(at + 512u);
    uint2* zr = reinterpret_cast<uint2*>(a.z + t * N);
    if (4 * lane < N) zr[lane] = lo;
    if (128 + 4 * lane < N) zr[32 + lane] = hi;
    if (!a.ro.b) continue;
    int e;
    float sc;
    const int K = a.ro.K;
    // router_route's rows: at most 128 experts, four to a lane
    float s[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
    if (4 * lane < N) {
      const float4 bv = reinterpret_cast<const float4*>(bs)[lane];
      s[0] = bf16_lo(lo.x) + bv.x;
      s[1] = bf16_hi(lo.x) + bv.y;
      s[2] = bf16_lo(lo.y) + bv.z;
      s[3] = bf16_hi(lo.y) + bv.w;
    }
    const float lmax = fmax_nan(fmax_nan(s[0], s[1]), fmax_nan(s[2], s[3]));
    const int r = warp_route(s, lmax, N, K, cand[warp], lane, a.err, e, sc);
    if (r == K) {
      a.ro.tau[t] = sc;
      if (!isfinite(sc)) raise_flag(a.err, kErrNonfinite);
    }
    if (r < K && a.ro.idx) a.ro.idx[t * K + r] = e;
    if (a.ro.loads) {
      if (t < tile_mb_hi) {
        if (r < K) atomicAdd(cnt + e, 1);
        continue;
      }
      if (!(t >= mb_lo && t < mb_hi)) {
        mb = warp_microbatch_of(a.ro.off, a.ro.M, t, lane);
        mb_lo = __ldg(a.ro.off + mb);
        mb_hi = __ldg(a.ro.off + mb + 1);
      }
      if (r < K) atomicAdd(a.ro.loads + (int64_t)mb * N + e, 1);
    }
  }
  cluster_sync();  // no block leaves while another reads its partial; cnt is complete
  if (a.ro.loads)
    for (int e = threadIdx.x; e < N; e += kThreads)
      if (cnt[e]) atomicAdd(a.ro.loads + (int64_t)tile_mb * N + e, cnt[e]);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u) : "memory");
  }
  if (threadIdx.x == 0 && *abort_flag) {
    drain_loads(issued, S, full);
    raise_flag(a.err, kErrCuda);
  }
}

}  // namespace

// Blocks per 128-token tile: 8, 4 or 2 while clusters of that size
// hold all tiles at once (8 tiles of 8 blocks run together, 16 do
// not; 32 of 4; 64 of 2), from d = 1,024 on.  Logits alone, us, for n = 1 / 2 /
// 4 / 8: T = 128, d = 4,096, E = 128 19.9 / 13.8 / 9.5 / 7.8; d = 1,024 7.9 /
// 7.8 / 6.4 / 6.1, E = 256 9.3 / 8.4 / 8.4 / 8.5; T = 2,048, d = 4,096, E =
// 128 20.5 / 14.2 / 9.9 / 15.0; T = 8,192 20.7 / 15.1 / 19.9 / 36.9; d = 512,
// E = 256, T = 128 7.2 / 7.4 / 7.8 / 8.2.  With routing, 64 tokens a block by a
// warp each take longer than 128 from the accumulator beside the next tile's
// MMAs, so two blocks pay from more columns on (T = 4,225, n = 1 / 2): E = 64 9.8
// / 12.6 at d = 1,024, 13.9 / 14.8 at 2,048, 18.0 / 16.9 at 3,072; E = 128 11.8 /
// 12.4 at 1,024, 13.9 / 13.4 at 1,536.  The rule does not ask whether there is
// routing: logits must not depend on it.
int router_splits(int64_t T, int d, int E, int sm_count) {
  const int64_t tiles = (T + kBM - 1) / kBM;
  if (d < 1024) return 1;
  if (tiles * 16 <= sm_count * 7 / 8) return 8;
  if (tiles * 4 <= sm_count * 7 / 8) return 4;
  const int least = E == 64 ? 3072 : E <= 128 ? 1536 : 1024;  // columns from which two pay
  return d >= least && tiles * 2 <= sm_count * 7 / 8 ? 2 : 1;
}

int launch_router_split(const uint16_t* x, const uint16_t* W, int64_t T, int d, int E, int n, uint16_t* z,
                        const SplitRoute& ro, int32_t* err, cudaStream_t s) {
  DeviceInfo di;
  if (int rc = device_info(&di)) return rc;
  if (ro.b && E > 128) return kErrUnsupported;
  const int most = di.max_smem_optin - 7 * 1024;  // beside the static arrays
  // before the maps: encoding them needs a context, which a thread's first runtime call makes current
  auto kern = n == 8 ? router_split_kernel<8> : n == 4 ? router_split_kernel<4> : router_split_kernel<2>;
  if (!allow_smem(kern, most)) return kErrCuda;
  CUtensorMap tmx, tmw;
  if (!make_map(&tmx, x, static_cast<uint64_t>(T), static_cast<uint64_t>(d), kBM)) return kErrCuda;
  if (!make_map(&tmw, W, static_cast<uint64_t>(E), static_cast<uint64_t>(d), static_cast<uint32_t>(E)))
    return kErrCuda;
  SplitArgs a{z, static_cast<int>(T), d, E, 0, err, ro};
  const int stage_bytes = (kBM + E) * kBK * 2;
  const int part = kBM * (E + 4) * 4;
  int S = (most - 1024) / stage_bytes;            // 1 KiB of alignment slack
  if (S > 8) S = 8;
  const int blocks = d / kBK / n + 1;  // k-blocks of the longest part
  if (S > blocks) S = blocks;
  if (S < 2) S = 2;
  a.S = S;
  int smem = S * stage_bytes;
  if (smem < part) smem = part;
  smem += 1024;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((T + kBM - 1) / kBM * n));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = n;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, tmx, tmw, a) == cudaSuccess ? kOk : kErrCuda;
}

}  // namespace eqb
