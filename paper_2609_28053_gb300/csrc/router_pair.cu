// router_pair.cu -- router logits z_t = W_r x_t (arXiv 2609.28053, Sec. 2,
// Eq. 1) for many experts, columns and tokens: the projection by pairs of SMs.
//
// With E = 256 a 64-column stage of the one-SM kernel (router_gemm.cu) is
// 16 KiB of x and 32 KiB of W_r, and what an SM takes in by TMA (about 55 B a
// clock) bounds it, not the tensor cores.  Here a cluster of two blocks takes
// 256 tokens, 128 each; each block stages its tokens' rows and one half of the
// experts' rows of W_r, and the tensor cores of both SMs read the two halves
// from both shared memories (tcgen05.mma.cta_group::2, M = 256): 32 KiB a
// stage and block.  Roles and buffers are those of router_gemm.cu, per block,
// except that block 0 alone issues the MMAs:
//   warp 0      TMA producer of the block's own tiles; both blocks' loads
//               complete on block 0's `full` barrier;
//   warp 1      (block 0) MMAs; tcgen05.commit frees the stage in both blocks
//               and signals both accumulators full;
//   warps 2..5  epilogue of the block's 128 tokens; both blocks' epilogues
//               release the accumulator on block 0's `acce` barrier.
// A pair costs about 1.3 us more to start and finish than two blocks on their
// own; each 64-column stage takes it 0.30 us where it took 0.38 (72 SMs busy),
// 0.39 against 0.58 (130, x from DRAM).  z is the same bit for bit.
//
// Every wait is bounded as in router_gemm.cu, and every thread reaches both
// cluster barriers whether or not a wait ran out.  After one that did, each
// block's producer waits (bounded again) for its loads in flight before the
// last of them: block 0 on the barriers that they complete on, block 1, which
// cannot poll those, for the MMAs that read its stages.
#include "tcgen05.cuh"

namespace eqb {

namespace {

struct PairArgs {
  uint16_t* z;
  int T, d, N, S;
  int32_t* err;
};

// Block 0's barrier at this block's address `bar`.
__device__ __forceinline__ uint32_t leader_bar(uint32_t bar) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(bar));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Bounded wait for arrivals from both blocks.
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  for (uint32_t i = 0; i < kSpinLimit; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(1000u)
        : "memory");
    if (ok) return true;
    if ((i & 63u) == 63u && *abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}
// A tile into this block's shared memory, completing on a barrier of either block.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.cta_group::2"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// The MMAs issued so far arrive, once done, on the barrier at this offset in
// the blocks of `mask` (3: both).
__device__ __forceinline__ void umma_commit_pair(uint32_t bar, uint16_t mask) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"(mask)
      : "memory");
}

__global__ void __launch_bounds__(192, 1)
    router_pair_kernel(const __grid_constant__ CUtensorMap tmx, const __grid_constant__ CUtensorMap tmw, PairArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * 8 + 5];  // full, empty, accumulators full and empty, drain
  __shared__ uint32_t tmem_holder;
  __shared__ int abort_word;
  volatile int* abort_flag = &abort_word;
  const int T = a.T, N = a.N, S = a.S;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;  // 1 KiB alignment for the swizzle atoms
  const uint32_t a_bytes = kBM * kBK * 2;
  const uint32_t stage_bytes = a_bytes + static_cast<uint32_t>(N / 2) * kBK * 2;
  auto full = [&](int s) { return smem_u32(bars + s); };
  auto empty = [&](int s) { return smem_u32(bars + 8 + s); };
  auto accf = [&](int b) { return smem_u32(bars + 16 + b); };
  auto acce = [&](int b) { return smem_u32(bars + 18 + b); };
  const uint32_t drain = smem_u32(bars + 20);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_rank());
  const int pairs = (T + 2 * kBM - 1) / (2 * kBM);
  const int first = static_cast<int>(blockIdx.x >> 1), step = static_cast<int>(gridDim.x >> 1);
  const int KB = a.d / kBK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full(s), 1);
      mbar_init(empty(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf(b), 1);
      mbar_init(acce(b), 256);
    }
    mbar_init(drain, 1);
    abort_word = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_holder)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync();  // both blocks' barriers stand before either is signalled from the other
  tc_fence_after();
  const uint32_t tmem = tmem_holder;
  griddep_wait();

  if (warp == 0) {
    if (lane == 0) {
      int stage = 0, issued = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int p = first; p < pairs && ok; p += step) {
        for (int kb = 0; kb < KB; ++kb, ++issued) {
          if (!mbar_wait(empty(stage), phase ^ 1u, abort_flag)) { ok = false; break; }
          const uint32_t dst = base + static_cast<uint32_t>(stage) * stage_bytes;
          if (rank == 0) mbar_expect_tx(full(stage), 2u * stage_bytes);  // both blocks' loads
          const uint32_t bar = leader_bar(full(stage));
          tma_load_2d_pair(dst, &tmx, bar, kb * kBK, (2 * p + rank) * kBM);
          tma_load_2d_pair(dst + a_bytes, &tmw, bar, kb * kBK, rank * (N / 2));
          if (++stage == S) { stage = 0; phase ^= 1u; }
        }
      }
      // the last stages are free: no arrival from the other block is outstanding
      for (int s = 0; s < S && ok; ++s) {
        ok = mbar_wait(empty(stage), phase ^ 1u, abort_flag);
        if (++stage == S) { stage = 0; phase ^= 1u; }
      }
      if (!ok) {
        if (rank == 0) drain_loads(issued, S, full);
        else drain_loads(issued, S, empty);  // MMA i's commit is phase i / S of its stage's `empty`
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      const uint32_t idesc = umma_idesc_bf16(2 * kBM, N);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      int it = 0;
      for (int p = first; p < pairs && ok; p += step, ++it) {
        const int buf = it & 1;
        const uint32_t use = static_cast<uint32_t>(it >> 1);
        if (!mbar_wait_cluster(acce(buf), (use & 1u) ^ 1u, abort_flag)) break;
        tc_fence_after();
        const uint32_t dt = tmem + static_cast<uint32_t>(buf * N);
        for (int kb = 0; kb < KB; ++kb) {
          if (!mbar_wait_cluster(full(stage), phase, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = base + static_cast<uint32_t>(stage) * stage_bytes;
          const uint64_t ad = sw128_desc(sa), bd = sw128_desc(sa + a_bytes);
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk)  // K = 16 per MMA: +32 bytes in the atom
            umma_bf16_pair(dt, ad + 2u * kk, bd + 2u * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
          umma_commit_pair(empty(stage), 3);
          if (++stage == S) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        umma_commit_pair(accf(buf), 3);
      }
      // Drain: all MMAs issued above complete before TMEM is released.
      umma_commit_pair(drain, 1);
      for (uint32_t i = 0; i < kSpinLimit; ++i)
        if (mbar_try_wait(drain, 0u)) break;
    }
  } else {
    const int q = warp & 3;  // TMEM lane quarter accessible to this warp
    const uint32_t lane_base = static_cast<uint32_t>(q * 32) << 16;
    int it = 0;
    for (int p = first; p < pairs; p += step, ++it) {
      const int buf = it & 1;
      const uint32_t use = static_cast<uint32_t>(it >> 1);
      // the warp leaves together (the loop body has warp-wide operations)
      if (!__all_sync(kFull, mbar_wait(accf(buf), use & 1u, abort_flag))) break;
      tc_fence_after();
      const int64_t row = static_cast<int64_t>(2 * p + rank) * kBM + q * 32 + lane;
      for (int c = 0; c < N; c += 32) {
        uint32_t r[32];
        tmem_ld32(tmem + lane_base + static_cast<uint32_t>(buf * N + c), r);
        if (row < T) {
          uint4* dst = reinterpret_cast<uint4*>(a.z + row * N + c);
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            uint4 o;
            o.x = pack_bf16x2_rn(__uint_as_float(r[8 * v + 0]), __uint_as_float(r[8 * v + 1]));
            o.y = pack_bf16x2_rn(__uint_as_float(r[8 * v + 2]), __uint_as_float(r[8 * v + 3]));
            o.z = pack_bf16x2_rn(__uint_as_float(r[8 * v + 4]), __uint_as_float(r[8 * v + 5]));
            o.w = pack_bf16x2_rn(__uint_as_float(r[8 * v + 6]), __uint_as_float(r[8 * v + 7]));
            dst[v] = o;
          }
        }
      }
      tc_fence_before();
      mbar_arrive_cluster(leader_bar(acce(buf)));
    }
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync();  // neither block leaves while the other's MMAs or arrivals reach it
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
  if (threadIdx.x == 0 && *abort_flag) raise_flag(a.err, kErrCuda);
}

}  // namespace

int launch_router_pair(const uint16_t* x, const uint16_t* W, int64_t T, int d, int E, uint16_t* z, int32_t* err,
                       cudaStream_t s) {
  if (E > 256 || E % 32 != 0) return kErrUnsupported;  // one UMMA N over two SMs, two accumulators
  DeviceInfo di;
  if (int rc = device_info(&di)) return rc;
  const int most = di.max_smem_optin - 1024;  // beside the static arrays
  // before the maps: encoding them needs a context, which a thread's first runtime call makes current
  if (!allow_smem(router_pair_kernel, most)) return kErrCuda;
  CUtensorMap tmx, tmw;
  if (!make_map(&tmx, x, static_cast<uint64_t>(T), static_cast<uint64_t>(d), kBM)) return kErrCuda;
  if (!make_map(&tmw, W, static_cast<uint64_t>(E), static_cast<uint64_t>(d), static_cast<uint32_t>(E / 2)))
    return kErrCuda;
  PairArgs a{z, static_cast<int>(T), d, E, 0, err};
  const int stage_bytes = (kBM + E / 2) * kBK * 2;
  int S = (most - 1024) / stage_bytes;        // 1 KiB of alignment slack
  if (S > 8) S = 8;
  a.S = S;
  const int smem = S * stage_bytes + 1024;
  const int64_t pairs = (T + 2 * kBM - 1) / (2 * kBM);
  const int64_t resident = di.sm_count / 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(2 * (pairs < resident ? pairs : resident)));
  cfg.blockDim = dim3(192);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, router_pair_kernel, tmx, tmw, a) == cudaSuccess ? kOk : kErrCuda;
}

}  // namespace eqb
