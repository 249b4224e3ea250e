// Two-SM form of the tcgen05 contraction engine: a cluster of two CTAs works on one
// 256-row tile with tcgen05.mma.cta_group::2.
//
// Each CTA stages 128 rows of A and half of the tile's B rows, and the pair's tensor
// cores read both halves of B; each CTA's TMEM receives its 128 rows x 256 columns. A
// stage of the same 64 KB feeds twice the products of the one-SM engine's 128 x 128
// tiles, which ask L2 for 85 bytes per clock and SM and their shared memory for 128 at
// the tensor cores' full rate: what L2 delivers to an SM bounded them.
//
//   warp 0        TMA producer (one thread of each CTA): its own stage, signalled on the
//                 leader's (rank 0) full barrier, which counts both CTAs' bytes
//   warp 1        MMA issuer (one thread of the leader); its commits free the stages and
//                 hand over the accumulators in both CTAs
//   warps 2..     epilogue, 8 warps: TMEM lane quadrant warp % 4, columns in two parts;
//                 they free an accumulator on the leader's barrier
//
// The products of a k-block, their order and the chunks of the reduction are those of
// the one-SM engine, so results are the same bit for bit (the tests compare both).
//
// A pair policy adapts a one-SM policy P of 128-column tiles:
//   Item decode_pair(int64_t) const;  int64_t total_pair() const;       (256 rows x TN columns)
//   Item sub(const Item&, int rank, int part) const;   (the 128 x (TN / 2) tile of a CTA's epilogue part)
// and its epilogue functions are P's, called with the sub-tile.
//
// Both CTAs meet at cluster barriers before TMEM is freed and before they exit; every
// other wait is bounded as in the one-SM engine, so each thread reaches them.
#pragma once
#include <atomic>

#include "tc_engine.cuh"

namespace gift {
namespace tc {

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// address of the leader's copy of a shared-memory location, in the cluster's shared window
__device__ __forceinline__ uint32_t leader_addr(uint32_t addr) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, "
      "p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// as mbar_wait, for arrivals from both CTAs of the pair
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, int* err, int site) {
  if (mbar_try_wait_cluster(bar, parity)) return true;
  const long long t0 = clock64();
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if ((i & 255u) == 0) {
      if (*reinterpret_cast<volatile int*>(err) != 0) return false;
      if (clock64() - t0 > kWaitCycles) {
        atomicCAS(err, 0, site);
        return false;
      }
    }
  }
}
// 2-D tile load into this CTA's shared memory, its bytes counted on a barrier of either CTA of the pair
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y,
                                                 uint32_t cluster_bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(cluster_bar)
      : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void mma_f16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// arrive once on the barrier at this offset in both CTAs when every MMA issued so far has completed
__device__ __forceinline__ void mma_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"((uint16_t)3)
      : "memory");
}

constexpr int kPairThreads = 64 + 256;  // producer, MMA issuer, eight epilogue warps

template <class P>
struct PairLayout {
  static_assert(P::EB == 2, "BF16 operands");
  static constexpr int TN = P::TN_PAIR;
  static_assert(TN == 256, "columns of the pair's tile");
  static constexpr int kABytes = kTM * 128;
  static constexpr int kBBytes = TN / 2 * 128;
  static constexpr int kPartsA = P::SPLIT == 1 ? 1 : 2;
  static constexpr int kPartsB = P::SPLIT == 3 ? 2 : 1;
  static constexpr int kStageBytes = kPartsA * kABytes + kPartsB * kBBytes;
  static constexpr int kBufs = 512 / TN;  // TMEM accumulators
  static constexpr int kBarBytes = 256;
  static constexpr int kFit = (232448 - 1024 - kBarBytes - 8 * P::kWarpSmem) / kStageBytes;
  static constexpr int STAGES = kFit > 8 ? 8 : kFit;
  static_assert(STAGES >= 2, "at least two stages");
  static_assert((2 * STAGES + 2 * kBufs) * 8 + 4 <= kBarBytes, "barriers and TMEM address fit");
  static constexpr int kSmem = 1024 + STAGES * kStageBytes + kBarBytes + 8 * P::kWarpSmem;
  static_assert(kSmem <= 232448, "shared memory per CTA");
};

template <class P>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
    tc_pair(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
            const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB2, const P p, int* err) {
  using L = PairLayout<P>;
  constexpr int S = L::STAGES;
  constexpr int NB = L::kBufs;
  constexpr int TN = L::TN;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S * L::kStageBytes);
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 2 * S + 2 * NB);
  uint8_t* wsm = smem + S * L::kStageBytes + L::kBarBytes;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank();
  const uint32_t full0 = smem_u32(bars);
  const uint32_t empty0 = full0 + 8 * S;
  const uint32_t tfull0 = empty0 + 8 * S;
  const uint32_t tempty0 = tfull0 + 8 * NB;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full0 + 8 * s, 1);   // (the leader's: its producer; both CTAs' bytes)
      mbar_init(empty0 + 8 * s, 1);  // the MMA issuer's commit
    }
    for (int b = 0; b < NB; ++b) {
      mbar_init(tfull0 + 8 * b, 1);     // the MMA issuer's commit
      mbar_init(tempty0 + 8 * b, 16);   // (the leader's: both CTAs' epilogue warps)
    }
    fence_barrier_init();
  }
  if (warp == 0) {
    tmem_alloc_pair(smem_u32(tmem_holder), 512);
    tmem_relinquish_pair();
  }
  fence_before_sync();
  __syncthreads();
  cluster_sync_all();  // the peer's barriers are initialised too
  fence_after_sync();
  const uint32_t tmem = *tmem_holder;
  const int64_t total = p.total_pair();
  const int64_t first = blockIdx.x >> 1, step = gridDim.x >> 1;
  constexpr uint32_t kIdesc = idesc_bf16(256, TN);
  bool ok = true;

  if (warp == 0) {
    if (lane == 0) {
      prefetch_tmap(&tmA);
      prefetch_tmap(&tmB);
      int stage = 0;
      uint32_t phase = 0;
      int last_phase[S];
#pragma unroll
      for (int s = 0; s < S; ++s) last_phase[s] = -1;
      for (int64_t item = first; ok && item < total; item += step) {
        const typename P::Item it = p.decode_pair(item);
        const int ar = p.a_row(it) + rank * kTM;
        const int nch = p.nchunks(it);
        for (int c = 0; ok && c < nch; ++c) {
          int br, kb0, kb1;
          p.chunk(it, c, br, kb0, kb1);
          br += rank * (TN / 2);
          for (int kb = kb0; kb < kb1; ++kb) {
            if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, err, kErrProducer)) {
              ok = false;
              break;
            }
            const uint32_t st = smem_u32(smem + stage * L::kStageBytes);
            const uint32_t bar = leader_addr(full0 + 8 * stage);
            if (rank == 0) mbar_expect_tx(full0 + 8 * stage, 2 * L::kStageBytes);
            tma_load_2d_pair(st, &tmA, kb * kTK, ar, bar);
            tma_load_2d_pair(st + L::kABytes, &tmB, kb * kTK, br, bar);
            if (P::SPLIT >= 2) tma_load_2d_pair(st + L::kABytes + L::kBBytes, &tmA2, kb * kTK, ar, bar);
            if (P::SPLIT == 3) tma_load_2d_pair(st + 2 * L::kABytes + L::kBBytes, &tmB2, kb * kTK, br, bar);
            last_phase[stage] = (int)phase;
            if (++stage == S) {
              stage = 0;
              phase ^= 1;
            }
          }
        }
      }
      // every stage consumed: its copies have landed and the commit's arrival has reached this CTA
      for (int s = 0; ok && s < S; ++s)
        if (last_phase[s] >= 0) ok = mbar_wait(empty0 + 8 * s, (uint32_t)last_phase[s], err, kErrProducer);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      int stage = 0;
      uint32_t phase = 0;
      int buf = 0;
      uint32_t bphase = 0;
      for (int64_t item = first; ok && item < total; item += step) {
        const typename P::Item it = p.decode_pair(item);
        const int nch = p.nchunks(it);
        for (int c = 0; ok && c < nch; ++c) {
          int br, kb0, kb1;
          p.chunk(it, c, br, kb0, kb1);
          if (!mbar_wait_cluster(tempty0 + 8 * buf, bphase ^ 1, err, kErrMma)) {
            ok = false;
            break;
          }
          fence_after_sync();
          const uint32_t d = tmem + buf * TN;
          for (int kb = kb0; kb < kb1; ++kb) {
            if (!mbar_wait_cluster(full0 + 8 * stage, phase, err, kErrMma)) {
              ok = false;
              break;
            }
            fence_after_sync();
            const uint32_t sa = smem_u32(smem + stage * L::kStageBytes);
            const uint32_t sb = sa + L::kABytes;
            const uint32_t sa2 = sb + L::kBBytes;
            const uint32_t sb2 = sa2 + L::kABytes;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {  // 16 BF16 elements of K each
              const uint32_t acc_in = (kb != kb0 || kk != 0) ? 1u : 0u;
              mma_f16_pair(d, sdesc_sw128(sa + kk * 32), sdesc_sw128(sb + kk * 32), kIdesc, acc_in);
              if (P::SPLIT == 3) mma_f16_pair(d, sdesc_sw128(sa + kk * 32), sdesc_sw128(sb2 + kk * 32), kIdesc, 1u);
              if (P::SPLIT >= 2) mma_f16_pair(d, sdesc_sw128(sa2 + kk * 32), sdesc_sw128(sb + kk * 32), kIdesc, 1u);
            }
            mma_commit_pair(empty0 + 8 * stage);
            if (++stage == S) {
              stage = 0;
              phase ^= 1;
            }
          }
          if (!ok) break;
          mma_commit_pair(tfull0 + 8 * buf);
          if (++buf == NB) {
            buf = 0;
            bphase ^= 1;
          }
        }
      }
    }
    __syncwarp();
  } else {
    const int quad = warp & 3, part = (warp - 2) >> 2;
    const int m = quad * 32 + lane;
    const int ew = warp - 2;
    uint8_t* my = wsm + ew * P::kWarpSmem;
    int buf = 0;
    uint32_t bphase = 0;
    for (int64_t item = first; ok && item < total; item += step) {
      const typename P::Item whole = p.decode_pair(item);
      const typename P::Item it = p.sub(whole, rank, part);
      typename P::Ctx ctx;
      __syncwarp();
      p.epi_begin(it, ctx, m, ew, my);
      __syncwarp();
      const int nch = p.nchunks(whole);
      for (int c = 0; c < nch; ++c) {
        if (!mbar_wait(tfull0 + 8 * buf, bphase, err, kErrTmemFull)) {
          ok = false;
          break;
        }
        fence_after_sync();
        p.epi_chunk(it, c, tmem + (static_cast<uint32_t>(quad * 32) << 16) + buf * TN + part * (TN / 2), ctx, m, my);
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(leader_addr(tempty0 + 8 * buf));
        if (++buf == NB) {
          buf = 0;
          bphase ^= 1;
        }
      }
      if (!ok) break;
      p.epi_end(it, ctx, m, my);
    }
    if constexpr (report_of<P>::value)
      if (!ok && lane == 0) report_wait(err);
  }
  if (!ok) {  // copies and MMAs of either CTA may still be on their way: let them land (bounded)
    const long long t0 = clock64();
    while (clock64() - t0 < kWaitCycles / 4) {
    }
  }
  __syncwarp();
  fence_before_sync();
  __syncthreads();
  cluster_sync_all();  // neither CTA's barriers, stages or TMEM are used any more
  if (warp == 0) {
    fence_after_sync();
    tmem_dealloc_pair(tmem, 512);
  }
  cluster_sync_all();
}

// clusters of two that run on the current device at once (a property of the device and the kernel, asked once)
template <class P>
int pair_clusters() {
  using L = PairLayout<P>;
  constexpr int kDevices = 64;
  static std::atomic<int> known[kDevices];
  int dev = 0;
  GIFT_CUDA(cudaGetDevice(&dev));
  if (dev < kDevices && known[dev].load() > 0) return known[dev].load();
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2);
  cfg.blockDim = dim3(kPairThreads);
  cfg.dynamicSmemBytes = L::kSmem;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = 2;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int n = 0;
  GIFT_CUDA(cudaFuncSetAttribute(tc_pair<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kSmem));
  GIFT_CUDA(cudaOccupancyMaxActiveClusters(&n, tc_pair<P>, &cfg));
  n = std::max(n, 1);
  if (dev < kDevices) known[dev].store(n);
  return n;
}

// Launch on as many pairs of SMs as run at once, at most `items` of them. B's tensor maps have boxes of TN / 2 rows.
template <class P>
void launch_pair(const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& a2, const CUtensorMap& b2, const P& p,
                 int* err, int64_t items, cudaStream_t s) {
  using L = PairLayout<P>;
  const unsigned grid = 2 * (unsigned)std::max<int64_t>(1, std::min<int64_t>(pair_clusters<P>(), items));
  GIFT_CUDA(cudaFuncSetAttribute(tc_pair<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kSmem));
  tc_pair<P><<<grid, kPairThreads, L::kSmem, s>>>(a, b, a2, b2, p, err);
  GIFT_LAUNCHED("tc_pair");
}

}  // namespace tc
}  // namespace gift
