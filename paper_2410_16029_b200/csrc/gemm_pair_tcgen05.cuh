// Grouped GEMM with 256 x 256 output tiles on pairs of SMs (a cluster of two CTAs, tcgen05 cta_group::2): the products of a refresh
// with G, out = A B for a table of problems, where the bases are more than 192 columns wide and K is short.
//
// What bounds them with a CTA of its own for every 128 x 256 tile is the path from L2 to the SMs, 10 to 11 TB/s: it stages 80 KB
// of operands for 64 steps of K with two parts of B, 48 KB with one.  A CTA of a pair stages its own 128 rows of A and half of
// B's columns, 48 KB or 32 KB, and the pair's MMA reads both halves.  The other way to share B, two accumulators of one CTA, takes
// all of the tensor memory and leaves the epilogue of a tile nothing to hide behind; here each CTA holds its 128 rows of
// the tile, 256 columns, twice, so that the epilogue overlaps the next tile's MMAs.
// 86 matrices of the 130M shapes, r = 256 (12 to 32 K blocks a tile): two parts 141 -> 107 us a product, one 88 -> 81.
// Where K is long the epilogue matters less and the pairs lose: with them a refresh of the 1.1B shapes took 52.0 ms, with two
// accumulators a CTA 51.3 although that still had a slower factorisation.  Tried for the projection of a step as well: 350M
// shapes 225 -> 199 us, 130M shapes 94 -> 99 us, the steps as they were to half a percent; not taken.
//
// Both CTAs of a pair walk the same tiles.  In each: warp 0 loads (the transaction counts of both go to the barriers of the first
// CTA), warps 2 to 9 drain the accumulators; warp 1 of the first issues the MMAs, whose commits free the stages and announce the
// accumulators in both.  No load is multicast.  Every wait is bounded (mbar_wait); the CTAs leave together.
#pragma once

#include "gemm_tcgen05.cuh"

namespace ngalore {

constexpr int kPairThreads = 64 + 32 * 8;
constexpr int kPairBN = 256;

template <int NB>
struct PairSmem {
  static constexpr int kABytes = kTcBM * kTcBK * 2;                   // 16 KB: this CTA's rows
  static constexpr int kBChunkBytes = 64 * kTcBK * 2;                 // 8 KB: 64 columns x 64 K rows
  static constexpr int kBBytes = 2 * kBChunkBytes;                    // this CTA's half of the columns, a part
  static constexpr int kStageBytes = kABytes + NB * kBBytes;
  static constexpr int kStages = NB == 1 ? 6 : 4;
  static constexpr int kEpiOffset = kStages * kStageBytes;
  static constexpr int kBarOffset = kEpiOffset + 8 * 32 * 32 * 4;
  static constexpr int kTotal = kBarOffset + 256 + 1024;
};
static_assert(PairSmem<1>::kTotal <= 232448 && PairSmem<2>::kTotal <= 232448, "shared memory budget of one CTA");

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}
// The address of a barrier in the first CTA of the pair.
__device__ __forceinline__ uint32_t first_cta(uint64_t* bar) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"(smem_u32(bar)));
  return a;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tma_load_pair(void* dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tc_mma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives at the barrier of the same place in both CTAs when the MMAs so far have ended.
__device__ __forceinline__ void tc_commit_pair(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(smem_u32(bar)), "h"(static_cast<uint16_t>(3)) : "memory");
}
// A wait for something that the other CTA has a part in (acquire at the scope of the cluster).
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  const uint32_t addr = smem_u32(bar);
  unsigned long long t0 = 0;
  for (unsigned it = 0;; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(addr), "r"(parity) : "memory");
    if (done) return true;
    if ((it & 63u) == 63u) {
      if (*abort_flag) return false;
      const unsigned long long now = global_timer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > kTcWaitLimitNs) break;
    }
  }
  *abort_flag = 1;
  return false;
}

// Columns of a tile as the MMA takes them (a multiple of 32, half of it from either CTA).
__device__ __forceinline__ int pair_columns(const TcTile& t) {
  const int rem = t.cols - t.n0;
  return rem >= kPairBN ? kPairBN : ((rem + 31) & ~31);
}

// NB: parts of B (as in tc_gemm_kernel; A has one).  A_MN: A is stored with its row index contiguous.
template <int NB, bool A_MN>
__global__ void __launch_bounds__(kPairThreads, 1)
tc_pair_kernel(const CUtensorMap* __restrict__ tmaps, const TcTile* __restrict__ tiles, const int* __restrict__ pair_first, Ctrl* ctrl,
               const TcProblem* __restrict__ probs) {
  using L = PairSmem<NB>;
  constexpr int STAGES = L::kStages;
  extern __shared__ unsigned char tc_smem_raw[];
  // (the same place in both CTAs: their windows of shared memory start alike)
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOffset);
  uint64_t* full_bar = bars;                     // [STAGES] (first CTA) both CTAs' operands landed
  uint64_t* empty_bar = bars + STAGES;           // [STAGES] operands consumed
  uint64_t* tfull_bar = bars + 2 * STAGES;       // [2] accumulators complete
  uint64_t* tempty_bar = bars + 2 * STAGES + 2;  // [2] (first CTA) accumulators drained, in both
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_rank());
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar + s, 1); mbar_init(empty_bar + s, 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(tfull_bar + b, 1); mbar_init(tempty_bar + b, 8); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const int pair = blockIdx.x >> 1;
  const int t_begin = pair_first[pair], t_end = pair_first[pair + 1];   // this pair's tiles

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      TcTile tile = tiles[t_begin];
      const CUtensorMap *mapA = tmaps + probs[tile.mat].map_a, *mapB = tmaps + probs[tile.mat].map_b;
      for (int t = t_begin; t < t_end && ok; ++t) {
        const TcTile next = tiles[min(t + 1, t_end - 1)];
        const int half = pair_columns(tile) >> 1, nchunks = (half + 63) >> 6;
        const int m0 = tile.m0 + rank * kTcBM, n0 = tile.n0 + rank * half;
        const uint32_t bytes = 2 * (L::kABytes + NB * nchunks * L::kBChunkBytes);   // of both CTAs
        for (int kb = 0; kb < tile.kblocks; ++kb) {
          if (!mbar_wait_cluster(empty_bar + stage, phase ^ 1u, abort_flag)) { ok = false; break; }
          unsigned char* sA = smem + stage * L::kStageBytes;
          const uint32_t bar = first_cta(full_bar + stage);
          if (rank == 0) mbar_expect_tx(full_bar + stage, bytes);
          const int k = tile.k0 + kb * kTcBK;
          if (A_MN) {
            tma_load_pair(sA, mapA, m0, k, bar);
            tma_load_pair(sA + L::kBChunkBytes, mapA, m0 + 64, k, bar);
          } else {
            tma_load_pair(sA, mapA, k, m0, bar);
          }
#pragma unroll
          for (int nb = 0; nb < NB; ++nb)
            for (int c = 0; c < nchunks; ++c)
              tma_load_pair(sA + L::kABytes + nb * L::kBBytes + c * L::kBChunkBytes, mapB + nb, n0 + c * 64, k, bar);
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
        if (next.mat != tile.mat) { mapA = tmaps + probs[next.mat].map_a; mapB = tmaps + probs[next.mat].map_b; }
        tile = next;
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (first CTA)
    if (lane == 0 && rank == 0) {
      int stage = 0;
      uint32_t phase = 0;
      int local = 0;
      bool ok = true;
      TcTile next = tiles[t_begin];
      for (int t = t_begin; t < t_end && ok; ++t, ++local) {
        const TcTile tile = next;
        next = tiles[min(t + 1, t_end - 1)];
        const int n_eff = pair_columns(tile);
        // M = 256: two tiles of the one-CTA instruction's 128 rows
        const uint32_t idesc = instr_desc(n_eff, A_MN, false) + (static_cast<uint32_t>(kTcBM >> 4) << 24);
        const int buf = local & 1;
        const uint32_t tphase = (local >> 1) & 1u;
        if (!mbar_wait_cluster(tempty_bar + buf, tphase ^ 1u, abort_flag)) { ok = false; break; }
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + buf * kPairBN;
        for (int kb = 0; kb < tile.kblocks; ++kb) {
          if (!mbar_wait_cluster(full_bar + stage, phase, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t aaddr = smem_u32(smem + stage * L::kStageBytes);
#pragma unroll
          for (int nb = 0; nb < NB; ++nb) {
            const uint32_t baddr = aaddr + L::kABytes + nb * L::kBBytes;
#pragma unroll
            for (int kk = 0; kk < kTcBK / 16; ++kk) {
              const uint64_t adesc = A_MN ? smem_desc(aaddr + kk * 2048, L::kBChunkBytes, 1024) : smem_desc(aaddr + kk * 32, 16, 1024);
              const uint64_t bdesc = smem_desc(baddr + kk * 2048, L::kBChunkBytes, 1024);
              tc_mma_pair(tmem_d, adesc, bdesc, idesc, (kb | nb | kk) != 0 ? 1u : 0u);
            }
          }
          tc_commit_pair(empty_bar + stage);
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
        if (ok) tc_commit_pair(tfull_bar + buf);
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2 .. 9): group g drains buffer g
    const int quarter = warp & 3;  // TMEM lanes 32 * quarter .. + 31 belong to this warp
    const int group = (warp - 2) >> 2;
    float* stg = reinterpret_cast<float*>(smem + L::kEpiOffset + (warp - 2) * 32 * 32 * 4);
    const int sub_row = lane >> 3, sub_col = (lane & 7) * 4;
    TcTile tile;
    if (t_begin + group < t_end) tile = tiles[t_begin + group];
    for (int local = group; t_begin + local < t_end; local += 2) {
      const TcTile next = tiles[min(t_begin + local + 2, t_end - 1)];
      const TcProblem pr = probs[tile.mat];
      const int n_eff = pair_columns(tile);
      const int buf = local & 1;
      const uint32_t tphase = (local >> 1) & 1u;
      const int row_base = tile.m0 + rank * kTcBM + quarter * 32;
      // (every lane polls; the warp goes on only if all of them saw the barrier complete)
      if (!__all_sync(0xffffffffu, mbar_wait_cluster(tfull_bar + buf, tphase, abort_flag))) break;
      tc_fence_after();
#pragma unroll
      for (int c0 = 0; c0 < kPairBN; c0 += 32) {
        if (c0 < n_eff) {
          uint32_t r[32];
          tc_ld32(tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + static_cast<uint32_t>(buf * kPairBN + c0), r);
          tc_wait_ld();
          if (c0 + 32 >= n_eff) {
            // all TMEM reads of this tile are done: hand the buffer back before the global traffic
            tc_fence_before();
            if (lane == 0) mbar_arrive_cluster(first_cta(tempty_bar + buf));
          }
#pragma unroll
          for (int j = 0; j < 8; ++j)
            *reinterpret_cast<float4*>(stg + lane * 32 + ((j ^ (lane & 7)) << 2)) =
                make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]), __uint_as_float(r[4 * j + 2]),
                            __uint_as_float(r[4 * j + 3]));
          __syncwarp();
          const int col = tile.n0 + c0 + sub_col;
          if (col < pr.out_cols) {
#pragma unroll
            for (int it = 0; it < 8; ++it) {
              const int rr = it * 4 + sub_row;
              const int row = row_base + rr;
              if (row < pr.out_rows) {
                const float4 acc = *reinterpret_cast<const float4*>(stg + rr * 32 + (((lane ^ rr) & 7) << 2));
                store_result<TC_EPI_STORE>(acc, row, col, pr.out, pr.ld_out, pr.out_hi, pr.out_lo, pr.ld16, tile.atomic);
              }
            }
          }
          __syncwarp();
        }
      }
      tile = next;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // a wait ran out: give bulk copies that may still be in flight time to land before the CTAs retire
    for (int i = 0; i < 200; ++i) __nanosleep(1000);
    if (threadIdx.x == 0) atomicExch(&ctrl->timeout_flag, 1);
  }
  cluster_sync();   // (neither goes while the other may still signal it or multiply from its shared memory)
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

template <int NB, bool A_MN>
inline bool tc_pair_set_smem() {
  return cudaFuncSetAttribute(tc_pair_kernel<NB, A_MN>, cudaFuncAttributeMaxDynamicSharedMemorySize, PairSmem<NB>::kTotal) == cudaSuccess;
}

// Launch-time setup of the kernels above: the number of pairs that run side by side on this device (0: none).  The tiles are handed out
// beforehand: a pair that had to wait for another to end would double the time of the launch.  (All four have an SM to themselves, so
// one of them is asked about.  A call that fails here means no pairs and nothing else: its error is not left for the next launch.)
inline int tc_pair_init() {
  if (!tc_pair_set_smem<1, false>() || !tc_pair_set_smem<1, true>() || !tc_pair_set_smem<2, false>() || !tc_pair_set_smem<2, true>()) {
    cudaGetLastError();
    return 0;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = 2;
  cfg.blockDim = kPairThreads;
  cfg.dynamicSmemBytes = PairSmem<2>::kTotal;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 2; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int pairs = 0;
  if (cudaOccupancyMaxActiveClusters(&pairs, tc_pair_kernel<2, true>, &cfg) == cudaSuccess) return pairs;
  cudaGetLastError();
  return 0;
}

template <int NB, bool A_MN>
inline cudaError_t tc_pair_launch(int pairs, cudaStream_t stream, const CUtensorMap* maps, const TcTile* tiles, const int* first, Ctrl* ctrl,
                                  const TcProblem* probs) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = 2 * pairs;
  cfg.blockDim = kPairThreads;
  cfg.dynamicSmemBytes = PairSmem<NB>::kTotal;
  cfg.stream = stream;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 2; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, tc_pair_kernel<NB, A_MN>, maps, tiles, first, ctrl, probs);
}

}  // namespace ngalore
