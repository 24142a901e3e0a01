// One persistent kernel for the whole history phase of a step: the Gram row of every matrix,
// the s x s solves, and the natural-gradient combination with the Adam moments (Sec. 2.4, 2.2).
//
// Structure: one CTA per SM; a producer warp streams the history (and m, v) through a ring of
// shared-memory stages with bulk asynchronous copies (cp.async.bulk + mbarrier), eight to sixteen consumer
// warps compute from shared memory, a finishing warp turns the partial sums of a Gram tile into its partial row
// and, after a matrix's last one, solves its s x s system while the consumers go on with the next item.  The producer runs ahead of the consumers across tile and
// matrix boundaries, so the SM always has several stages of loads in flight.
//
// Work items (Gram tiles and combination tiles of all matrices) are fetched in order from a global
// counter by the producer.  Gram items never wait; the finishing warp of the CTA that has a matrix's last Gram
// tile solves its s x s system and publishes the weights; the consumers of a combination item wait
// (bounded) for that flag.  Every item a combination item depends on sits earlier in the list and
// has been fetched by a CTA that consumes its items in order, so the kernel cannot deadlock.
// All Gram items precede all combination items, so the wait is short except at the very end of the Gram items.
#pragma once

#include <vector>

#include "../../include/ngalore.h"
#include "common.cuh"
#include "gemm_tcgen05.cuh"  // mbarrier wrappers
#include "kernels_stream.cuh"

namespace ngalore {

struct FusedItem {
  int mat;
  int local;
  int kind;  // 0 = Gram tile, 1 = combination tile
  int pad;
};

struct FusedPlan {
  FusedItem* d_items = nullptr;
  int n_items = 0;
  int grid = 0;
  bool hist16 = false;  // the state keeps its history ring in bf16
  bool mom16 = false;   // the state keeps its moments in bf16
};

constexpr long long kSpinLimit = 4000000;  // polls of ~100 ns each before a flag wait is abandoned

struct StageMeta {
  int mat, kind, local, first, last, count;
  int cur, c;  // ring position and number of valid slots of this step (the same for every stage of a launch)
  long long e0;
};

// Stage layout.  fp32 history: SMAX slots of CE floats, then m, then v.  bf16 history (HIST16): SMAX slots of CE
// bf16 values (the current slot's place stays unused), then the current gradient, m and v as floats.
// MOM16: the moments are stored as bf16 (half the bytes of their stages).
template <int SMAX, bool HIST16, bool MOM16 = false>
struct FusedCfg {
  // Elements per stage and slot.  The bf16 history costs more instructions per byte (conversion, two Gram rows),
  // and the per-stage bookkeeping of a consumer thread weighs as much as its arithmetic on two elements, so up to sixteen slots its
  // threads take four, and its stages are as long as three of them fit: with two, a stage of which is worked on, the SM has too little
  // under way.  350M shapes, s = 16, bf16 moments: two stages of 2048 elements 950 us, three of 1792 (14 warps) 805.  (Beyond
  // sixteen slots: five stages of 512 elements, two a thread.)
  static constexpr int CE = !HIST16 ? (SMAX <= 16 ? 1024 : 512) : (SMAX <= 8 ? 2048 : (SMAX <= 16 ? (MOM16 ? 1792 : 1536) : 512));
  // Consumer threads: a warp issues the 100 to 250 instructions of a stage one after another, so eight warps take 1 us for it
  // whatever it holds.  The bf16 history costs more instructions per byte (conversion, two Gram rows), and a stage of
  // eight slots at most holds as little as 12 KB (history and moments of s = 0) to 40 KB, which arrive in 0.3 to 0.9 us; they get
  // sixteen warps.  Measured, eight against sixteen, stream phase: s = 5, 11 M elements, 154 -> 125 us; s = 0 on the 60M
  // shapes 39 -> 35; s = 8 on them 88 either way, as sixteen slots (1.1B shapes, 4.16 ms), which stay with eight warps.  So do bf16
  // moments beside an fp32 history: two elements a thread draw a block of the generator for two of its four words (130M shapes,
  // s = 5 and 8, 302 -> 308 and 353 -> 361 us; 350M shapes, s = 8, 870 -> 894; s = 0 no difference).
  static constexpr int kConsumers = HIST16 && SMAX <= 16 ? CE / 4 : (SMAX <= 8 && !MOM16 ? 512 : 256);
  static constexpr int kThreads = kConsumers + 64;  // and the producer and the finishing warp
  static constexpr int kHistBytes = SMAX * CE * (HIST16 ? 2 : 4);
  static constexpr int kCurOff = kHistBytes;                          // HIST16: fp32 gradient of this step
  static constexpr int kMOff = kHistBytes + (HIST16 ? CE * 4 : 0);
  static constexpr int kVOff = kMOff + CE * (MOM16 ? 2 : 4);
  static constexpr int kStageBytes = kVOff + CE * (MOM16 ? 2 : 4);
  static constexpr int kStages = HIST16 ? (SMAX <= 16 ? 3 : 5) : (SMAX <= 8 ? 5 : 3);
  static constexpr int kBase = kStages * kStageBytes;
  static constexpr int kFullOff = kBase, kEmptyOff = kBase + 64, kMetaOff = kBase + 128, kFlagOff = kBase + 512;
  static constexpr int kMeetOff = kBase + 640, kRedBarOff = kBase + 768, kRedMetaOff = kBase + 800, kRedOff = kBase + 896;
  static constexpr int kRows = HIST16 ? 2 : 1;                  // Gram rows per tile
  static constexpr int kRedDoubles = (kConsumers / 32) * SMAX;  // one Gram row per consumer warp
  static constexpr int kTotal = kRedOff + 2 * kRows * kRedDoubles * 8;   // (two tiles in flight to the finishing warp)
  static_assert(kStages * sizeof(StageMeta) <= 384, "stage metadata overflows its slot");
  static_assert(kTotal <= 232448, "shared memory budget of one CTA exceeded");
};

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
// Sums of S values over the 32 lanes of a warp: afterwards lane l holds the sum of value l / (32 / S).  S - 1 exchanges
// instead of the 5 S of one butterfly per value: each step halves the values a lane is responsible for.
template <int S>
__device__ __forceinline__ double warp_sums(double (&v)[S]) {
  const int lane = threadIdx.x & 31;
  int n = S, off = 16;
#pragma unroll
  for (int step = 0; step < 5; ++step, off >>= 1) {
    if (n > 1) {
      n >>= 1;
      const bool upper = (lane & off) != 0;
#pragma unroll
      for (int i = 0; i < S / 2; ++i) {
        if (i < n) {
          const double mine = upper ? v[i + n] : v[i], other = upper ? v[i] : v[i + n];
          v[i] = mine + __shfl_xor_sync(0xffffffffu, other, off);
        }
      }
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
    }
  }
  return v[0];
}

// A wait of a whole warp: all lanes see the barrier complete, or all of them give up (lanes that part here could not come
// together again in what follows).  The vote costs the bf16 history 2 % of the kernel (350M shapes, s = 16: 887 -> 907 us),
// the fp32 history half a percent at most; put off to the release of the stage, or with one lane polling for all, it costs more.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag));
}

// What the finishing warp needs to know about a finished Gram tile (mat < 0: the CTA has no more).
struct RedMeta {
  int mat, local, cur, c;
};

template <int THREADS>
__device__ __forceinline__ void consumer_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
}

__device__ __forceinline__ float bf16_bits_to_float(uint32_t bits16) { return __uint_as_float(bits16 << 16); }
__device__ __forceinline__ uint32_t float_to_bf16_bits(float x) {
  return static_cast<uint32_t>(__bfloat16_as_ushort(__float2bfloat16_rn(x)));
}

// Two floats in a 64-bit register, and the packed multiply-add on them.
__device__ __forceinline__ uint64_t pack_pair(float lo, float hi) {
  uint64_t p;
  asm("mov.b64 %0, {%1, %2};" : "=l"(p) : "f"(lo), "f"(hi));
  return p;
}
__device__ __forceinline__ void unpack_pair(uint64_t p, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p)); }
__device__ __forceinline__ uint64_t widen_pair(uint32_t bf16x2) { return pack_pair(__uint_as_float(bf16x2 << 16), __uint_as_float(bf16x2 & 0xFFFF0000u)); }
__device__ __forceinline__ uint64_t fma_pair(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// HIST16: the ring holds bf16 values; the gradient of the current step is read in fp32 from its own buffer
// (MatDesc::H) and its bf16 rounding is written into ring slot `cur` by the combination pass.  The Gram pass
// then also recomputes the row of the slot that was current one step ago, now that it is a rounded value, so
// that Kraw stays the Gram matrix of exactly the values the combination uses.
// MOM16: the moments are read and written as bf16: m rounded to nearest, v rounded stochastically (one step changes
// v by a relative 1 - beta2, less than half a bf16 unit, so rounding to nearest would freeze it) with bits from a
// counter-based generator keyed by (element group, matrix, step index); the direction u of the step comes from
// the unrounded values.
template <int SMAX, bool HIST16, bool MOM16>
__global__ void __launch_bounds__((FusedCfg<SMAX, HIST16, MOM16>::kThreads), 1)
fused_stream_kernel(const MatDesc* __restrict__ mats, const FusedItem* __restrict__ items, int n_items, Ctrl* ctrl,
                    const Hyper* __restrict__ hyper) {
  using C = FusedCfg<SMAX, HIST16, MOM16>;
  constexpr int CE = C::CE;
  constexpr int kConsumerThreads = C::kConsumers;
  constexpr int kWarps = kConsumerThreads / 32;
  constexpr int VEC = CE / kConsumerThreads;  // 4 or 2 elements per thread and stage
  static_assert(VEC == 2 || VEC == 4, "a thread handles two or four elements of a stage");
  extern __shared__ __align__(128) unsigned char fs_smem[];
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(fs_smem + C::kFullOff);
  uint64_t* empty_bar = reinterpret_cast<uint64_t*>(fs_smem + C::kEmptyOff);
  StageMeta* meta = reinterpret_cast<StageMeta*>(fs_smem + C::kMetaOff);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(fs_smem + C::kFlagOff);
  volatile int* s_flag = abort_flag + 1;                                        // [2] 1: the weights of a combination item came
  uint64_t* meet_bar = reinterpret_cast<uint64_t*>(fs_smem + C::kMeetOff);      // all consumer warps
  uint64_t* red_full = reinterpret_cast<uint64_t*>(fs_smem + C::kRedBarOff);   // [2] all consumer warps have left their sums
  uint64_t* red_empty = red_full + 2;                                           // [2] the finishing warp has taken them
  RedMeta* red_meta = reinterpret_cast<RedMeta*>(fs_smem + C::kRedMetaOff);     // [2]
  double* red = reinterpret_cast<double*>(fs_smem + C::kRedOff);                // [2][rows][warps][SMAX]

  const int tid = threadIdx.x;
  if (tid == 0) {
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(full_bar + s, 1);
      mbar_init(empty_bar + s, kConsumerThreads / 32);
    }
    for (int b = 0; b < 2; ++b) { mbar_init(red_full + b, kWarps); mbar_init(red_empty + b, 1); }
    mbar_init(meet_bar, kWarps);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  // (The tables are laid out for good: the item that this CTA will probably claim first, and its matrix, come to the SM ahead of
  // the wait for the kernel before.  It is claimed like the others all the same: an item that belonged to a CTA which another kernel
  // keeps from starting could be waited for by that kernel's neighbours for good.)
  if (tid == kConsumerThreads && static_cast<int>(blockIdx.x) < n_items) {
    const MatDesc& d0 = mats[items[blockIdx.x].mat];
    asm volatile("" ::"l"(d0.H), "l"(d0.m), "r"(d0.te), "r"(mats[0].s));
  }
  pdl_begin();
  const int tag = ctrl->epoch + 1;

  if (tid >= kConsumerThreads + 32) {
    // ------------------------------------------------------------------ finishing warp
    const int lane = tid & 31;
    const double lambda = hyper->lambda;
    for (unsigned int n = 0;; ++n) {
      const int buf = n & 1;
      if (!mbar_wait_warp(red_full + buf, (n >> 1) & 1u, abort_flag)) break;
      const RedMeta mt = red_meta[buf];
      double part[C::kRows];
#pragma unroll
      for (int r = 0; r < C::kRows; ++r) {
        part[r] = 0.0;
        if (lane < SMAX) {
          const double* src = red + (buf * C::kRows + r) * C::kRedDoubles + lane;
          double t0 = 0.0, t1 = 0.0;
#pragma unroll
          for (int w = 0; w < kWarps; w += 2) { t0 += src[w * SMAX]; t1 += src[(w + 1) * SMAX]; }
          part[r] = t0 + t1;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(red_empty + buf);
      if (mt.mat < 0) break;
      const MatDesc& d = mats[mt.mat];
      const int cur = mt.cur, c = mt.c;
      // per-tile partial rows: [tile][s] (fp32 history) or [tile][2][s] (HIST16: row of `cur`, row of `prev`)
      if (d.ntiles > 1) {
        int last = 0;
        if (lane < d.s) {
#pragma unroll
          for (int r = 0; r < C::kRows; ++r) __stcg(d.gpart + (static_cast<long long>(mt.local) * C::kRows + r) * d.s + lane, part[r]);
          __threadfence();
        }
        __syncwarp();
        if (lane == 0) last = atomicAdd(d.gram_done, 1) == d.ntiles - 1 ? 1 : 0;
        if (!__shfl_sync(0xffffffffu, last, 0)) continue;
        __threadfence();
      }
      // the matrix's last tile
      if (d.ntiles > 1) {
#pragma unroll
        for (int r = 0; r < C::kRows; ++r) part[r] = gram_row_sum<SMAX>(d, lane, c, C::kRows, r);
      }
      const bool two = HIST16 && c >= 2;
      solve_matrix<SMAX>(d, cur, c, lambda, lane < c ? part[0] : 0.0, two, two ? (cur == 0 ? d.s : cur) - 1 : 0, part[C::kRows - 1]);
      __threadfence();
      __syncwarp();
      if (lane == 0) {
        *d.gram_done = 0;
        __threadfence();
        if (ctrl->debug_withhold != mt.mat + 1) atomicExch(d.w_ready, tag);
      }
    }
  } else if (tid >= kConsumerThreads) {
    // ------------------------------------------------------------------ producer warp
    // Lane 0 claims items and arms the barriers; every lane issues the bulk copy of "its" slot (lane j copies
    // history slot j, the next two lanes m and v), so a stage's copies are issued in parallel.  The next item is
    // claimed and its descriptor fetched while the stages of the current one go out, one round trip to memory per
    // stage: three round trips in a row between two items cost more than streaming 4096 elements of eight slots.
    const int lane = tid & 31;
    const int s_all = mats[0].s;                       // (the same for every matrix, and so are ring position and count)
    const int c = ring_count(ctrl, s_all), cur_slot = ring_cur(ctrl, s_all);
    struct Source {
      int mat, kind, local;
      long long e0, e1;
      const unsigned char* src[2];                     // this lane's copies: number lane, and lane + 32 where there is one
    };
    // copy number k of an item: history slot k, then m and v; its place in a stage and bytes per element
    auto place = [&](int k) {
      if (k < c) return !HIST16 ? k * CE * 4 : (k == cur_slot ? C::kCurOff : k * CE * 2);
      return k == c ? C::kMOff : C::kVOff;
    };
    auto width = [&](int k) { return k < c ? (HIST16 && k != cur_slot ? 2 : 4) : (MOM16 ? 2 : 4); };
    auto describe = [&](const FusedItem& item, Source& o) {
      const MatDesc& d = mats[item.mat];
      o.mat = item.mat; o.kind = item.kind; o.local = item.local;
      o.e0 = static_cast<long long>(item.local) * d.te;
      o.e1 = (o.e0 + d.te < d.rn) ? o.e0 + d.te : d.rn;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int k = lane + 32 * q;
        const void* base = nullptr;
        if (k < c) base = !HIST16 ? static_cast<const void*>(d.H + static_cast<long long>(k) * d.rn)
                                  : (k == cur_slot ? static_cast<const void*>(d.H) : static_cast<const void*>(d.H16 + static_cast<long long>(k) * d.rn));
        else if (k == c) base = MOM16 ? static_cast<const void*>(d.m16) : static_cast<const void*>(d.m);
        else if (k == c + 1) base = MOM16 ? static_cast<const void*>(d.v16) : static_cast<const void*>(d.v);
        o.src[q] = static_cast<const unsigned char*>(base);
      }
    };
    int stage = 0;
    uint32_t phase = 0;
    int it = 0;
    FusedItem item{};
    Source now{}, next{};
    if (lane == 0) it = static_cast<int>(atomicAdd(&ctrl->work_counter, 1u));
    it = __shfl_sync(0xffffffffu, it, 0);
    if (it < n_items) { item = items[it]; describe(item, now); }
    while (true) {
      if (it >= n_items) {
        if (lane == 0 && mbar_wait(empty_bar + stage, phase ^ 1u, abort_flag)) {
          meta[stage].kind = -1;
          mbar_arrive(full_bar + stage);
        }
        break;
      }
      const int ncopies = c + (now.kind == 1 ? 2 : 0);
      int step = 0;   // how far the next item is known: 0 claimed, 1 fetched, 2 described
      auto look_ahead = [&]() {
        if (step == 0) {
          if (lane == 0) it = static_cast<int>(atomicAdd(&ctrl->work_counter, 1u));
        } else if (step == 1) {
          it = __shfl_sync(0xffffffffu, it, 0);
          if (it < n_items) item = items[it];
        } else if (step == 2) {
          if (it < n_items) describe(item, next);
        }
        ++step;
      };
      bool ok = true;
      for (long long e = now.e0; e < now.e1; e += CE) {
        const int cnt = (now.e1 - e < CE) ? static_cast<int>(now.e1 - e) : CE;
        int good = 1;
        if (lane == 0) good = mbar_wait(empty_bar + stage, phase ^ 1u, abort_flag) ? 1 : 0;
        good = __shfl_sync(0xffffffffu, good, 0);
        if (!good) { ok = false; break; }
        unsigned char* sb = fs_smem + stage * C::kStageBytes;
        const uint32_t bytes = static_cast<uint32_t>(cnt) * 4u;
        if (lane == 0) {
          StageMeta mt;
          mt.mat = now.mat; mt.kind = now.kind; mt.local = now.local;
          mt.first = (e == now.e0) ? 1 : 0; mt.last = (e + CE >= now.e1) ? 1 : 0; mt.count = cnt; mt.e0 = e;
          mt.cur = cur_slot; mt.c = c;
          meta[stage] = mt;
          const uint32_t hist_bytes = HIST16 ? bytes * static_cast<uint32_t>(c) - (bytes / 2) * static_cast<uint32_t>(c - 1)
                                             : bytes * static_cast<uint32_t>(c);
          const uint32_t mom_bytes = now.kind == 1 ? (MOM16 ? bytes : 2u * bytes) : 0u;
          mbar_expect_tx(full_bar + stage, hist_bytes + mom_bytes);
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int k = lane + 32 * q;
          if (k < ncopies) {
            const int w = width(k);
            bulk_load(sb + place(k), now.src[q] + e * w, static_cast<uint32_t>(cnt * w), full_bar + stage);
          }
        }
        if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
        look_ahead();
      }
      if (!ok) break;
      while (step < 3) look_ahead();
      now = next;
    }
  } else {
    // ------------------------------------------------------------------ consumers (8 to 16 warps)
    // One loop over the stages of an item for either kind, so that the sums of a Gram tile and the weights of a
    // combination tile do not both occupy registers.
    const int warp = tid >> 5, lane = tid & 31;
    const Hyper hp = *hyper;
    const int idx = tid * VEC;     // this thread's elements of a stage
    int stage = 0;
    uint32_t phase = 0;
    unsigned int tiles_done = 0;   // Gram tiles handed to the finishing warp
    unsigned int combined = 0;     // combination items whose weights have been waited for
    // Tell the finishing warp that the CTA has no more of them (every Gram item is ahead of every combination item).  That
    // is done as soon as it is known, so that none of its waits spans more than a Gram tile: a wait is given up after a
    // time, and the combination items of a CTA may take longer than that without anything being wrong.
    bool gram_open = true;
    auto close_gram = [&]() {
      if (tid == 0) red_meta[tiles_done & 1].mat = -1;
      __syncwarp();
      if (lane == 0) mbar_arrive(red_full + (tiles_done & 1));
      gram_open = false;
    };
    if (HIST16) {
      // the current slot's place in a stage stays zero for the whole launch: its gradient takes part in fp32 instead
      const int cur = ring_cur(ctrl, mats[0].s);
      for (int x = 0; x < C::kStages; ++x)
        for (int i = tid; i < CE / 2; i += kConsumerThreads)
          reinterpret_cast<uint32_t*>(fs_smem + x * C::kStageBytes + cur * CE * 2)[i] = 0u;
      consumer_sync<kConsumerThreads>();
    }
    // hand the stage back and go on to the next one of the item
    auto release = [&]() {
      __syncwarp();
      if (lane == 0) mbar_arrive(empty_bar + stage);
      if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
    };
    // this thread's elements of fp32 slot j, of bf16 slot j (as pairs), of the fp32 gradient of the step, of a moment
    auto load32 = [&](int j, float (&h)[VEC]) {
      const float* q = reinterpret_cast<const float*>(fs_smem + stage * C::kStageBytes) + j * CE + idx;
#pragma unroll
      for (int x = 0; x < VEC; ++x) h[x] = q[x];
    };
    auto load16 = [&](int j, uint64_t (&h)[VEC / 2]) {
      const uint32_t* q = reinterpret_cast<const uint32_t*>(fs_smem + stage * C::kStageBytes + (j * CE + idx) * 2);
#pragma unroll
      for (int x = 0; x < VEC / 2; ++x) h[x] = widen_pair(q[x]);
    };
    auto load_current = [&](float (&h)[VEC]) {
      const float* q = reinterpret_cast<const float*>(fs_smem + stage * C::kStageBytes + C::kCurOff) + idx;
#pragma unroll
      for (int x = 0; x < VEC; ++x) h[x] = q[x];
    };
    auto load_moment = [&](int off, float (&h)[VEC]) {
      if (!MOM16) {
        const float* q = reinterpret_cast<const float*>(fs_smem + stage * C::kStageBytes + off) + idx;
#pragma unroll
        for (int x = 0; x < VEC; ++x) h[x] = q[x];
      } else {
        const uint32_t* q = reinterpret_cast<const uint32_t*>(fs_smem + stage * C::kStageBytes + off + idx * 2);
#pragma unroll
        for (int x = 0; x < VEC; x += 2) {
          const uint32_t pair = q[x >> 1];
          h[x] = bf16_bits_to_float(pair & 0xFFFFu);
          h[x + 1] = bf16_bits_to_float(pair >> 16);
        }
      }
    };
    while (true) {
      if (!mbar_wait_warp(full_bar + stage, phase, abort_flag)) break;
      StageMeta mt = meta[stage];
      if (mt.kind < 0) {   // no more items
        if (gram_open && mbar_wait_warp(red_empty + (tiles_done & 1), ((tiles_done >> 1) & 1u) ^ 1u, abort_flag)) close_gram();
        break;
      }
      const int cur = mt.cur, c = mt.c;
      bool alive = true;
      if (mt.kind == 0) {
        // ---- Gram tile
        const int buf = tiles_done & 1;
        // this warp's sums of row r over its lanes, into the buffer of the finishing warp
        auto hand_over = [&](int r, double (&v)[SMAX]) {
          const double t = warp_sums<SMAX>(v);
          if ((lane & (32 / SMAX - 1)) == 0) red[((buf * C::kRows + r) * kWarps + warp) * SMAX + lane / (32 / SMAX)] = t;
        };
        if constexpr (!HIST16) {
          float acc[SMAX];
#pragma unroll
          for (int j = 0; j < SMAX; ++j) acc[j] = 0.f;
          while (true) {
            if (idx < mt.count) {
              float x[VEC];
              load32(cur, x);
#pragma unroll
              for (int j = 0; j < SMAX; ++j) {
                if (j >= c) break;
                float h[VEC];
                load32(j, h);
                float t = 0.f;
#pragma unroll
                for (int q = 0; q < VEC; ++q) t += x[q] * h[q];
                acc[j] += t;
              }
            }
            const bool last = mt.last != 0;
            release();
            if (last) break;
            if (!mbar_wait_warp(full_bar + stage, phase, abort_flag)) { alive = false; break; }
            mt = meta[stage];
          }
          if (!alive || !mbar_wait_warp(red_empty + buf, ((tiles_done >> 1) & 1u) ^ 1u, abort_flag)) break;
          double v[SMAX];
#pragma unroll
          for (int j = 0; j < SMAX; ++j) v[j] = static_cast<double>(acc[j]);
          hand_over(0, v);
        } else {
          // rows of `cur` and of the slot that was current one step ago, in pairs: the inner loop is bound by the
          // instructions it issues, and the packed multiply-add halves those
          uint64_t acc[SMAX], acc2[SMAX];
          // The product of the fp32 gradient with itself, in the operations and the order of the other products: a
          // gradient that repeats bit for bit has to give an exactly singular Gram matrix, not one that a rounding makes
          // indefinite.
          uint64_t axx = 0ull;
#pragma unroll
          for (int j = 0; j < SMAX; ++j) acc[j] = acc2[j] = 0ull;
          const int prev = c >= 2 ? (cur == 0 ? mats[mt.mat].s : cur) - 1 : cur;
          while (true) {
            if (idx < mt.count) {
              float x[VEC];
              uint64_t xx[VEC / 2], xp[VEC / 2];
              load_current(x);
              load16(prev, xp);            // (a single gradient: the zeros of its own place)
#pragma unroll
              for (int q = 0; q < VEC / 2; ++q) {
                xx[q] = pack_pair(x[2 * q], x[2 * q + 1]);
                axx = fma_pair(xx[q], xx[q], axx);
              }
#pragma unroll
              for (int j = 0; j < SMAX; ++j) {
                if (j >= c) break;
                uint64_t h[VEC / 2];
                load16(j, h);
#pragma unroll
                for (int q = 0; q < VEC / 2; ++q) {
                  acc[j] = fma_pair(xx[q], h[q], acc[j]);
                  acc2[j] = fma_pair(xp[q], h[q], acc2[j]);
                }
              }
            }
            const bool last = mt.last != 0;
            release();
            if (last) break;
            if (!mbar_wait_warp(full_bar + stage, phase, abort_flag)) { alive = false; break; }
            mt = meta[stage];
          }
          if (!alive || !mbar_wait_warp(red_empty + buf, ((tiles_done >> 1) & 1u) ^ 1u, abort_flag)) break;
          {
            double v[SMAX];
#pragma unroll
            for (int j = 0; j < SMAX; ++j) {
              float s0, s1;
              unpack_pair(j == cur ? axx : acc[j], s0, s1);
              v[j] = static_cast<double>(s0 + s1);
            }
            hand_over(0, v);
          }
          __syncwarp();
          {
            double v[SMAX];
#pragma unroll
            for (int j = 0; j < SMAX; ++j) {
              float s0, s1;
              unpack_pair(acc2[j], s0, s1);
              v[j] = static_cast<double>(s0 + s1);   // (entry `cur` is not used: row `cur` has it)
            }
            hand_over(C::kRows - 1, v);
          }
        }
        ++tiles_done;
        if (tid == 0) red_meta[buf] = RedMeta{mt.mat, mt.local, cur, c};
        __syncwarp();
        if (lane == 0) mbar_arrive(red_full + buf);
      } else {
        // ---- combination tile
        // (where the finishing warp still has two tiles to take, the next item will do)
        if (gram_open && __all_sync(0xffffffffu, mbar_test(red_empty + (tiles_done & 1), ((tiles_done >> 1) & 1u) ^ 1u))) close_gram();
        const MatDesc& d = mats[mt.mat];
        bool item_ok = true;
        if (d.s > 0) {
          // One thread waits for the weights; the others meet it at a barrier that they leave, like every other wait, when
          // one of the CTA's warps has given up.  (A bar.sync would wait for good for a warp that is gone.)  What it found
          // goes through one of two places in turn: nobody is more than one item ahead.
          if (tid == 0) {
            const volatile int* flag = d.w_ready;
            const long long limit = ctrl->spin_limit > 0 ? ctrl->spin_limit : kSpinLimit;
            long long spins = 0;
            int ok = 1;
            while (*flag != tag) {
              if (++spins > limit) { ok = 0; break; }
              __nanosleep(100);
            }
            if (!ok) {
              // The weights never came: this matrix takes no update in this step (the back-projection skips it)
              // and says why.  Tiles of it that other CTAs did combine have advanced their part of m and v.
              atomicExch(&ctrl->timeout_flag, 1);
              atomicExch(d.step_bad, 1);
              atomicCAS(d.status, 0, 8 /* NGALORE_ERR_TIMEOUT */);
            }
            s_flag[combined & 1] = ok;
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(meet_bar);
          if (!mbar_wait_warp(meet_bar, combined & 1, abort_flag)) break;
          item_ok = s_flag[combined & 1] != 0;
          ++combined;
          __threadfence();
        }
        const float my_w = __ldcg(d.wsol + lane);
        const bool item_bad = __ldcg(d.step_bad) != 0;
        float *const it_m = d.m, *const it_v = d.v, *const it_cur = current_gradient(d, cur);
        __half* const it_u = d.u16;
        uint16_t *const it_m16 = d.m16, *const it_v16 = d.v16;
        uint16_t* const it_h16 = HIST16 ? d.H16 + static_cast<long long>(cur) * d.rn : nullptr;
        const unsigned int it_mat = static_cast<unsigned int>(d.index), it_step = static_cast<unsigned int>(ctrl->k);
        float w[SMAX];
#pragma unroll
        for (int j = 0; j < SMAX; ++j) w[j] = __shfl_sync(0xffffffffu, my_w, j);
        const float wc = HIST16 ? __shfl_sync(0xffffffffu, my_w, cur) : 0.f;
        while (true) {
          if (item_ok && idx < mt.count) {
            const long long e = mt.e0 + idx;
            if (item_bad) {
              // The poisoned slot becomes a zero gradient; m, v are left alone and the update is zero.
#pragma unroll
              for (int q = 0; q < VEC; ++q) {
                it_cur[e + q] = 0.f;
                it_u[e + q] = __float2half_rn(0.f);
                if (HIST16) it_h16[e + q] = 0;
              }
            } else {
              float n[VEC], mm[VEC], vv[VEC], uu[VEC];
              if constexpr (!HIST16) {
#pragma unroll
                for (int q = 0; q < VEC; ++q) n[q] = 0.f;
#pragma unroll
                for (int j = 0; j < SMAX; ++j) {
                  if (j >= c) break;
                  float h[VEC];
                  load32(j, h);
#pragma unroll
                  for (int q = 0; q < VEC; ++q) n[q] = fmaf(w[j], h[q], n[q]);
                }
              } else {
                float x[VEC];
                load_current(x);
                uint64_t np[VEC / 2];
#pragma unroll
                for (int q = 0; q < VEC / 2; ++q) np[q] = pack_pair(wc * x[2 * q], wc * x[2 * q + 1]);
#pragma unroll
                for (int j = 0; j < SMAX; ++j) {
                  if (j >= c) break;
                  uint64_t h[VEC / 2];
                  load16(j, h);
                  const uint64_t ww = pack_pair(w[j], w[j]);
#pragma unroll
                  for (int q = 0; q < VEC / 2; ++q) np[q] = fma_pair(ww, h[q], np[q]);
                }
#pragma unroll
                for (int q = 0; q < VEC / 2; ++q) unpack_pair(np[q], n[2 * q], n[2 * q + 1]);
                // from the next step on this gradient is an old one: store its bf16 rounding in the ring
                uint32_t* dst = reinterpret_cast<uint32_t*>(it_h16 + e);
#pragma unroll
                for (int q = 0; q < VEC; q += 2) dst[q >> 1] = float_to_bf16_bits(x[q]) | (float_to_bf16_bits(x[q + 1]) << 16);
              }
              load_moment(C::kMOff, mm);
              load_moment(C::kVOff, vv);
#pragma unroll
              for (int q = 0; q < VEC; ++q) {
                mm[q] = hp.beta1 * mm[q] + (1.f - hp.beta1) * n[q];
                vv[q] = hp.beta2 * vv[q] + (1.f - hp.beta2) * n[q] * n[q];
                uu[q] = mm[q] / sqrtf(vv[q] + hp.eps);
              }
              if (MOM16) {
                // elements 4 g .. 4 g + 3 take the upper halves of the four words of one generator call
                uint32_t* dm = reinterpret_cast<uint32_t*>(it_m16 + e);
                uint32_t* dv = reinterpret_cast<uint32_t*>(it_v16 + e);
#pragma unroll
                for (int q0 = 0; q0 < VEC; q0 += 4) {
                  const unsigned long long grp = static_cast<unsigned long long>(e + q0) >> 2;
                  const uint4 rnd = philox4x32_10(make_uint4(static_cast<unsigned int>(grp), static_cast<unsigned int>(grp >> 32),
                                                             it_mat, it_step), hp.seed_lo, hp.seed_hi);
                  const unsigned int rb[4] = {rnd.x >> 16, rnd.y >> 16, rnd.z >> 16, rnd.w >> 16};
#pragma unroll
                  for (int q = q0; q < q0 + 4 && q < VEC; q += 2) {
                    // (VEC = 2: e is a multiple of 2, the pair is words 0, 1 or words 2, 3 of its group)
                    const int w0 = VEC == 2 ? static_cast<int>(e & 2) : q - q0;
                    dm[q >> 1] = float_to_bf16_bits(mm[q]) | (float_to_bf16_bits(mm[q + 1]) << 16);
                    dv[q >> 1] = stochastic_bf16_bits(vv[q], rb[w0]) | (stochastic_bf16_bits(vv[q + 1], rb[w0 + 1]) << 16);
                  }
                }
                if (VEC == 4) *reinterpret_cast<uint2*>(it_u + e) = pack_f16x4(uu[0], uu[1], uu[2 % VEC], uu[3 % VEC]);
                else *reinterpret_cast<uint32_t*>(it_u + e) = pack_f16x4(uu[0], uu[1], 0.f, 0.f).x;
              } else if (VEC == 4) {
                *reinterpret_cast<float4*>(it_m + e) = make_float4(mm[0], mm[1], mm[2 % VEC], mm[3 % VEC]);
                *reinterpret_cast<float4*>(it_v + e) = make_float4(vv[0], vv[1], vv[2 % VEC], vv[3 % VEC]);
                *reinterpret_cast<uint2*>(it_u + e) = pack_f16x4(uu[0], uu[1], uu[2 % VEC], uu[3 % VEC]);
              } else {
                *reinterpret_cast<float2*>(it_m + e) = make_float2(mm[0], mm[1]);
                *reinterpret_cast<float2*>(it_v + e) = make_float2(vv[0], vv[1]);
                *reinterpret_cast<uint32_t*>(it_u + e) = pack_f16x4(uu[0], uu[1], 0.f, 0.f).x;
              }
            }
          }
          const bool last = mt.last != 0;
          release();
          if (last) break;
          if (!mbar_wait_warp(full_bar + stage, phase, abort_flag)) { alive = false; break; }
          mt = meta[stage];
        }
        if (!alive) break;
      }
    }
  }
  __syncthreads();
  if (*abort_flag) {
    // a wait ran out: give bulk copies that may still be in flight time to land before the CTA retires
    for (int i = 0; i < 200; ++i) __nanosleep(1000);
    if (tid == 0) atomicExch(&ctrl->timeout_flag, 1);
  }
}

template <int SMAX, bool HIST16, bool MOM16>
inline cudaError_t fused_set_smem() {
  return cudaFuncSetAttribute(fused_stream_kernel<SMAX, HIST16, MOM16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              FusedCfg<SMAX, HIST16, MOM16>::kTotal);
}

template <bool HIST16, bool MOM16>
inline cudaError_t fused_set_smem_for(int s) {
  return s <= 8 ? fused_set_smem<8, HIST16, MOM16>() : (s <= 16 ? fused_set_smem<16, HIST16, MOM16>() : fused_set_smem<32, HIST16, MOM16>());
}

// skip_gram (optional, one entry per matrix): 1 where the Gram row and the solve of a matrix are done before this
// kernel runs (projection with the Gram row in its epilogue); such a matrix gets combination tiles only.
inline ngalore_status fused_plan_create(FusedPlan& plan, const std::vector<MatDesc>& mats, int s, int sm_count,
                                        const std::vector<int>* skip_gram = nullptr) {
  plan.grid = sm_count;
  // Item order: every Gram tile (matrix order), then every combination tile (same order).  A CTA that picks
  // up a combination tile then never waits for a Gram tile that is still running, except for the last few
  // matrices.  Measured against keeping a matrix's combination pass close behind its Gram pass (in the hope
  // of L2 hits on its history): the stalls of the close order cost far more than the hits gain; on the 1.1B
  // shapes the phase went from 4.85 ms to 4.2 ms, on the 130M shapes from 0.51 ms to 0.35 ms.
  std::vector<FusedItem> items;
  const int n = static_cast<int>(mats.size());
  for (int i = 0; i < n; ++i) {
    if (mats[i].s == 0) continue;
    if (skip_gram != nullptr && (*skip_gram)[i]) continue;
    for (int t = 0; t < mats[i].ntiles; ++t) items.push_back(FusedItem{i, t, 0, 0});
  }
  for (int i = 0; i < n; ++i)
    for (int t = 0; t < mats[i].ntiles; ++t) items.push_back(FusedItem{i, t, 1, 0});
  plan.n_items = static_cast<int>(items.size());
  if (plan.grid > plan.n_items) plan.grid = plan.n_items;
  if (cudaMalloc(&plan.d_items, sizeof(FusedItem) * items.size()) != cudaSuccess) {
    plan.d_items = nullptr;
    return NGALORE_ERR_ALLOC;
  }
  if (cudaMemcpy(plan.d_items, items.data(), sizeof(FusedItem) * items.size(), cudaMemcpyHostToDevice) != cudaSuccess)
    return NGALORE_ERR_CUDA;
  plan.hist16 = !mats.empty() && mats[0].H16 != nullptr;
  plan.mom16 = !mats.empty() && mats[0].m16 != nullptr;
  const cudaError_t e = plan.hist16 ? (plan.mom16 ? fused_set_smem_for<true, true>(s) : fused_set_smem_for<true, false>(s))
                                    : (plan.mom16 ? fused_set_smem_for<false, true>(s) : fused_set_smem_for<false, false>(s));
  return e == cudaSuccess ? NGALORE_OK : NGALORE_ERR_CUDA;
}

inline void fused_plan_destroy(FusedPlan& plan) {
  if (plan.d_items) cudaFree(plan.d_items);
  plan.d_items = nullptr;
}

template <int SMAX, bool HIST16, bool MOM16>
inline void fused_launch_one(const FusedPlan& plan, const MatDesc* d_mats, Ctrl* d_ctrl, const Hyper* d_hyper,
                             bool short_step, cudaStream_t stream) {
  using C = FusedCfg<SMAX, HIST16, MOM16>;
  launch_step(short_step, fused_stream_kernel<SMAX, HIST16, MOM16>, plan.grid, C::kThreads, C::kTotal, stream, d_mats, plan.d_items,
              plan.n_items, d_ctrl, d_hyper);
}

template <bool HIST16, bool MOM16>
inline void fused_launch_for(const FusedPlan& plan, const MatDesc* d_mats, Ctrl* d_ctrl, const Hyper* d_hyper, int s,
                             bool short_step, cudaStream_t stream) {
  if (s <= 8) fused_launch_one<8, HIST16, MOM16>(plan, d_mats, d_ctrl, d_hyper, short_step, stream);
  else if (s <= 16) fused_launch_one<16, HIST16, MOM16>(plan, d_mats, d_ctrl, d_hyper, short_step, stream);
  else fused_launch_one<32, HIST16, MOM16>(plan, d_mats, d_ctrl, d_hyper, short_step, stream);
}

inline ngalore_status fused_stream_launch(FusedPlan& plan, const MatDesc* d_mats, int /*n_mats*/, Ctrl* d_ctrl,
                                          const Hyper* d_hyper, int s, bool short_step, cudaStream_t stream, int64_t* launches) {
  if (plan.hist16) {
    if (plan.mom16) fused_launch_for<true, true>(plan, d_mats, d_ctrl, d_hyper, s, short_step, stream);
    else fused_launch_for<true, false>(plan, d_mats, d_ctrl, d_hyper, s, short_step, stream);
  } else {
    if (plan.mom16) fused_launch_for<false, true>(plan, d_mats, d_ctrl, d_hyper, s, short_step, stream);
    else fused_launch_for<false, false>(plan, d_mats, d_ctrl, d_hyper, s, short_step, stream);
  }
  *launches += 1;
  return cudaGetLastError() == cudaSuccess ? NGALORE_OK : NGALORE_ERR_CUDA;
}

}  // namespace ngalore
