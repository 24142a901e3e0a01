// One persistent kernel for the whole history phase of a step: the Gram row of every matrix,
// the s x s solves, and the natural-gradient combination with the Adam moments (Sec. 2.4, 2.2).
//
// Structure: one CTA per SM; a producer warp streams the history (and m, v) through a ring of
// shared-memory stages with bulk asynchronous copies (cp.async.bulk + mbarrier), eight to sixteen consumer
// warps compute from shared memory, and a finishing warp turns the partial sums of a Gram tile into its partial row,
// solves the s x s system of the matrices whose last Gram tile the CTA has and fetches the weights of its
// combination items, each ahead of the consumers.  The producer runs ahead of them across tile and
// matrix boundaries, so the SM always has several stages of loads in flight.
//
// Work items (Gram tiles and combination tiles of all matrices) are fetched in order from a global
// counter by the producer.  The consumers of a Gram item wait for nothing but its data; the finishing warp of the CTA that has a
// matrix's last Gram tile waits (bounded) for the partial rows of the others and publishes the weights, that of a
// CTA with a combination item waits (bounded) for those.  Every item that is waited for sits earlier in the list and
// has been fetched by a CTA that consumes its items in order, so the kernel cannot deadlock.
// All Gram items precede all combination items, so the wait is short except at the very end of the Gram items.
//
// No consumer reads anything but shared memory before its results go out: where one of them fetched the weights itself (flag, fence,
// weights, descriptor: 2 to 3 us an item during which nothing left the full ring), a CTA of the 60M shapes, s = 8, spent 12 to 20
// of 72 us on it, of the encoder shapes at r = 8 13 of 25.
#pragma once

#include <algorithm>
#include <type_traits>
#include <vector>

#include "../../include/ngalore.h"
#include "common.cuh"
#include "gemm_tcgen05.cuh"  // mbarrier wrappers
#include "kernels_stream.cuh"

namespace ngalore {

// All that the producer needs of an item, so that one trip to memory fetches it.
struct __align__(16) FusedItem {
  int mat;
  int kind;        // 0 = Gram tile, 1 = combination tile
  int solve;       // a Gram tile: whether it is its matrix's last one
  int count;       // elements, of a run at most
  long long e0;    // first element
  long long rn;    // elements of a history slot
  const void* hist;      // the ring: fp32, or bf16 where the state keeps its history so
  const float* current;  // bf16 history: the fp32 gradient of this step
  const void *m, *v;     // moments, fp32 or bf16
  uintptr_t rows;        // where the partial rows of a Gram tile go (StageMeta)
  int rest;              // elements of a Gram tile beyond its first run: products are summed in fp32 run by run, runs in fp64
  int pad;
};

struct FusedPlan {
  FusedItem* d_items = nullptr;
  int n_items = 0;
  int grid = 0;
  bool hist16 = false;  // the state keeps its history ring in bf16
  bool mom16 = false;   // the state keeps its moments in bf16
  bool runs = false;    // some Gram tile has more than one run
};

// The finishing warp's waits for what other CTAs publish, the partial rows of a matrix and its weights, in time, since what a poll takes
// depends on what else goes on (0.33 us for a weight that nothing writes).  The consumers and the producer wait for this warp in turn, until
// kTcWaitLimitNs, and give the whole CTA up then, with items of matrices that have nothing to do with it: so all that it may spend
// before a combination item has its weights, the rows of two slots and the weights themselves, has to be less.  And the rows are given up before the
// weights that depend on them, so that no solve ends after somebody has flagged its matrix.
constexpr unsigned long long kRowsLimitNs = 300000000ull, kWeightsLimitNs = 900000000ull;
static_assert(2 * kRowsLimitNs < kWeightsLimitNs && 2 * kRowsLimitNs + kWeightsLimitNs <= kTcWaitLimitNs / 4 * 3, "waits that depend on each other end in turn");

struct StageMeta {
  int kind, last, count, pad;   // last: the sums of a Gram tile's run are complete, or a combination item is
  long long e0;
  uintptr_t rows;               // where the rows of the Gram tile go; odd: its next run is still to come
};

// What the finishing warp is told to do, in the order of the CTA's items: solve for a matrix, or fetch the weights of a combination item
// (kind < 0: there are no more).
struct WeightsJob {
  int mat, kind;
};

// ... and what it leaves for the consumers of a combination item.
struct __align__(16) ItemWeights {
  float w[kMaxHistory];
  float *m, *v, *cur;
  __half* u;
  uint16_t *m16, *v16, *h16;
  int index;
  int ok, bad;     // ok 0: the weights never came; bad 1: the step is flagged for the matrix
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
  static constexpr int kJobs = 4;                               // jobs under way to the finishing warp
  static constexpr int kJobBarOff = kBase + 528, kJobOff = kJobBarOff + 16 * kJobs, kWBarOff = kJobOff + 8 * kJobs;
  static constexpr int kRedBarOff = kWBarOff + 32, kRedRowsOff = kRedBarOff + 32, kWeightsOff = kBase + 768;
  static constexpr int kRedOff = kWeightsOff + 2 * static_cast<int>(sizeof(ItemWeights));
  static_assert(kRedRowsOff + 16 <= kWeightsOff && kRedOff % 8 == 0, "shared memory regions overlap");
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
// RUNS: some Gram tile has more than one run.  An instance of its own, since the code for it costs sets without 0.2 us of 20.6 (one 512 x 1376
// matrix) to 0.3 of 196.5 (60M shapes).
template <int SMAX, bool HIST16, bool MOM16, bool RUNS>
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
  uint64_t* job_full = reinterpret_cast<uint64_t*>(fs_smem + C::kJobBarOff);    // [kJobs] the producer has left a job
  uint64_t* job_empty = job_full + C::kJobs;                                    // [kJobs] the finishing warp has taken it
  WeightsJob* jobs = reinterpret_cast<WeightsJob*>(fs_smem + C::kJobOff);       // [kJobs]
  uint64_t* w_full = reinterpret_cast<uint64_t*>(fs_smem + C::kWBarOff);        // [2] the weights of a combination item are there
  uint64_t* w_empty = w_full + 2;                                               // [2] all consumer warps are through with them
  ItemWeights* weights = reinterpret_cast<ItemWeights*>(fs_smem + C::kWeightsOff);  // [2]
  uint64_t* red_full = reinterpret_cast<uint64_t*>(fs_smem + C::kRedBarOff);   // [2] all consumer warps have left their sums
  uint64_t* red_empty = red_full + 2;                                           // [2] the finishing warp has taken them
  ulonglong2** red_rows = reinterpret_cast<ulonglong2**>(fs_smem + C::kRedRowsOff); // [2] where a tile's rows go (null: there are no more)
  double* red = reinterpret_cast<double*>(fs_smem + C::kRedOff);                // [2][rows][warps][SMAX]

  const int tid = threadIdx.x;
  if (tid == 0) {
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(full_bar + s, 1);
      mbar_init(empty_bar + s, kConsumerThreads / 32);
    }
    for (int b = 0; b < 2; ++b) { mbar_init(red_full + b, kWarps); mbar_init(red_empty + b, 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(w_full + b, 1); mbar_init(w_empty + b, kWarps); }
    for (int b = 0; b < C::kJobs; ++b) { mbar_init(job_full + b, 1); mbar_init(job_empty + b, 1); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  // (The tables are laid out for good: the item that this CTA will probably claim first comes to the SM ahead of
  // the wait for the kernel before.  It is claimed like the others all the same: an item that belonged to a CTA which another kernel
  // keeps from starting could be waited for by that kernel's neighbours for good.)
  if (tid == kConsumerThreads && static_cast<int>(blockIdx.x) < n_items) {
    const FusedItem& i0 = items[blockIdx.x];
    asm volatile("" ::"r"(i0.mat), "l"(i0.hist), "l"(i0.rows), "r"(mats[0].s));
  }
  pdl_begin();
  int it = 0;      // the producer's item: claimed ahead of everything else
  if (tid == kConsumerThreads) it = static_cast<int>(atomicAdd(&ctrl->work_counter, 1u));
  const unsigned int tag = static_cast<unsigned int>(ctrl->epoch + 1);
  const int s_all = mats[0].s;                       // (the same for every matrix, and so are ring position and count)
  const int c = ring_count(ctrl, s_all), cur = ring_cur(ctrl, s_all);
  const int prev = HIST16 && c >= 2 ? (cur == 0 ? s_all : cur) - 1 : -1;   // the slot whose row is worked out again

  if (tid >= kConsumerThreads + 32) {
    // ------------------------------------------------------------------ finishing warp
    // Two kinds of work: the partial row of every Gram tile that the consumers leave, and the producer's jobs.  Whatever it
    // waits for, it looks after the rows meanwhile: another CTA may be waiting for them, or the consumers for their place.
    const int lane = tid & 31;
    const double lambda = hyper->lambda;
    const int withheld = ctrl->debug_withhold - 1;
    const unsigned int polls = static_cast<unsigned int>(ctrl->spin_limit);   // (testing aid; 0: the limit in time alone)
    unsigned long long rows_limit = kRowsLimitNs;   // (what did not come in time for one matrix is not waited for again)
    bool jobs_open = true, rows_open = true;
    unsigned int taken = 0, tiles = 0, fetched = 0;   // jobs, Gram tiles and combination items so far
    auto look_after_rows = [&]() {
      const int buf = tiles & 1;
      if (!rows_open || !__all_sync(0xffffffffu, mbar_test(red_full + buf, (tiles >> 1) & 1u))) return;
      ulonglong2* const rows = red_rows[buf];   // [rows][s]: row of `cur` and (HIST16) of `prev`
      double part[C::kRows];
#pragma unroll
      for (int r = 0; r < C::kRows; ++r) {
        const double* src = red + (buf * C::kRows + r) * C::kRedDoubles + min(lane, SMAX - 1);
        double t0 = 0.0, t1 = 0.0;
#pragma unroll
        for (int w = 0; w < kWarps; w += 2) { t0 += src[w * SMAX]; t1 += src[(w + 1) * SMAX]; }
        part[r] = t0 + t1;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(red_empty + buf);
      ++tiles;
      if (rows == nullptr) {
        rows_open = false;
      } else if (lane < s_all) {
#pragma unroll
        for (int r = 0; r < C::kRows; ++r) st_tagged(rows + r * s_all + lane, part[r], tag);
      }
      __syncwarp();
    };
    // mbar_wait of the whole warp, which looks after the rows between two looks
    auto wait_for = [&](uint64_t* bar, uint32_t parity) {
      unsigned long long t0 = 0;
      for (unsigned int it = 0; !__all_sync(0xffffffffu, mbar_test(bar, parity)); ++it) {
        look_after_rows();
        if ((it & 63u) == 63u) {
          const unsigned long long now = global_timer_ns();
          if (t0 == 0) t0 = now;
          if (__any_sync(0xffffffffu, *abort_flag != 0 || now - t0 > kTcWaitLimitNs)) { *abort_flag = 1; return false; }
        }
      }
      return true;
    };
    while (jobs_open) {
      const int at = taken % C::kJobs;
      if (!wait_for(job_full + at, (taken / C::kJobs) & 1u)) break;
      const WeightsJob job = jobs[at];
      __syncwarp();
      if (lane == 0) mbar_arrive(job_empty + at);
      ++taken;
      if (job.kind < 0) { jobs_open = false; break; }
      const MatDesc& d = mats[job.mat];
      if (job.kind == 0) {
        GramSolve<SMAX> solve;
        solve.prepare(d, cur, prev, c, lambda, lane);
        double row = 0.0, rowp = 0.0;
        bool here = tagged_row_sum<SMAX>(d, lane, c, C::kRows, 0, tag, rows_limit, abort_flag, row, look_after_rows);
        if (HIST16 && prev >= 0 && here) here = tagged_row_sum<SMAX>(d, lane, c, C::kRows, C::kRows - 1, tag, rows_limit, abort_flag, rowp, look_after_rows);
        if (!here) { rows_limit = 0; continue; }   // (nobody gets weights, and says so)
        solve.finish(d, cur, prev, c, lambda, lane, row, rowp, tag, withheld == job.mat);
        continue;
      }
      float w;
      int ok = 1, bad;
      if (s_all > 0) {
        unsigned long long word, t0 = 0;
        for (unsigned int spins = 0;; ++spins) {
          word = ld_relaxed(d.wpub + lane);
          if (__all_sync(0xffffffffu, static_cast<unsigned int>(word >> 32) >> 1 == (tag & 0x7fffffffu))) break;
          if (polls != 0 && spins >= polls) ok = 0;
          if ((spins & 63u) == 63u) {
            const unsigned long long now = global_timer_ns();
            if (t0 == 0) t0 = now;
            if (__any_sync(0xffffffffu, *abort_flag != 0 || now - t0 > kWeightsLimitNs)) ok = 0;
          }
          if (!ok) break;
          look_after_rows();
          if (spins > 16) __nanosleep(100);
        }
        w = __uint_as_float(static_cast<unsigned int>(word));
        bad = static_cast<int>(word >> 32) & 1;
        if (!ok && lane == 0) {
          // The weights never came: this matrix takes no update in this step (the back-projection skips it)
          // and says why.  Tiles of it that other CTAs did combine have advanced their part of m and v.
          atomicExch(&ctrl->timeout_flag, 1);
          atomicExch(d.step_bad, 1);
          atomicCAS(d.status, 0, 8 /* NGALORE_ERR_TIMEOUT */);
        }
      } else {
        w = __ldcg(d.wsol + lane);
        bad = __ldcg(d.step_bad) != 0 ? 1 : 0;
      }
      const int slot = fetched & 1;
      if (!wait_for(w_empty + slot, ((fetched >> 1) & 1u) ^ 1u)) break;
      ++fetched;
      ItemWeights& o = weights[slot];
      o.w[lane] = w;
      if (lane == 0) {
        o.m = d.m; o.v = d.v; o.cur = current_gradient(d, cur); o.u = d.u16; o.m16 = d.m16; o.v16 = d.v16;
        o.h16 = HIST16 ? d.H16 + static_cast<long long>(cur) * d.rn : nullptr;
        o.index = d.index; o.ok = ok; o.bad = bad;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(w_full + slot);
    }
    // (the consumers say so when they have left the last Gram tile's sums)
    while (rows_open) {
      if (!wait_for(red_full + (tiles & 1), (tiles >> 1) & 1u)) break;
      look_after_rows();
    }
  } else if (tid >= kConsumerThreads) {
    // ------------------------------------------------------------------ producer warp
    // Lane 0 claims items and arms the barriers; every lane issues the bulk copy of "its" slot (lane j copies
    // history slot j, the next two lanes m and v), so a stage's copies are issued in parallel.  The next item is
    // claimed and fetched while the stages of the current one go out, one round trip to memory per
    // stage: round trips in a row between two items cost as much as streaming 4096 elements of eight slots.
    const int lane = tid & 31;
    // copy number k of an item: history slot k, then m and v; its place in a stage, bytes per element and source
    auto place = [&](int k) {
      if (k < c) return !HIST16 ? k * CE * 4 : (k == cur ? C::kCurOff : k * CE * 2);
      return k == c ? C::kMOff : C::kVOff;
    };
    auto width = [&](int k) { return k < c ? (HIST16 && k != cur ? 2 : 4) : (MOM16 ? 2 : 4); };
    auto source = [&](const FusedItem& o, int k) {
      const void* base = k == c ? o.m : o.v;
      if (k < c) base = HIST16 && k == cur ? static_cast<const void*>(o.current) : static_cast<const unsigned char*>(o.hist) + k * o.rn * width(k);
      return static_cast<const unsigned char*>(base);
    };
    // Tells the finishing warp what this CTA needs of it for an item.  block: wait until there is room (without it, false where
    // there is none).
    unsigned int told = 0;
    bool ok = true;
    auto tell = [&](int mat, int kind, bool block) {
      const int at = told % C::kJobs;
      const uint32_t parity = ((told / C::kJobs) & 1u) ^ 1u;
      int good = 1;
      if (lane == 0) {
        good = block ? (mbar_wait(job_empty + at, parity, abort_flag) ? 1 : 0) : (mbar_test(job_empty + at, parity) ? 1 : 0);
        if (good) {
          jobs[at] = WeightsJob{mat, kind};
          mbar_arrive(job_full + at);
        }
      }
      good = __shfl_sync(0xffffffffu, good, 0);
      if (good) ++told;
      else if (block) ok = false;
      return good != 0;
    };
    auto wanted = [](const FusedItem& o) { return o.kind == 1 || o.solve != 0; };
    int stage = 0;
    uint32_t phase = 0;
    FusedItem now{}, next{};
    bool told_ahead = false;   // the finishing warp knows of the next item
    it = __shfl_sync(0xffffffffu, it, 0);
    if (it < n_items) now = items[it];
    while (true) {
      if (it >= n_items) {
        tell(0, -1, true);
        if (lane == 0 && mbar_wait(empty_bar + stage, phase ^ 1u, abort_flag)) {
          meta[stage].kind = -1;
          mbar_arrive(full_bar + stage);
        }
        break;
      }
      if (wanted(now) && !told_ahead) tell(now.mat, now.kind, true);
      if (!ok) break;
      told_ahead = false;
      const int ncopies = c + (now.kind == 1 ? 2 : 0);
      const unsigned char* src[2] = {source(now, lane), source(now, lane + 32)};   // this lane's copies
      int step = 0;   // how far the next item is known: 0 claimed, 1 fetched, 2 on: told to the finishing warp, where that has room
      auto look_ahead = [&]() {
        if (step == 0) {
          if (lane == 0) it = static_cast<int>(atomicAdd(&ctrl->work_counter, 1u));
        } else if (step == 1) {
          it = __shfl_sync(0xffffffffu, it, 0);
          if (it < n_items) next = items[it];
        } else if (!told_ahead && it < n_items && wanted(next)) {
          told_ahead = tell(next.mat, next.kind, false);
        }
        ++step;
      };
      while (true) {
        const long long e1 = now.e0 + now.count;
        for (long long e = now.e0; e < e1; e += CE) {
          const int cnt = (e1 - e < CE) ? static_cast<int>(e1 - e) : CE;
          int good = 1;
          if (lane == 0) good = mbar_wait(empty_bar + stage, phase ^ 1u, abort_flag) ? 1 : 0;
          good = __shfl_sync(0xffffffffu, good, 0);
          if (!good) { ok = false; break; }
          unsigned char* sb = fs_smem + stage * C::kStageBytes;
          const uint32_t bytes = static_cast<uint32_t>(cnt) * 4u;
          if (lane == 0) {
            meta[stage] = StageMeta{now.kind, e + CE >= e1 ? 1 : 0, cnt, 0, e, now.rows};
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
              bulk_load(sb + place(k), src[q] + e * w, static_cast<uint32_t>(cnt * w), full_bar + stage);
            }
          }
          if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
          look_ahead();
        }
        if (!RUNS || !ok || now.rest == 0) break;
        // the next run of the tile, like one of its own to the consumers
        now.e0 += now.count;
        now.count = min(now.count, now.rest);
        now.rest -= now.count;
        if (now.rest == 0) now.rows &= ~static_cast<uintptr_t>(1);
      }
      if (!ok) break;
      while (step < 2) look_ahead();
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
    bool later = false;            // this run of a Gram tile is not its first
    unsigned int combined = 0;     // combination items whose weights have been taken
    const unsigned int it_step = static_cast<unsigned int>(ctrl->k);
    // Tells the finishing warp that the CTA has no more Gram tiles (all of them are ahead of the combination items), as soon as that is
    // known: at the end of the kernel it would be the last thing everybody waits for.
    bool gram_open = true;
    auto close_gram = [&]() {
      if (tid == 0) red_rows[tiles_done & 1] = nullptr;
      __syncwarp();
      if (lane == 0) mbar_arrive(red_full + (tiles_done & 1));
      gram_open = false;
    };
    if (HIST16) {
      // the current slot's place in a stage stays zero for the whole launch: its gradient takes part in fp32 instead
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
      bool alive = true;
      if (mt.kind == 0) {
        // ---- Gram tile, or a run of one
        const int buf = tiles_done & 1;
        // this warp's sums of row r over its lanes, into the buffer of the finishing warp (runs of a tile one after another)
        auto hand_over = [&](int r, double (&v)[SMAX]) {
          const double t = warp_sums<SMAX>(v);
          double* const at = red + ((buf * C::kRows + r) * kWarps + warp) * SMAX + lane / (32 / SMAX);
          if ((lane & (32 / SMAX - 1)) == 0) *at = RUNS && later ? *at + t : t;
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
          const int old = prev >= 0 ? prev : cur;
          while (true) {
            if (idx < mt.count) {
              float x[VEC];
              uint64_t xx[VEC / 2], xp[VEC / 2];
              load_current(x);
              load16(old, xp);             // (a single gradient: the zeros of its own place)
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
        later = RUNS && (mt.rows & 1) != 0;
        if (later) continue;
        ++tiles_done;
        if (tid == 0) red_rows[buf] = reinterpret_cast<ulonglong2*>(mt.rows);
        __syncwarp();
        if (lane == 0) mbar_arrive(red_full + buf);
      } else {
        // ---- combination tile
        // (where the finishing warp still has two tiles to take, the next item will do)
        if (gram_open && __all_sync(0xffffffffu, mbar_test(red_empty + (tiles_done & 1), ((tiles_done >> 1) & 1u) ^ 1u))) close_gram();
        const ItemWeights& iw = weights[combined & 1];
        if (!mbar_wait_warp(w_full + (combined & 1), (combined >> 1) & 1u, abort_flag)) break;
        const bool item_ok = iw.ok != 0, item_bad = iw.bad != 0;
        float *const it_m = iw.m, *const it_v = iw.v, *const it_cur = iw.cur;
        __half* const it_u = iw.u;
        uint16_t *const it_m16 = iw.m16, *const it_v16 = iw.v16, *const it_h16 = iw.h16;
        const unsigned int it_mat = static_cast<unsigned int>(iw.index);
        float w[SMAX];
#pragma unroll
        for (int j = 0; j < SMAX; j += 4) {
          const float4 x = *reinterpret_cast<const float4*>(iw.w + j);
          w[j] = x.x; w[j + 1] = x.y; w[j + 2] = x.z; w[j + 3] = x.w;
        }
        const float wc = HIST16 ? iw.w[cur] : 0.f;
        __syncwarp();
        if (lane == 0) mbar_arrive(w_empty + (combined & 1));
        ++combined;
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

template <int SMAX, bool HIST16, bool MOM16, bool RUNS>
struct FusedKernel {
  using C = FusedCfg<SMAX, HIST16, MOM16>;
  static constexpr auto kernel = fused_stream_kernel<SMAX, HIST16, MOM16, RUNS>;
};
// f with the kernel of a plan
template <typename F>
inline auto fused_with_kernel(const FusedPlan& plan, int s, F&& f) {
  auto instance = [&](auto hist16, auto mom16, auto runs) {
    constexpr bool H = decltype(hist16)::value, M = decltype(mom16)::value, R = decltype(runs)::value;
    return s <= 8 ? f(FusedKernel<8, H, M, R>{}) : (s <= 16 ? f(FusedKernel<16, H, M, R>{}) : f(FusedKernel<32, H, M, R>{}));
  };
  auto moments = [&](auto hist16, auto mom16) {
    return plan.runs ? instance(hist16, mom16, std::true_type{}) : instance(hist16, mom16, std::false_type{});
  };
  auto history = [&](auto hist16) { return plan.mom16 ? moments(hist16, std::true_type{}) : moments(hist16, std::false_type{}); };
  return plan.hist16 ? history(std::true_type{}) : history(std::false_type{});
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
  plan.hist16 = !mats.empty() && mats[0].H16 != nullptr;
  plan.mom16 = !mats.empty() && mats[0].m16 != nullptr;
  auto add = [&](int i, int t, int kind) {
    const MatDesc& d = mats[i];
    FusedItem o{};
    o.mat = i; o.kind = kind; o.solve = kind == 0 && t == d.ntiles - 1 ? 1 : 0;
    o.e0 = static_cast<long long>(t) * d.te;
    o.count = static_cast<int>(std::min<long long>(d.te, d.rn - o.e0));
    o.rn = d.rn;
    o.hist = plan.hist16 ? static_cast<const void*>(d.H16) : static_cast<const void*>(d.H);
    o.current = d.H;
    o.m = plan.mom16 ? static_cast<const void*>(d.m16) : static_cast<const void*>(d.m);
    o.v = plan.mom16 ? static_cast<const void*>(d.v16) : static_cast<const void*>(d.v);
    o.rows = reinterpret_cast<uintptr_t>(d.grow + static_cast<long long>(t) * (plan.hist16 ? 2 : 1) * s);
    if (kind == 0 && o.count > d.run) {
      o.rest = o.count - d.run; o.count = d.run; o.rows |= 1;
      plan.runs = true;
    }
    items.push_back(o);
  };
  for (int i = 0; i < n; ++i) {
    if (mats[i].s == 0) continue;
    if (skip_gram != nullptr && (*skip_gram)[i]) continue;
    for (int t = 0; t < mats[i].ntiles; ++t) add(i, t, 0);
  }
  for (int i = 0; i < n; ++i)
    for (int t = 0; t < mats[i].ntiles; ++t) add(i, t, 1);
  plan.n_items = static_cast<int>(items.size());
  if (plan.grid > plan.n_items) plan.grid = plan.n_items;
  if (cudaMalloc(&plan.d_items, sizeof(FusedItem) * items.size()) != cudaSuccess) {
    plan.d_items = nullptr;
    return NGALORE_ERR_ALLOC;
  }
  if (cudaMemcpy(plan.d_items, items.data(), sizeof(FusedItem) * items.size(), cudaMemcpyHostToDevice) != cudaSuccess)
    return NGALORE_ERR_CUDA;
  const cudaError_t e = fused_with_kernel(plan, s, [](auto k) {
    return cudaFuncSetAttribute(k.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, decltype(k)::C::kTotal);
  });
  return e == cudaSuccess ? NGALORE_OK : NGALORE_ERR_CUDA;
}

inline void fused_plan_destroy(FusedPlan& plan) {
  if (plan.d_items) cudaFree(plan.d_items);
  plan.d_items = nullptr;
}

inline ngalore_status fused_stream_launch(FusedPlan& plan, const MatDesc* d_mats, int /*n_mats*/, Ctrl* d_ctrl,
                                          const Hyper* d_hyper, int s, bool short_step, cudaStream_t stream, int64_t* launches) {
  fused_with_kernel(plan, s, [&](auto k) {
    using C = typename decltype(k)::C;
    return launch_step(short_step, k.kernel, plan.grid, C::kThreads, C::kTotal, stream, d_mats, plan.d_items, plan.n_items, d_ctrl, d_hyper);
  });
  *launches += 1;
  return cudaGetLastError() == cudaSuccess ? NGALORE_OK : NGALORE_ERR_CUDA;
}

}  // namespace ngalore
