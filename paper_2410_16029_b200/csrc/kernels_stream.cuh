// Streaming kernels of the step: Gram row of the history ring, the s x s Cholesky solve,
// and the fused natural-gradient combination + Adam moments (Sec. 2.4 and Sec. 2.2).
#pragma once

#include "common.cuh"

namespace ngalore {

__device__ __forceinline__ float4 ldg4(const float* p) {
  return *reinterpret_cast<const float4*>(p);
}

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Partial inner products <H_cur, H_j> over one tile of the flattened r' x N index range.
// Products and short per-thread sums are fp32; everything across threads is fp64.
template <int SMAX>
__device__ __forceinline__ void gram_tile(const MatDesc& d, int local, int cur, int c, int tile_elems,
                                          double* red /* smem: (kStreamThreads/32) * SMAX */) {
  const long long e0 = static_cast<long long>(local) * tile_elems;
  const long long e1 = (e0 + tile_elems < d.rn) ? e0 + tile_elems : d.rn;
  float acc[SMAX];
#pragma unroll
  for (int j = 0; j < SMAX; ++j) acc[j] = 0.f;
  const float* Hc = d.H + static_cast<long long>(cur) * d.rn;
  for (long long e = e0 + threadIdx.x * 4; e < e1; e += kStreamThreads * 4) {
    const float4 x = ldg4(Hc + e);
#pragma unroll
    for (int j = 0; j < SMAX; ++j) {
      if (j < c) {
        const float4 y = ldg4(d.H + static_cast<long long>(j) * d.rn + e);
        acc[j] += x.x * y.x + x.y * y.y + x.z * y.z + x.w * y.w;
      }
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int j = 0; j < SMAX; ++j) {
    const double t = warp_sum(static_cast<double>(acc[j]));
    if (lane == 0) red[warp * SMAX + j] = t;
  }
  __syncthreads();
  if (threadIdx.x < SMAX) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kStreamThreads / 32; ++w) t += red[w * SMAX + threadIdx.x];
    if (static_cast<int>(threadIdx.x) < d.s) {
      d.gpart[static_cast<long long>(local) * d.s + threadIdx.x] = t;
      __threadfence();  // a later reader may run in another CTA of the same launch
    }
  }
  __syncthreads();
}

// Lane j's share of the Gram row (zero from lane c on): the sum over the matrix's tiles of partial product j, in a fixed
// order, so that the result is reproducible.
// The partial rows of early tiles have left L2 by then, so it is the number of loads under way that decides: 32 / SMAX lanes
// share a column, sixteen loads each (352 tiles, s = 16: 37 us with one lane a column and eight loads, 19 us so).
template <int SMAX>
__device__ __forceinline__ double gram_row_sum(const MatDesc& d, int lane, int c) {
  constexpr int G = 32 / SMAX, U = 16;
  const double* gp = d.gpart + min(lane % SMAX, c - 1);
  const long long st = d.s;
  double t[4] = {0.0, 0.0, 0.0, 0.0};
  for (int t0 = 0; t0 < d.ntiles; t0 += G * U) {
    double x[U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const int tile = t0 + q * G + lane / SMAX;
      const double v = __ldcg(gp + min(tile, d.ntiles - 1) * st);
      x[q] = tile < d.ntiles ? v : 0.0;
    }
#pragma unroll
    for (int q = 0; q < U; ++q) t[q & 3] += x[q];
  }
  double sum = (t[0] + t[1]) + (t[2] + t[3]);
#pragma unroll
  for (int o = SMAX; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  return lane < c ? sum : 0.0;
}

// One warp: put the new Gram row (lane j: <H_cur, H_j>) into Kraw, form lambda I + K with K = Kraw / c and solve for
// the weights w of N~ = sum_i w_i H_i, i.e. (lambda I + K) w = e_cur.  This is F^-1 applied to the
// current gradient by the Woodbury identity, written for the case where the current gradient is a
// column of the stacked matrix; it avoids the cancellation of the two-term form.
// Lane i keeps row i of the matrix in registers; the elimination (Gauss-Jordan without pivoting: the matrix is
// symmetric positive definite, its pivots are the squares of Cholesky's, and the same pivots tell when it is not)
// broadcasts row k by shuffles, so the chain per step is one shuffle, one reciprocal and one multiply-add.  In shared
// memory with serial substitutions the solve took 9 us for s = 8 and 25 us for s = 16; so 2 and 4 us.
// What bounds it is that the 32 lanes run together.  Lanes that a branch on the lane number has parted are not brought back
// together by a shuffle that all of them take part in: each one then costs two turns of the scheduler, 500 cycles instead of
// 30 (one 1024 x 1024 matrix, s = 20: 125 us a solve, 10 so).  So nothing ahead of the elimination, here and in
// gram_row_sum, branches on the lane, and what is stored is stored after it.
template <int SMAX>
__device__ __forceinline__ void solve_matrix(const MatDesc& d, int cur, int c, double lambda, double row) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  double a[SMAX];
  {
    const double* old = d.Kraw + min(lane, c - 1) * d.s;
#pragma unroll
    for (int j = 0; j < SMAX; ++j) {
      const double v = __ldcg(old + min(j, c - 1));
      a[j] = lane < c && j < c ? v : 0.0;
    }
  }
  const bool finite = __all_sync(0xffffffffu, lane >= c || isfinite(row));
  int bad = finite ? 0 : 7 /* NGALORE_ERR_NONFINITE */;
  const double val = finite && lane < c ? row : 0.0;
  const double ic = 1.0 / static_cast<double>(c);
#pragma unroll
  for (int j = 0; j < SMAX; ++j) {
    const double v = __shfl_sync(0xffffffffu, val, j);
    a[j] = lane == cur ? v : a[j];
    a[j] = j == cur ? val : a[j];
    a[j] *= ic;
    a[j] += j == lane ? lambda : 0.0;
  }
  double b = lane == cur ? 1.0 : 0.0, diag = 1.0;
#pragma unroll
  for (int k = 0; k < SMAX; ++k) {
    if (k >= c || bad != 0) break;
    const double p = __shfl_sync(0xffffffffu, a[k], k);
    if (!(p > 0.0) || !isfinite(p)) {
      bad = isfinite(p) ? 6 /* NGALORE_ERR_NOT_SPD */ : 7;
      break;
    }
    diag = lane == k ? p : diag;
    const double ip = 1.0 / p;
    const double f = lane == k ? 0.0 : a[k] * ip;
#pragma unroll
    for (int j = k + 1; j < SMAX; ++j) a[j] -= f * __shfl_sync(0xffffffffu, a[j], k);
    b -= f * __shfl_sync(0xffffffffu, b, k);
  }
  d.wsol[lane] = bad == 0 && lane < c ? static_cast<float>(b / diag) : 0.f;
  // (where the step is flagged the poisoned slot becomes a zero gradient: its Gram row and column vanish)
  if (lane < (bad != 0 ? d.s : c)) {
    d.Kraw[cur * d.s + lane] = bad != 0 ? 0.0 : val;
    d.Kraw[lane * d.s + cur] = bad != 0 ? 0.0 : val;
  }
  if (lane == 0) {
    *d.step_bad = bad != 0 ? 1 : 0;
    if (bad != 0) atomicCAS(d.status, 0, bad);
  }
  __syncwarp();
}

// ---------------------------------------------------------------- the same solve in the fused stream kernel
//
// What one warp has for another CTA there (partial rows, weights) goes through words of eight bytes that hold four bytes of the value
// and the tag of the step: a reader polls the words themselves, so that a value is one trip to L2 behind its writer.  (Value, fence,
// counter, fence, read took three to four trips each way: one 512 x 1376 matrix, s = 8, waited 10 us from its last Gram tile to its
// weights, and 4 so.)
__device__ __forceinline__ void st_relaxed(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void ld_relaxed_2(const ulonglong2* p, unsigned long long& a, unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ unsigned long long tagged(unsigned int value, unsigned int tag) {
  return static_cast<unsigned long long>(value) | (static_cast<unsigned long long>(tag) << 32);
}
__device__ __forceinline__ void st_tagged(ulonglong2* p, double x, unsigned int tag) {
  const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(x));
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};"
               ::"l"(p), "l"(tagged(static_cast<unsigned int>(bits), tag)), "l"(tagged(static_cast<unsigned int>(bits >> 32), tag)) : "memory");
}
// Lane j's weight, for the combination tiles (the tag carries whether the step is flagged for the matrix).
__device__ __forceinline__ void publish_weights(const MatDesc& d, int lane, float w, bool bad, unsigned int tag) {
  st_relaxed(d.wpub + lane, tagged(__float_as_uint(w), 2u * tag + (bad ? 1u : 0u)));
}

// gram_row_sum over tagged rows ([tile][rows][s]; row: which of them), each waited for; sums in the same order.  False where they do not come within
// limit_ns.
// meanwhile: what the warp does between two looks.
template <int SMAX, typename F>
__device__ __forceinline__ bool tagged_row_sum(const MatDesc& d, int lane, int c, int rows, int row, unsigned int tag, unsigned long long limit_ns,
                                               const volatile int* abort_flag, double& out, F&& meanwhile) {
  constexpr int G = 32 / SMAX, U = 8;   // (sixteen take the registers of eight slots and more: 0.7 us slower for one matrix)
  const ulonglong2* gp = d.grow + static_cast<long long>(row) * d.s + min(lane % SMAX, c - 1);
  const long long st = static_cast<long long>(rows) * d.s;
  double t[4] = {0.0, 0.0, 0.0, 0.0};
  unsigned int spins = 0;
  unsigned long long begin = 0;
  for (int t0 = 0; t0 < d.ntiles; t0 += G * U) {
    unsigned long long lo[U], hi[U];
    while (true) {
#pragma unroll
      for (int q = 0; q < U; ++q) ld_relaxed_2(gp + min(t0 + q * G + lane / SMAX, d.ntiles - 1) * st, lo[q], hi[q]);
      bool here = true;
#pragma unroll
      for (int q = 0; q < U; ++q) here = here && static_cast<unsigned int>(lo[q] >> 32) == tag && static_cast<unsigned int>(hi[q] >> 32) == tag;
      if (__all_sync(0xffffffffu, here)) break;
      if ((++spins & 63u) == 0u) {
        const unsigned long long now = global_timer_ns();
        if (begin == 0) begin = now;
        if (__any_sync(0xffffffffu, *abort_flag != 0 || now - begin > limit_ns)) return false;
      }
      meanwhile();
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const double v = __longlong_as_double(static_cast<long long>((lo[q] & 0xffffffffull) | (hi[q] << 32)));
      t[q & 3] += t0 + q * G + lane / SMAX < d.ntiles ? v : 0.0;
    }
  }
  double sum = (t[0] + t[1]) + (t[2] + t[3]);
#pragma unroll
  for (int o = SMAX; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  out = lane < c ? sum : 0.0;
  return true;
}

// solve_matrix in two parts.  prepare eliminates the slots whose products are known when the step begins (all but `cur`, and with a
// bf16 history `prev`) while the Gram tiles are still on their way; finish takes the columns of the new ones through the same
// steps, two trips through the lanes for each slot (s = 8: 0.3 us where the whole elimination takes 2, s = 16: 0.6 instead of 4), and
// solves the system of one or two unknowns that is left.  As there, nothing branches on the lane ahead of the shuffles.
template <int SMAX>
struct GramSolve {
  double f[SMAX];    // row `lane`: the multiplier of every step
  double rdiag;      // one over its pivot
  double old_prev;   // <H_lane, H_prev> as it was
  int bad;

  __device__ __forceinline__ static bool known(int j, int cur, int prev, int c) { return j < c && j != cur && j != prev; }

  __device__ __forceinline__ void prepare(const MatDesc& d, int cur, int prev, int c, double lambda, int lane) {
    const double* old = d.Kraw + min(lane, c - 1) * d.s;
    const double ic = 1.0 / static_cast<double>(c);
    const bool mine = known(lane, cur, prev, c);
    old_prev = __ldcg(old + max(prev, 0));
#pragma unroll
    for (int j = 0; j < SMAX; ++j) f[j] = __ldcg(old + min(j, c - 1));
#pragma unroll
    for (int j = 0; j < SMAX; ++j) {
      f[j] = mine && known(j, cur, prev, c) ? f[j] * ic : 0.0;
      f[j] += j == lane ? (mine ? lambda : 1.0) : 0.0;
    }
    double diag = 1.0;
    bad = 0;
#pragma unroll
    for (int k = 0; k < SMAX; ++k) {
      if (k >= c || bad != 0) break;
      if (k == cur || k == prev) continue;
      const double p = __shfl_sync(0xffffffffu, f[k], k);
      if (!(p > 0.0) || !isfinite(p)) {
        bad = isfinite(p) ? 6 /* NGALORE_ERR_NOT_SPD */ : 7 /* NGALORE_ERR_NONFINITE */;
        break;
      }
      diag = lane == k ? p : diag;
      const double ip = 1.0 / p;
      f[k] = lane == k ? 0.0 : f[k] * ip;
#pragma unroll
      for (int j = k + 1; j < SMAX; ++j) f[j] -= f[k] * __shfl_sync(0xffffffffu, f[j], k);
    }
    rdiag = 1.0 / diag;
  }

  // row, rowp: lane j's <H_cur, H_j> and <H_prev, H_j>.  Publishes the weights (unless withheld), then leaves the Gram matrix, the
  // weights and the status of the matrix for the next kernels and steps.
  __device__ __forceinline__ void finish(const MatDesc& d, int cur, int prev, int c, double lambda, int lane, double row, double rowp,
                                         unsigned int tag, bool withhold) {
    const bool finite = __all_sync(0xffffffffu, lane >= c || isfinite(row));
    bad = finite ? bad : 7;
    const double val = finite && lane < c ? row : 0.0;
    const double ic = 1.0 / static_cast<double>(c);
    const int use = prev >= 0 && lane < c && lane != cur && isfinite(rowp) ? 1 : 0;
    const double val_prev = __shfl_sync(0xffffffffu, val, max(prev, 0));   // <H_cur, H_prev>
    const double valp = lane == cur ? val_prev : (use ? rowp : old_prev);
    const bool mine = known(lane, cur, prev, c);
    const double kc = mine ? val * ic : 0.0, kp = mine && prev >= 0 ? valp * ic : 0.0;
    double yc = kc, yp = kp;
#pragma unroll
    for (int k = 0; k < SMAX; ++k) {
      if (k >= c || bad != 0) break;
      if (k == cur || k == prev) continue;
      const double sc = __shfl_sync(0xffffffffu, yc, k);
      yc -= f[k] * sc;
      if (prev >= 0) {
        const double sp = __shfl_sync(0xffffffffu, yp, k);
        yp -= f[k] * sp;
      }
    }
    const double zc = mine ? yc * rdiag : 0.0, zp = mine ? yp * rdiag : 0.0;
    const double ccur = __shfl_sync(0xffffffffu, val, cur) * ic + lambda;
    double xc, xp = 0.0, s_cc;
    if (prev >= 0) {
      const double s_pp = __shfl_sync(0xffffffffu, valp, prev) * ic + lambda - warp_sum(kp * zp);
      const double s_pc = val_prev * ic - warp_sum(kp * zc);
      const double l = s_pc / s_pp;
      s_cc = ccur - warp_sum(kc * zc) - l * s_pc;
      if (bad == 0 && (!(s_pp > 0.0) || !isfinite(s_pp))) bad = isfinite(s_pp) ? 6 : 7;
      xc = 1.0 / s_cc;
      xp = -l * xc;
    } else {
      s_cc = ccur - warp_sum(kc * zc);
      xc = 1.0 / s_cc;
    }
    if (bad == 0 && (!(s_cc > 0.0) || !isfinite(s_cc))) bad = isfinite(s_cc) ? 6 : 7;
    const double x = lane == cur ? xc : (lane == prev ? xp : -(zc * xc + zp * xp));
    const float w = bad == 0 && lane < c ? static_cast<float>(x) : 0.f;
    if (!withhold) publish_weights(d, lane, w, bad != 0, tag);
    d.wsol[lane] = w;
    if (use) {
      d.Kraw[prev * d.s + lane] = rowp;
      d.Kraw[lane * d.s + prev] = rowp;
    }
    __syncwarp();
    // (where the step is flagged the poisoned slot becomes a zero gradient: its Gram row and column vanish)
    if (lane < (bad != 0 ? d.s : c)) {
      d.Kraw[cur * d.s + lane] = bad != 0 ? 0.0 : val;
      d.Kraw[lane * d.s + cur] = bad != 0 ? 0.0 : val;
    }
    if (lane == 0) {
      *d.step_bad = bad != 0 ? 1 : 0;
      if (bad != 0) atomicCAS(d.status, 0, bad);
    }
    __syncwarp();
  }
};

// N~ = sum_j w_j H_j, then the Adam moments as printed in Sec. 2.2 (eps inside the root, no bias
// correction), then u rounded to fp16 for the back-projection GEMM.
template <int SMAX>
__device__ __forceinline__ void combine_tile(const MatDesc& d, int local, int cur, int c, int tile_elems,
                                             const Hyper& hp, const float* wsm /* smem weights */) {
  const long long e0 = static_cast<long long>(local) * tile_elems;
  const long long e1 = (e0 + tile_elems < d.rn) ? e0 + tile_elems : d.rn;
  if (__ldcg(d.step_bad)) {
    float* Hc = d.H + static_cast<long long>(cur) * d.rn;
    for (long long e = e0 + threadIdx.x * 4; e < e1; e += kStreamThreads * 4) {
      *reinterpret_cast<float4*>(Hc + e) = make_float4(0.f, 0.f, 0.f, 0.f);
      *reinterpret_cast<uint2*>(d.u16 + e) = make_uint2(0u, 0u);
    }
    return;
  }
  float w[SMAX];
#pragma unroll
  for (int j = 0; j < SMAX; ++j) w[j] = wsm[j];
  const float b1 = hp.beta1, b2 = hp.beta2, eps = hp.eps;
  for (long long e = e0 + threadIdx.x * 4; e < e1; e += kStreamThreads * 4) {
    float4 n = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < SMAX; ++j) {
      if (j < c) {
        const float4 y = ldg4(d.H + static_cast<long long>(j) * d.rn + e);
        n.x = fmaf(w[j], y.x, n.x);
        n.y = fmaf(w[j], y.y, n.y);
        n.z = fmaf(w[j], y.z, n.z);
        n.w = fmaf(w[j], y.w, n.w);
      }
    }
    float4 m = ldg4(d.m + e), v = ldg4(d.v + e);
    m.x = b1 * m.x + (1.f - b1) * n.x;
    m.y = b1 * m.y + (1.f - b1) * n.y;
    m.z = b1 * m.z + (1.f - b1) * n.z;
    m.w = b1 * m.w + (1.f - b1) * n.w;
    v.x = b2 * v.x + (1.f - b2) * n.x * n.x;
    v.y = b2 * v.y + (1.f - b2) * n.y * n.y;
    v.z = b2 * v.z + (1.f - b2) * n.z * n.z;
    v.w = b2 * v.w + (1.f - b2) * n.w * n.w;
    *reinterpret_cast<float4*>(d.m + e) = m;
    *reinterpret_cast<float4*>(d.v + e) = v;
    const float u0 = m.x / sqrtf(v.x + eps), u1 = m.y / sqrtf(v.y + eps);
    const float u2 = m.z / sqrtf(v.z + eps), u3 = m.w / sqrtf(v.w + eps);
    *reinterpret_cast<uint2*>(d.u16 + e) = pack_f16x4(u0, u1, u2, u3);
  }
}

// ---------------------------------------------------------------- plain (debug) kernels: one launch per phase

template <int SMAX>
__global__ void __launch_bounds__(kStreamThreads) gram_kernel(const MatDesc* mats, const StreamTile* tiles,
                                                              const Ctrl* ctrl) {
  __shared__ double red[(kStreamThreads / 32) * SMAX];
  const StreamTile t = tiles[blockIdx.x];
  const MatDesc& d = mats[t.mat];
  if (d.s == 0) return;
  gram_tile<SMAX>(d, t.local, ring_cur(ctrl, d.s), ring_count(ctrl, d.s), d.te, red);
}

__global__ void __launch_bounds__(128) solve_kernel(const MatDesc* mats, int n_mats, const Ctrl* ctrl,
                                                    const Hyper* hyper) {
  const int warp = threadIdx.x >> 5;
  const int mat = blockIdx.x * 4 + warp;
  if (mat >= n_mats) return;
  const MatDesc& d = mats[mat];
  if (d.s == 0) return;
  const int c = ring_count(ctrl, d.s);
  solve_matrix<kMaxHistory>(d, ring_cur(ctrl, d.s), c, hyper->lambda, gram_row_sum<kMaxHistory>(d, threadIdx.x & 31, c));
}

template <int SMAX>
__global__ void __launch_bounds__(kStreamThreads) combine_kernel(const MatDesc* mats, const StreamTile* tiles,
                                                                 const Ctrl* ctrl, const Hyper* hyper) {
  __shared__ float wsm[kMaxHistory];
  const StreamTile t = tiles[blockIdx.x];
  const MatDesc& d = mats[t.mat];
  if (threadIdx.x < kMaxHistory) wsm[threadIdx.x] = d.wsol[threadIdx.x];
  __syncthreads();
  combine_tile<SMAX>(d, t.local, ring_cur(ctrl, d.s), ring_count(ctrl, d.s), d.te, *hyper, wsm);
}

__global__ void advance_kernel(Ctrl* ctrl) { advance_step(ctrl); }

// Ends a step of which some launches are missing: the next one takes its place in the ring.
__global__ void abandon_kernel(Ctrl* ctrl) { reset_work(ctrl); }

}  // namespace ngalore
