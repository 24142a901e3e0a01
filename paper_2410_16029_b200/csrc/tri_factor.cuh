// R^-1 of a Cholesky QR: from the Gram matrix C = Y^T Y of a basis to the upper triangular R^-1 with (Y R^-1) orthonormal,
// written as two bf16 parts for the tensor-core product Q = Y R^-1.  One CTA per matrix, one launch for all of them.
//
// C's columns are scaled to unit norm (D^-1 C D^-1 + shift I = Lf Lf^T, R^-1 = D^-1 Lf^-T) and Lf is factored and
// inverted at once, by block elimination on [C | I] in blocks of 32: with the inverse of the diagonal block's factor,
//   S_i = C_ik Inv_k^T   for the block rows i below k   (the panel of the factor)
//   S_j = (Inv_k B_kj)^T for the block columns j up to k (row k of Lf^-1, transposed)
//   block (i, j) -= S_i S_j^T for every i > k, j <= i
// where block (i, j) holds C's trailing part for j > k and the accumulated right-hand side B for j <= k: both live in
// one lower triangle of 32 x 32 blocks, and a step is a single symmetric-looking rank-32 update of it.  Row k of Lf^-1 is
// final after its step and goes out as columns of R^-1.
//
// All of it is fp64, the products on the fp64 tensor cores (which here have the rate of the vector units, but need a
// fraction of the instructions and operand reads), also where C comes as fp32 from the tensor cores: scaled, such a matrix has
// a condition of up to 65536, which takes four digits off whatever precision the elimination has.  In fp32 with the
// products as three TF32 products of operands in two parts it took two thirds of the time (58 matrices of 128
// columns 35 us, 84 of 256 86, 156 of up to 512 493), but left R^-1 two to ten times as far from 64 bits as a plain fp32
// factorisation does (the sums of the tensor cores are truncated); fp32 multiply-adds on the vector units take as long as
// fp64 tensor cores and are no closer at 32 and 64 columns.  As it is, the two bf16 parts of the result are what decides.
// One warp factors and inverts the next diagonal block as soon as that has its update, while the others update
// the rest.  The blocks live in shared memory where they fit (up to 160 columns), else in L2.
// It replaced a scaling kernel, a Cholesky factorisation with one CTA per matrix, a recursive triangular inverse (two
// batched products per level) and a conversion: 12 launches, in fp32 125, 310 and 1600 us for 58 matrices of 128 columns, 86 of 256 and
// 156 of up to 512, in fp64 190, 490 and 2900.  As first built 49, 148 and 827 us: a step waited for all of S before the next
// diagonal block had its update, one warp formed that (2 000 cycles) and took 8 000 for its factor, a square root and a
// round through shared memory for each pivot, and the load took one entry at a time.  Now 31, 120 and 708 us: 9 000 cycles a step up
// to 128 columns, two thirds of them the chain of pivots; beyond, the fp64 tensor cores are busy for half of the time, which neither
// more of the blocks in shared memory, nor halves of blocks sent for ahead of time (123 and 760 us), nor columns collected in
// registers (183 and 1070 us) changed.
#pragma once

#include "common.cuh"
#include "gemm_tcgen05.cuh"   // smem_u32

namespace ngalore {

constexpr int kTfThreads = 512;
constexpr int kTfNB = 32;
constexpr int kTfLd = kTfNB + 4;     // row length of the operands in shared memory (fragments without bank conflicts)
constexpr int kTfLdS8 = 12;          // ... and of an 8 x 8 tile

struct FactorMat {
  const float* C32;     // the Gram matrix, L x L, lower triangle valid: fp32 ...
  const double* C64;    // ... or fp64
  double* work;         // blocks of the lower triangle, where they do not fit shared memory
  double* spill;        // rows of S, where they do not fit shared memory
  __nv_bfloat16* Rhi;   // L x ld: high part of R^-1
  __nv_bfloat16* Rlo;
  int L, ld;
  double* R64 = nullptr;         // if set: R^-1 goes here (L x L, fp64) instead; may be C, which is read before
  const int* only_if = nullptr;  // conditional launches: nothing is done where this word is 0
};

// Shared memory without the blocks.
__host__ __device__ inline size_t tf_base_smem(int L, bool s_global) {
  const size_t np = static_cast<size_t>((L + kTfNB - 1) / kTfNB) * kTfNB;
  return sizeof(double) * ((s_global ? 0 : np * kTfLd) + np + 3 * kTfNB * kTfLd + 8 * kTfLdS8);
}
// Rows of S in global memory.
__host__ __device__ inline size_t tf_spill_doubles(int L) { return static_cast<size_t>((L + kTfNB - 1) / kTfNB) * kTfNB * kTfLd; }
__host__ __device__ inline size_t tf_block_bytes(int L) {
  const size_t nb = (L + kTfNB - 1) / kTfNB;
  return sizeof(double) * nb * (nb + 1) / 2 * kTfNB * kTfNB;
}

__device__ __forceinline__ int tf_at(int row, int col) { return row * kTfNB + (col ^ ((row & 3) * 8)); }   // inside a block

// fp64 tensor-core product of 8 x 4 (row = lane / 4, k = lane % 4) and 4 x 8 (k = lane % 4, column = lane / 4); the result's row is
// lane / 4, its columns 2 (lane % 4) and the next.
__device__ __forceinline__ void tf_dmma(double (&c)[2], double a, double b) {
  asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}

// 1 / d and 1 / sqrt(d) for d > 0 far from the ends of the range: the hardware's approximation (20 bits) and one step of
// Householder's third-order iteration, y (1 + e + e^2) with e = 1 - d y and y (1 + e / 2 + 3 e^2 / 8) with e = 1 - d y^2, whose error is
// of the order of e^3.  Measured over 1e-280 .. 1e280, they are off by at most 1.001 and 1.24 units of 2^-53 of the value
// (test_gpu_fp64_scalars.py; half a unit in the last place is up to one of these).  No branches, so that the pivots of a block and their square
// roots overlap.
__device__ __forceinline__ double tf_reciprocal(double d) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  const double e = fma(-d, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double tf_inverse_root(double d) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  const double e = fma(-d * y, y, 1.0);
  return fma(y, e * fma(e, 0.375, 0.5), y);
}

// One warp: Inv = inverse of the Cholesky factor of the 32 x 32 block in W (row length kTfLd, lower triangle), by the elimination
// described at the top once more, in blocks of eight.  The ten 8 x 8 tiles of the lower triangle stay in registers: tile (i, j) is that of
// the matrix until step j and from then on that of the right-hand side, transposed.  So a tile of S is computed from tiles in
// the layout of a result, and is both operands of the update in that layout (the index of summation may be permuted at
// will): only the diagonal tile, which every lane factors for itself, and its inverse go through shared memory (I8).
// A pivot that is not above tiny is replaced by it, so that the factor of a rank-deficient matrix stays finite.
// What bounds it is the chain of 32 pivots, a reciprocal and two multiply-adds each; their square roots are taken beside it.
// (With the block in shared memory and the square roots in the chain 8 000 cycles; column by column, 32 steps, 19 000.)
__device__ __forceinline__ void tf_diagonal(const double* W, double tiny, double* I8, double* Inv, int lane) {
  const int fr = lane >> 2, fk = lane & 3;
  double acc[4][4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j <= i; ++j) {
      const double2 v = *reinterpret_cast<const double2*>(W + (8 * i + fr) * kTfLd + 8 * j + 2 * fk);
      acc[i][j][0] = v.x; acc[i][j][1] = v.y;
    }
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    __syncwarp();
    *reinterpret_cast<double2*>(I8 + fr * kTfLdS8 + 2 * fk) = make_double2(acc[s][s][0], acc[s][s][1]);
    __syncwarp();
    // U D U^T of the tile, then column lane % 8 of D^-1/2 U^-1
    double r[8][8], x[8], d[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j <= i; j += 2) {
        const double2 v = *reinterpret_cast<const double2*>(I8 + i * kTfLdS8 + j);
        r[i][j] = v.x; r[i][j + 1] = v.y;
      }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      d[t] = r[t][t] > tiny ? r[t][t] : tiny;
      const double ip = tf_reciprocal(d[t]);
      double l[8];
#pragma unroll
      for (int i = t + 1; i < 8; ++i) l[i] = r[i][t] * ip;
#pragma unroll
      for (int j = t + 1; j < 8; ++j)
#pragma unroll
        for (int i = j; i < 8; ++i) r[i][j] -= l[i] * r[j][t];
#pragma unroll
      for (int i = t + 1; i < 8; ++i) r[i][t] = l[i];
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = i == (lane & 7) ? 1.0 : 0.0;
#pragma unroll
    for (int t = 0; t < 8; ++t)
#pragma unroll
      for (int i = t + 1; i < 8; ++i) x[i] -= r[i][t] * x[t];
    __syncwarp();
    if (lane < 8) {
#pragma unroll
      for (int t = 0; t < 8; ++t) I8[t * kTfLdS8 + lane] = x[t] * tf_inverse_root(d[t]);
    }
    __syncwarp();
    const double2 b = *reinterpret_cast<const double2*>(I8 + fr * kTfLdS8 + 2 * fk);
    double S[4][2];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (j == s) {
        S[j][0] = I8[2 * fk * kTfLdS8 + fr];
        S[j][1] = I8[(2 * fk + 1) * kTfLdS8 + fr];
      } else {
        double (&from)[2] = j > s ? acc[j][s] : acc[s][j];
        S[j][0] = S[j][1] = 0.0;
        tf_dmma(S[j], from[0], b.x);
        tf_dmma(S[j], from[1], b.y);
      }
    }
    // the tiles right of s first: the next diagonal tile is one of them
#pragma unroll
    for (int i = s + 1; i < 4; ++i)
#pragma unroll
      for (int j = s + 1; j <= i; ++j) {
        tf_dmma(acc[i][j], -S[i][0], S[j][0]);
        tf_dmma(acc[i][j], -S[i][1], S[j][1]);
      }
#pragma unroll
    for (int i = s + 1; i < 4; ++i)
#pragma unroll
      for (int j = 0; j <= s; ++j) {
        if (j == s) acc[i][j][0] = acc[i][j][1] = 0.0;
        tf_dmma(acc[i][j], -S[j][0], S[i][0]);
        tf_dmma(acc[i][j], -S[j][1], S[i][1]);
      }
    // rows 8 s .. 8 s + 7 of the result
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) Inv[(8 * s + 2 * fk + h) * kTfLd + 8 * j + fr] = j <= s ? S[j][h] : 0.0;
  }
}

// Warp 0 is the chain: it factors diagonal block k + 1 (tf_diagonal) while the others do the rest of step k.  Warps 1 to 3, which sit
// on other schedulers, help it to get there: the four form a quarter each of S_(k+1) and of the update of block
// (k + 1, k + 1), before anything else takes the tensor cores.  Then the twelve warps that do not share warp 0's scheduler form the
// rest of S, a quarter of a block row at a time, and update the rest of the matrix; warps 4, 8 and 12, which would hold up the chain
// (a multiply-add of it waits for every product that is under way), join them when it has ended, and so does warp 0.
template <bool S_GLOBAL>
__global__ void __launch_bounds__(kTfThreads, 1) tri_factor_kernel(const FactorMat* mats, int smem_bytes, double shift_scale, int conditional) {
  constexpr int NB = kTfNB, LD = kTfLd, WARPS = kTfThreads / 32;
  extern __shared__ __align__(16) unsigned char tf_smem[];
  __shared__ int counter;
  const FactorMat m = mats[blockIdx.x];
  pdl_begin();
  if (conditional && *m.only_if == 0) return;
  const int L = m.L, nb = (L + NB - 1) / NB, np = nb * NB;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, fr = lane >> 2, fk = lane & 3;
  double* Inv0 = reinterpret_cast<double*>(tf_smem);            // [2][NB][LD]
  double* W = Inv0 + 2 * NB * LD;                           // [NB][LD] the next diagonal block
  double* I8 = W + NB * LD;                                 // [8][kTfLdS8]
  double* rd = I8 + 8 * kTfLdS8;                            // [np] 1 / column norm
  double* Ssh = rd + np;
  double* S = S_GLOBAL ? m.spill : Ssh;    // [np][LD]
  const bool resident = tf_base_smem(L, S_GLOBAL) + tf_block_bytes(L) <= static_cast<size_t>(smem_bytes);
  double* B = resident ? (S_GLOBAL ? Ssh : Ssh + np * LD) : m.work;
  auto block = [&](int i, int j) -> double* { return B + (i * (i + 1) / 2 + j) * (NB * NB); };
  const double tiny = 1e-28, one = 1.0 + (m.C32 != nullptr ? shift_scale * static_cast<double>(L) / 65536.0 : shift_scale);
  if (tid == 0) counter = 0;

  // the scaled matrix (beyond L: the identity), 16 rows of a block at a time; a warp's first ones are under way while the norms are
  // worked out
  {
    double raw[16];
    int i = 0, j = 0, row0 = 0;
    auto fetch = [&](int u) {
      const int b = u >> 1;
      i = static_cast<int>((sqrtf(8.f * b + 1.f) - 1.f) * 0.5f);
      while ((i + 1) * (i + 2) / 2 <= b) ++i;
      while (i * (i + 1) / 2 > b) --i;
      j = b - i * (i + 1) / 2;
      row0 = (u & 1) * 16;
      const int c = min(j * NB + lane, L - 1), r = i * NB + row0;
      auto rows = [&](const auto* p) {
#pragma unroll
        for (int q = 0; q < 16; ++q) raw[q] = static_cast<double>(p[static_cast<long long>(min(r + q, L - 1)) * L + c]);
      };
      if (m.C32 != nullptr) rows(m.C32); else rows(m.C64);
    };
    const int units = nb * (nb + 1);
    if (warp < units) fetch(warp);
    for (int x = tid; x < np; x += kTfThreads) {
      const long long o = static_cast<long long>(min(x, L - 1)) * (L + 1);
      double d = m.C32 != nullptr ? static_cast<double>(m.C32[o]) : m.C64[o];
      if (x >= L) d = 1.0;
      if (!(d > 1e-60)) d = d == d ? 1e-60 : d;          // (a NaN stays one, and the basis check finds it)
      rd[x] = rsqrt(d);
    }
    __syncthreads();
    for (int u = warp; u < units;) {
      const int c = j * NB + lane;
      double* dst = B + (u >> 1) * (NB * NB);
      const double scale = rd[c];
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int row = row0 + q, r = i * NB + row;
        const double v = raw[q] * rd[r] * scale;
        dst[tf_at(row, lane)] = r == c ? (r < L ? one : 1.0) : (r < L && c < r ? v : 0.0);
      }
      u += WARPS;
      if (u < units) fetch(u);
    }
  }
  __syncthreads();

  for (int k = -1; k < nb; ++k) {
    const double* Inv = Inv0 + (k & 1) * NB * LD;
    // rows 8 q .. 8 q + 7 of S_i, and of the block (i, k) of R^-1
    auto form = [&](int i, int q) {
      double acc[4][2];
#pragma unroll
      for (int y = 0; y < 4; ++y) acc[y][0] = acc[y][1] = 0.0;
      if (i != k) {
        const double* blk = i > k ? block(i, k) : block(k, i);
        double a[8];
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) a[kk] = blk[i > k ? tf_at(8 * q + fr, 4 * kk + fk) : tf_at(4 * kk + fk, 8 * q + fr)];
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
#pragma unroll
          for (int y = kk / 2; y < 4; ++y) tf_dmma(acc[y], a[kk], Inv[(8 * y + fr) * LD + 4 * kk + fk]);   // (Inv is lower triangular)
      } else {
#pragma unroll
        for (int y = 0; y < 4; ++y)
#pragma unroll
          for (int h = 0; h < 2; ++h) acc[y][h] = Inv[(8 * y + 2 * fk + h) * LD + 8 * q + fr];
      }
      const int row = i * NB + 8 * q + fr;
      const double scale = rd[row];
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const int kk = 8 * y + 2 * fk, col = k * NB + kk;
        *reinterpret_cast<double2*>(S + row * LD + kk) = make_double2(acc[y][0], acc[y][1]);
        if (m.R64 != nullptr) {
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (row < L && col + h < L) m.R64[static_cast<long long>(row) * L + col + h] = i <= k ? acc[y][h] * scale : 0.0;
        } else if (row < L && col < L) {   // (L is a multiple of 4: the pair is inside together)
          float f[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float v = i <= k ? static_cast<float>(acc[y][h] * scale) : 0.f;
            f[h] = v == v ? fminf(fmaxf(v, -1e30f), 1e30f) : v;
          }
          const __nv_bfloat162 hv = __floats2bfloat162_rn(f[0], f[1]);
          const __nv_bfloat162 lv = __floats2bfloat162_rn(f[0] - __low2float(hv), f[1] - __high2float(hv));
          const long long o = static_cast<long long>(row) * m.ld + col;
          *reinterpret_cast<__nv_bfloat162*>(m.Rhi + o) = hv;
          *reinterpret_cast<__nv_bfloat162*>(m.Rlo + o) = lv;
        }
      }
    };
    if (k + 1 == nb) {   // the last block column of R^-1
      for (int t = warp; t < 4 * nb; t += WARPS) form(t >> 2, t & 3);
      break;
    }
    const int t0 = (k + 1) * (k + 2) / 2, t1 = nb * (nb + 1) / 2, td = t0 + k + 1;   // td: block (k + 1, k + 1)
    const bool beside = (warp & 3) != 0;   // not on the scheduler of the chain
    if (warp < 4) {
      double acc[4][2];
      const double* blk = block(k + 1, k + 1);
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const double2 v = *reinterpret_cast<const double2*>(blk + tf_at(8 * warp + fr, 8 * y + 2 * fk));
        acc[y][0] = v.x; acc[y][1] = v.y;
      }
      if (k >= 0) {
        form(k + 1, warp);
        asm volatile("bar.sync 1, 128;" ::: "memory");
        const double* Sk = S + (k + 1) * NB * LD;
#pragma unroll
        for (int kk = 0; kk < NB; kk += 4) {
          const double a = -Sk[(8 * warp + fr) * LD + kk + fk];
#pragma unroll
          for (int y = 0; y < 4; ++y)
            if (y <= warp) tf_dmma(acc[y], a, Sk[(8 * y + fr) * LD + kk + fk]);
        }
      }
#pragma unroll
      for (int y = 0; y < 4; ++y)
        *reinterpret_cast<double2*>(W + (8 * warp + fr) * LD + 8 * y + 2 * fk) = make_double2(acc[y][0], acc[y][1]);
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (warp == 0) tf_diagonal(W, tiny, I8, Inv0 + ((k + 1) & 1) * NB * LD, lane);
    }
    if (k >= 0) {
      if (beside) {
        for (int t = warp - 1 - (warp >> 2); t < 4 * (nb - 1); t += 12) {
          const int i = t >> 2;
          form(i > k ? i + 1 : i, t & 3);
        }
        asm volatile("bar.arrive 3, %0;" ::"n"(kTfThreads) : "memory");
        asm volatile("bar.sync 2, 384;" ::: "memory");
      } else {
        asm volatile("bar.sync 3, %0;" ::"n"(kTfThreads) : "memory");   // (S is complete, and so is the chain's step)
      }
    }
    // block (i, j) -= S_i S_j^T; block column k starts from zero (its old contents were the panel)
    auto next = [&]() {
      int t = 0;
      if (lane == 0) t = atomicAdd(&counter, 1);
      return __shfl_sync(0xffffffffu, t, 0) + t0;
    };
    for (int t = k >= 0 ? next() : t1; t < t1; t = next()) {
      if (t == td) continue;
      int i = static_cast<int>((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
      while ((i + 1) * (i + 2) / 2 <= t) ++i;
      while (i * (i + 1) / 2 > t) --i;
      const int j = t - i * (i + 1) / 2;
      double* blk = block(i, j);
      double acc[4][4][2];
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const double2 v = j == k ? make_double2(0.0, 0.0) : *reinterpret_cast<const double2*>(blk + tf_at(8 * x + fr, 8 * y + 2 * fk));
          acc[x][y][0] = v.x; acc[x][y][1] = v.y;
        }
      const double *Si = S + i * NB * LD + fr * LD + fk, *Sj = S + j * NB * LD + fr * LD + fk;
#pragma unroll
      for (int k0 = 0; k0 < NB; k0 += 4) {
        double a[4], b[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) { a[x] = -Si[8 * x * LD + k0]; b[x] = Sj[8 * x * LD + k0]; }
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          if (j == k && k0 < 8 * y) continue;     // (S_k is the transpose of Inv, upper triangular)
#pragma unroll
          for (int x = 0; x < 4; ++x)
            if (x >= y || i != j) tf_dmma(acc[x][y], a[x], b[y]);   // (the upper part of a diagonal block is not used)
        }
      }
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y)
          *reinterpret_cast<double2*>(blk + tf_at(8 * x + fr, 8 * y + 2 * fk)) = make_double2(acc[x][y][0], acc[x][y][1]);
    }
    __syncthreads();
    if (tid == 0) counter = 0;   // (read again only after the next barriers)
  }
}

// The same with a cluster of CTAs to a matrix, for wide matrices of which there are few: what takes the time of one CTA beyond the
// chain of diagonal blocks are the fp64 tensor cores of its SM.  Blocks and S live in global memory (L2); rank 0 has the chain, its
// warps 0, 4, 8 and 12 nothing else, and the other warps of all CTAs share the rest of S and of the update.  Two cluster barriers a step:
// S is complete (the chain has arrived by then and waits for it later), and the step has ended.  What other SMs write is read past L1.
constexpr int kTfClusterMax = 4, kTfClusterFrom = 256;
constexpr size_t kTfClusterSmem = 49152;   // without raising the kernel's limit

__device__ __forceinline__ void tf_cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void tf_cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

__global__ void __launch_bounds__(kTfThreads, 1) tri_factor_cluster_kernel(const FactorMat* mats, int cluster, double shift_scale, int conditional) {
  constexpr int NB = kTfNB, LD = kTfLd, WARPS = kTfThreads / 32;
  extern __shared__ __align__(16) unsigned char tf_smem[];
  const int rank = static_cast<int>(blockIdx.x) % cluster;
  const FactorMat m = mats[blockIdx.x / cluster];
  pdl_begin();
  if (conditional && *m.only_if == 0) return;   // (all of the cluster)
  const int L = m.L, nb = (L + NB - 1) / NB, np = nb * NB;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, fr = lane >> 2, fk = lane & 3;
  double* Inv0 = reinterpret_cast<double*>(tf_smem);        // [2][NB][LD]
  double* W = Inv0 + 2 * NB * LD;                           // [NB][LD] the next diagonal block
  double* I8 = W + NB * LD;                                 // [8][kTfLdS8]
  double* Sc = I8 + 8 * kTfLdS8;                            // [NB][LD] S of the next diagonal block's rows, for the chain
  double* rd = Sc + NB * LD;                                // [np] 1 / column norm
  double *S = m.spill, *B = m.work;
  auto block = [&](int i, int j) -> double* { return B + (i * (i + 1) / 2 + j) * (NB * NB); };
  const double tiny = 1e-28, one = 1.0 + (m.C32 != nullptr ? shift_scale * static_cast<double>(L) / 65536.0 : shift_scale);
  const int all = cluster * WARPS, mine = rank * WARPS + warp;   // all warps, and this one's number
  // the warps that share a step: all but those on the scheduler of the chain
  const bool chain_side = rank == 0 && (warp & 3) == 0;
  const int sharers = all - 4, share = rank == 0 ? warp - 1 - (warp >> 2) : mine - 4;

  // the scaled matrix (beyond L: the identity), 16 rows of a block at a time
  for (int x = tid; x < np; x += kTfThreads) {
    const long long o = static_cast<long long>(min(x, L - 1)) * (L + 1);
    double d = m.C32 != nullptr ? static_cast<double>(m.C32[o]) : m.C64[o];
    if (x >= L) d = 1.0;
    if (!(d > 1e-60)) d = d == d ? 1e-60 : d;          // (a NaN stays one, and the basis check finds it)
    rd[x] = rsqrt(d);
  }
  __syncthreads();
  for (int u = mine; u < nb * (nb + 1); u += all) {
    const int b = u >> 1, row0 = (u & 1) * 16;
    int i = static_cast<int>((sqrtf(8.f * b + 1.f) - 1.f) * 0.5f);
    while ((i + 1) * (i + 2) / 2 <= b) ++i;
    while (i * (i + 1) / 2 > b) --i;
    const int j = b - i * (i + 1) / 2;
    double raw[16];
    auto rows = [&](const auto* p) {
#pragma unroll
      for (int q = 0; q < 16; ++q)
        raw[q] = static_cast<double>(p[static_cast<long long>(min(i * NB + row0 + q, L - 1)) * L + min(j * NB + lane, L - 1)]);
    };
    if (m.C32 != nullptr) rows(m.C32); else rows(m.C64);
    const int c = j * NB + lane;
    const double scale = rd[c];
    double* dst = B + b * (NB * NB);
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int row = row0 + q, r = i * NB + row;
      const double v = raw[q] * rd[r] * scale;
      dst[tf_at(row, lane)] = r == c ? (r < L ? one : 1.0) : (r < L && c < r ? v : 0.0);
    }
  }
  tf_cluster_arrive();
  tf_cluster_wait();

  for (int k = -1; k < nb; ++k) {
    double* Inv = Inv0 + (k & 1) * NB * LD;
    if (k >= 0 && rank != 0) {   // the inverse that the chain has left in the first CTA
      uint32_t from;
      asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(from) : "r"(smem_u32(Inv)));
      for (int x = tid; x < NB * LD / 2; x += kTfThreads) {
        double2 v;
        asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(from + 16u * x) : "memory");
        reinterpret_cast<double2*>(Inv)[x] = v;
      }
      __syncthreads();
    }
    // rows 8 q .. 8 q + 7 of S_i, and of the block (i, k) of R^-1
    auto form = [&](int i, int q, bool for_chain) {
      double acc[4][2];
#pragma unroll
      for (int y = 0; y < 4; ++y) acc[y][0] = acc[y][1] = 0.0;
      if (i != k) {
        const double* blk = i > k ? block(i, k) : block(k, i);
        double a[8];
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) a[kk] = __ldcg(blk + (i > k ? tf_at(8 * q + fr, 4 * kk + fk) : tf_at(4 * kk + fk, 8 * q + fr)));
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
#pragma unroll
          for (int y = kk / 2; y < 4; ++y) tf_dmma(acc[y], a[kk], Inv[(8 * y + fr) * LD + 4 * kk + fk]);   // (Inv is lower triangular)
      } else {
#pragma unroll
        for (int y = 0; y < 4; ++y)
#pragma unroll
          for (int h = 0; h < 2; ++h) acc[y][h] = Inv[(8 * y + 2 * fk + h) * LD + 8 * q + fr];
      }
      const int row = i * NB + 8 * q + fr;
      const double scale = rd[row];
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const int kk = 8 * y + 2 * fk, col = k * NB + kk;
        *reinterpret_cast<double2*>(S + row * LD + kk) = make_double2(acc[y][0], acc[y][1]);
        if (for_chain) *reinterpret_cast<double2*>(Sc + (8 * q + fr) * LD + kk) = make_double2(acc[y][0], acc[y][1]);
        if (m.R64 != nullptr) {
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (row < L && col + h < L) m.R64[static_cast<long long>(row) * L + col + h] = i <= k ? acc[y][h] * scale : 0.0;
        } else if (row < L && col < L) {   // (L is a multiple of 4: the pair is inside together)
          float f[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float v = i <= k ? static_cast<float>(acc[y][h] * scale) : 0.f;
            f[h] = v == v ? fminf(fmaxf(v, -1e30f), 1e30f) : v;
          }
          const __nv_bfloat162 hv = __floats2bfloat162_rn(f[0], f[1]);
          const __nv_bfloat162 lv = __floats2bfloat162_rn(f[0] - __low2float(hv), f[1] - __high2float(hv));
          const long long o = static_cast<long long>(row) * m.ld + col;
          *reinterpret_cast<__nv_bfloat162*>(m.Rhi + o) = hv;
          *reinterpret_cast<__nv_bfloat162*>(m.Rlo + o) = lv;
        }
      }
    };
    if (k + 1 == nb) {   // the last block column of R^-1
      for (int t = mine; t < 4 * nb; t += all) form(t >> 2, t & 3, false);
      break;
    }
    if (rank == 0 && warp < 4) {
      double acc[4][2];
      const double* blk = block(k + 1, k + 1);
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const double2 v = __ldcg(reinterpret_cast<const double2*>(blk + tf_at(8 * warp + fr, 8 * y + 2 * fk)));
        acc[y][0] = v.x; acc[y][1] = v.y;
      }
      if (k >= 0) {
        form(k + 1, warp, true);
        asm volatile("bar.sync 1, 128;" ::: "memory");
#pragma unroll
        for (int kk = 0; kk < NB; kk += 4) {
          const double a = -Sc[(8 * warp + fr) * LD + kk + fk];
#pragma unroll
          for (int y = 0; y < 4; ++y)
            if (y <= warp) tf_dmma(acc[y], a, Sc[(8 * y + fr) * LD + kk + fk]);
        }
      }
#pragma unroll
      for (int y = 0; y < 4; ++y)
        *reinterpret_cast<double2*>(W + (8 * warp + fr) * LD + 8 * y + 2 * fk) = make_double2(acc[y][0], acc[y][1]);
      asm volatile("bar.sync 1, 128;" ::: "memory");
    }
    if (chain_side) {
      tf_cluster_arrive();
      if (warp == 0) tf_diagonal(W, tiny, I8, Inv0 + ((k + 1) & 1) * NB * LD, lane);
      tf_cluster_wait();
    } else {
      if (k >= 0)
        for (int t = share; t < 4 * (nb - 1); t += sharers) form((t >> 2) > k ? (t >> 2) + 1 : t >> 2, t & 3, false);
      tf_cluster_arrive();
      tf_cluster_wait();
      // block (i, j) -= S_i S_j^T; block column k starts from zero (its old contents were the panel)
      const int t0 = (k + 1) * (k + 2) / 2, t1 = nb * (nb + 1) / 2, td = t0 + k + 1;   // td: block (k + 1, k + 1)
      for (int t = k >= 0 ? t0 + share : t1; t < t1; t += sharers) {
        if (t == td) continue;
        int i = static_cast<int>((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
        while ((i + 1) * (i + 2) / 2 <= t) ++i;
        while (i * (i + 1) / 2 > t) --i;
        const int j = t - i * (i + 1) / 2;
        double* blk = block(i, j);
        double acc[4][4][2];
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            const double2 v = j == k ? make_double2(0.0, 0.0) : __ldcg(reinterpret_cast<const double2*>(blk + tf_at(8 * x + fr, 8 * y + 2 * fk)));
            acc[x][y][0] = v.x; acc[x][y][1] = v.y;
          }
        const double *Si = S + i * NB * LD + fr * LD + fk, *Sj = S + j * NB * LD + fr * LD + fk;
#pragma unroll
        for (int k0 = 0; k0 < NB; k0 += 4) {
          double a[4], b[4];
#pragma unroll
          for (int x = 0; x < 4; ++x) { a[x] = -__ldcg(Si + 8 * x * LD + k0); b[x] = __ldcg(Sj + 8 * x * LD + k0); }
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            if (j == k && k0 < 8 * y) continue;     // (S_k is the transpose of Inv, upper triangular)
#pragma unroll
            for (int x = 0; x < 4; ++x)
              if (x >= y || i != j) tf_dmma(acc[x][y], a[x], b[y]);   // (the upper part of a diagonal block is not used)
          }
        }
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y)
            *reinterpret_cast<double2*>(blk + tf_at(8 * x + fr, 8 * y + 2 * fk)) = make_double2(acc[x][y][0], acc[x][y][1]);
      }
    }
    tf_cluster_arrive();
    tf_cluster_wait();
  }
  // (the first CTA stays until nobody reads its shared memory any more)
  tf_cluster_arrive();
  tf_cluster_wait();
}

constexpr int kTfSmemLimit = 232448 - 256;   // (the kernel has 128 bytes of its own)

inline size_t tf_cluster_smem(int l_max) {
  return sizeof(double) * (4 * kTfNB * kTfLd + 8 * kTfLdS8 + static_cast<size_t>((l_max + kTfNB - 1) / kTfNB) * kTfNB);
}
inline void tf_cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& attr, int n, int cluster, int l_max) {
  cfg.gridDim = n * cluster;
  cfg.blockDim = kTfThreads;
  cfg.dynamicSmemBytes = tf_cluster_smem(l_max);
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = cluster; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
}
// CTAs that factor a matrix together, for n matrices, the widest l_max wide: four or two where all matrices still go at once (a cluster
// has its SMs in one group of them, so that 148 SMs hold fewer than 37 clusters of four; 37 matrices of 480 columns in two waves 8.4 ms a
// refresh, with one CTA each 7.8) and are so wide that it pays: refresh, one CTA / a cluster, nine matrices of 196 columns 2.24 / 2.23
// ms, of 256 3.06 / 2.97, of 416 5.24 / 4.19, three of 512 7.13 / 4.80; pairs, 74 of 256 4.40 / 4.40, of 328 6.36 / 6.11, 60 of 480 8.99 / 8.21.
// Beyond 1440 columns the norms of a matrix's columns no longer fit beside the blocks in the 48 KB that every kernel has, and one CTA takes it as
// before: what a cluster would give there has not been measured.
inline int tf_cluster(int n, int l_max) {
  if (l_max <= kTfClusterFrom || tf_cluster_smem(l_max) > kTfClusterSmem) return 1;
  for (int c = kTfClusterMax; c > 1; c /= 2) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr{};
    tf_cluster_config(cfg, attr, n, c, l_max);
    int fit = 0;
    if (cudaOccupancyMaxActiveClusters(&fit, tri_factor_cluster_kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    if (n <= fit) return c;
  }
  return 1;
}

// Factor n matrices, the widest l_max wide (widest first in the list: CTAs are handed out in order).  shift_scale: what
// is added to the unit diagonal, for fp32 matrices in units of L / 65536.  dependent: launched as a programmatic dependent.  cluster: CTAs to a
// matrix (tf_cluster; more than one: work and spill hold all blocks and rows of S of every matrix).
inline cudaError_t tri_factor_launch(const FactorMat* d_mats, int n, int l_max, double shift_scale, cudaStream_t stream,
                                     int64_t* launches, bool conditional = false, bool dependent = false, int cluster = 1) {
  // as much shared memory as the widest matrix that fits with its blocks, and at least what the widest needs without
  size_t smem = tf_base_smem(l_max, false);
  const bool s_global = smem > static_cast<size_t>(kTfSmemLimit);
  if (s_global) smem = tf_base_smem(l_max, true);
  for (int l = l_max; l > 0; l -= 4) {
    const size_t need = tf_base_smem(l, s_global) + tf_block_bytes(l);
    if (need <= static_cast<size_t>(kTfSmemLimit)) { smem = need > smem ? need : smem; break; }
  }
  if (cluster > 1) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[2]{};
    tf_cluster_config(cfg, attr[0], n, cluster, l_max);
    cfg.stream = stream;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 2 : 1;
    *launches += 1;
    return cudaLaunchKernelEx(&cfg, tri_factor_cluster_kernel, d_mats, cluster, shift_scale, conditional ? 1 : 0);
  }
  // (the limit to its largest value, since it belongs to the process and not to one state, and here, so that only a kernel
  // that is launched gets loaded)
  auto run = [&](auto kernel) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTfSmemLimit);
    if (e != cudaSuccess) return e;
    launch_step(dependent, kernel, n, kTfThreads, smem, stream, d_mats, static_cast<int>(smem), shift_scale, conditional ? 1 : 0);
    *launches += 1;
    return cudaGetLastError();
  };
  return s_global ? run(tri_factor_kernel<true>) : run(tri_factor_kernel<false>);
}

}  // namespace ngalore
