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
// One warp factors and inverts the next diagonal block as soon as that has its update, while the other fifteen update
// the rest.  The blocks live in shared memory where they fit (up to 160 columns), else in L2.
// It replaced a scaling kernel, a Cholesky factorisation with one CTA per matrix, a recursive triangular inverse (two
// batched products per level) and a conversion: 12 launches.  Measured per orthonormalisation: 58 matrices of 128 columns 50 us,
// 86 of 256 150, 156 of up to 512 840 (those launches: in fp32 125, 310 and 1600 us, in fp64 190, 490 and 2900).  What is left
// is the chain of diagonal blocks up to 256 columns (8 000 cycles each) and the fp64 tensor cores' rate beyond.
#pragma once

#include "common.cuh"
#include "gemm_tcgen05.cuh"   // smem_u32

namespace ngalore {

constexpr int kTfThreads = 512;
constexpr int kTfNB = 32;
constexpr int kTfLd = kTfNB + 4;     // row length of the operands in shared memory (fragments without bank conflicts)
constexpr int kTfLdW = kTfNB + 8;    // row length of the diagonal block's work space
constexpr int kTfLdS8 = 12;          // ... and of its operands

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
  return sizeof(double) * ((s_global ? 0 : np * kTfLd) + np + kTfNB * (2 * kTfLd + kTfLdW + kTfLdS8) + 64);
}
// Rows of S in global memory.
__host__ __device__ inline size_t tf_spill_doubles(int L) { return static_cast<size_t>((L + kTfNB - 1) / kTfNB) * kTfNB * kTfLd; }
__host__ __device__ inline size_t tf_block_bytes(int L) {
  const size_t nb = (L + kTfNB - 1) / kTfNB;
  return sizeof(double) * nb * (nb + 1) / 2 * kTfNB * kTfNB;
}

// acc[mt][nt][h] (entry (8 mt + lane / 4, 8 nt + 2 (lane % 4) + h) of a 32 x 32 block) += left(row, k) right(col, k),
// summed over K values of k.
template <int K, typename FL, typename FR>
__device__ __forceinline__ void tf_product(double (&acc)[4][4][2], FL left, FR right, int fr, int fk) {
#pragma unroll
  for (int k0 = 0; k0 < K; k0 += 4) {
    double a[4], b[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) a[m] = left(8 * m + fr, k0 + fk);
#pragma unroll
    for (int n = 0; n < 4; ++n) b[n] = right(8 * n + fr, k0 + fk);
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int n = 0; n < 4; ++n)
        asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                     : "+d"(acc[m][n][0]), "+d"(acc[m][n][1]) : "d"(a[m]), "d"(b[n]));
  }
}

__device__ __forceinline__ int tf_at(int row, int col) { return row * kTfNB + (col ^ ((row & 3) * 8)); }   // inside a block

// Eight consecutive numbers.
__device__ __forceinline__ void tf_load8(const double* p, double (&v)[8]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const double2 x = reinterpret_cast<const double2*>(p)[q];
    v[2 * q] = x.x; v[2 * q + 1] = x.y;
  }
}
__device__ __forceinline__ void tf_store8(double* p, const double (&v)[8]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) reinterpret_cast<double2*>(p)[q] = make_double2(v[2 * q], v[2 * q + 1]);
}

// One warp: Inv = inverse of the Cholesky factor of the 32 x 32 block at blk, by the elimination described at the top
// once more, in blocks of eight.  A pivot that is not above tiny is replaced by it, so that the factor of a
// rank-deficient matrix stays finite.  (Column by column, 32 steps of shuffle, square root, scaling and update, it took
// 19 000 cycles and bounded the kernel.)
__device__ __forceinline__ void tf_diagonal(const double* blk, double tiny, double* W, double* S8, double* I8, double* Inv, int lane) {
  const int fr = lane >> 2, fk = lane & 3;
  {
    double r[kTfNB];
#pragma unroll
    for (int q = 0; q < kTfNB; ++q) r[q] = blk[tf_at(q, lane)];
#pragma unroll
    for (int q = 0; q < kTfNB; ++q) W[q * kTfLdW + lane] = r[q];
  }
  __syncwarp();
#pragma unroll 1
  for (int c0 = 0; c0 < kTfNB; c0 += 8) {
    // the 8 x 8 block: every lane computes all of its factor (shuffles would double the length of the chain), then one
    // column of the inverse
    {
      double r[8][8], x[8], inv[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) tf_load8(W + (c0 + i) * kTfLdW + c0, r[i]);
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        double d = r[t][t];
        if (!(d > tiny)) d = tiny;
        inv[t] = rsqrt(d);
#pragma unroll
        for (int i = t + 1; i < 8; ++i) r[i][t] *= inv[t];
#pragma unroll
        for (int j = t + 1; j < 8; ++j)
#pragma unroll
          for (int i = j; i < 8; ++i) r[i][j] -= r[i][t] * r[j][t];
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = i == (lane & 7) ? 1.0 : 0.0;
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        x[t] *= inv[t];
#pragma unroll
        for (int i = t + 1; i < 8; ++i) x[i] -= r[i][t] * x[t];
      }
      if (lane < 8) {
#pragma unroll
        for (int t = 0; t < 8; ++t) I8[t * 8 + lane] = x[t];
      }
    }
    __syncwarp();
    // the operands, lane = row, and rows c0 .. c0 + 7 of the result
    {
      double v[8], o[8];
      if (lane >= c0 + 8) {
        tf_load8(W + lane * kTfLdW + c0, v);
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = lane < c0 ? W[(c0 + q) * kTfLdW + lane] : (lane == c0 + q ? 1.0 : 0.0);
      }
#pragma unroll
      for (int n = 0; n < 8; ++n) {
        double row[8];
        tf_load8(I8 + n * 8, row);
        o[n] = 0.0;
#pragma unroll
        for (int q = 0; q <= n; ++q) o[n] += row[q] * v[q];
        Inv[(c0 + n) * kTfLd + lane] = lane < c0 + 8 ? o[n] : 0.0;
      }
      tf_store8(S8 + lane * kTfLdS8, o);
      __syncwarp();
      if (lane >= c0 + 8) {
        const double zero[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        tf_store8(W + lane * kTfLdW + c0, zero);
      }
    }
    __syncwarp();
    if (c0 + 8 == kTfNB) break;
    // (rows up to c0 + 7 are not read any more: they may take part)
    double acc[4][4][2];
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y)
#pragma unroll
        for (int h = 0; h < 2; ++h) acc[x][y][h] = W[(8 * x + fr) * kTfLdW + 8 * y + 2 * fk + h];
    tf_product<8>(acc, [&](int r, int kk) { return -S8[r * kTfLdS8 + kk]; }, [&](int n, int kk) { return S8[n * kTfLdS8 + kk]; }, fr, fk);
    __syncwarp();
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y)
#pragma unroll
        for (int h = 0; h < 2; ++h) W[(8 * x + fr) * kTfLdW + 8 * y + 2 * fk + h] = acc[x][y][h];
    __syncwarp();
  }
}

template <bool S_GLOBAL>
__global__ void __launch_bounds__(kTfThreads, 1) tri_factor_kernel(const FactorMat* mats, int smem_bytes, double shift_scale, int conditional) {
  constexpr int NB = kTfNB, LD = kTfLd, WARPS = kTfThreads / 32;
  extern __shared__ __align__(16) unsigned char tf_smem[];
  __shared__ int counter;
  const FactorMat m = mats[blockIdx.x];
  if (conditional && *m.only_if == 0) return;
  const int L = m.L, nb = (L + NB - 1) / NB, np = nb * NB;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, fr = lane >> 2, fk = lane & 3;
  double* Inv0 = reinterpret_cast<double*>(tf_smem);            // [2][NB][LD]
  double* W = Inv0 + 2 * NB * LD;                           // work space of the diagonal block: [NB][kTfLdW],
  double* S8 = W + NB * kTfLdW;                             // [NB][kTfLdS8],
  double* I8 = S8 + NB * kTfLdS8;                           // [8][8]
  double* rd = I8 + 64;                                     // [np] 1 / column norm
  double* Ssh = rd + np;
  double* S = S_GLOBAL ? m.spill : Ssh;    // [np][LD]
  const bool resident = tf_base_smem(L, S_GLOBAL) + tf_block_bytes(L) <= static_cast<size_t>(smem_bytes);
  double* B = resident ? (S_GLOBAL ? Ssh : Ssh + np * LD) : m.work;
  auto gram = [&](int r, int c) {
    const long long o = static_cast<long long>(r) * L + c;
    return m.C32 != nullptr ? static_cast<double>(m.C32[o]) : m.C64[o];
  };
  auto block = [&](int i, int j) -> double* { return B + (i * (i + 1) / 2 + j) * (NB * NB); };
  const double tiny = 1e-28, one = 1.0 + (m.C32 != nullptr ? shift_scale * static_cast<double>(L) / 65536.0 : shift_scale);

  for (int i = tid; i < np; i += kTfThreads) {
    double d = i < L ? gram(i, i) : 1.0;
    if (!(d > 1e-60)) d = d == d ? 1e-60 : d;          // (a NaN stays one, and the basis check finds it)
    rd[i] = rsqrt(d);
  }
  __syncthreads();
  // the scaled matrix (beyond L: the identity)
  for (int b = warp; b < nb * (nb + 1) / 2; b += WARPS) {
    int i = static_cast<int>((sqrtf(8.f * b + 1.f) - 1.f) * 0.5f);
    while ((i + 1) * (i + 2) / 2 <= b) ++i;
    while (i * (i + 1) / 2 > b) --i;
    const int j = b - i * (i + 1) / 2;
    const int c = j * NB + lane;
    double* dst = B + b * (NB * NB);
#pragma unroll 1
    for (int row0 = 0; row0 < NB; row0 += 16) {
      double raw[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) raw[q] = gram(min(i * NB + row0 + q, L - 1), min(c, L - 1));
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int row = row0 + q, r = i * NB + row;
        const double v = raw[q] * rd[r] * rd[c];
        dst[tf_at(row, lane)] = r == c ? (r < L ? one : 1.0) : (r < L && c < r ? v : 0.0);
      }
    }
  }
  if (tid == 0) counter = 0;
  __syncthreads();

  for (int k = -1; k < nb; ++k) {
    const double* Inv = Inv0 + (k & 1) * NB * LD;
    // S, and block column k of R^-1
    for (int i = warp; i < nb && k >= 0; i += WARPS) {
      double acc[4][4][2];
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x][y][0] = acc[x][y][1] = 0.0;
      auto right = [&](int n, int kk) { return Inv[n * LD + kk]; };
      if (i > k) {
        const double* blk = block(i, k);
        tf_product<NB>(acc, [&](int r, int kk) { return blk[tf_at(r, kk)]; }, right, fr, fk);
      } else if (i < k) {
        const double* blk = block(k, i);
        tf_product<NB>(acc, [&](int r, int kk) { return blk[tf_at(kk, r)]; }, right, fr, fk);
      } else {
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y)
#pragma unroll
            for (int h = 0; h < 2; ++h) acc[x][y][h] = Inv[(8 * y + 2 * fk + h) * LD + 8 * x + fr];
      }
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int row = i * NB + 8 * x + fr;
        const double scale = rd[row];
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const int kk = 8 * y + 2 * fk, col = k * NB + kk;
          S[row * LD + kk] = acc[x][y][0];
          S[row * LD + kk + 1] = acc[x][y][1];
          if (m.R64 != nullptr) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
              if (row < L && col + h < L) m.R64[static_cast<long long>(row) * L + col + h] = i <= k ? acc[x][y][h] * scale : 0.0;
          } else if (row < L && col < L) {   // (L is a multiple of 4: the pair is inside together)
            float f[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const float v = i <= k ? static_cast<float>(acc[x][y][h] * scale) : 0.f;
              f[h] = v == v ? fminf(fmaxf(v, -1e30f), 1e30f) : v;
            }
            const __nv_bfloat162 hv = __floats2bfloat162_rn(f[0], f[1]);
            const __nv_bfloat162 lv = __floats2bfloat162_rn(f[0] - __low2float(hv), f[1] - __high2float(hv));
            const long long o = static_cast<long long>(row) * m.ld + col;
            *reinterpret_cast<__nv_bfloat162*>(m.Rhi + o) = hv;
            *reinterpret_cast<__nv_bfloat162*>(m.Rlo + o) = lv;
          }
        }
      }
    }
    __syncthreads();
    if (k + 1 == nb) break;
    // block (i, j) -= S_i S_j^T; block column k starts from zero (its old contents were the panel).  Warp 0 begins with
    // the next diagonal block, the others take the rest in order.
    const int t0 = (k + 1) * (k + 2) / 2, t1 = nb * (nb + 1) / 2, td = t0 + k + 1;   // td: block (k + 1, k + 1)
    auto next = [&]() {
      int t = 0;
      if (lane == 0) t = atomicAdd(&counter, 1);
      return __shfl_sync(0xffffffffu, t, 0) + t0;
    };
    // (warps 4, 8 and 12 sit on the scheduler of warp 0, whose diagonal block the next step waits for: they rest
    // until it is done)
    if (warp != 0 && (warp & 3) == 0) asm volatile("bar.sync 1, 128;" ::: "memory");
    int t = warp == 0 ? td : (k >= 0 ? next() : t1);
    bool first = warp == 0;
    while (t < t1) {
      if (k >= 0 && (first || t != td)) {
        int i = static_cast<int>((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
        while ((i + 1) * (i + 2) / 2 <= t) ++i;
        while (i * (i + 1) / 2 > t) --i;
        const int j = t - i * (i + 1) / 2;
        double* blk = block(i, j);
        double acc[4][4][2];
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y)
#pragma unroll
            for (int h = 0; h < 2; ++h) acc[x][y][h] = j == k ? 0.0 : blk[tf_at(8 * x + fr, 8 * y + 2 * fk) + h];
        const double *Si = S + i * NB * LD, *Sj = S + j * NB * LD;
        tf_product<NB>(acc, [&](int r, int kk) { return -Si[r * LD + kk]; }, [&](int n, int kk) { return Sj[n * LD + kk]; }, fr, fk);
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y)
#pragma unroll
            for (int h = 0; h < 2; ++h) blk[tf_at(8 * x + fr, 8 * y + 2 * fk) + h] = acc[x][y][h];
      }
      if (first) {
        __syncwarp();
        tf_diagonal(block(k + 1, k + 1), tiny, W, S8, I8, Inv0 + ((k + 1) & 1) * NB * LD, lane);
        first = false;
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (k < 0) break;
      }
      t = next();
    }
    __syncthreads();
    if (tid == 0) counter = 0;   // (read again only after the next barrier)
  }
}

constexpr int kTfSmemLimit = 232448 - 256;   // (the kernel has 128 bytes of its own)

// Factor n matrices, the widest l_max wide (widest first in the list: CTAs are handed out in order).  shift_scale: what
// is added to the unit diagonal, for fp32 matrices in units of L / 65536.
inline cudaError_t tri_factor_launch(const FactorMat* d_mats, int n, int l_max, double shift_scale, cudaStream_t stream,
                                     int64_t* launches, bool conditional = false) {
  // as much shared memory as the widest matrix that fits with its blocks, and at least what the widest needs without
  size_t smem = tf_base_smem(l_max, false);
  const bool s_global = smem > static_cast<size_t>(kTfSmemLimit);
  if (s_global) smem = tf_base_smem(l_max, true);
  for (int l = l_max; l > 0; l -= 4) {
    const size_t need = tf_base_smem(l, s_global) + tf_block_bytes(l);
    if (need <= static_cast<size_t>(kTfSmemLimit)) { smem = need > smem ? need : smem; break; }
  }
  // (the limit to its largest value, since it belongs to the process and not to one state, and here, so that only a kernel
  // that is launched gets loaded)
  auto run = [&](auto kernel) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTfSmemLimit);
    if (e != cudaSuccess) return e;
    kernel<<<n, kTfThreads, smem, stream>>>(d_mats, static_cast<int>(smem), shift_scale, conditional ? 1 : 0);
    *launches += 1;
    return cudaGetLastError();
  };
  return s_global ? run(tri_factor_kernel<true>) : run(tri_factor_kernel<false>);
}

}  // namespace ngalore
