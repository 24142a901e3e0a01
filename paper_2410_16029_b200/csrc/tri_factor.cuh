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
// All products run on the tensor cores: fp64 matrices on the fp64 ones (which here have the rate of the vector units,
// but need a fraction of the instructions and operand reads), fp32 matrices as three TF32 products of operands split in
// two parts of eleven bits (2^-21 of a product is lost, with the Gram matrix good to 2^-17).  One warp factors and
// inverts the next diagonal block as soon as that has its update, while the other fifteen update the rest.  The
// blocks live in shared memory where they fit (fp32: up to 256 columns, fp64: up to 160), else in L2.
// It replaced a scaling kernel, a Cholesky factorisation with one CTA per matrix, a recursive triangular inverse (two
// batched products per level) and a conversion: 12 launches.  Measured per orthonormalisation, fp32: 58 matrices of 128
// columns 125 -> 36 us, 84 of 256 310 -> 89 us, 156 of up to 512 1600 -> 493 us; the fp64 pass of the same sets 190 -> 52,
// 490 -> 150 and 2900 -> 900 us.  What is left is the chain of diagonal blocks up to 256 columns (6 400 cycles each) and
// the tensor cores' rate for TF32 beyond.
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
  const void* C;        // L x L (T), lower triangle valid
  void* work;           // blocks of the lower triangle, where they do not fit shared memory
  void* spill;          // rows of S, where they do not fit shared memory
  __nv_bfloat16* Rhi;   // L x ld: high part of R^-1
  __nv_bfloat16* Rlo;
  int L, ld;
  double* R64 = nullptr;         // if set: R^-1 goes here (L x L, fp64) instead; may be C, which is read before
  const int* only_if = nullptr;  // conditional launches: nothing is done where this word is 0
};

// Shared memory without the blocks.
template <typename T>
__host__ __device__ inline size_t tf_base_smem(int L, bool s_global) {
  const size_t np = static_cast<size_t>((L + kTfNB - 1) / kTfNB) * kTfNB;
  return sizeof(T) * ((s_global ? 0 : np * kTfLd) + np + kTfNB * (2 * kTfLd + kTfLdW + kTfLdS8) + 64);
}
// Rows of S in global memory.
__host__ __device__ inline size_t tf_spill_doubles(int L) { return static_cast<size_t>((L + kTfNB - 1) / kTfNB) * kTfNB * kTfLd; }
template <typename T>
__host__ __device__ inline size_t tf_block_bytes(int L) {
  const size_t nb = (L + kTfNB - 1) / kTfNB;
  return sizeof(T) * nb * (nb + 1) / 2 * kTfNB * kTfNB;
}

__device__ __forceinline__ void tf_mma(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
__device__ __forceinline__ void tf_split(float x, uint32_t& hi, uint32_t& lo) {
  hi = __float_as_uint(x) & 0xffffe000u;
  lo = __float_as_uint(x - __uint_as_float(hi));
}

// acc[mt][nt][h] (entry (8 mt + lane / 4, 8 nt + 2 (lane % 4) + h) of a 32 x 32 block) += left(row, k) right(col, k),
// summed over K values of k.
template <int K, typename FL, typename FR>
__device__ __forceinline__ void tf_product(float (&acc)[4][4][2], FL left, FR right, int fr, int fk) {
#pragma unroll
  for (int k0 = 0; k0 < K; k0 += 8) {
    uint32_t ah[2][4], al[2][4], bh[4][2], bl[4][2];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int e = 0; e < 4; ++e) tf_split(left(16 * m + 8 * (e & 1) + fr, k0 + 4 * (e >> 1) + fk), ah[m][e], al[m][e]);
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int e = 0; e < 2; ++e) tf_split(right(8 * n + fr, k0 + 4 * e + fk), bh[n][e], bl[n][e]);
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        float c[4] = {acc[2 * m][n][0], acc[2 * m][n][1], acc[2 * m + 1][n][0], acc[2 * m + 1][n][1]};
        tf_mma(c, al[m], bh[n]);
        tf_mma(c, ah[m], bl[n]);
        tf_mma(c, ah[m], bh[n]);
        acc[2 * m][n][0] = c[0]; acc[2 * m][n][1] = c[1]; acc[2 * m + 1][n][0] = c[2]; acc[2 * m + 1][n][1] = c[3];
      }
  }
}
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
// 1 / sqrt(x): the approximation and one Newton step (fp32, to about one unit in the last place), the function (fp64).
__device__ __forceinline__ float tf_rsqrt(float x) {
  const float y = rsqrtf(x);
  return y * (1.5f - 0.5f * x * y * y);
}
__device__ __forceinline__ double tf_rsqrt(double x) { return rsqrt(x); }

template <typename T>
struct alignas(16) TfVec { T v[16 / sizeof(T)]; };
// Eight consecutive numbers.
template <typename T>
__device__ __forceinline__ void tf_load8(const T* p, T (&v)[8]) {
  constexpr int N = 16 / sizeof(T);
#pragma unroll
  for (int q = 0; q < 8 / N; ++q) {
    const TfVec<T> x = reinterpret_cast<const TfVec<T>*>(p)[q];
#pragma unroll
    for (int y = 0; y < N; ++y) v[q * N + y] = x.v[y];
  }
}
template <typename T>
__device__ __forceinline__ void tf_store8(T* p, const T (&v)[8]) {
  constexpr int N = 16 / sizeof(T);
#pragma unroll
  for (int q = 0; q < 8 / N; ++q) {
    TfVec<T> x;
#pragma unroll
    for (int y = 0; y < N; ++y) x.v[y] = v[q * N + y];
    reinterpret_cast<TfVec<T>*>(p)[q] = x;
  }
}

// One warp: Inv = inverse of the Cholesky factor of the 32 x 32 block at blk, by the elimination described at the top
// once more, in blocks of eight.  A pivot that is not above tiny is replaced by it, so that the factor of a
// rank-deficient matrix stays finite.  (Column by column, 32 steps of shuffle, square root, scaling and update, it took
// 19 000 cycles and bounded the kernel.)
template <typename T>
__device__ __forceinline__ void tf_diagonal(const T* blk, T tiny, T* W, T* S8, T* I8, T* Inv, int lane) {
  const int fr = lane >> 2, fk = lane & 3;
  {
    T r[kTfNB];
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
      T r[8][8], x[8], inv[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) tf_load8(W + (c0 + i) * kTfLdW + c0, r[i]);
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        T d = r[t][t];
        if (!(d > tiny)) d = tiny;
        inv[t] = tf_rsqrt(d);
#pragma unroll
        for (int i = t + 1; i < 8; ++i) r[i][t] *= inv[t];
#pragma unroll
        for (int j = t + 1; j < 8; ++j)
#pragma unroll
          for (int i = j; i < 8; ++i) r[i][j] -= r[i][t] * r[j][t];
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = i == (lane & 7) ? T(1) : T(0);
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
      T v[8], o[8];
      if (lane >= c0 + 8) {
        tf_load8(W + lane * kTfLdW + c0, v);
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = lane < c0 ? W[(c0 + q) * kTfLdW + lane] : (lane == c0 + q ? T(1) : T(0));
      }
#pragma unroll
      for (int n = 0; n < 8; ++n) {
        T row[8];
        tf_load8(I8 + n * 8, row);
        o[n] = T(0);
#pragma unroll
        for (int q = 0; q <= n; ++q) o[n] += row[q] * v[q];
        Inv[(c0 + n) * kTfLd + lane] = lane < c0 + 8 ? o[n] : T(0);
      }
      tf_store8(S8 + lane * kTfLdS8, o);
      __syncwarp();
      if (lane >= c0 + 8) {
        const T zero[8] = {T(0), T(0), T(0), T(0), T(0), T(0), T(0), T(0)};
        tf_store8(W + lane * kTfLdW + c0, zero);
      }
    }
    __syncwarp();
    if (c0 + 8 == kTfNB) break;
    // (rows up to c0 + 7 are not read any more: they may take part)
    T acc[4][4][2];
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

template <typename T, bool S_GLOBAL>
__global__ void __launch_bounds__(kTfThreads, 1) tri_factor_kernel(const FactorMat* mats, int smem_bytes, double shift_scale, int conditional) {
  constexpr int NB = kTfNB, LD = kTfLd, WARPS = kTfThreads / 32;
  extern __shared__ __align__(16) unsigned char tf_smem[];
  __shared__ int counter;
  const FactorMat m = mats[blockIdx.x];
  if (conditional && *m.only_if == 0) return;
  const int L = m.L, nb = (L + NB - 1) / NB, np = nb * NB;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, fr = lane >> 2, fk = lane & 3;
  T* Inv0 = reinterpret_cast<T*>(tf_smem);            // [2][NB][LD]
  T* W = Inv0 + 2 * NB * LD;                           // work space of the diagonal block: [NB][kTfLdW],
  T* S8 = W + NB * kTfLdW;                             // [NB][kTfLdS8],
  T* I8 = S8 + NB * kTfLdS8;                           // [8][8]
  T* rd = I8 + 64;                                     // [np] 1 / column norm
  T* Ssh = rd + np;
  T* S = S_GLOBAL ? static_cast<T*>(m.spill) : Ssh;    // [np][LD]
  const bool resident = tf_base_smem<T>(L, S_GLOBAL) + tf_block_bytes<T>(L) <= static_cast<size_t>(smem_bytes);
  T* B = resident ? (S_GLOBAL ? Ssh : Ssh + np * LD) : static_cast<T*>(m.work);
  const T* C = static_cast<const T*>(m.C);
  auto block = [&](int i, int j) -> T* { return B + (i * (i + 1) / 2 + j) * (NB * NB); };
  const T tiny = sizeof(T) == 8 ? T(1e-28) : T(1e-12);
  const T one = T(1.0 + (sizeof(T) == 8 ? shift_scale : shift_scale * static_cast<double>(L) / 65536.0));

  for (int i = tid; i < np; i += kTfThreads) {
    T d = i < L ? C[static_cast<long long>(i) * L + i] : T(1);
    const T floor = sizeof(T) == 8 ? T(1e-60) : T(1e-37);
    if (!(d > floor)) d = d == d ? floor : d;          // (a NaN stays one, and the basis check finds it)
    rd[i] = tf_rsqrt(d);
  }
  __syncthreads();
  // the scaled matrix (beyond L: the identity)
  for (int b = warp; b < nb * (nb + 1) / 2; b += WARPS) {
    int i = static_cast<int>((sqrtf(8.f * b + 1.f) - 1.f) * 0.5f);
    while ((i + 1) * (i + 2) / 2 <= b) ++i;
    while (i * (i + 1) / 2 > b) --i;
    const int j = b - i * (i + 1) / 2;
    const int c = j * NB + lane;
    T* dst = B + b * (NB * NB);
#pragma unroll 1
    for (int row0 = 0; row0 < NB; row0 += 16) {
      T raw[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) raw[q] = C[static_cast<long long>(min(i * NB + row0 + q, L - 1)) * L + min(c, L - 1)];
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int row = row0 + q, r = i * NB + row;
        const T v = raw[q] * rd[r] * rd[c];
        dst[tf_at(row, lane)] = r == c ? (r < L ? one : T(1)) : (r < L && c < r ? v : T(0));
      }
    }
  }
  if (tid == 0) counter = 0;
  __syncthreads();

  for (int k = -1; k < nb; ++k) {
    const T* Inv = Inv0 + (k & 1) * NB * LD;
    // S, and block column k of R^-1
    for (int i = warp; i < nb && k >= 0; i += WARPS) {
      T acc[4][4][2];
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x][y][0] = acc[x][y][1] = T(0);
      auto right = [&](int n, int kk) { return Inv[n * LD + kk]; };
      if (i > k) {
        const T* blk = block(i, k);
        tf_product<NB>(acc, [&](int r, int kk) { return blk[tf_at(r, kk)]; }, right, fr, fk);
      } else if (i < k) {
        const T* blk = block(k, i);
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
        const T scale = rd[row];
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const int kk = 8 * y + 2 * fk, col = k * NB + kk;
          S[row * LD + kk] = acc[x][y][0];
          S[row * LD + kk + 1] = acc[x][y][1];
          if (m.R64 != nullptr) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
              if (row < L && col + h < L) m.R64[static_cast<long long>(row) * L + col + h] = i <= k ? static_cast<double>(acc[x][y][h] * scale) : 0.0;
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
        T* blk = block(i, j);
        T acc[4][4][2];
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y)
#pragma unroll
            for (int h = 0; h < 2; ++h) acc[x][y][h] = j == k ? T(0) : blk[tf_at(8 * x + fr, 8 * y + 2 * fk) + h];
        const T *Si = S + i * NB * LD, *Sj = S + j * NB * LD;
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
        tf_diagonal<T>(block(k + 1, k + 1), tiny, W, S8, I8, Inv0 + ((k + 1) & 1) * NB * LD, lane);
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

// (to their largest values: the limit of a kernel belongs to the process, not to one state)
inline cudaError_t tri_factor_init() {
  cudaError_t e;
  auto set = [](const void* f) { return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kTfSmemLimit); };
  if ((e = set(reinterpret_cast<const void*>(tri_factor_kernel<float, false>))) != cudaSuccess) return e;
  if ((e = set(reinterpret_cast<const void*>(tri_factor_kernel<double, false>))) != cudaSuccess) return e;
  return set(reinterpret_cast<const void*>(tri_factor_kernel<double, true>));
}

// Factor n matrices, the widest l_max wide (widest first in the list: CTAs are handed out in order).  shift_scale: what
// is added to the unit diagonal, for fp32 matrices in units of L / 65536.
template <typename T>
inline cudaError_t tri_factor_launch(const FactorMat* d_mats, int n, int l_max, double shift_scale, cudaStream_t stream,
                                     int64_t* launches, bool conditional = false) {
  // as much shared memory as the widest matrix that fits with its blocks, and at least what the widest needs without
  size_t smem = tf_base_smem<T>(l_max, false);
  const bool s_global = smem > static_cast<size_t>(kTfSmemLimit);
  if (s_global) smem = tf_base_smem<T>(l_max, true);
  for (int l = l_max; l > 0; l -= 4) {
    const size_t need = tf_base_smem<T>(l, s_global) + tf_block_bytes<T>(l);
    if (need <= static_cast<size_t>(kTfSmemLimit)) { smem = need > smem ? need : smem; break; }
  }
  if (s_global) {
    if (sizeof(T) == 4) return cudaErrorInvalidValue;   // (an fp32 basis of 875 columns needs 147 KB)
    tri_factor_kernel<double, true><<<n, kTfThreads, smem, stream>>>(d_mats, static_cast<int>(smem), shift_scale, conditional ? 1 : 0);
  } else {
    tri_factor_kernel<T, false><<<n, kTfThreads, smem, stream>>>(d_mats, static_cast<int>(smem), shift_scale, conditional ? 1 : 0);
  }
  *launches += 1;
  return cudaGetLastError();
}

}  // namespace ngalore
