// Pieces of the subspace refresh (Sec. 1: P spans the leading left singular vectors of G,
// "updated periodically").  The refresh is a randomized subspace iteration; every application of
// G or G^T is followed by an orthonormalisation Q = Y R^-1 with R^T R = Y^T Y (Cholesky QR with
// the Gram matrix and the factorisation in fp64).
#pragma once

#include <algorithm>

#include "common.cuh"

namespace ngalore {

// ---------------------------------------------------------------- random test matrix

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

// Standard normal entries from a counter-based hash (Box-Muller on two hashed uniforms).
__global__ void fill_normal_kernel(float* X, long long n, unsigned long long seed, unsigned long long stream_id) {
  const long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const unsigned long long h =
      splitmix64(seed ^ splitmix64(stream_id * 0x100000001B3ull + static_cast<unsigned long long>(i)));
  const float u1 = (static_cast<float>(h >> 40) + 1.0f) * (1.0f / 16777217.0f);
  const float u2 = static_cast<float>((h >> 8) & 0xFFFFFFull) * (1.0f / 16777216.0f);
  X[i] = sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
}

// The same values as two bf16 parts for a list of matrices in one launch: blockIdx.y selects the matrix (its stream of
// random numbers is stream_base + blockIdx.y), blockIdx.x strides over its entries, two neighbours of a row at a time.
// Bound by the instructions of the hash and the Box-Muller functions (4 bytes leave for about 90 of them); with one entry a
// thread, its own division into row and column and 64 blocks a matrix, however large: 60M shapes 38 us, 130M 150, 1.1B
// 1144; now 34, 130 and 1133.
struct FillJob {
  __nv_bfloat16 *hi, *lo;   // rows x ld
  long long n;              // rows x cols
  int cols, ld;
};

__global__ void __launch_bounds__(256) fill_normal_grouped_kernel(const FillJob* jobs, unsigned long long seed, unsigned long long stream_base) {
  const FillJob jb = jobs[blockIdx.y];
  const unsigned long long stream_id = stream_base + blockIdx.y;
  auto normal = [&](long long i) {
    const unsigned long long h =
        splitmix64(seed ^ splitmix64(stream_id * 0x100000001B3ull + static_cast<unsigned long long>(i)));
    const float u1 = (static_cast<float>(h >> 40) + 1.0f) * (1.0f / 16777217.0f);
    const float u2 = static_cast<float>((h >> 8) & 0xFFFFFFull) * (1.0f / 16777216.0f);
    return sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
  };
  const long long stride = 2ll * gridDim.x * blockDim.x;
  for (long long i = 2 * (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x); i < jb.n; i += stride) {
    const float x = normal(i), y = normal(i + 1);   // (cols is a multiple of 4)
    const __nv_bfloat162 hi = __floats2bfloat162_rn(x, y);
    const long long row = i < (1ll << 32) ? static_cast<unsigned int>(i) / static_cast<unsigned int>(jb.cols) : i / jb.cols;
    const long long o = row * jb.ld + (i - row * jb.cols);
    *reinterpret_cast<__nv_bfloat162*>(jb.hi + o) = hi;
    *reinterpret_cast<__nv_bfloat162*>(jb.lo + o) = __floats2bfloat162_rn(x - __low2float(hi), y - __high2float(hi));
  }
}

// ---------------------------------------------------------------- batched Cholesky (fp64, right-looking, blocked)

struct CholProblem {
  double* C;    // L x L row-major; lower triangle in, lower Cholesky factor out (C = Lf Lf^T)
  int L;
  int pad;
  double tiny;  // pivot floor, written by chol_begin_kernel
};

constexpr int kCholNB = 32;  // panel width

// Pivot floor of every matrix from its diagonal before the factorisation starts.  A pivot that is not above it
// (rank-deficient Y) is replaced by it so that the factor stays finite; the caller runs a second
// orthonormalisation pass at the end of the refresh.  One warp per matrix.
__global__ void __launch_bounds__(32) chol_begin_kernel(CholProblem* probs) {
  CholProblem& p = probs[blockIdx.x];
  double md = 0.0;
  for (int i = threadIdx.x; i < p.L; i += 32) md = fmax(md, p.C[static_cast<long long>(i) * p.L + i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) md = fmax(md, __shfl_xor_sync(0xffffffffu, md, o));
  if (threadIdx.x == 0) p.tiny = fmax(md * 1e-28, 1e-300);   // never zero: a matrix of zeros still factors
}

// Panel step at column j0, one CTA per matrix: factor the diagonal block in shared memory (one warp, lane = row),
// then solve the rows below it against the block (x D^T = c, forward substitution, one thread per row).
__global__ void __launch_bounds__(256) chol_panel_kernel(const CholProblem* probs, int j0) {
  constexpr int NB = kCholNB;
  __shared__ double D[NB][NB + 1];
  const CholProblem p = probs[blockIdx.x];
  double* C = p.C;
  const int L = p.L;
  if (j0 >= L) return;
  const int tid = threadIdx.x;
  const int nbj = (L - j0 < NB) ? (L - j0) : NB;
  const double tiny = p.tiny;
  for (int x = tid; x < NB * NB; x += 256) {
    const int a = x / NB, b = x % NB;
    D[a][b] = (a < nbj && b < nbj) ? C[static_cast<long long>(j0 + a) * L + j0 + b] : 0.0;
  }
  __syncthreads();
  if (tid < 32) {
    const int lane = tid;
    for (int k = 0; k < nbj; ++k) {
      double dkk = D[k][k];
      if (!(dkk > tiny)) dkk = tiny;
      const double lkk = sqrt(dkk);
      __syncwarp();
      if (lane == k) D[k][k] = lkk;
      if (lane > k && lane < nbj) D[lane][k] /= lkk;
      __syncwarp();
      if (lane > k && lane < nbj) {
        const double lik = D[lane][k];
        for (int j = k + 1; j <= lane; ++j) D[lane][j] -= lik * D[j][k];
      }
      __syncwarp();
    }
  }
  __syncthreads();
  for (int x = tid; x < NB * NB; x += 256) {
    const int a = x / NB, b = x % NB;
    if (a < nbj && b <= a) C[static_cast<long long>(j0 + a) * L + j0 + b] = D[a][b];
  }
  for (int i = j0 + nbj + tid; i < L; i += 256) {
    double xr[NB];
    double* crow = C + static_cast<long long>(i) * L + j0;
#pragma unroll
    for (int jj = 0; jj < NB; ++jj) {
      if (jj < nbj) {
        double a = crow[jj];
#pragma unroll
        for (int t = 0; t < NB; ++t)
          if (t < jj) a -= xr[t] * D[jj][t];
        xr[jj] = a / D[jj][jj];
      }
    }
#pragma unroll
    for (int jj = 0; jj < NB; ++jj)
      if (jj < nbj) crow[jj] = xr[jj];
  }
}

// Trailing update after the panel at column j0: C[i][j] -= sum_k C[i][j0 + k] C[j][j0 + k] on the lower triangle
// beyond the panel.  blockIdx.y selects the matrix, blockIdx.x a pair (ti >= tj) of 64-row tiles.
__global__ void __launch_bounds__(256) chol_trailing_kernel(const CholProblem* probs, int j0) {
  constexpr int NB = kCholNB;
  __shared__ double As[NB][64 + 1];
  __shared__ double Bs[NB][64 + 1];
  const CholProblem p = probs[blockIdx.y];
  const int L = p.L, base = j0 + NB;
  if (base >= L) return;
  const int nt = (L - base + 63) / 64;
  int ti = static_cast<int>((sqrtf(8.f * blockIdx.x + 1.f) - 1.f) * 0.5f);
  while ((ti + 1) * (ti + 2) / 2 <= static_cast<int>(blockIdx.x)) ++ti;
  while (ti * (ti + 1) / 2 > static_cast<int>(blockIdx.x)) --ti;
  const int tj = blockIdx.x - ti * (ti + 1) / 2;
  if (ti >= nt) return;
  const int i0 = base + ti * 64, c0 = base + tj * 64;
  const int t = threadIdx.x;
  for (int x = t; x < NB * 64; x += 256) {
    const int r = x / NB, k = x % NB;  // k contiguous in memory
    As[k][r] = (i0 + r < L) ? p.C[static_cast<long long>(i0 + r) * L + j0 + k] : 0.0;
    Bs[k][r] = (c0 + r < L) ? p.C[static_cast<long long>(c0 + r) * L + j0 + k] : 0.0;
  }
  __syncthreads();
  const int tx = t & 15, ty = t >> 4;
  double acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
#pragma unroll 8
  for (int k = 0; k < NB; ++k) {
    double a[4], b[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) { a[x] = As[k][ty * 4 + x]; b[x] = Bs[k][tx * 4 + x]; }
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) acc[x][y] += a[x] * b[y];
  }
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    const int i = i0 + ty * 4 + x;
    if (i >= L) continue;
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const int j = c0 + tx * 4 + y;
      if (j <= i) p.C[static_cast<long long>(i) * L + j] -= acc[x][y];
    }
  }
}

// Factor n matrices (the largest of size Lmax).  Panels of 32 columns: the panel step runs one CTA per matrix, the
// trailing update spreads over the whole GPU; 2 Lmax / 32 launches.
inline cudaError_t chol_batched_launch(CholProblem* d_probs, int n, int Lmax, cudaStream_t stream, int64_t* launches) {
  chol_begin_kernel<<<n, 32, 0, stream>>>(d_probs);
  *launches += 1;
  for (int j0 = 0; j0 < Lmax; j0 += kCholNB) {
    chol_panel_kernel<<<n, 256, 0, stream>>>(d_probs, j0);
    *launches += 1;
    const int rows = Lmax - j0 - kCholNB;
    if (rows > 0) {
      const int nt = (rows + 63) / 64;
      chol_trailing_kernel<<<dim3(nt * (nt + 1) / 2, n), 256, 0, stream>>>(d_probs, j0);
      *launches += 1;
    }
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------- Q = Y Lf^-T (rows are independent)

// One CTA owns 32 rows of Y (rows x L, fp32) and produces the same rows of Q (fp32) with
// Q Lf^T = Y, Lf the lower Cholesky factor of Y^T Y (fp64).  Column blocks of 32 are solved in
// order; finished columns of Q stay in shared memory (fp64).
struct OrthApply {
  const float* Y;
  float* Q;
  const double* Lf;
  int rows, L;
};

inline size_t orth_apply_smem_bytes(int L) {
  return (static_cast<size_t>(32) * L + 32 * 33) * sizeof(double);
}

__global__ void __launch_bounds__(256) orth_apply_kernel(OrthApply p) {
  constexpr int NB = 32, RB = 32;
  extern __shared__ __align__(16) unsigned char orth_smem_raw[];
  double* Qs = reinterpret_cast<double*>(orth_smem_raw);  // RB x L (finished columns)
  double* Ls = Qs + static_cast<size_t>(RB) * p.L;        // NB x (NB + 1) chunk of Lf
  const int tid = threadIdx.x;
  const int r0 = blockIdx.x * RB;
  const int L = p.L;
  const int row = tid >> 3;      // 0..31
  const int cg = (tid & 7) * 4;  // 4 columns of the current block
  for (int j0 = 0; j0 < L; j0 += NB) {
    const int nbj = (L - j0 < NB) ? (L - j0) : NB;
    double acc[4];
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const int col = j0 + cg + y;
      acc[y] = (r0 + row < p.rows && col < L)
                   ? static_cast<double>(p.Y[static_cast<long long>(r0 + row) * L + col])
                   : 0.0;
    }
    for (int k0 = 0; k0 < j0; k0 += NB) {
      __syncthreads();
      for (int x = tid; x < NB * NB; x += 256) {
        const int a = x / NB, b = x % NB;
        Ls[a * (NB + 1) + b] = (a < nbj) ? p.Lf[static_cast<long long>(j0 + a) * L + k0 + b] : 0.0;
      }
      __syncthreads();
#pragma unroll 8
      for (int b = 0; b < NB; ++b) {
        const double qv = Qs[static_cast<size_t>(row) * L + k0 + b];
        acc[0] -= qv * Ls[(cg + 0) * (NB + 1) + b];
        acc[1] -= qv * Ls[(cg + 1) * (NB + 1) + b];
        acc[2] -= qv * Ls[(cg + 2) * (NB + 1) + b];
        acc[3] -= qv * Ls[(cg + 3) * (NB + 1) + b];
      }
    }
    __syncthreads();
#pragma unroll
    for (int y = 0; y < 4; ++y)
      if (cg + y < nbj) Qs[static_cast<size_t>(row) * L + j0 + cg + y] = acc[y];
    for (int x = tid; x < NB * NB; x += 256) {
      const int a = x / NB, b = x % NB;
      Ls[a * (NB + 1) + b] = (a < nbj && b < nbj) ? p.Lf[static_cast<long long>(j0 + a) * L + j0 + b] : 0.0;
    }
    __syncthreads();
    if (tid < RB) {
      double* q = Qs + static_cast<size_t>(tid) * L + j0;
      for (int jj = 0; jj < nbj; ++jj) {
        double a = q[jj];
        for (int t = 0; t < jj; ++t) a -= q[t] * Ls[jj * (NB + 1) + t];
        q[jj] = a / Ls[jj * (NB + 1) + jj];
      }
    }
    __syncthreads();
  }
  for (int x = tid; x < RB * L; x += 256) {
    const int a = x / L, b = x % L;
    if (r0 + a < p.rows)
      p.Q[static_cast<long long>(r0 + a) * L + b] = static_cast<float>(Qs[static_cast<size_t>(a) * L + b]);
  }
}

// ---------------------------------------------------------------- working copies of P

// Working copies of a projector P32 (rows x rp): P16 (rows x ldp) and its transpose Pt16 (rp x ldpt), both
// holding the bf16-rounded values.  One of the two is stored as bf16 and the other as fp16 (p16_is_half says
// which): a bf16 number converts to fp16 without error unless it is below 2^-17 in magnitude, where the error is
// at most 2^-25, far below the resolution of an orthonormal column's entries.
// Block (32, 8).
__device__ __forceinline__ uint16_t working_bits(float val, bool as_half) {
  const __nv_bfloat16 b = __float2bfloat16_rn(val);
  if (!as_half) return __bfloat16_as_ushort(b);
  return __half_as_ushort(__float2half_rn(__bfloat162float(b)));
}

__global__ void working_copies_kernel(const float* P32, uint16_t* P16, uint16_t* Pt16, int rows, int rp, int ldp,
                                      int ldpt, int p16_is_half) {
  __shared__ float tile[32][33];
  const int i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
  for (int a = threadIdx.y; a < 32; a += blockDim.y) {
    const int i = i0 + a, j = j0 + threadIdx.x;
    float val = 0.f;
    if (i < rows && j < rp) {
      val = P32[static_cast<long long>(i) * rp + j];
      P16[static_cast<long long>(i) * ldp + j] = working_bits(val, p16_is_half != 0);
    }
    tile[a][threadIdx.x] = val;
  }
  __syncthreads();
  for (int a = threadIdx.y; a < 32; a += blockDim.y) {
    const int j = j0 + a, i = i0 + threadIdx.x;
    if (i < rows && j < rp) Pt16[static_cast<long long>(j) * ldpt + i] = working_bits(tile[threadIdx.x][a], p16_is_half == 0);
  }
}

// The end of a refresh for a list of matrices in two launches, each reading the new basis once: the column norms, and the
// master and working copies of the basis with its columns scaled to unit norm.  Scaling: the products of the refresh go
// through operands split in two bf16 parts; the rounding of the diagonal of a triangular factor or of a rotation (a
// relative 2^-17) scales a whole column, which is the largest part of what the last product leaves of
// non-orthonormality.  The norms also tell a basis that is none (see basis_check_kernel): all of them zero, or one not
// finite; such a matrix gets the first r' unit vectors, in the second case with its status word set.
// CTAs take tiles of norm_rows x kEndCols (norms) and kEndRows x kEndCols entries (copies); tile_start[j] is the first tile of
// job j (n_jobs + 1 entries, ascending).  Up to 2048 rows make two tiles for the norms, whose sums give the same bits in either
// order.  Bound by memory traffic: 4 bytes an entry read, then 12.  They replaced five
// kernels of five passes with one CTA count for every matrix, so that a 32000-row embedding took as many CTAs as a
// 512-row matrix: 60M shapes 316 us, 130M 680 us, 1.1B 2620 us before, 52, 121 and 596 us now.
struct WorkingJob {
  const float* src;   // rows x rp, dense; rp a multiple of 4
  double* sums;       // rp sums of squares (cleared beforehand)
  float* P32;
  uint16_t* P16;
  uint16_t* Pt16;
  int* status;
  int rows, rp, ldp, ldpt;
  int p16_is_half;
  int tiles_x;        // tiles along the rp columns
  int norm_rows;      // rows of a tile for the norms (end_norm_rows)
};
constexpr int kEndRows = 128, kEndCols = 64;
inline int end_norm_rows(int rows) { return rows <= 2048 ? std::max((rows + 1) / 2, kEndRows) : 2 * kEndRows; }

__device__ __forceinline__ int end_job(const int* tile_start, int n_jobs) {
  int lo = 0, hi = n_jobs;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (tile_start[mid] <= static_cast<int>(blockIdx.x)) lo = mid; else hi = mid;
  }
  return lo;
}

__global__ void __launch_bounds__(256) basis_norms_kernel(const WorkingJob* jobs, const int* tile_start, int n_jobs) {
  const int j = end_job(tile_start, n_jobs);
  const WorkingJob jb = jobs[j];
  const int t = static_cast<int>(blockIdx.x) - tile_start[j];
  const int r0 = (t / jb.tiles_x) * jb.norm_rows, r1 = min(r0 + jb.norm_rows, jb.rows);
  // thread: four neighbouring columns and every sixteenth row
  __shared__ double part[16][kEndCols + 2];
  const int q = threadIdx.x & 15, g = threadIdx.x >> 4, c = (t % jb.tiles_x) * kEndCols + 4 * q;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  if (c < jb.rp) {
#pragma unroll 8
    for (int r = r0 + g; r < r1; r += 16) {
      const float4 x = *reinterpret_cast<const float4*>(jb.src + static_cast<long long>(r) * jb.rp + c);
      s[0] += static_cast<double>(x.x) * x.x; s[1] += static_cast<double>(x.y) * x.y;
      s[2] += static_cast<double>(x.z) * x.z; s[3] += static_cast<double>(x.w) * x.w;
    }
  }
#pragma unroll
  for (int y = 0; y < 4; ++y) part[g][4 * q + y] = s[y];
  __syncthreads();
  const int col = (t % jb.tiles_x) * kEndCols + threadIdx.x;
  if (threadIdx.x < kEndCols && col < jb.rp) {
    double sum = 0.0;
#pragma unroll
    for (int x = 0; x < 16; ++x) sum += part[x][threadIdx.x];
    atomicAdd(jb.sums + col, sum);
  }
}

__global__ void __launch_bounds__(256) working_copies_grouped_kernel(const WorkingJob* jobs, const int* tile_start, int n_jobs) {
  __shared__ __align__(8) uint16_t tile[kEndCols][kEndRows + 4];   // (rows of 264 bytes, read eight at a time)
  const int j = end_job(tile_start, n_jobs);
  const WorkingJob jb = jobs[j];
  const int t = static_cast<int>(blockIdx.x) - tile_start[j];
  const int i0 = (t / jb.tiles_x) * kEndRows, j0 = (t % jb.tiles_x) * kEndCols;
  bool bad = false, any = false;
  for (int c = threadIdx.x; c < jb.rp; c += 256) {
    const double v = jb.sums[c];
    bad = bad || !isfinite(v);
    any = any || v > 0.0;
  }
  const bool nonfinite = __syncthreads_or(bad ? 1 : 0) != 0;
  const bool repair = nonfinite || __syncthreads_or(any ? 1 : 0) == 0;
  if (nonfinite && t == 0 && threadIdx.x == 0) atomicCAS(jb.status, 0, 7 /* NGALORE_ERR_NONFINITE */);
  const int q = threadIdx.x & 15, c = j0 + 4 * q;
  float f[4] = {0.f, 0.f, 0.f, 0.f};
  if (c < jb.rp) {
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const double v = jb.sums[c + y];
      f[y] = v > 0.0 ? static_cast<float>(1.0 / sqrt(v)) : 0.f;
    }
  }
#pragma unroll
  for (int p = 0; p < kEndRows / 16; ++p) {
    const int a = (threadIdx.x >> 4) + 16 * p, i = i0 + a;
    if (i >= jb.rows || c >= jb.rp) continue;
    const float4 x = *reinterpret_cast<const float4*>(jb.src + static_cast<long long>(i) * jb.rp + c);
    float v[4] = {x.x * f[0], x.y * f[1], x.z * f[2], x.w * f[3]};
    if (repair) {
#pragma unroll
      for (int y = 0; y < 4; ++y) v[y] = i == c + y ? 1.f : 0.f;
    }
    *reinterpret_cast<float4*>(jb.P32 + static_cast<long long>(i) * jb.rp + c) = make_float4(v[0], v[1], v[2], v[3]);
    uint2 w;
    w.x = working_bits(v[0], jb.p16_is_half != 0) | (static_cast<uint32_t>(working_bits(v[1], jb.p16_is_half != 0)) << 16);
    w.y = working_bits(v[2], jb.p16_is_half != 0) | (static_cast<uint32_t>(working_bits(v[3], jb.p16_is_half != 0)) << 16);
    *reinterpret_cast<uint2*>(jb.P16 + static_cast<long long>(i) * jb.ldp + c) = w;
#pragma unroll
    for (int y = 0; y < 4; ++y) tile[4 * q + y][a] = working_bits(v[y], jb.p16_is_half == 0);
  }
  __syncthreads();
  // the transposed copy: a warp writes 128 rows of a column, four a lane
  const int lane = threadIdx.x & 31, i = i0 + 4 * lane;
  for (int y = threadIdx.x >> 5; y < kEndCols; y += 8) {
    if (j0 + y >= jb.rp || i >= jb.rows) continue;
    uint16_t* dst = jb.Pt16 + static_cast<long long>(j0 + y) * jb.ldpt + i;
    if (i + 3 < jb.rows) {
      *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(&tile[y][4 * lane]);
    } else {
      for (int x = 0; x < 4 && i + x < jb.rows; ++x) dst[x] = tile[y][4 * lane + x];
    }
  }
}

// A refreshed basis that is no basis: all zeros (the gradient of a frozen layer: every product of the iteration is
// zero and nothing can be normalised) or with entries that are not finite (a gradient with such entries).  Any
// orthonormal basis serves a zero gradient, so such a matrix gets the first r' unit vectors; the second case also
// raises the matrix's status word.  Two launches over a list of matrices: sums, then the repair.
struct BasisJob {
  float* Ya;       // rows x rp, dense: the basis, in one of the two buffers of the refresh
  float* Yb;
  double* acc;     // [0]: sum of squares, [1]: number of entries that are not finite (cleared by the caller)
  int* status;
  int rows, rp;
};

__global__ void __launch_bounds__(256) basis_check_kernel(const BasisJob* jobs, int in_a) {
  __shared__ double red[8];
  __shared__ int bad_any;
  const BasisJob jb = jobs[blockIdx.y];
  const float* Y = in_a ? jb.Ya : jb.Yb;
  const long long n = static_cast<long long>(jb.rows) * jb.rp;
  if (threadIdx.x == 0) bad_any = 0;
  __syncthreads();
  double s = 0.0;
  int bad = 0;
  for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += 256ll * gridDim.x) {
    const float x = Y[i];
    if (isfinite(x)) s += static_cast<double>(x) * static_cast<double>(x);
    else bad = 1;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  if (bad) bad_any = 1;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += red[w];
    if (t != 0.0) atomicAdd(jb.acc, t);
    if (bad_any) atomicAdd(jb.acc + 1, 1.0);
  }
}

__global__ void __launch_bounds__(256) basis_repair_kernel(const BasisJob* jobs, int in_a) {
  const BasisJob jb = jobs[blockIdx.y];
  const bool nonfinite = jb.acc[1] > 0.0;
  if (!nonfinite && jb.acc[0] > 0.0) return;
  float* Y = in_a ? jb.Ya : jb.Yb;
  const long long n = static_cast<long long>(jb.rows) * jb.rp;
  for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += 256ll * gridDim.x)
    Y[i] = (i / jb.rp == i % jb.rp) ? 1.f : 0.f;
  if (nonfinite && blockIdx.x == 0 && threadIdx.x == 0) atomicCAS(jb.status, 0, 7 /* NGALORE_ERR_NONFINITE */);
}

// dst (rows x cols, dense fp32) = src (rows x cols, leading dimension ld; fp16 or bf16 bits)
__global__ void widen_16_kernel(const uint16_t* src, float* dst, long long n, int cols, int ld, int is_half) {
  const long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const uint16_t bits = src[(i / cols) * ld + (i % cols)];
  dst[i] = is_half ? __half2float(__ushort_as_half(bits)) : __bfloat162float(__ushort_as_bfloat16(bits));
}

// dst (cols x ld_dst, bf16, padding columns left untouched) = src^T for src (rows x cols, bf16).  Block (32, 8).
__global__ void transpose_bf16_kernel(const uint16_t* src, uint16_t* dst, int rows, int cols, int ld_dst) {
  __shared__ uint16_t tile[32][33];
  const int i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
  for (int a = threadIdx.y; a < 32; a += blockDim.y) {
    const int i = i0 + a, j = j0 + threadIdx.x;
    tile[a][threadIdx.x] = (i < rows && j < cols) ? src[static_cast<long long>(i) * cols + j] : uint16_t(0);
  }
  __syncthreads();
  for (int a = threadIdx.y; a < 32; a += blockDim.y) {
    const int j = j0 + a, i = i0 + threadIdx.x;
    if (i < rows && j < cols) dst[static_cast<long long>(j) * ld_dst + i] = tile[threadIdx.x][a];
  }
}

}  // namespace ngalore
