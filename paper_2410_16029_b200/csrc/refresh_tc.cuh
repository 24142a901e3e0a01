// Subspace refresh on the tensor cores (Sec. 1: P spans the leading left singular vectors of G).
//
// Randomized subspace iteration with L = r' columns: Y = G Omega, then q sweeps of
//   Z = G^T Q_Y,  Q_Z = orth(Z),  Y = G Q_Z,  Q_Y = orth(Y).
// Every product runs through the grouped tcgen05 GEMM with the iterate split into a high and a low
// bf16 part (16 mantissa bits).  Between products the iterate only has to stay well conditioned, so
// orth() is a *shifted* Cholesky QR: the Gram matrix Y^T Y comes from the tensor cores (three bf16
// products, fp32 accumulation), its columns are scaled to unit norm and a small multiple of the identity
// is added before the fp64 factorisation (tri_factor.cuh) so that the fp32 accumulation error cannot make it
// indefinite, and Q = Y R^-1 is again a tensor-core GEMM with R^-1 split in two bf16 parts.  The last basis is then
// orthonormalised exactly (Gram matrix, factorisation and triangular inverse in fp64) and by two Newton steps, and rotated to
// the Ritz vectors of G inside the subspace (Z = G^T Q, eigenvectors V of Z^T Z by the kernels of ritz_eigen.cuh, P = Q V on
// the tensor cores, columns in falling order of their singular value and scaled to unit norm).
#pragma once

#include <cstring>
#include <vector>

#include <algorithm>
#include <type_traits>

#include "gemm_pair_tcgen05.cuh"
#include "gemm_tcgen05.cuh"
#include "kernels_refresh.cuh"
#include "ritz_eigen.cuh"
#include "tri_factor.cuh"

namespace ngalore {

// hi = bf16(x), lo = bf16(x - hi); rows x cols fp32 (dense) -> rows x ld bf16 (padding untouched: it is zero).
struct SplitJob {
  const float* src;
  __nv_bfloat16 *hi, *lo;
  long long n;
  int cols, ld;
};

// All matrices in one launch: blockIdx.y selects the matrix, blockIdx.x strides over its elements, four at a
// time where the row length allows it (the kernel is a pure stream: 4 bytes in, 4 bytes out per element).
__global__ void split_hilo_grouped_kernel(const SplitJob* jobs) {
  pdl_begin();
  const SplitJob jb = jobs[blockIdx.y];
  const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
  const long long t0 = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if ((jb.cols & 3) == 0 && (jb.ld & 3) == 0) {
    const int quads_per_row = jb.cols >> 2;
    for (long long q = t0; q < (jb.n >> 2); q += stride) {
      const float4 x = reinterpret_cast<const float4*>(jb.src)[q];
      const long long row = q / quads_per_row;
      const long long o = row * jb.ld + ((q - row * quads_per_row) << 2);
      const __nv_bfloat162 h01 = __floats2bfloat162_rn(x.x, x.y), h23 = __floats2bfloat162_rn(x.z, x.w);
      const __nv_bfloat162 l01 = __floats2bfloat162_rn(x.x - __low2float(h01), x.y - __high2float(h01));
      const __nv_bfloat162 l23 = __floats2bfloat162_rn(x.z - __low2float(h23), x.w - __high2float(h23));
      uint2 hv, lv;
      hv.x = *reinterpret_cast<const uint32_t*>(&h01); hv.y = *reinterpret_cast<const uint32_t*>(&h23);
      lv.x = *reinterpret_cast<const uint32_t*>(&l01); lv.y = *reinterpret_cast<const uint32_t*>(&l23);
      *reinterpret_cast<uint2*>(jb.hi + o) = hv;
      *reinterpret_cast<uint2*>(jb.lo + o) = lv;
    }
    return;
  }
  for (long long i = t0; i < jb.n; i += stride) {
    const float x = jb.src[i];
    const __nv_bfloat16 h = __float2bfloat16_rn(x);
    const long long o = (i / jb.cols) * jb.ld + (i % jb.cols);
    jb.hi[o] = h;
    jb.lo[o] = __float2bfloat16_rn(x - __bfloat162float(h));
  }
}

// Clear a list of buffers in one launch (a memset per buffer costs more in launch overhead than in work when
// there are hundreds of small ones): blockIdx.y selects the buffer, blockIdx.x strides over its 16-byte words.
struct ZeroJob {
  float4* p;
  long long n16;
};

__global__ void zero_jobs_kernel(const ZeroJob* jobs) {
  pdl_begin();
  const ZeroJob jb = jobs[blockIdx.y];
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < jb.n16;
       i += static_cast<long long>(gridDim.x) * blockDim.x)
    jb.p[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// Shift added to the unit-diagonal Gram matrix: L / 65536 (tri_factor_kernel).  Each entry carries a relative error of at
// most about 3 * 2^-18 from the two-part bf16 split (the dropped lo*lo product and the rounding of lo) plus the fp32
// accumulation error, so the error matrix has norm below 2^-16 L; with this shift the Cholesky factorisation
// cannot meet a negative pivot.  The price is that directions closer than sqrt(shift) are not pulled
// apart, which is harmless between products.  Scaling the columns to unit norm first makes the shift act on every
// column alike, whatever its norm, so weak directions are still orthogonalised against each other and re-normalised.

struct SyrkTile {
  int mat, ti, tj, k0, k1;  // output tile (ti, tj <= ti) of 64 x 64, rows k0 .. k1 - 1 of Y
};
// Rows of a slab: long ones save atomics, short ones balance the SMs where there are few tiles.  58 matrices of r' = 128
// (232 tiles of 1024 rows) 138 us against 117 with short ones, 84 of r' = 256 (1080) 473 / 448 us, 156 of the 1.1B shapes
// (15 thousand) 4.14 / 4.33 ms.
// Up to 2048 rows make no more than two slabs: two sums added to zero give the same bits in either order.
constexpr int kSyrkRows = 1024, kSyrkRowsFew = 256;
constexpr int kSyrkFewTiles = 16;   // per SM

struct SyrkMat {
  const __nv_bfloat16 *hi, *lo;   // rows x ld: the two parts of the basis, L columns of which are valid ...
  const float* f32;               // ... or the basis itself, rows x L
  double* C;       // L x L fp64 accumulator (zeroed before the launch); lower tiles are written
  int rows, L, ld;
};

// Exact Gram matrix C += Y^T Y in fp64 of the basis as its two bf16 parts hold it (which is what the product with R^-1
// multiplies), grouped over all matrices: one CTA per 64 x 64 lower tile and slab of rows, partial sums added with fp64
// atomics.  On the fp64 tensor cores: bound by their rate, which is that of the vector units (34 TFLOP/s), but reached
// with a quarter of the instructions and a third of the shared-memory reads; the next 16 rows are fetched and widened
// while the current ones are multiplied.  156 matrices of the 1.1B shapes, 115 GFLOP: 7.2 ms with 4 x 4 register tiles on
// the vector units, 4.1 ms so.  F32: of a basis in fp32 (refresh_tc_short).
template <bool F32>
__global__ void __launch_bounds__(256) syrk_f64_kernel(const SyrkMat* mats, const SyrkTile* tiles) {
  constexpr int LD = 64 + 8;      // rows 8 modulo 16 doubles apart: fragments without bank conflicts
  __shared__ __align__(16) double As[2][16][LD];
  __shared__ __align__(16) double Bs[2][16][LD];
  const SyrkTile t = tiles[blockIdx.x];
  const SyrkMat m = mats[t.mat];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, fr = lane >> 2, fk = lane & 3;
  const int i0 = t.ti * 64, j0 = t.tj * 64;
  const int k1 = t.k1;
  const int lc = (tid & 15) * 4, lk = tid >> 4;   // this thread fetches four columns of one row of either operand
  const int wr = (warp >> 1) * 16, wc = (warp & 1) * 32;
  const bool idle = t.ti == t.tj && wc > wr + 15;   // (all of it above the diagonal)
  double acc[2][4][2];
#pragma unroll
  for (int x = 0; x < 2; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y][0] = acc[x][y][1] = 0.0;
  uint2 ah, al, bh, bl;
  float4 af, bf;
  auto fetch = [&](int k0) {
    const int k = k0 + lk;
    const bool in_a = k < k1 && i0 + lc < m.L, in_b = k < k1 && j0 + lc < m.L;
    if constexpr (F32) {
      const float* row = m.f32 + static_cast<long long>(min(k, k1 - 1)) * m.L;
      const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
      af = in_a ? *reinterpret_cast<const float4*>(row + i0 + lc) : zero;
      bf = in_b ? *reinterpret_cast<const float4*>(row + j0 + lc) : zero;
      return;
    }
    const long long row = static_cast<long long>(min(k, k1 - 1)) * m.ld;
    const uint2 zero = make_uint2(0u, 0u);
    ah = in_a ? *reinterpret_cast<const uint2*>(m.hi + row + i0 + lc) : zero;
    al = in_a ? *reinterpret_cast<const uint2*>(m.lo + row + i0 + lc) : zero;
    bh = in_b ? *reinterpret_cast<const uint2*>(m.hi + row + j0 + lc) : zero;
    bl = in_b ? *reinterpret_cast<const uint2*>(m.lo + row + j0 + lc) : zero;
  };
  auto widen = [](uint32_t h, uint32_t l) {
    return make_double2(static_cast<double>(__uint_as_float(h << 16)) + static_cast<double>(__uint_as_float(l << 16)),
                        static_cast<double>(__uint_as_float(h & 0xffff0000u)) + static_cast<double>(__uint_as_float(l & 0xffff0000u)));
  };
  auto put = [&](int buf) {
    double2* a = reinterpret_cast<double2*>(&As[buf][lk][lc]);
    double2* b = reinterpret_cast<double2*>(&Bs[buf][lk][lc]);
    if constexpr (F32) {
      a[0] = make_double2(af.x, af.y); a[1] = make_double2(af.z, af.w);
      b[0] = make_double2(bf.x, bf.y); b[1] = make_double2(bf.z, bf.w);
    } else {
      a[0] = widen(ah.x, al.x); a[1] = widen(ah.y, al.y);
      b[0] = widen(bh.x, bl.x); b[1] = widen(bh.y, bl.y);
    }
  };
  fetch(t.k0);
  put(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = t.k0; k0 < k1; k0 += 16, buf ^= 1) {
    const bool more = k0 + 16 < k1;
    if (more) fetch(k0 + 16);
    if (!idle) {
#pragma unroll
      for (int kk = 0; kk < 16; kk += 4) {
        double a[2], b[4];
#pragma unroll
        for (int x = 0; x < 2; ++x) a[x] = As[buf][kk + fk][wr + 8 * x + fr];
#pragma unroll
        for (int y = 0; y < 4; ++y) b[y] = Bs[buf][kk + fk][wc + 8 * y + fr];
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y) dmma(acc[x][y], a[x], b[y]);
      }
    }
    if (more) put(buf ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int x = 0; x < 2; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = i0 + wr + 8 * x + fr, j = j0 + wc + 8 * y + 2 * fk + h;
        if (i < m.L && j <= i) atomicAdd(m.C + static_cast<long long>(i) * m.L + j, acc[x][y][h]);
      }
}

// Q = Y R^-1 in fp64 from an fp32 basis, rounded to fp32 once: the last pass over matrices with few rows (refresh_tc_short).
// One CTA per 64 x 64 tile of Q on the fp64 tensor cores; R^-1 is upper triangular, so a tile sums over the rows of R^-1 down to
// its own last column only.
struct ShortMat {
  const float* Y;       // rows x L
  const double* R;      // L x L
  float* Q;             // rows x L
  int rows, L;
};
struct ShortTile {
  int mat, m0, n0;
};
__global__ void __launch_bounds__(256) apply_f64_kernel(const ShortMat* mats, const ShortTile* tiles) {
  constexpr int LD = 64 + 8;      // (as in syrk_f64_kernel)
  __shared__ __align__(16) double As[2][16][LD];   // [k][row]
  __shared__ __align__(16) double Bs[2][16][LD];   // [k][column]
  const ShortTile t = tiles[blockIdx.x];
  const ShortMat m = mats[t.mat];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, fr = lane >> 2, fk = lane & 3;
  const int k1 = min(t.n0 + 64, m.L);
  const int ar = tid >> 2, ak = (tid & 3) * 4;     // of Y this thread fetches four columns of a row ...
  const int bk = tid >> 4, bc = (tid & 15) * 4;    // ... and of R^-1 as well
  const int wr = (warp >> 1) * 16, wc = (warp & 1) * 32;
  double acc[2][4][2];
#pragma unroll
  for (int x = 0; x < 2; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y][0] = acc[x][y][1] = 0.0;
  float4 a4;
  double2 b4[2];
  auto fetch = [&](int k0) {   // (L is a multiple of 4: four columns are inside together)
    a4 = t.m0 + ar < m.rows && k0 + ak < k1 ? *reinterpret_cast<const float4*>(m.Y + static_cast<long long>(t.m0 + ar) * m.L + k0 + ak)
                                            : make_float4(0.f, 0.f, 0.f, 0.f);
    const bool in_b = k0 + bk < k1 && t.n0 + bc < m.L;
    const double2* row = reinterpret_cast<const double2*>(m.R + static_cast<long long>(k0 + bk) * m.L + t.n0 + bc);
    b4[0] = in_b ? row[0] : make_double2(0.0, 0.0);
    b4[1] = in_b ? row[1] : make_double2(0.0, 0.0);
  };
  auto put = [&](int buf) {
    As[buf][ak][ar] = a4.x; As[buf][ak + 1][ar] = a4.y; As[buf][ak + 2][ar] = a4.z; As[buf][ak + 3][ar] = a4.w;
    double2* b = reinterpret_cast<double2*>(&Bs[buf][bk][bc]);
    b[0] = b4[0]; b[1] = b4[1];
  };
  fetch(0);
  put(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < k1; k0 += 16, buf ^= 1) {
    const bool more = k0 + 16 < k1;
    if (more) fetch(k0 + 16);
#pragma unroll
    for (int kk = 0; kk < 16; kk += 4) {
      double a[2], b[4];
#pragma unroll
      for (int x = 0; x < 2; ++x) a[x] = As[buf][kk + fk][wr + 8 * x + fr];
#pragma unroll
      for (int y = 0; y < 4; ++y) b[y] = Bs[buf][kk + fk][wc + 8 * y + fr];
#pragma unroll
      for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) dmma(acc[x][y], a[x], b[y]);
    }
    if (more) put(buf ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int x = 0; x < 2; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const int i = t.m0 + wr + 8 * x + fr, j = t.n0 + wc + 8 * y + 2 * fk;
      if (i < m.rows && j < m.L)
        *reinterpret_cast<float2*>(m.Q + static_cast<long long>(i) * m.L + j) = make_float2(static_cast<float>(acc[x][y][0]), static_cast<float>(acc[x][y][1]));
    }
}

struct NewtonJob {
  const float* C32;     // L x L, lower triangle valid
  __nv_bfloat16 *Rhi, *Rlo;
  int L, ld;
};

// Second-order orthonormalisation of a basis that is orthonormal to first order already: with C = Q^T Q = I + E,
// Q (I - E / 2) has Q^T Q = I + O(E^2).  C comes from the tensor cores (its error, about 1e-7 on an entry for columns
// of unit norm, is what is left of E afterwards); S = I - E / 2 = 1.5 I - C / 2 is written in two bf16 parts where the
// product Q = Y R^-1 expects R^-1.  blockIdx.x = matrix, blockIdx.y = share of the 32 x 32 blocks of its lower triangle: a block is
// read once, row by row, and goes out as itself and transposed through shared memory (read column by column for the upper
// half, 156 matrices of up to 512 columns took 133 us and 86 of 256 20.5; so 72 and 16).
__global__ void __launch_bounds__(256) newton_prep_kernel(const NewtonJob* jobs) {
  __shared__ float tile[32][33];
  const NewtonJob g = jobs[blockIdx.x];
  pdl_begin();
  const int nb = (g.L + 31) >> 5, lane = threadIdx.x & 31, row = threadIdx.x >> 5;
  auto put = [&](int j, int i, float c) {
    const float f = i == j ? 1.5f - 0.5f * c : -0.5f * c;
    const __nv_bfloat16 h = __float2bfloat16_rn(f);
    g.Rhi[j * g.ld + i] = h;
    g.Rlo[j * g.ld + i] = __float2bfloat16_rn(f - __bfloat162float(h));
  };
  for (int b = blockIdx.y; b < nb * (nb + 1) / 2; b += gridDim.y) {
    int bi = static_cast<int>((sqrtf(8.f * b + 1.f) - 1.f) * 0.5f);
    while ((bi + 1) * (bi + 2) / 2 <= b) ++bi;
    while (bi * (bi + 1) / 2 > b) --bi;
    const int r0 = bi * 32, c0 = (b - bi * (bi + 1) / 2) * 32;
    __syncthreads();
#pragma unroll
    for (int y = row; y < 32; y += 8) {
      const int j = r0 + y, i = c0 + lane;
      if (j < g.L && i <= j) {
        const float c = g.C32[j * g.L + i];
        tile[y][lane] = c;
        put(j, i, c);
      }
    }
    __syncthreads();
#pragma unroll
    for (int y = row; y < 32; y += 8) {
      const int j = c0 + y, i = r0 + lane;
      if (i < g.L && i > j) put(j, i, tile[lane][y]);
    }
  }
}

// ------------------------------------------------------------------------------------------ plan

// RG_APPLY_TRI: RG_APPLY_Y with an upper triangular right operand (its blocks of zeros are left out)
enum RefreshGemm { RG_Y_FROM_Z = 0, RG_Z_FROM_Y, RG_GRAM_Y, RG_GRAM_Z, RG_APPLY_Y, RG_APPLY_TRI, RG_COUNT };
// The basis Y is kept as two bf16 parts, in two sets that take turns: a product with G leaves it in set 0, Q = Y R^-1 goes
// from one set to the other (its tiles read whole rows of Y while others write).  Set 1 shares the memory of the fp32
// buffer Yf, which only the result of the refresh and the products with a split K use.
enum RefreshMap { RM_G_A = 0, RM_G_MN, RM_Z_B, RM_Z_B_LO, RM_Y_B, RM_Y_B_LO, RM_Y_A, RM_Y_A_LO,
                  RM_Y1_B, RM_Y1_B_LO, RM_Y1_A, RM_Y1_A_LO, RM_RINV, RM_RINV_LO, RM_COUNT };
// The problem tables: a kind of product (RefreshGemm: its tiles) with its operands' and result's place.
enum RefreshProb { RP_Y_FROM_Z = 0, RP_Z_FROM_Y0, RP_Z_FROM_Y1, RP_GRAM_Y0, RP_GRAM_Y1, RP_GRAM_Z, RP_APPLY_01, RP_APPLY_10,
                   RP_APPLY_0F, RP_COUNT };

struct RefreshMat {
  int M, N, L, ldl;
  float *Yf, *Zf;                       // fp32 GEMM outputs (M x L, N x L)
  __nv_bfloat16 *Yhi, *Ylo, *Zhi, *Zlo; // bf16 parts of the iterates (rows x ldl), Y in set 0
  __nv_bfloat16 *Y1hi, *Y1lo;           // Y in set 1 (the memory of Yf, M x ldl floats)
  float* C32;                           // L x L
  double *C64, *X64, *T64;              // L x L each
  double* D;                            // L column norms (sums of squares) of the result
  __nv_bfloat16 *Rhi, *Rlo;             // L x ldl
};

constexpr int kRefBN = 128;
// The products with G take tiles of 256 columns where most of the work has bases that wide: a 128 x 256 tile needs
// three quarters of the shared-memory reads per multiply-add, and G is read half as often.
constexpr int kRefWideBN = 256;
// A product with G (one part of A, NB parts of B): 192 KB of stages, as many as go.
template <int BN, int NB, int MT, bool MN>
struct RefProduct {
  static constexpr int kEpiWarps = 8, kThreads = 64 + 32 * kEpiWarps;
  static constexpr int kStages = 192 / (16 * MT + NB * BN / 8);
  static constexpr int kSmem = TcSmem<BN, 1, NB, kStages, kEpiWarps, MT>::kTotal;
  static constexpr auto kernel = tc_gemm_kernel<BN, 1, NB, kStages, TC_EPI_STORE, kEpiWarps, MN, false, MT>;
};
// Matrices with fewer rows than this end with a pass in fp64 (refresh_tc_short).
constexpr int kShortRows = 512;
constexpr int kRefStages2 = 3;  // NA = 2, NB = 2: 64 KB per stage

struct RefreshPlan {
  bool ready = false;
  size_t device_bytes = 0;
  EncodeTiledFn encode = nullptr;
  int n = 0;
  std::vector<RefreshMat> mats;
  std::vector<CUtensorMap> h_maps;  // RM_COUNT per matrix
  std::vector<const void*> last_G;
  char* buf = nullptr;
  CUtensorMap* d_maps = nullptr;
  TcProblem* d_probs[RP_COUNT] = {};
  TcTile* d_tiles[RG_COUNT] = {};
  int* d_first[RG_COUNT] = {};   // first tile of every CTA
  int n_tiles[RG_COUNT] = {};
  int grid[RG_COUNT] = {};
  bool wide = false;           // the products with G take tiles of kRefWideBN columns ...
  bool tall = false;           // ... and of 256 rows
  bool pair = false;           // ... on pairs of SMs
  bool brief = false;          // the kernels between the products are programmatic dependents
  std::vector<int> atomic_mats[RG_COUNT];  // matrices whose K is split for this GEMM (output must be zeroed)
  // buffers to clear before GEMM kind g (the outputs of atomic_mats[g]); entry RG_COUNT: every matrix's X64
  ZeroJob* d_zero[RG_COUNT + 1] = {};
  int n_zero[RG_COUNT + 1] = {};
  char* zero_tables = nullptr;
  NewtonJob* d_newton = nullptr;
  FactorMat* d_factor32 = nullptr;   // R^-1 from C32 (tri_factor.cuh), widest first
  FactorMat* d_factor64 = nullptr;   // R^-1 from the exact Gram matrix in X64
  int l_max = 0;  // largest basis width L of the set
  int cluster = 1, short_cluster = 1;   // CTAs that factor a matrix together, of all and of the short ones
  // the matrices whose product with G splits K (their result arrives as fp32 and is split afterwards; all others
  // leave the product as bf16 parts already)
  SplitJob* d_split_y_rest = nullptr;
  SplitJob* d_split_z_rest = nullptr;
  int n_split_y_rest = 0, n_split_z_rest = 0;
  SyrkMat* d_syrk_mats = nullptr;
  SyrkTile* d_syrk_tiles = nullptr;
  int n_syrk_tiles = 0;
  // Rayleigh-Ritz rotation: the eigensolver works in the X64, T64 and C64 buffers
  EigMat* d_eig = nullptr;
  FactorMat* d_eig_factor = nullptr;
  int eig_max = 0;             // largest matrix it diagonalises
  int sm_count = 0;
  FillJob* d_fill = nullptr;   // the random start Z = Omega of every matrix
  int fill_blocks = 1;         // blocks a matrix: eight entries a thread in the largest
  // the last exact pass over the matrices with fewer than kShortRows rows (refresh_tc_short)
  std::vector<char> is_short;
  int n_short = 0, short_l_max = 0, n_short_syrk = 0, n_short_tiles = 0;
  SyrkMat* d_short_syrk_mats = nullptr;
  SyrkTile* d_short_syrk_tiles = nullptr;
  FactorMat* d_short_factor = nullptr;
  ShortMat* d_short = nullptr;
  ShortTile* d_short_tiles = nullptr;
  ZeroJob* d_short_zero = nullptr;
  ZeroJob* d_zero_d = nullptr;   // clears every matrix's D (as 16-byte words)
};

inline void refresh_plan_destroy(RefreshPlan& plan) {
  if (plan.buf) cudaFree(plan.buf);
  if (plan.zero_tables) cudaFree(plan.zero_tables);
  plan.zero_tables = nullptr;
  plan.buf = nullptr;
  plan.ready = false;
}

inline ngalore_status refresh_plan_create(RefreshPlan& plan, const std::vector<MatDesc>& mats,
                                          const std::vector<float*>& Yf, const std::vector<float*>& Zf,
                                          const std::vector<float*>& Yshort, int sm_count, int ritz_columns) {
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || fn == nullptr)
    return NGALORE_ERR_CUDA;
  plan.encode = reinterpret_cast<EncodeTiledFn>(fn);
  const int n = static_cast<int>(mats.size());
  plan.n = n;
  plan.sm_count = sm_count;
  plan.mats.resize(n);
  plan.last_G.assign(n, nullptr);

  // ---- tile and problem tables (host)
  std::vector<TcProblem> probs[RP_COUNT];
  std::vector<TcTile> tiles[RG_COUNT];
  for (int g = 0; g < RP_COUNT; ++g) probs[g].resize(n);
  {
    double all = 0.0, wide = 0.0;
    for (int i = 0; i < n; ++i) {
      const double w = static_cast<double>(mats[i].M) * mats[i].N * mats[i].rp;
      all += w;
      if (mats[i].rp > 192) wide += w;
    }
    plan.wide = 2.0 * wide >= all;
  }
  int pairs = 0;
  {
    // Tiles of 256 rows: what bounds the products with G is the L2 bandwidth (10 TB/s), and two accumulators that share
    // the basis halve its part of the traffic.  1.1B shapes, a product with two parts 1.86 -> 1.59 ms, with one 1.02 ->
    // 0.94; 60M 44 -> 40 and 36 -> 34 us.  Not where that leaves SMs without a tile.  256 x 256 accumulators fill the
    // tensor memory, so the epilogue of a tile is not hidden behind the next: of 15 K blocks a tile (130M shapes) 140 us
    // become 146 (two parts) and 88 become 96 (one), of 40 (1.1B) it pays.
    const int bn = plan.wide ? kRefWideBN : kRefBN;
    long long tiles_tall = 0, blocks = 0;
    for (const MatDesc& d : mats) {
      const long long cols = (d.rp + bn - 1) / bn, ty = (d.M + 2 * kTcBM - 1) / (2 * kTcBM) * cols, tz = (d.N + 2 * kTcBM - 1) / (2 * kTcBM) * cols;
      tiles_tall += ty + tz;
      blocks += ty * ((d.N + kTcBK - 1) / kTcBK) + tz * ((d.M + kTcBK - 1) / kTcBK);
    }
    plan.tall = tiles_tall >= 2 * sm_count && (!plan.wide || blocks >= 24 * tiles_tall);
    // 256 x 256 tiles on pairs of SMs (gemm_pair_tcgen05.cuh, which has the figures) where they are too short for the two
    // accumulators of one CTA, and enough of them to balance the pairs.
    if (plan.wide && !plan.tall && tiles_tall >= 2 * sm_count) {
      pairs = std::min(tc_pair_init(), sm_count / 2);
      plan.pair = 2 * pairs >= sm_count - 4;
    }
  }
  auto tile_rows = [&](int g) { return (plan.tall || plan.pair) && (g == RG_Y_FROM_Z || g == RG_Z_FROM_Y) ? 2 * kTcBM : kTcBM; };
  auto tile_cols = [&](int g) { return plan.wide && (g == RG_Y_FROM_Z || g == RG_Z_FROM_Y) ? kRefWideBN : kRefBN; };
  auto add_tiles = [&](int g, int i, int out_rows, int out_cols, int K, long long target_kb) {
    const int kb_total = (K + kTcBK - 1) / kTcBK;
    if (g == RG_APPLY_Y || g == RG_APPLY_TRI) {
      // the tiles that read the same rows of Y one after another, the longest first: side by side in time they share
      // them in L2 (sorted by length over all matrices, Y came from DRAM once per column tile: 1.1B shapes 500 -> 465 us a
      // product, 84 matrices of r' = 256 69 -> 66 us)
      for (int m0 = 0; m0 < out_rows; m0 += kTcBM)
        for (int n0 = (out_cols - 1) / kRefBN * kRefBN; n0 >= 0; n0 -= kRefBN)
          tiles[g].push_back(TcTile{i, m0, n0, 0, g == RG_APPLY_TRI ? std::min(kb_total, (n0 + kRefBN) / kTcBK) : kb_total, 0, out_rows, out_cols});
      return;
    }
    // (to the nearest number: a K a little over the target costs less balance than two tiles cost atomics)
    int splits = static_cast<int>((kb_total + target_kb / 2) / target_kb);
    if (splits < 1) splits = 1;
    // Gram matrices have few tiles, of three products a K block: two halves from 16 blocks on (58 of r' = 128 24 -> 20.5 us; three
    // sums and more would depend on the order of the atomics)
    if ((g == RG_GRAM_Y || g == RG_GRAM_Z) && splits == 1 && kb_total >= 16 && target_kb == 16) splits = 2;
    const int kb_per = (kb_total + splits - 1) / splits;
    splits = (kb_total + kb_per - 1) / kb_per;
    if (splits > 1) plan.atomic_mats[g].push_back(i);
    const bool symmetric = g == RG_GRAM_Y || g == RG_GRAM_Z;   // the lower triangle is enough
    for (int n0 = 0; n0 < out_cols; n0 += tile_cols(g))
      for (int sp = 0; sp < splits; ++sp)
        for (int m0 = symmetric ? n0 / kTcBM * kTcBM : 0; m0 < out_rows; m0 += tile_rows(g)) {
          const int kb0 = sp * kb_per;
          const int kbn = std::min(kb_per, kb_total - kb0);
          tiles[g].push_back(TcTile{i, m0, n0, kb0 * kTcBK, kbn, splits > 1 ? 1 : 0, out_rows, out_cols});
        }
  };

  // ---- device buffer layout
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) / 256 * 256; return o; };
  struct Offs { size_t Yhi, Ylo, Zhi, Zlo, C32, C64, X64, T64, D, Rhi, Rlo; };
  std::vector<Offs> offs(n);
  for (int i = 0; i < n; ++i) {
    RefreshMat& m = plan.mats[i];
    m.M = mats[i].M; m.N = mats[i].N; m.L = mats[i].rp; m.ldl = (m.L + 7) / 8 * 8;
    m.Yf = Yf[i]; m.Zf = Zf[i];
    offs[i].Yhi = take(sizeof(__nv_bfloat16) * m.M * m.ldl);
    offs[i].Ylo = take(sizeof(__nv_bfloat16) * m.M * m.ldl);
    offs[i].Zhi = take(sizeof(__nv_bfloat16) * m.N * m.ldl);
    offs[i].Zlo = take(sizeof(__nv_bfloat16) * m.N * m.ldl);
    offs[i].C32 = take(sizeof(float) * m.L * m.L);
    offs[i].C64 = take(std::max(sizeof(double) * m.L * m.L, tf_block_bytes(m.L)));   // (also holds the factor's blocks)
    const size_t l2 = std::max(static_cast<size_t>(m.L) * m.L, tf_spill_doubles(m.L));   // (both also hold the factor's rows)
    offs[i].X64 = take(sizeof(double) * l2);
    offs[i].T64 = take(sizeof(double) * l2);
    offs[i].D = take(sizeof(double) * m.L);
    offs[i].Rhi = take(sizeof(__nv_bfloat16) * m.L * m.ldl);
    offs[i].Rlo = take(sizeof(__nv_bfloat16) * m.L * m.ldl);
  }
  const size_t o_maps = take(sizeof(CUtensorMap) * RM_COUNT * n);
  size_t o_probs[RP_COUNT], o_tiles[RG_COUNT], o_first[RG_COUNT];
  std::vector<int> tile_first[RG_COUNT];
  for (int g = 0; g < RP_COUNT; ++g) o_probs[g] = take(sizeof(TcProblem) * n);

  // work estimate for the split-K targets: per GEMM kind, k-blocks per CTA if perfectly balanced
  for (int g = 0; g < RG_COUNT; ++g) {
    long long total_kb = 0;
    for (int i = 0; i < n; ++i) {
      const RefreshMat& m = plan.mats[i];
      int rows, cols, K;
      switch (g) {
        case RG_Y_FROM_Z: rows = m.M; cols = m.L; K = m.N; break;
        case RG_Z_FROM_Y: rows = m.N; cols = m.L; K = m.M; break;
        case RG_GRAM_Y: rows = m.L; cols = m.L; K = m.M; break;
        case RG_GRAM_Z: rows = m.L; cols = m.L; K = m.N; break;
        default: rows = m.M; cols = m.L; K = m.L; break;  // RG_APPLY_Y, RG_APPLY_TRI
      }
      total_kb += static_cast<long long>((rows + tile_rows(g) - 1) / tile_rows(g)) * ((cols + tile_cols(g) - 1) / tile_cols(g)) *
                  ((K + kTcBK - 1) / kTcBK);
    }
    long long target = (total_kb * (tile_rows(g) / kTcBM) + sm_count - 1) / sm_count / 4;
    if (target < 16) target = 16;
    for (int i = 0; i < n; ++i) {
      const RefreshMat& m = plan.mats[i];
      int rows, cols, K;
      switch (g) {
        case RG_Y_FROM_Z: rows = m.M; cols = m.L; K = m.N; break;
        case RG_Z_FROM_Y: rows = m.N; cols = m.L; K = m.M; break;
        case RG_GRAM_Y: rows = m.L; cols = m.L; K = m.M; break;
        case RG_GRAM_Z: rows = m.L; cols = m.L; K = m.N; break;
        default: rows = m.M; cols = m.L; K = m.L; break;  // RG_APPLY_Y, RG_APPLY_TRI
      }
      add_tiles(g, i, rows, cols, K, target);
    }
    o_tiles[g] = take(sizeof(TcTile) * tiles[g].size());
    plan.n_tiles[g] = static_cast<int>(tiles[g].size());
    plan.grid[g] = std::min(plan.n_tiles[g], plan.pair && (g == RG_Y_FROM_Z || g == RG_Z_FROM_Y) ? pairs : sm_count);   // (CTAs, or pairs)
    tc_assign_tiles(tiles[g], plan.grid[g], tile_first[g], g == RG_APPLY_Y || g == RG_APPLY_TRI);
    o_first[g] = take(sizeof(int) * tile_first[g].size());
  }
  // Programmatic dependents, for what has one wave of CTAs and is short: the start of a kernel (launch, barriers, tensor memory) and
  // the end of the one before are a third of it.  Refresh, with ordinary launches / so: three small matrices 610 / 490 us, 824-wide
  // layers at r = 48 943 / 819, 1264-wide at r = 8 1240 / 1069, 60M shapes (5 tiles a CTA in the products with R^-1) 2200 / 2117,
  // 37 and 74 matrices of 768 rows at r = 160 1881 / 1817 and 2427 / 2356.  Not with wide bases, whose factorisations are long: at
  // r = 224 2974 / 3048 and 3644 / 3658, at r = 256 3660 / 3808 and 4410 / 4452, 130M shapes 6777 / 6820; nor the kernels of the
  // eigensolver: 60M shapes 2200 / 2292.
  plan.brief = !plan.wide && plan.n_tiles[RG_APPLY_TRI] <= 8 * sm_count;
  const size_t o_newton = take(sizeof(NewtonJob) * n);
  const size_t o_factor32 = take(sizeof(FactorMat) * n);
  const size_t o_factor64 = take(sizeof(FactorMat) * n);
  std::vector<SyrkTile> syrk_tiles;
  plan.is_short.resize(n);
  for (int i = 0; i < n; ++i) plan.is_short[i] = plan.mats[i].M < kShortRows ? 1 : 0;
  auto slabs = [&](int slab, bool short_only = false) {
    syrk_tiles.clear();
    for (int i = 0; i < n; ++i) {
      if (short_only && !plan.is_short[i]) continue;
      const int nt = (plan.mats[i].L + 63) / 64, rows = plan.mats[i].M;
      const int step = rows <= 2 * kSyrkRows ? std::max(slab, (rows / 2 + 15) & ~15) : slab;
      for (int k0 = 0; k0 < rows; k0 += step)
        for (int ti = 0; ti < nt; ++ti)
          for (int tj = 0; tj <= ti; ++tj) syrk_tiles.push_back(SyrkTile{i, ti, tj, k0, std::min(k0 + step, rows)});
    }
  };
  slabs(kSyrkRows);
  if (static_cast<int>(syrk_tiles.size()) < kSyrkFewTiles * sm_count) slabs(kSyrkRowsFew);
  const std::vector<SyrkTile> all_syrk_tiles = syrk_tiles;
  slabs(kSyrkRowsFew, true);
  const std::vector<SyrkTile> short_syrk_tiles = syrk_tiles;
  syrk_tiles = all_syrk_tiles;
  std::vector<ShortTile> short_tiles;
  for (int i = 0; i < n; ++i)
    if (plan.is_short[i])
      for (int n0 = (plan.mats[i].L - 1) / 64 * 64; n0 >= 0; n0 -= 64)   // (the longest sums first)
        for (int m0 = 0; m0 < plan.mats[i].M; m0 += 64) short_tiles.push_back(ShortTile{i, m0, n0});
  plan.n_short_syrk = static_cast<int>(short_syrk_tiles.size());
  plan.n_short_tiles = static_cast<int>(short_tiles.size());
  plan.n_syrk_tiles = static_cast<int>(syrk_tiles.size());
  const size_t o_syrk_m = take(sizeof(SyrkMat) * n);
  const size_t o_syrk_t = take(sizeof(SyrkTile) * syrk_tiles.size());
  const size_t o_sy_rest = take(sizeof(SplitJob) * n);
  const size_t o_sz_rest = take(sizeof(SplitJob) * n);
  const size_t o_eig = take(sizeof(EigMat) * n);
  const size_t o_eig_factor = take(sizeof(FactorMat) * n);
  const size_t o_eig_redo = take(sizeof(int) * n);
  const size_t o_fill = take(sizeof(FillJob) * n);
  const size_t o_zero_d = take(sizeof(ZeroJob) * n);
  const size_t o_short_syrk_m = take(sizeof(SyrkMat) * n);
  const size_t o_short_syrk_t = take(sizeof(SyrkTile) * short_syrk_tiles.size());
  const size_t o_short_factor = take(sizeof(FactorMat) * n);
  const size_t o_short_m = take(sizeof(ShortMat) * n);
  const size_t o_short_t = take(sizeof(ShortTile) * short_tiles.size());
  const size_t o_short_zero = take(sizeof(ZeroJob) * n);
  std::vector<size_t> o_eig_tri(n);
  for (int i = 0; i < n; ++i) o_eig_tri[i] = take(sizeof(double) * eig_tri_doubles(plan.mats[i].L));
  if (cudaMalloc(&plan.buf, off) != cudaSuccess) { plan.buf = nullptr; return NGALORE_ERR_ALLOC; }
  if (cudaMemset(plan.buf, 0, off) != cudaSuccess) return NGALORE_ERR_CUDA;
  plan.device_bytes = off;

  std::vector<NewtonJob> newton(n);
  std::vector<FactorMat> factor32(n), factor64(n);
  plan.l_max = 0;
  for (const RefreshMat& m : plan.mats) plan.l_max = m.L > plan.l_max ? m.L : plan.l_max;
  std::vector<SplitJob> sy_rest, sz_rest;
  std::vector<SyrkMat> syrk_m(n), short_syrk_m(n);
  std::vector<FactorMat> short_factor;
  std::vector<ShortMat> short_m(n);
  std::vector<ZeroJob> short_zero;
  std::vector<EigMat> eig(n);
  std::vector<FactorMat> eig_factors(n);
  plan.h_maps.resize(static_cast<size_t>(RM_COUNT) * n);
  std::memset(plan.h_maps.data(), 0, sizeof(CUtensorMap) * plan.h_maps.size());
  for (int i = 0; i < n; ++i) {
    RefreshMat& m = plan.mats[i];
    m.Yhi = reinterpret_cast<__nv_bfloat16*>(plan.buf + offs[i].Yhi);
    m.Ylo = reinterpret_cast<__nv_bfloat16*>(plan.buf + offs[i].Ylo);
    m.Zhi = reinterpret_cast<__nv_bfloat16*>(plan.buf + offs[i].Zhi);
    m.Zlo = reinterpret_cast<__nv_bfloat16*>(plan.buf + offs[i].Zlo);
    m.C32 = reinterpret_cast<float*>(plan.buf + offs[i].C32);
    m.C64 = reinterpret_cast<double*>(plan.buf + offs[i].C64);
    m.X64 = reinterpret_cast<double*>(plan.buf + offs[i].X64);
    m.T64 = reinterpret_cast<double*>(plan.buf + offs[i].T64);
    m.D = reinterpret_cast<double*>(plan.buf + offs[i].D);
    m.Rhi = reinterpret_cast<__nv_bfloat16*>(plan.buf + offs[i].Rhi);
    m.Rlo = reinterpret_cast<__nv_bfloat16*>(plan.buf + offs[i].Rlo);
    newton[i] = NewtonJob{m.C32, m.Rhi, m.Rlo, m.L, m.ldl};
    factor32[i] = FactorMat{m.C32, nullptr, m.C64, m.T64, m.Rhi, m.Rlo, m.L, m.ldl};
    factor64[i] = FactorMat{nullptr, m.X64, m.C64, m.T64, m.Rhi, m.Rlo, m.L, m.ldl};
    m.Y1hi = reinterpret_cast<__nv_bfloat16*>(m.Yf);
    m.Y1lo = m.Y1hi + static_cast<size_t>(m.M) * m.ldl;
    syrk_m[i] = SyrkMat{m.Y1hi, m.Y1lo, nullptr, m.X64, m.M, m.L, m.ldl};
    short_syrk_m[i] = SyrkMat{nullptr, nullptr, m.Yf, m.X64, m.M, m.L, m.L};
    short_m[i] = ShortMat{m.Yf, m.X64, Yshort[i], m.M, m.L};
    if (plan.is_short[i]) {
      short_factor.push_back(FactorMat{nullptr, m.X64, m.C64, m.T64, nullptr, nullptr, m.L, 0, m.X64});
      short_zero.push_back(ZeroJob{reinterpret_cast<float4*>(m.X64), static_cast<long long>(m.L) * m.L * 8 / 16});
      plan.short_l_max = std::max(plan.short_l_max, m.L);
    }
    if (std::find(plan.atomic_mats[RG_Y_FROM_Z].begin(), plan.atomic_mats[RG_Y_FROM_Z].end(), i) != plan.atomic_mats[RG_Y_FROM_Z].end())
      sy_rest.push_back(SplitJob{m.Yf, m.Yhi, m.Ylo, static_cast<long long>(m.M) * m.L, m.L, m.ldl});
    if (std::find(plan.atomic_mats[RG_Z_FROM_Y].begin(), plan.atomic_mats[RG_Z_FROM_Y].end(), i) != plan.atomic_mats[RG_Z_FROM_Y].end())
      sz_rest.push_back(SplitJob{m.Zf, m.Zhi, m.Zlo, static_cast<long long>(m.N) * m.L, m.L, m.ldl});
    // (the rotated part: all of the basis, or its leading ritz_columns, kept a multiple of 4)
    const int Lj = std::min(m.L, (ritz_columns + 3) & ~3);
    int* redo = reinterpret_cast<int*>(plan.buf + o_eig_redo) + i;
    eig[i] = EigMat{m.C32, nullptr, m.L, Lj, Lj, m.X64, m.T64, m.C64, reinterpret_cast<double*>(plan.buf + o_eig_tri[i]),
                    redo, nullptr, 0, m.Rhi, m.Rlo, m.ldl, m.L};
    eig_factors[i] = eig_factor(eig[i]);
    plan.eig_max = std::max(plan.eig_max, Lj);
    CUtensorMap* mp = &plan.h_maps[static_cast<size_t>(i) * RM_COUNT];
    const uint64_t sl = static_cast<uint64_t>(m.ldl) * 2;
    bool ok = true;
    ok &= tc_encode_2d(plan.encode, mp + RM_Z_B, m.Zhi, m.L, m.N, sl, 64, kTcBK);
    ok &= tc_encode_2d(plan.encode, mp + RM_Z_B_LO, m.Zlo, m.L, m.N, sl, 64, kTcBK);
    ok &= tc_encode_2d(plan.encode, mp + RM_Y_B, m.Yhi, m.L, m.M, sl, 64, kTcBK);
    ok &= tc_encode_2d(plan.encode, mp + RM_Y_B_LO, m.Ylo, m.L, m.M, sl, 64, kTcBK);
    ok &= tc_encode_2d(plan.encode, mp + RM_Y_A, m.Yhi, m.L, m.M, sl, kTcBK, kTcBM);
    ok &= tc_encode_2d(plan.encode, mp + RM_Y_A_LO, m.Ylo, m.L, m.M, sl, kTcBK, kTcBM);
    ok &= tc_encode_2d(plan.encode, mp + RM_Y1_B, m.Y1hi, m.L, m.M, sl, 64, kTcBK);
    ok &= tc_encode_2d(plan.encode, mp + RM_Y1_B_LO, m.Y1lo, m.L, m.M, sl, 64, kTcBK);
    ok &= tc_encode_2d(plan.encode, mp + RM_Y1_A, m.Y1hi, m.L, m.M, sl, kTcBK, kTcBM);
    ok &= tc_encode_2d(plan.encode, mp + RM_Y1_A_LO, m.Y1lo, m.L, m.M, sl, kTcBK, kTcBM);
    ok &= tc_encode_2d(plan.encode, mp + RM_RINV, m.Rhi, m.L, m.L, sl, 64, kTcBK);
    ok &= tc_encode_2d(plan.encode, mp + RM_RINV_LO, m.Rlo, m.L, m.L, sl, 64, kTcBK);
    if (!ok) return NGALORE_ERR_CUDA;
    const int base = i * RM_COUNT;
    // result as bf16 parts (hi == nullptr: as fp32)
    auto problem = [&](float* out, int rows, int map_a, int map_b, __nv_bfloat16* hi, __nv_bfloat16* lo) {
      TcProblem q{out, rows, m.L, m.L, base + map_a, base + map_b, 0};
      if (hi != nullptr) { q.ld16 = m.ldl; q.out_hi = hi; q.out_lo = lo; }
      return q;
    };
    auto is_split = [&](int g) {
      const std::vector<int>& a = plan.atomic_mats[g];
      return std::find(a.begin(), a.end(), i) != a.end();
    };
    probs[RP_Y_FROM_Z][i] = problem(m.Yf, m.M, RM_G_A, RM_Z_B, is_split(RG_Y_FROM_Z) ? nullptr : m.Yhi, m.Ylo);
    probs[RP_Z_FROM_Y0][i] = problem(m.Zf, m.N, RM_G_MN, RM_Y_B, is_split(RG_Z_FROM_Y) ? nullptr : m.Zhi, m.Zlo);
    probs[RP_Z_FROM_Y1][i] = problem(m.Zf, m.N, RM_G_MN, RM_Y1_B, is_split(RG_Z_FROM_Y) ? nullptr : m.Zhi, m.Zlo);
    probs[RP_GRAM_Y0][i] = problem(m.C32, m.L, RM_Y_B, RM_Y_B, nullptr, nullptr);
    probs[RP_GRAM_Y1][i] = problem(m.C32, m.L, RM_Y1_B, RM_Y1_B, nullptr, nullptr);
    probs[RP_GRAM_Z][i] = problem(m.C32, m.L, RM_Z_B, RM_Z_B, nullptr, nullptr);
    probs[RP_APPLY_01][i] = problem(nullptr, m.M, RM_Y_A, RM_RINV, m.Y1hi, m.Y1lo);
    probs[RP_APPLY_10][i] = problem(nullptr, m.M, RM_Y1_A, RM_RINV, m.Yhi, m.Ylo);
    probs[RP_APPLY_0F][i] = problem(m.Yf, m.M, RM_Y_A, RM_RINV, nullptr, nullptr);
  }
  plan.d_maps = reinterpret_cast<CUtensorMap*>(plan.buf + o_maps);
  for (int g = 0; g < RP_COUNT; ++g) {
    plan.d_probs[g] = reinterpret_cast<TcProblem*>(plan.buf + o_probs[g]);
    if (cudaMemcpy(plan.d_probs[g], probs[g].data(), sizeof(TcProblem) * n, cudaMemcpyHostToDevice) != cudaSuccess) return NGALORE_ERR_CUDA;
  }
  for (int g = 0; g < RG_COUNT; ++g) {
    plan.d_tiles[g] = reinterpret_cast<TcTile*>(plan.buf + o_tiles[g]);
    plan.d_first[g] = reinterpret_cast<int*>(plan.buf + o_first[g]);
    if (cudaMemcpy(plan.d_first[g], tile_first[g].data(), sizeof(int) * tile_first[g].size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(plan.d_tiles[g], tiles[g].data(), sizeof(TcTile) * tiles[g].size(), cudaMemcpyHostToDevice) != cudaSuccess)
      return NGALORE_ERR_CUDA;
  }
  plan.d_newton = reinterpret_cast<NewtonJob*>(plan.buf + o_newton);
  plan.d_factor32 = reinterpret_cast<FactorMat*>(plan.buf + o_factor32);
  plan.d_factor64 = reinterpret_cast<FactorMat*>(plan.buf + o_factor64);
  auto wider = [](const FactorMat& a, const FactorMat& b) { return a.L > b.L; };
  std::stable_sort(factor32.begin(), factor32.end(), wider);
  std::stable_sort(factor64.begin(), factor64.end(), wider);
  plan.d_syrk_mats = reinterpret_cast<SyrkMat*>(plan.buf + o_syrk_m);
  plan.d_syrk_tiles = reinterpret_cast<SyrkTile*>(plan.buf + o_syrk_t);
  plan.d_split_y_rest = reinterpret_cast<SplitJob*>(plan.buf + o_sy_rest);
  plan.d_split_z_rest = reinterpret_cast<SplitJob*>(plan.buf + o_sz_rest);
  plan.n_split_y_rest = static_cast<int>(sy_rest.size());
  plan.n_split_z_rest = static_cast<int>(sz_rest.size());
  plan.d_eig = reinterpret_cast<EigMat*>(plan.buf + o_eig);
  plan.d_eig_factor = reinterpret_cast<FactorMat*>(plan.buf + o_eig_factor);
  std::stable_sort(eig_factors.begin(), eig_factors.end(), wider);
  plan.d_fill = reinterpret_cast<FillJob*>(plan.buf + o_fill);
  {
    std::vector<FillJob> fill(n);
    for (int i = 0; i < n; ++i) {
      const RefreshMat& m = plan.mats[i];
      fill[i] = FillJob{m.Zhi, m.Zlo, static_cast<long long>(m.N) * m.L, m.L, m.ldl};
      plan.fill_blocks = std::max(plan.fill_blocks, static_cast<int>(std::min<long long>(512, (fill[i].n + 2047) / 2048)));
    }
    if (cudaMemcpy(plan.d_fill, fill.data(), sizeof(FillJob) * n, cudaMemcpyHostToDevice) != cudaSuccess) return NGALORE_ERR_CUDA;
  }
  plan.d_zero_d = reinterpret_cast<ZeroJob*>(plan.buf + o_zero_d);
  {
    std::vector<ZeroJob> zd(n);
    for (int i = 0; i < n; ++i)
      zd[i] = ZeroJob{reinterpret_cast<float4*>(plan.mats[i].D), static_cast<long long>(plan.mats[i].L) * 8 / 16};  // L is a multiple of 4
    if (cudaMemcpy(plan.d_zero_d, zd.data(), sizeof(ZeroJob) * n, cudaMemcpyHostToDevice) != cudaSuccess) return NGALORE_ERR_CUDA;
  }
  if (cudaMemcpy(plan.d_newton, newton.data(), sizeof(NewtonJob) * n, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(plan.d_factor32, factor32.data(), sizeof(FactorMat) * n, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(plan.d_factor64, factor64.data(), sizeof(FactorMat) * n, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(plan.d_syrk_mats, syrk_m.data(), sizeof(SyrkMat) * n, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(plan.d_syrk_tiles, syrk_tiles.data(), sizeof(SyrkTile) * syrk_tiles.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(plan.d_split_y_rest, sy_rest.data(), sizeof(SplitJob) * sy_rest.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(plan.d_split_z_rest, sz_rest.data(), sizeof(SplitJob) * sz_rest.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(plan.d_eig, eig.data(), sizeof(EigMat) * n, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(plan.d_eig_factor, eig_factors.data(), sizeof(FactorMat) * n, cudaMemcpyHostToDevice) != cudaSuccess)
    return NGALORE_ERR_CUDA;

  plan.cluster = tf_cluster(n, plan.l_max);
  plan.n_short = static_cast<int>(short_factor.size());
  plan.short_cluster = tf_cluster(plan.n_short, plan.short_l_max);
  if (plan.n_short > 0) {
    std::stable_sort(short_factor.begin(), short_factor.end(), wider);
    bool ok = true;
    auto put = [&](auto*& dst, size_t at, const auto& src) {
      using T = typename std::remove_reference_t<decltype(src)>::value_type;
      dst = reinterpret_cast<T*>(plan.buf + at);
      ok = ok && cudaMemcpy(dst, src.data(), sizeof(T) * src.size(), cudaMemcpyHostToDevice) == cudaSuccess;
    };
    put(plan.d_short_syrk_mats, o_short_syrk_m, short_syrk_m);
    put(plan.d_short_syrk_tiles, o_short_syrk_t, short_syrk_tiles);
    put(plan.d_short_factor, o_short_factor, short_factor);
    put(plan.d_short, o_short_m, short_m);
    put(plan.d_short_tiles, o_short_t, short_tiles);
    put(plan.d_short_zero, o_short_zero, short_zero);
    if (!ok) return NGALORE_ERR_CUDA;
  }

  // ---- tables of buffers to clear
  {
    std::vector<ZeroJob> jobs;
    int first[RG_COUNT + 2];
    for (int g = 0; g <= RG_COUNT; ++g) {
      first[g] = static_cast<int>(jobs.size());
      if (g == RG_COUNT) {
        for (const RefreshMat& m : plan.mats)
          jobs.push_back(ZeroJob{reinterpret_cast<float4*>(m.X64), static_cast<long long>(m.L) * m.L * 8 / 16});
        continue;
      }
      auto clear = [&](int kind) {
        for (int i : plan.atomic_mats[kind]) {
          const RefreshMat& m = plan.mats[i];
          float* out; long long bytes;
          switch (kind) {
            case RG_Y_FROM_Z: out = m.Yf; bytes = 4ll * m.M * m.L; break;
            case RG_Z_FROM_Y: out = m.Zf; bytes = 4ll * m.N * m.L; break;
            default: out = m.C32; bytes = 4ll * m.L * m.L; break;
          }
          jobs.push_back(ZeroJob{reinterpret_cast<float4*>(out), bytes / 16});  // L is a multiple of 4
        }
      };
      // Y = G Z is the first product of a sweep: before it go the outputs of all that follows up to the next one, which
      // are free by then (a launch less each: 14 of 3 us in a refresh of six sweeps)
      if (g == RG_Y_FROM_Z) { clear(RG_Y_FROM_Z); clear(RG_GRAM_Y); clear(RG_Z_FROM_Y); }
      else if (g != RG_Z_FROM_Y) clear(g);
    }
    first[RG_COUNT + 1] = static_cast<int>(jobs.size());
    if (cudaMalloc(&plan.zero_tables, sizeof(ZeroJob) * (jobs.size() + 1)) != cudaSuccess) {
      plan.zero_tables = nullptr;
      return NGALORE_ERR_ALLOC;
    }
    if (!jobs.empty() && cudaMemcpy(plan.zero_tables, jobs.data(), sizeof(ZeroJob) * jobs.size(), cudaMemcpyHostToDevice) != cudaSuccess)
      return NGALORE_ERR_CUDA;
    for (int g = 0; g <= RG_COUNT; ++g) {
      plan.d_zero[g] = reinterpret_cast<ZeroJob*>(plan.zero_tables) + first[g];
      plan.n_zero[g] = first[g + 1] - first[g];
    }
    plan.device_bytes += sizeof(ZeroJob) * (jobs.size() + 1);
  }

  using L2 = TcSmem<kRefBN, 2, 2, kRefStages2, 8>;
  // (the four products with G that this plan takes: setting an attribute loads a kernel, the first state of a process would
  // pay for all sixteen)
  auto init = [](auto p) { return cudaFuncSetAttribute(p.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, p.kSmem) == cudaSuccess; };
  auto init_all = [&](auto bn, auto mt) {
    constexpr int BN = decltype(bn)::value, MT = decltype(mt)::value;
    return init(RefProduct<BN, 1, MT, false>{}) && init(RefProduct<BN, 1, MT, true>{}) && init(RefProduct<BN, 2, MT, false>{}) &&
           init(RefProduct<BN, 2, MT, true>{});
  };
  using Wide = std::integral_constant<int, kRefWideBN>;
  using Narrow = std::integral_constant<int, kRefBN>;
  using Tall = std::integral_constant<int, 2>;
  using Flat = std::integral_constant<int, 1>;
  if (!plan.pair &&
      !(plan.wide ? (plan.tall ? init_all(Wide{}, Tall{}) : init_all(Wide{}, Flat{}))
                  : (plan.tall ? init_all(Narrow{}, Tall{}) : init_all(Narrow{}, Flat{}))))
    return NGALORE_ERR_CUDA;
  if (cudaFuncSetAttribute(tc_gemm_kernel<kRefBN, 2, 2, kRefStages2, TC_EPI_STORE, 8, false>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, L2::kTotal) != cudaSuccess ||
      cudaFuncSetAttribute(tc_gemm_kernel<kRefBN, 2, 2, kRefStages2, TC_EPI_STORE, 8, true>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, L2::kTotal) != cudaSuccess)
    return NGALORE_ERR_CUDA;
  plan.ready = true;
  return NGALORE_OK;
}


// g: the kind of product, problem: its operands' and result's place (RefreshProb).
// high_only: the products with G take only the high bf16 part of the basis (half the tensor-core work; the basis
// then enters with 8 bits instead of 16, which the early sweeps of the iteration do not notice).
// cleared: the outputs have been cleared with those of the last Y = G Z.
inline ngalore_status refresh_tc_gemm(RefreshPlan& plan, int g, int problem, Ctrl* d_ctrl, cudaStream_t stream, int64_t* launches,
                                      bool high_only = false, bool cleared = false) {
  // outputs that several K slices accumulate into start from zero
  if (plan.n_zero[g] > 0 && !cleared) {
    launch_step(plan.brief, zero_jobs_kernel, dim3(32, plan.n_zero[g]), 256, 0, stream, plan.d_zero[g]);
    *launches += 1;
  }
  using L2 = TcSmem<kRefBN, 2, 2, kRefStages2, 8>;
  const int threads = 64 + 32 * 8;
  cudaError_t pair_err = cudaSuccess;
  auto product = [&](auto a_mn) {   // a product with G; a_mn: with G^T
    constexpr bool MN = decltype(a_mn)::value;
    auto run = [&](auto p) {
      launch_step(plan.brief, p.kernel, plan.grid[g], p.kThreads, p.kSmem, stream, plan.d_maps, plan.d_tiles[g], plan.d_first[g], nullptr,
                  d_ctrl, plan.d_probs[problem], nullptr, 0);
    };
    if (plan.pair) {
      auto pair = [&](auto parts) {
        pair_err = tc_pair_launch<decltype(parts)::value, MN>(plan.grid[g], stream, plan.d_maps, plan.d_tiles[g], plan.d_first[g], d_ctrl, plan.d_probs[problem]);
      };
      if (high_only) pair(std::integral_constant<int, 1>{}); else pair(std::integral_constant<int, 2>{});
    } else if (plan.wide && plan.tall) {
      if (high_only) run(RefProduct<kRefWideBN, 1, 2, MN>{}); else run(RefProduct<kRefWideBN, 2, 2, MN>{});
    } else if (plan.wide) {
      if (high_only) run(RefProduct<kRefWideBN, 1, 1, MN>{}); else run(RefProduct<kRefWideBN, 2, 1, MN>{});
    } else if (plan.tall) {
      if (high_only) run(RefProduct<kRefBN, 1, 2, MN>{}); else run(RefProduct<kRefBN, 2, 2, MN>{});
    } else {
      if (high_only) run(RefProduct<kRefBN, 1, 1, MN>{}); else run(RefProduct<kRefBN, 2, 1, MN>{});
    }
  };
  switch (g) {
    case RG_Y_FROM_Z: product(std::false_type{}); break;
    case RG_Z_FROM_Y: product(std::true_type{}); break;
    case RG_GRAM_Y:
    case RG_GRAM_Z:
      launch_step(plan.brief, tc_gemm_kernel<kRefBN, 2, 2, kRefStages2, TC_EPI_STORE, 8, true>, plan.grid[g], threads, L2::kTotal, stream,
                  plan.d_maps, plan.d_tiles[g], plan.d_first[g], nullptr, d_ctrl, plan.d_probs[problem], nullptr, 0);
      break;
    default:
      launch_step(plan.brief, tc_gemm_kernel<kRefBN, 2, 2, kRefStages2, TC_EPI_STORE, 8, false>, plan.grid[g], threads, L2::kTotal, stream,
                  plan.d_maps, plan.d_tiles[g], plan.d_first[g], nullptr, d_ctrl, plan.d_probs[problem], nullptr, 0);
      break;
  }
  *launches += 1;
  return pair_err == cudaSuccess && cudaGetLastError() == cudaSuccess ? NGALORE_OK : NGALORE_ERR_CUDA;
}

// The products with G write the bf16 parts of their result themselves, except for the matrices whose K they split.
inline ngalore_status refresh_tc_split(RefreshPlan& plan, bool y_side, cudaStream_t stream, int64_t* launches) {
  const int n_jobs = y_side ? plan.n_split_y_rest : plan.n_split_z_rest;
  if (n_jobs == 0) return NGALORE_OK;
  launch_step(plan.brief, split_hilo_grouped_kernel, dim3(64, n_jobs), 256, 0, stream, y_side ? plan.d_split_y_rest : plan.d_split_z_rest);
  *launches += 1;
  return cudaGetLastError() == cudaSuccess ? NGALORE_OK : NGALORE_ERR_CUDA;
}

// iterate (as it leaves the product Y = G Z, in set 0) -> well-conditioned basis, in set 1.
inline ngalore_status refresh_tc_orth(RefreshPlan& plan, Ctrl* d_ctrl, cudaStream_t stream, int64_t* launches,
                                      double shift_scale = 1.0) {
  ngalore_status rc;
  if ((rc = refresh_tc_split(plan, true, stream, launches))) return rc;
  if ((rc = refresh_tc_gemm(plan, RG_GRAM_Y, RP_GRAM_Y0, d_ctrl, stream, launches, false, true))) return rc;
  if (tri_factor_launch(plan.d_factor32, plan.n, plan.l_max, shift_scale, stream, launches, false, plan.brief, plan.cluster) != cudaSuccess) return NGALORE_ERR_CUDA;
  return refresh_tc_gemm(plan, RG_APPLY_TRI, RP_APPLY_01, d_ctrl, stream, launches);
}

// Final pass: Cholesky QR of the last basis with the Gram matrix accumulated exactly in fp64 (no shift beyond
// 1e-12), Cholesky and triangular inverse in fp64; only Q = Y R^-1 goes through the tensor cores in two bf16
// parts, whose rounding averages out over the rows.  Matrices with few rows are re-done entirely in fp64 by
// the caller.  From set 1 to set 0.
inline ngalore_status refresh_tc_final(RefreshPlan& plan, Ctrl* d_ctrl, cudaStream_t stream, int64_t* launches) {
  zero_jobs_kernel<<<dim3(32, plan.n_zero[RG_COUNT]), 256, 0, stream>>>(plan.d_zero[RG_COUNT]);
  *launches += 1;
  syrk_f64_kernel<false><<<plan.n_syrk_tiles, 256, 0, stream>>>(plan.d_syrk_mats, plan.d_syrk_tiles);
  *launches += 1;
  if (tri_factor_launch(plan.d_factor64, plan.n, plan.l_max, 1e-12, stream, launches, false, false, plan.cluster) != cudaSuccess) return NGALORE_ERR_CUDA;
  return refresh_tc_gemm(plan, RG_APPLY_TRI, RP_APPLY_10, d_ctrl, stream, launches);
}

// Pass after refresh_tc_final: the basis is orthonormal to first order by then (1e-5, up to 1e-3 for a gradient of
// low numerical rank), and a Newton step with the tensor-core Gram matrix squares what is missing, down to the
// accuracy of that Gram matrix; a second exact pass gave the same at ten times the cost.
// From set `set` to the other.
inline ngalore_status refresh_tc_refine(RefreshPlan& plan, int set, Ctrl* d_ctrl, cudaStream_t stream, int64_t* launches) {
  ngalore_status rc;
  if ((rc = refresh_tc_gemm(plan, RG_GRAM_Y, set == 0 ? RP_GRAM_Y0 : RP_GRAM_Y1, d_ctrl, stream, launches))) return rc;
  launch_step(plan.brief, newton_prep_kernel, dim3(plan.n, 8), 256, 0, stream, plan.d_newton);
  *launches += 1;
  return refresh_tc_gemm(plan, RG_APPLY_Y, set == 0 ? RP_APPLY_01 : RP_APPLY_10, d_ctrl, stream, launches);
}

// The matrices with few rows: the rounding of the last product's operands to two bf16 parts does not average out over their
// rows, so their bases get one more Cholesky QR, all of it in fp64, from Yf to the buffer given for it when the plan was made.  Four
// launches for all of them; matrix by matrix, on the vector units and with two launches for every 32 columns of a factor, it was most of
// a refresh: 42 matrices of 328 rows at r' = 328 43.2 ms, now 5.8, of them 0.09 the Gram matrices, 0.21 the factors and 0.11 the
// product; 36 of 200 rows at r' = 196 11.3 -> 2.6; 49 of 328 rows at r' = 44 8.4 -> 1.3.
inline ngalore_status refresh_tc_short(RefreshPlan& plan, cudaStream_t stream, int64_t* launches) {
  if (plan.n_short == 0) return NGALORE_OK;
  zero_jobs_kernel<<<dim3(8, plan.n_short), 256, 0, stream>>>(plan.d_short_zero);
  syrk_f64_kernel<true><<<plan.n_short_syrk, 256, 0, stream>>>(plan.d_short_syrk_mats, plan.d_short_syrk_tiles);
  *launches += 2;
  if (tri_factor_launch(plan.d_short_factor, plan.n_short, plan.short_l_max, 1e-12, stream, launches, false, false, plan.short_cluster) != cudaSuccess) return NGALORE_ERR_CUDA;
  apply_f64_kernel<<<plan.n_short_tiles, 256, 0, stream>>>(plan.d_short, plan.d_short_tiles);
  *launches += 1;
  return cudaGetLastError() == cudaSuccess ? NGALORE_OK : NGALORE_ERR_CUDA;
}

// Whole-set refresh; leaves the basis in Yf, of the matrices with few rows (is_short) in the buffer given for it.
inline ngalore_status refresh_tc_run(RefreshPlan& plan, const uint16_t* const* G, int q, unsigned long long seed,
                                     unsigned long long stream_base, Ctrl* d_ctrl, cudaStream_t stream,
                                     int64_t* launches) {
  bool changed = false;
  for (int i = 0; i < plan.n; ++i) {
    if (plan.last_G[i] != G[i]) {
      plan.last_G[i] = G[i];
      const RefreshMat& m = plan.mats[i];
      CUtensorMap* mp = &plan.h_maps[static_cast<size_t>(i) * RM_COUNT];
      if (!tc_encode_2d(plan.encode, mp + RM_G_A, G[i], m.N, m.M, static_cast<uint64_t>(m.N) * 2, kTcBK, kTcBM) ||
          !tc_encode_2d(plan.encode, mp + RM_G_MN, G[i], m.N, m.M, static_cast<uint64_t>(m.N) * 2, 64, kTcBK))
        return NGALORE_ERR_CUDA;
      changed = true;
    }
  }
  if (changed && cudaMemcpyAsync(plan.d_maps, plan.h_maps.data(), sizeof(CUtensorMap) * plan.h_maps.size(),
                                 cudaMemcpyHostToDevice, stream) != cudaSuccess)
    return NGALORE_ERR_CUDA;
  ngalore_status rc;
  fill_normal_grouped_kernel<<<dim3(plan.fill_blocks, plan.n), 256, 0, stream>>>(plan.d_fill, seed, stream_base);
  *launches += 1;
  if (cudaGetLastError() != cudaSuccess) return NGALORE_ERR_CUDA;
  if ((rc = refresh_tc_gemm(plan, RG_Y_FROM_Z, RP_Y_FROM_Z, d_ctrl, stream, launches))) return rc;
  if ((rc = refresh_tc_orth(plan, d_ctrl, stream, launches))) return rc;
  // A sweep applies G G^T to the basis and orthonormalises the result.  Z = G^T Q is not orthonormalised in between:
  // its columns are images of orthonormal ones, and the two-part bf16 operands keep 16 bits of every entry whatever
  // the norm of its column, so the second product loses nothing that an orthonormalisation of Z would have saved
  // (measured on the 1.1B shapes: the same Ritz vectors to all printed digits, a quarter of the refresh time less).
  for (int it = 0; it < q; ++it) {
    // the first half of the sweeps multiplies with the high bf16 part of the basis only: what that rounding adds
    // (2^-9 of an entry) shrinks with every later sweep like any other component outside the dominant subspace
    // (not with fewer than four sweeps, where every one of them counts)
    const bool coarse = q >= 4 && it < q / 2;
    if ((rc = refresh_tc_gemm(plan, RG_Z_FROM_Y, RP_Z_FROM_Y1, d_ctrl, stream, launches, coarse))) return rc;
    if ((rc = refresh_tc_split(plan, false, stream, launches))) return rc;
    if ((rc = refresh_tc_gemm(plan, RG_Y_FROM_Z, RP_Y_FROM_Z, d_ctrl, stream, launches, coarse))) return rc;
    if ((rc = refresh_tc_orth(plan, d_ctrl, stream, launches))) return rc;
  }
  // Exact orthonormalisation of the basis that leaves the sweeps: the basis can be ill conditioned in its weak
  // directions, so the product with the exact triangular factor leaves it orthonormal to 1e-5 .. 1e-3 only; two
  // Newton steps start from that and end at about 1e-6.  The Rayleigh-Ritz step below relies on it (it
  // solves C v = lambda v, not C v = lambda (Q^T Q) v, and what Q lacks in orthonormality goes into the Ritz vectors).
  if ((rc = refresh_tc_final(plan, d_ctrl, stream, launches))) return rc;
  if ((rc = refresh_tc_refine(plan, 0, d_ctrl, stream, launches))) return rc;
  if ((rc = refresh_tc_refine(plan, 1, d_ctrl, stream, launches))) return rc;
  // Rayleigh-Ritz: Z = G^T Q, C = Z^T Z (tensor cores: its entries are good to about 2^-17 of the diagonal, far
  // finer than the gaps that decide a Ritz vector), V = eigenvectors of C (or of its leading block, see
  // ritz_eigen.cuh), P = Q V.
  if ((rc = refresh_tc_gemm(plan, RG_Z_FROM_Y, RP_Z_FROM_Y0, d_ctrl, stream, launches))) return rc;
  if ((rc = refresh_tc_split(plan, false, stream, launches))) return rc;
  if ((rc = refresh_tc_gemm(plan, RG_GRAM_Z, RP_GRAM_Z, d_ctrl, stream, launches))) return rc;
  if (eig_batched_launch(plan.d_eig, plan.d_eig_factor, plan.n, plan.eig_max, plan.l_max, plan.sm_count, stream, launches) != cudaSuccess)
    return NGALORE_ERR_CUDA;
  // Q orthonormal to about 1e-6 and V orthogonal: so is their product, once its columns are scaled back to unit norm
  // (with the working copies, see finish_refresh; their norms go to D)
  if ((rc = refresh_tc_gemm(plan, RG_APPLY_Y, RP_APPLY_0F, d_ctrl, stream, launches))) return rc;
  if ((rc = refresh_tc_short(plan, stream, launches))) return rc;
  zero_jobs_kernel<<<dim3(1, plan.n), 256, 0, stream>>>(plan.d_zero_d);
  *launches += 1;
  return cudaGetLastError() == cudaSuccess ? NGALORE_OK : NGALORE_ERR_CUDA;
}

}  // namespace ngalore
