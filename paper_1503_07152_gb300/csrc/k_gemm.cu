// Sampling GEMM of the dense test operator: Y = A X or Y = A^T X with A a
// row-major N x N matrix and X, Y column-major N x ncols blocks (the black-box
// products A Omega / A^* Omega of Fig. "Randomized compression of a HODLR
// matrix").  The test matrices of the sweeps are zero on half of their rows
// (Omega_1 lives on left children, Omega_2 on right children) and the identity
// probe is zero outside one diagonal band, so a pre-pass marks the all-zero
// (K-tile, column-tile) blocks of X and the GEMM skips them: the work and the
// A bytes read follow the nonzero structure of X.
//
// These are the CUDA-core forms: FP32 (128 x 64 output tile per block of 256
// threads, 8 x 4 register tile per thread; every K-tile is accumulated in a fresh
// register tile and added to the running sum with Kahan compensation) and FP64
// sums over an FP64 or an FP32 operator (k_dense_gemm64).
#include <algorithm>
#include <cooperative_groups.h>

#include "df.cuh"
#include "hm_internal.h"

namespace hm {
namespace {

constexpr int BM = 128;
constexpr int BN = 64;

constexpr int BK = 32;

// flags[kt * nct + ct] = 1 iff X(kt*BK .. , ct*CN ..) has a nonzero entry.
template <typename T, int CN>
__global__ void k_tile_flags(const T* __restrict__ X, int64_t ldx, int64_t n, int64_t ncols,
                             uint8_t* __restrict__ flags, int nct) {
  const int kt = blockIdx.x, ct = blockIdx.y;
  bool nz = false;
  for (int idx = threadIdx.x; idx < BK * CN; idx += blockDim.x) {
    const int k = idx % BK, c = idx / BK;
    const int64_t row = (int64_t)kt * BK + k, col = (int64_t)ct * CN + c;
    if (row < n && col < ncols) nz |= (X[row + col * ldx] != (T)0);
  }
  nz = __syncthreads_or(nz);
  if (threadIdx.x == 0) flags[(int64_t)kt * nct + ct] = nz ? 1 : 0;
}

template <typename T, int TRANS>
__global__ __launch_bounds__(256) void k_dense_gemm(const T* __restrict__ A, int64_t lda,
                                                    int64_t n, int64_t ncols,
                                                    const T* __restrict__ X, int64_t ldx,
                                                    T* __restrict__ Y, int64_t ldy,
                                                    const uint8_t* __restrict__ flags, int nct) {
  __shared__ __align__(16) T As[BK][BM + 4];
  __shared__ __align__(16) T Xs[BK][BN + 4];
  const int64_t m0 = (int64_t)blockIdx.x * BM;
  const int ct = blockIdx.y;
  const int64_t c0 = (int64_t)ct * BN;
  const int tid = threadIdx.x;
  const int rg = tid >> 4, cg = tid & 15;

  T acc[8][4], cmp[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) { acc[i][j] = 0; cmp[i][j] = 0; }

  const int nkt = (int)((n + BK - 1) / BK);
  for (int kt = 0; kt < nkt; ++kt) {
    if (flags && !flags[(int64_t)kt * nct + ct]) continue;  // uniform over the block
    const int64_t k0 = (int64_t)kt * BK;
    // A tile: BM x BK values of op(A)
    if (!TRANS) {
      // element (m, k) = A[(m0 + m) * lda + k0 + k]; lanes run along k
      for (int idx = tid; idx < BM * BK; idx += 256) {
        const int k = idx % BK, m = idx / BK;
        const int64_t row = m0 + m, col = k0 + k;
        As[k][m] = (row < n && col < n) ? A[row * lda + col] : (T)0;
      }
    } else {
      // element (m, k) = A[(k0 + k) * lda + m0 + m]; lanes run along m
      for (int idx = tid; idx < BM * BK; idx += 256) {
        const int m = idx % BM, k = idx / BM;
        const int64_t row = k0 + k, col = m0 + m;
        As[k][m] = (row < n && col < n) ? A[row * lda + col] : (T)0;
      }
    }
    for (int idx = tid; idx < BK * BN; idx += 256) {
      const int k = idx % BK, c = idx / BK;
      const int64_t row = k0 + k, col = c0 + c;
      Xs[k][c] = (row < n && col < ncols) ? X[row + col * ldx] : (T)0;
    }
    __syncthreads();
    T tmp[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) tmp[i][j] = 0;
#pragma unroll 4
    for (int kk = 0; kk < BK; ++kk) {
      T a[8], x[4];
#pragma unroll
      for (int i = 0; i < 8; ++i) a[i] = As[kk][rg * 8 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = Xs[kk][cg * 4 + j];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) tmp[i][j] = fma(a[i], x[j], tmp[i][j]);
    }
    // compensated running sum
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const T y = tmp[i][j] - cmp[i][j];
        const T t = acc[i][j] + y;
        cmp[i][j] = (t - acc[i][j]) - y;
        acc[i][j] = t;
      }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int64_t col = c0 + cg * 4 + j;
    if (col >= ncols) continue;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int64_t row = m0 + rg * 8 + i;
      if (row < n) Y[row + col * ldy] = acc[i][j];
    }
  }
}

// FP64 samples with an FP64 operator, or an FP32 one (an FP32 value is an FP64 value;
// widened on the integer pipe): every product formed and summed in FP64.
//
// Bound by the FP64 pipe (64 cycles per warp FMA and scheduler), so the aim is FMAs
// on every scheduler and none for padding: a block of four warps takes 32 rows
// (lanes) x 32 columns (warp w: columns w, w + 4, ..), only columns that exist are
// multiplied, and where the row blocks alone would not fill the chip a cluster of S
// blocks shares a tile's K tiles and sums its shares over distributed shared memory in
// rank order (deterministic, no workspace).  N = 1024, 20 columns, half of K active:
// 1175 us as 8 blocks of 128 x 64 outputs, 41 us so.
//
// K tile t belongs to block t mod 2S, or its mirror image 2S - 1 - t mod 2S where that
// is not below S: half-active patterns of any period then spread over the blocks, and
// neither the other columns nor their zeros decide which sums a column's terms go to.
// Products are summed 32 at a time, 16 below N = 1024, and those sums added up: with m
// terms to a block the rounding grows as the root of 32 + m / 32 or 16 + m / 16, so that
// neither is above that of 16 at a time and no split over K.  A chain over all of K rounds
// 3 times as much at N = 8192 for one FP64 add in 33 less.
template <typename TA, int TRANS>
__global__ __launch_bounds__(128) void k_dense_gemm64(const TA* __restrict__ A, int64_t lda,
                                                      int64_t n, int64_t ncols,
                                                      const double* __restrict__ X, int64_t ldx,
                                                      double* __restrict__ Y, int64_t ldy,
                                                      const uint8_t* __restrict__ flags,
                                                      int nct, int S) {
  __shared__ double As[32][33];  // [k][row] (TRANS) or [row][k]
  __shared__ double Xs[32][33];  // [column][k], later the sums [column][row]
  const int64_t m0 = (int64_t)blockIdx.x * 32;
  const int part = blockIdx.y, ct = blockIdx.z;
  const int64_t c0 = (int64_t)ct * 32;
  const int nc = (int)min((int64_t)32, ncols - c0);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int nq = w < nc ? (nc - w + 3) / 4 : 0;  // this warp's columns
  const bool halves = n < 1024;                  // sums of 16 (of 32)
  double acc[8] = {};
  const int nkt = (int)((n + BK - 1) / BK);
  for (int kt = 0; kt < nkt; ++kt) {
    if (flags && !flags[(int64_t)kt * nct + ct]) continue;  // uniform over the block
    const int q = kt & (2 * S - 1);  // (S is a power of two)
    if ((q < S ? q : 2 * S - 1 - q) != part) continue;
    const int64_t k0 = (int64_t)kt * BK;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      // lanes along the contiguous index of A: k, or the row of op(A)
      const int r = w + 4 * i;
      const int64_t row = TRANS ? k0 + r : m0 + r, col = (TRANS ? m0 : k0) + lane;
      const TA a = (row < n && col < n) ? A[row * lda + col] : (TA)0;
      if constexpr (sizeof(TA) == 8) As[r][lane] = a;
      else As[r][lane] = df::widen(a);
      if (r < nc) Xs[r][lane] = (k0 + lane < n) ? X[k0 + lane + (c0 + r) * ldx] : 0.0;
    }
    __syncthreads();
    if (nq > 0)
      with_count<8>(nq, [&](auto cols) {
        double t[cols] = {};
#pragma unroll
        for (int k0 = 0; k0 < BK; k0 += 16) {
#pragma unroll 4
          for (int k = k0; k < k0 + 16; ++k) {
            const double a = TRANS ? As[k][lane] : As[lane][k];
#pragma unroll
            for (int q = 0; q < cols; ++q) t[q] = fma(a, Xs[w + 4 * q][k], t[q]);
          }
          if (k0 > 0 || halves)
#pragma unroll
            for (int q = 0; q < cols; ++q) {
              acc[q] += t[q];
              t[q] = 0.0;
            }
        }
      });
    __syncthreads();
  }
  if (S == 1) {
    if (m0 + lane < n)
      for (int q = 0; q < 8; ++q)
        if (q < nq) Y[m0 + lane + (c0 + w + 4 * q) * ldy] = acc[q];
    return;
  }
#pragma unroll
  for (int q = 0; q < 8; ++q)
    if (q < nq) Xs[w + 4 * q][lane] = acc[q];
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  cl.sync();
  for (int c = part + S * w; c < nc; c += 4 * S) {
    double s = 0.0;
    for (int p = 0; p < S; ++p) s += cl.map_shared_rank(&Xs[c][lane], p)[0];
    if (m0 + lane < n) Y[m0 + lane + (c0 + c) * ldy] = s;
  }
  cl.sync();  // no block leaves while another may still read its sums
}

}  // namespace

// The FP64 GEMM with its cluster size: doubled while one column tile's blocks are fewer
// than three per SM (152 SMs) and there is a K tile for each (N = 1024: 8 blocks a tile;
// from N ~ 15000 on: 1).  The number of columns plays no part: it would decide how a
// column's terms are grouped.
template <typename TA>
static void dense_gemm64(const TA* A, int64_t lda, int trans, int64_t n, int64_t ncols,
                         const double* X, int64_t ldx, double* Y, int64_t ldy, uint8_t* flags,
                         cudaStream_t st) {
  count_launches(flags ? 2 : 1);
  const int nct = (int)((ncols + 31) / 32), nkt = (int)((n + BK - 1) / BK);
  if (flags) k_tile_flags<double, 32><<<dim3(nkt, nct), 256, 0, st>>>(X, ldx, n, ncols, flags, nct);
  const int64_t rows = (n + 31) / 32;
  int S = 1;
  while (S < 8 && rows * S < 456 && 2 * S <= nkt) S *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)rows, (unsigned)S, (unsigned)nct);
  cfg.blockDim = dim3(128);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = (unsigned)S;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const uint8_t* fl = flags;
  if (trans)
    cudaLaunchKernelEx(&cfg, k_dense_gemm64<TA, 1>, A, lda, n, ncols, X, ldx, Y, ldy, fl, nct, S);
  else
    cudaLaunchKernelEx(&cfg, k_dense_gemm64<TA, 0>, A, lda, n, ncols, X, ldx, Y, ldy, fl, nct, S);
}

void launch_dense_gemm_a32(const float* A, int64_t lda, int trans, int64_t n, int64_t ncols,
                           const double* X, int64_t ldx, double* Y, int64_t ldy, uint8_t* flags,
                           cudaStream_t st) {
  dense_gemm64<float>(A, lda, trans, n, ncols, X, ldx, Y, ldy, flags, st);
}

template <typename T>
void launch_dense_gemm(const T* A, int64_t lda, int trans, int64_t n, int64_t ncols, const T* X,
                       int64_t ldx, T* Y, int64_t ldy, uint8_t* flags, cudaStream_t st) {
  if constexpr (sizeof(T) == 8) {
    dense_gemm64<double>(A, lda, trans, n, ncols, X, ldx, Y, ldy, flags, st);
  } else {
    count_launches(flags ? 2 : 1);
    const int nct = (int)((ncols + BN - 1) / BN);
    const int nkt = (int)((n + BK - 1) / BK);
    if (flags)
      k_tile_flags<T, BN><<<dim3(nkt, nct), 256, 0, st>>>(X, ldx, n, ncols, flags, nct);
    dim3 grid((unsigned)((n + BM - 1) / BM), (unsigned)nct);
    if (trans)
      k_dense_gemm<T, 1><<<grid, 256, 0, st>>>(A, lda, n, ncols, X, ldx, Y, ldy, flags, nct);
    else
      k_dense_gemm<T, 0><<<grid, 256, 0, st>>>(A, lda, n, ncols, X, ldx, Y, ldy, flags, nct);
  }
}

int64_t dense_flags_bytes(int64_t n, int64_t ncols, int is_double) {
  (void)is_double;
  // the smallest K tile and column tile of any variant
  return ((n + 15) / 16) * ((ncols + 31) / 32);
}

template void launch_dense_gemm<float>(const float*, int64_t, int, int64_t, int64_t,
                                       const float*, int64_t, float*, int64_t, uint8_t*,
                                       cudaStream_t);
template void launch_dense_gemm<double>(const double*, int64_t, int, int64_t, int64_t,
                                        const double*, int64_t, double*, int64_t, uint8_t*,
                                        cudaStream_t);

}  // namespace hm
