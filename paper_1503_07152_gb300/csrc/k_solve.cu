// Kernels of the HODLR direct solver (api_solve.cu): batched inversion of small
// dense matrices by Gauss-Jordan elimination with partial pivoting, and the
// assembly of the per-parent Woodbury matrices.
#include <algorithm>
#include <atomic>
#include <cooperative_groups.h>

#include "hm_internal.h"

namespace hm {
namespace {

// |x| as an integer of the same order (the bits of a non-negative number), NaN below all:
// a comparison on the integer pipe instead of one on the FP64 pipe.
__device__ __forceinline__ long long magnitude_key(double x) {
  const long long a = __double_as_longlong(x) & 0x7fffffffffffffffll;
  return a > 0x7ff0000000000000ll ? -1 : a;
}
__device__ __forceinline__ long long magnitude_key(float x) {
  const int a = __float_as_int(x) & 0x7fffffff;
  return a > 0x7f800000 ? -1 : a;
}

// Inverse of every matrix of a batch by Gauss-Jordan elimination with partial
// pivoting, in place (W: n x n, column-major, ld n, in global memory, read once and
// out[b] written once): row k of the inverse replaces the eliminated column k as the
// step goes, the row exchanges are undone as column exchanges at the end.  A zero
// pivot raises *singular and the step is skipped (the output is then garbage).
//
// Bound by the FP64 pipe (n^2 FMAs a step, 64 cycles a warp FMA on one scheduler), so
// a matrix is dealt out column by column over a cluster of S blocks (block p holds
// columns p, p + S, .. in shared memory) when the batch alone leaves SMs idle.  A
// step: the owner of column k finds the pivot and writes it and the column's
// multipliers into every block's shared memory, one cluster barrier, and each block
// exchanges the two rows of its columns and updates them.  The multipliers are double-
// buffered, so one barrier a step orders them: a block writes buffer k & 1 at step k
// only after the barrier of step k - 1, which every block passes after its last use of
// that buffer, at step k - 2.  32 leaves of 94: 1037 -> 204 us (one block a matrix, the
// augmented n x 2n form in L2); 36 x 36 Woodbury blocks: 188 -> 62 us (486 and 136 before
// the pivot search left the FP64 pipe: its comparisons held every scheduler; 218 and 68
// with three Newton steps from the FP32 reciprocal in the division's place).
template <typename T>
__global__ __launch_bounds__(256) void k_gauss_jordan(const T* __restrict__ W, int n,
                                                      T* __restrict__ out,
                                                      int* __restrict__ singular, int S) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ T fcol[2][256];   // the pivot column before the step, rows exchanged
  __shared__ int prow[2];      // its pivot row
  __shared__ T pinv[2];        // 1 / pivot
  __shared__ short swp[256];   // pivot row of every step
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int part = S > 1 ? (int)cl.block_rank() : 0;
  const int b = blockIdx.x / S;
  T* M = reinterpret_cast<T*>(smem_raw);  // local column c: global column part + S c
  const int nloc = part < n ? (n - part + S - 1) / S : 0;
  const T* Wb = W + (int64_t)b * n * n;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int e = tid; e < n * nloc; e += 256) {
    const int i = e % n, c = e / n;
    M[e] = Wb[i + (int64_t)(part + S * c) * n];
  }
  if (S > 1) cl.sync();  // every block of the cluster runs before its memory is written
  else __syncthreads();
  for (int k = 0; k < n; ++k) {
    const int buf = k & 1;
    if (k % S == part) {
      T* col = M + (int64_t)(k / S) * n;
      // pivot: the largest |A(i, k)|, i >= k (first on ties), found by every warp for itself
      long long best = -1;
      int p = n;
      for (int i = k + lane; i < n; i += 32) {
        const long long a = magnitude_key(col[i]);
        if (a > best) { best = a; p = i; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, p, o);
        if (ob > best || (ob == best && oi < p)) { best = ob; p = oi; }
      }
      if (best <= 0 || p >= n) {
        if (tid == 0) atomicExch(singular, 1);
        p = k;
      }
      for (int i = tid; i < n; i += 256) {
        const T v = col[i == k ? p : (i == p ? k : i)];
        for (int q = 0; q < S; ++q) (S > 1 ? cl.map_shared_rank(&fcol[buf][i], q) : &fcol[buf][i])[0] = v;
      }
      if (warp == 0) {  // (one warp: an FP64 division is a long chain on the FP64 pipe)
        const T pv = col[p];
        const T iv = (pv != (T)0) ? (T)1 / pv : (T)0;
        if (lane < S) {
          (S > 1 ? cl.map_shared_rank(&prow[buf], lane) : &prow[buf])[0] = p;
          (S > 1 ? cl.map_shared_rank(&pinv[buf], lane) : &pinv[buf])[0] = iv;
        }
      }
    }
    if (S > 1) cl.sync();
    else __syncthreads();
    const int p = prow[buf];
    const T inv = pinv[buf];
    if (tid == 0) swp[k] = (short)p;
    // a warp takes a column: exchange rows k and p, scale the pivot row's entry, update
    for (int c = warp; c < nloc; c += 8) {
      T* col = M + (int64_t)c * n;
      if (part + S * c == k) {  // the column of the inverse that replaces column k
        for (int i = lane; i < n; i += 32) col[i] = i == k ? inv : -fcol[buf][i] * inv;
        continue;
      }
      const T xp = col[p], xk = col[k];
      const T x = xp * inv;
      __syncwarp();
      for (int i = lane; i < n; i += 32) {
        const T y = i == p ? xk : col[i];
        col[i] = i == k ? x : fma(-fcol[buf][i], x, y);
      }
      __syncwarp();
    }
    __syncthreads();  // the owner of column k + 1 reads what one of its warps updated
  }
  if (S > 1) cl.sync();  // no block leaves while another may still write to it
  else __syncthreads();
  // undo the exchanges: column k and column swp[k], k = n - 1 .. 0.  Thread c follows
  // its column to the place it ends up at.
  T* ob = out + (int64_t)b * n * n;
  for (int c = warp; c < nloc; c += 8) {
    int dst = part + S * c;
    for (int k = n - 1; k >= 0; --k) {
      const int p = swp[k];
      if (dst == k) dst = p;
      else if (dst == p) dst = k;
    }
    for (int i = lane; i < n; i += 32) ob[i + (int64_t)dst * n] = M[(int64_t)c * n + i];
  }
}

// D_leaf padded to nmax (identity beyond the leaf size), one block per leaf.
template <typename T>
__global__ void k_gj_load_leaves(const T* __restrict__ D, int nmax,
                                 const int64_t* __restrict__ size, int L, T* __restrict__ W) {
  const int leaf = blockIdx.x;
  const int ns = (int)size[(1 << L) + leaf];
  const T* Dl = D + (int64_t)leaf * nmax * nmax;
  T* Wl = W + (int64_t)leaf * nmax * nmax;
  for (int e = threadIdx.x; e < nmax * nmax; e += blockDim.x) {
    const int i = e % nmax, j = e / nmax;
    Wl[e] = (i < ns && j < ns) ? Dl[e] : (T)(i == j ? 1 : 0);
  }
}

// [[I, P_b], [P_a, I]] for every parent p of a level (children a = 2p, b = 2p + 1):
// P holds V_x^T W_x (r x r, ld r) for the children, indexed by x - child0.
template <typename T>
__global__ void k_gj_load_woodbury(const T* __restrict__ P, int r, T* __restrict__ W) {
  const int pi = blockIdx.x;  // parent index within its level
  const int n = 2 * r;
  const T* Pa = P + (int64_t)(2 * pi) * r * r;
  const T* Pb = P + (int64_t)(2 * pi + 1) * r * r;
  T* Wp = W + (int64_t)pi * n * n;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int i = e % n, j = e / n;
    T v;
    if ((i < r) == (j < r)) v = (T)(i == j ? 1 : 0);
    else if (i < r) v = Pb[i + (int64_t)(j - r) * r];  // top right: V_b^T W_b
    else v = Pa[(i - r) + (int64_t)j * r];             // bottom left: V_a^T W_a
    Wp[e] = v;
  }
}

}  // namespace

// Cluster size: doubled (up to 8) while two blocks per SM are not reached and a block
// would keep at least eight columns, and further while a block's columns do not fit its
// shared memory (n = 256 in FP64: 512 KB over 4 blocks).
template <typename T>
void launch_gauss_jordan(T* work, int batch, int n, T* out, int* singular, cudaStream_t st) {
  count_launches(1);
  int S = 1;
  while (S < 8 && ((int64_t)batch * 2 * S <= 304 && n >= 16 * S)) S *= 2;
  auto smem = [&](int s) { return (size_t)n * ((n + s - 1) / s) * sizeof(T); };
  while (S < 8 && smem(S) > 200 * 1024) S *= 2;
  static std::atomic<uint32_t> done{0};
  raise_smem_limit((const void*)k_gauss_jordan<T>, done);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(batch * S));
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem(S);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)S;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const T* W = work;
  cudaLaunchKernelEx(&cfg, k_gauss_jordan<T>, W, n, out, singular, S);
}

template <typename T>
void launch_gj_load_leaves(const T* D, int nmax, const int64_t* d_size, int L, T* work,
                           cudaStream_t st) {
  count_launches(1);
  k_gj_load_leaves<T><<<1 << L, 256, 0, st>>>(D, nmax, d_size, L, work);
}

template <typename T>
void launch_gj_load_woodbury(const T* P, int r, int nparents, T* work, cudaStream_t st) {
  count_launches(1);
  k_gj_load_woodbury<T><<<nparents, 256, 0, st>>>(P, r, work);
}

#define HM_INST(T)                                                                              \
  template void launch_gauss_jordan<T>(T*, int, int, T*, int*, cudaStream_t);                  \
  template void launch_gj_load_leaves<T>(const T*, int, const int64_t*, int, T*, cudaStream_t); \
  template void launch_gj_load_woodbury<T>(const T*, int, int, T*, cudaStream_t);
HM_INST(float)
HM_INST(double)
#undef HM_INST

}  // namespace hm

namespace hm {
namespace {

// Y = alpha A + beta B (column-major n x ncols blocks)
template <typename T>
__global__ void k_axpby(T* __restrict__ Y, int64_t ldy, T alpha, const T* __restrict__ A,
                        int64_t lda, T beta, const T* __restrict__ B, int64_t ldb, int64_t n,
                        int64_t ncols) {
  for (int64_t c = blockIdx.y; c < ncols; c += gridDim.y)
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
      Y[i + c * ldy] = alpha * A[i + c * lda] + (beta != (T)0 ? beta * B[i + c * ldb] : (T)0);
}

}  // namespace

template <typename T>
void launch_axpby(T* Y, int64_t ldy, T alpha, const T* A, int64_t lda, T beta, const T* B,
                  int64_t ldb, int64_t n, int64_t ncols, cudaStream_t st) {
  if (n <= 0 || ncols <= 0) return;
  count_launches(1);
  dim3 grid((unsigned)std::min<int64_t>((n + 255) / 256, 1024),
            (unsigned)std::min<int64_t>(ncols, 65535));
  k_axpby<T><<<grid, 256, 0, st>>>(Y, ldy, alpha, A, lda, beta, B, ldb, n, ncols);
}
template void launch_axpby<float>(float*, int64_t, float, const float*, int64_t, float,
                                  const float*, int64_t, int64_t, int64_t, cudaStream_t);
template void launch_axpby<double>(double*, int64_t, double, const double*, int64_t, double,
                                   const double*, int64_t, int64_t, int64_t, cudaStream_t);

}  // namespace hm
