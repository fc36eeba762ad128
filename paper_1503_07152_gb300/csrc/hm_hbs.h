// Declarations of the HBS / HBS-ID kernels.
#pragma once

#include "hm_internal.h"

namespace hm {

// One small GEMM: C (m x n, ldc) = alpha op(A) op(B) + beta C; op = transpose when ta/tb.
struct GemmItem {
  const void* A;
  const void* B;
  void* C;
  int32_t m, n, k;
  int32_t lda, ldb, ldc;
  int32_t ta, tb;
};

// One level's small FP64 products in one launch, the operands of every node found from
// its index on the device (no item list to build and copy): node x gets
//   C = op(A_0) B_0 [+ op(A_1) B_1],
// each product summed on its own and the two added last.  q, u hold one r x w block
// per heap node (the solver: per node of the level, x - node0).
struct NodeGemm {
  enum Mode {
    kUp,        // q[x] = op(A_0) q[2x] + op(A_1) q[2x + 1], A_h = A0 + (2x + h) r^2
    kDown,      // u[x] = B_x q[x ^ 1] + op(A) u[x / 2]: B_x = A0 + x r^2 (ta0: the sibling's,
                //   transposed), A = A1 + x r^2 (ta1); no second term when A1 is null
    kLeafUp,    // q[x] = A X(I_x), A = A0 + leaf r nmax (r x n_x)
    kLeafDown,  // Y(I_x) = A^T u[x], A as above
    kSolve      // u[x] = the rows of M [q_b; q_a] (ta0: of M^T [q_a; q_b]) that child x of
                //   its parent takes, M = A0 + parent (2r)^2, parents of level node0 / 2
  };
  int32_t mode;
  int32_t node0, r, w, nmax, ta0, ta1;
  const double *A0, *A1;
  double *q, *u;
  const double* X;
  double* Y;
  int64_t ldx, ldy;
  const int64_t *start, *size;
};
void launch_node_gemm(const NodeGemm& a, int nodes, cudaStream_t st, bool df);

template <typename T>
void launch_gather_parent_scaled(const T* U, int64_t ldu, T* P, int64_t ldp, int64_t n, int r,
                                 int lv, const int64_t* d_start, const T* y, int col0,
                                 cudaStream_t st);
template <typename T>
// max_m, max_n, max_k: the largest m, n and k of the items (the tiled form is used
// when its staging fits, else the plain one; the results are the same).  df: FP64
// items in double-float on the FP32 pipe (HM_A32).
void launch_batched_gemm(const GemmItem* items, int count, T alpha, T beta, cudaStream_t st,
                         int max_m, int max_n, int max_k, bool df = false);
template <typename TS, typename TD>
void launch_node_copy(int nnodes, int node0, const TS* src, int64_t sstride, int sld, TD* dst,
                      int64_t dstride, int dld, int rows, int cols, int flip, cudaStream_t st);
template <typename T>
void launch_id_prep_leaf(const T* U, int64_t ldu, const int64_t* d_start, const int64_t* d_size,
                         int L, const T* y, int r, double* Yt, int ncmax, cudaStream_t st);
template <typename T>
void launch_id_prep_parent(int nnodes, int node0, const double* Utmp, const T* y, int r,
                           double* Yt, cudaStream_t st);
// df: the pivoted QR and the substitution in double-float (HM_A32)
void launch_pivqr_id(int nnodes, const double* Yt, int r, int nc, double eps, int kcap,
                     int32_t* k, int32_t* J, double* T, cudaStream_t st, bool df = false);
template <typename T>
void launch_usamp_leaf(const T* U, int64_t ldu, const int64_t* d_start, int L, const int32_t* J,
                       int r, double* Us, int64_t* skel, cudaStream_t st);
void launch_usamp_parent(int nnodes, int node0, const double* Utmp, const int32_t* J, int r,
                         double* Us, int64_t* skel, cudaStream_t st);

}  // namespace hm
