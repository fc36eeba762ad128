// Segmented (per tree node) tall-skinny products, the workhorses of the peel
// and of the per-node linear algebra:
//   seg_tn:  out[node] = A(I_node, :)^T B(I_node, :)   (projections V^T x of the
//            HODLR product, Sec. 2.8; Gram matrices; the short-basis products
//            U_alpha^* U_tau(J_alpha,:) of Fig. "A basic scheme for compressing an
//            HBS matrix")
//   seg_nn:  Y(I_node, :) = alpha P(I_node, :) C[node'] + beta Y(I_node, :)
//            (expansions U t, basis updates U <- U \hat U, Q = P T).
// A node's rows are split into chunks; uneven node sizes go into one launch.
// Column offsets can depend on the node's parity (left child / right child), which
// is how the packed test matrices [Omega_2 | Omega_1] are addressed.
#include <algorithm>
#include <atomic>

#include "df.cuh"
#include "hm_internal.h"

namespace hm {
namespace {

constexpr int TN_ROWS = 32;   // rows staged per step
constexpr int TN_MAX = 128;   // max ka, kb

// Per-thread tile for a product of ka x kb outputs: 256 threads in a 16 x 16
// grid, thread (ti, tj) owning rows ti + 16 i (i < TI) and columns tj + 16 j
// (j < TJ), so a warp reads 16 consecutive staged columns of B (no bank
// conflicts) and only the 16 TI x 16 TJ outputs that cover ka x kb are computed.
// Which thread owns an output changes nothing in how it is summed.
constexpr int tn_tile(int k) { return k <= 32 ? 2 : (k <= 64 ? 4 : 8); }

// FP32 partial products of one chunk (<= 256 rows).
template <typename T, int TI, int TJ>
__global__ __launch_bounds__(256) void k_seg_tn_partial(
    const Chunk* __restrict__ chunks, const T* __restrict__ A, int64_t lda, int aoff_e,
    int aoff_o, int ka, const T* __restrict__ B, int64_t ldb, int boff_e, int boff_o, int kb,
    double* __restrict__ partial) {
  constexpr int KA = 16 * TI, KB = 16 * TJ, LDA = KA + 1, LDB = KB + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* As = reinterpret_cast<T*>(smem_raw);  // [TN_ROWS][LDA]
  T* Bs = As + TN_ROWS * LDA;              // [TN_ROWS][LDB]
  const Chunk ch = chunks[blockIdx.x];
  const int aoff = (ch.node & 1) ? aoff_o : aoff_e;
  const int boff = (ch.node & 1) ? boff_o : boff_e;
  const int tid = threadIdx.x;
  const int ti = tid >> 4, tj = tid & 15;
  // products summed in T over at most 16 rows, then added into FP64 sums: the
  // projections of the peel are differences of large sums, so a long FP32 sum
  // would cost far more than its unit roundoff
  double acc[TI][TJ];
#pragma unroll
  for (int i = 0; i < TI; ++i)
#pragma unroll
    for (int j = 0; j < TJ; ++j) acc[i][j] = 0.0;
  for (int64_t r0 = ch.r0; r0 < ch.r1; r0 += TN_ROWS) {
    const int rows = (int)((ch.r1 - r0) < TN_ROWS ? (ch.r1 - r0) : TN_ROWS);
    for (int idx = tid; idx < TN_ROWS * KA; idx += 256) {
      const int rr = idx % TN_ROWS, c = idx / TN_ROWS;
      As[rr * LDA + c] = (rr < rows && c < ka) ? A[r0 + rr + (int64_t)(aoff + c) * lda] : (T)0;
    }
    for (int idx = tid; idx < TN_ROWS * KB; idx += 256) {
      const int rr = idx % TN_ROWS, c = idx / TN_ROWS;
      Bs[rr * LDB + c] = (rr < rows && c < kb) ? B[r0 + rr + (int64_t)(boff + c) * ldb] : (T)0;
    }
    __syncthreads();
    for (int q0 = 0; q0 < rows; q0 += 16) {
      const int q1 = (q0 + 16 < rows) ? q0 + 16 : rows;
      T tmp[TI][TJ];
#pragma unroll
      for (int i = 0; i < TI; ++i)
#pragma unroll
        for (int j = 0; j < TJ; ++j) tmp[i][j] = 0;
      for (int rr = q0; rr < q1; ++rr) {
        T a[TI], b[TJ];
#pragma unroll
        for (int i = 0; i < TI; ++i) a[i] = As[rr * LDA + ti + 16 * i];
#pragma unroll
        for (int j = 0; j < TJ; ++j) b[j] = Bs[rr * LDB + tj + 16 * j];
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
          for (int j = 0; j < TJ; ++j) tmp[i][j] = fma(a[i], b[j], tmp[i][j]);
      }
#pragma unroll
      for (int i = 0; i < TI; ++i)
#pragma unroll
        for (int j = 0; j < TJ; ++j) acc[i][j] += (double)tmp[i][j];
    }
    __syncthreads();
  }
  double* out = partial + (int64_t)blockIdx.x * ka * kb;
#pragma unroll
  for (int i = 0; i < TI; ++i)
#pragma unroll
    for (int j = 0; j < TJ; ++j) {
      const int ii = ti + 16 * i, jj = tj + 16 * j;
      if (ii < ka && jj < kb) out[ii + jj * ka] = acc[i][j];
    }
}

// FP64 partial products of one chunk.  Bound by the FP64 pipe (a warp's FMA holds a
// scheduler's FP64 unit for 64 cycles on GB300), so what counts is that every
// scheduler has FMAs to issue and that none is issued for padding: the ka x kb
// outputs of a chunk are dealt out flat, M to a thread and 128 M to a block (a
// grid of output tiles would idle lanes at every edge, and one block per chunk
// left most of the chip idle: 64 chunks x 60 x 37 at N = 16384 took 278 us, this
// 81).  Products are summed over SUM64 rows and those sums added up: the rounding error
// of a 256-row chain is 2.7 times that, for one FP64 add in 17 less.
constexpr int SUM64 = 16;  // terms of a chain in the FP64 sums
template <int M>
__global__ __launch_bounds__(128) void k_seg_tn_partial64(
    const Chunk* __restrict__ chunks, const double* __restrict__ A, int64_t lda, int aoff_e,
    int aoff_o, int ka, const double* __restrict__ B, int64_t ldb, int boff_e, int boff_o,
    int kb, double* __restrict__ partial) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Chunk ch = chunks[blockIdx.x];
  const int aoff = (ch.node & 1) ? aoff_o : aoff_e;
  const int boff = (ch.node & 1) ? boff_o : boff_e;
  const int tid = threadIdx.x, mtot = ka * kb, e0 = blockIdx.y * 128 * M;
  // the columns of B that outputs e0 .. need
  const int jlo = e0 / ka, nb = (min(e0 + 128 * M, mtot) - 1) / ka - jlo + 1;
  const int pa = ka | 1, pb = nb | 1;
  double* As = reinterpret_cast<double*>(smem_raw);  // [TN_ROWS][pa]
  double* Bs = As + TN_ROWS * pa;                    // [TN_ROWS][pb]
  int ia[M], jb[M];
  double acc[M];
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const int e = e0 + tid + 128 * m;
    ia[m] = e < mtot ? e % ka : 0;
    jb[m] = e < mtot ? e / ka - jlo : 0;
    acc[m] = 0.0;
  }
  const int rr = tid & 31, cg = tid >> 5;
  for (int64_t r0 = ch.r0; r0 < ch.r1; r0 += TN_ROWS) {
    const int rows = (int)min((int64_t)TN_ROWS, ch.r1 - r0);
    if (rr < rows) {
      for (int c = cg; c < ka; c += 4) As[rr * pa + c] = A[r0 + rr + (int64_t)(aoff + c) * lda];
      for (int c = cg; c < nb; c += 4)
        Bs[rr * pb + c] = B[r0 + rr + (int64_t)(boff + jlo + c) * ldb];
    }
    __syncthreads();
    for (int q0 = 0; q0 < rows; q0 += SUM64) {
      const int q1 = min(rows, q0 + SUM64);
      double t[M] = {};
#pragma unroll 4
      for (int q = q0; q < q1; ++q)
#pragma unroll
        for (int m = 0; m < M; ++m) t[m] = fma(As[q * pa + ia[m]], Bs[q * pb + jb[m]], t[m]);
#pragma unroll
      for (int m = 0; m < M; ++m) acc[m] += t[m];
    }
    __syncthreads();
  }
  double* out = partial + (int64_t)blockIdx.x * mtot;  // output (i, j) at i + j ka
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const int e = e0 + tid + 128 * m;
    if (e < mtot) out[e] = acc[m];
  }
}

// The same for few chunks (a small operator): 32 outputs a block, the chunk's groups of
// SUM64 rows dealt out to its eight warps, the groups' sums added in row order as above
// (the same bits: a column's result does not depend on how many go along).  One thread per
// output would be a chain of 256 dependent FMAs (10 us) behind eight exposed rounds of
// loads (12 us); here all rows are staged at once and a chain is 16 long.  4 chunks x
// 20 x 40 (N = 1024): 23 -> 10 us (164 with one block per chunk).
__global__ __launch_bounds__(256) void k_seg_tn_partial64_split(
    const Chunk* __restrict__ chunks, const double* __restrict__ A, int64_t lda, int aoff_e,
    int aoff_o, int ka, const double* __restrict__ B, int64_t ldb, int boff_e, int boff_o,
    int kb, double* __restrict__ partial) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Chunk ch = chunks[blockIdx.x];
  const int rows = (int)(ch.r1 - ch.r0);  // <= 256
  const int aoff = (ch.node & 1) ? aoff_o : aoff_e;
  const int boff = (ch.node & 1) ? boff_o : boff_e;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int mtot = ka * kb, e0 = blockIdx.y * 32, ne = min(32, mtot - e0);
  const int jlo = e0 / ka, nb = (e0 + ne - 1) / ka - jlo + 1;
  const int pb = nb | 1;
  double* As = reinterpret_cast<double*>(smem_raw);  // [256][33]: column c of output e0 + c
  double* Bs = As + 256 * 33;                        // [256][pb]
  const int row = tid;
  if (row < rows) {
    const double* ap = A + ch.r0 + row + (int64_t)aoff * lda;
    const double* bp = B + ch.r0 + row + (int64_t)(boff + jlo) * ldb;
#pragma unroll 8
    for (int c = 0; c < ne; ++c) As[row * 33 + c] = ap[(int64_t)((e0 + c) % ka) * lda];
    for (int c = 0; c < nb; ++c) Bs[row * pb + c] = bp[(int64_t)c * ldb];
  }
  __syncthreads();
  const int groups = (rows + SUM64 - 1) / SUM64;
  if (lane < ne) {
    const int jb = (e0 + lane) / ka - jlo;
    for (int g = w; g < groups; g += 8) {
      const int q1 = min(rows, (g + 1) * SUM64);
      double t = 0.0;
#pragma unroll 4
      for (int q = g * SUM64; q < q1; ++q) t = fma(As[q * 33 + lane], Bs[q * pb + jb], t);
      As[g * SUM64 * 33 + lane] = t;  // over an entry that this lane alone reads
    }
  }
  __syncthreads();
  if (w == 0 && lane < ne) {
    double v = 0.0;
    for (int g = 0; g < groups; ++g) v += As[g * SUM64 * 33 + lane];
    partial[(int64_t)blockIdx.x * mtot + e0 + lane] = v;
  }
}

// The FP64 form of the partial products in double-float arithmetic on the FP32
// pipe (GB300's FP64 pipe runs at a small fraction of the FP32 rate).  Each FP64
// input is cut once, when staged, into x = hi + lo (two floats, 48 significant
// bits); a product a b is formed as hi_a hi_b exactly (TwoProduct by FMA) plus
// the cross terms, and summed per output in a double-float (s_hi, s_lo) through
// TwoSum.  The partial of a chunk (<= 256 rows) is accurate to ~1e-14 relative.
//
// Bound by the FP32 pipe: 12 instructions per product.  A block takes one chunk
// and a 32 x 32 tile of the outputs (a thread 2 x 2 of it), so that a level of a
// few dozen chunks still fills the chip; which thread owns an output changes
// nothing in how it is summed.  The next 32 rows are in flight in registers while
// the staged ones are multiplied.  A step whose 32 columns of B are all zero is
// skipped (its products are exact zeros): the packed test matrices [Omega_2 |
// Omega_1] are zero on every other child's rows, and the column tiles do not
// straddle the two halves when kb is split (`half`).  N = 16384, 64 chunks, 60 x
// 120: 230 -> 80 us (64 x 128 outputs a block, one block per chunk, FP64-pipe cuts
// before); 60 x 60: 126 -> 48.
constexpr int DT = 32;  // outputs of a block: DT x DT

__global__ __launch_bounds__(256) void k_seg_tn_partial_df(
    const Chunk* __restrict__ chunks, const double* __restrict__ A, int64_t lda, int aoff_e,
    int aoff_o, int ka, const double* __restrict__ B, int64_t ldb, int boff_e, int boff_o,
    int kb, int half, double* __restrict__ partial) {
  __shared__ float2 As[TN_ROWS][DT + 1], Bs[TN_ROWS][DT + 1];
  const Chunk ch = chunks[blockIdx.x];
  const int aoff = (ch.node & 1) ? aoff_o : aoff_e;
  const int boff = (ch.node & 1) ? boff_o : boff_e;
  const int tid = threadIdx.x;
  const int ti = tid >> 4, tj = tid & 15;
  // columns [a0, a1) of A, [b0, b1) of B
  const int a0 = blockIdx.y * DT, a1 = min(ka, a0 + DT);
  const int per = (half + DT - 1) / DT, hz = (int)blockIdx.z / per;
  const int b0 = hz * half + ((int)blockIdx.z - hz * per) * DT;
  const int b1 = min(min(kb, (hz + 1) * half), b0 + DT);
  const int rr = tid & 31, cg = tid >> 5;  // staging: row, columns cg + 8 i
  const double* Ap = A + ch.r0 + rr + (int64_t)(aoff + a0) * lda;
  const double* Bp = B + ch.r0 + rr + (int64_t)(boff + b0) * ldb;
  double va[4], vb[4];
  auto load = [&](int64_t r0) {
    const bool live = ch.r0 + r0 + rr < ch.r1;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = cg + 8 * i;
      va[i] = (live && a0 + c < a1) ? Ap[r0 + (int64_t)c * lda] : 0.0;
      vb[i] = (live && b0 + c < b1) ? Bp[r0 + (int64_t)c * ldb] : 0.0;
    }
  };
  float sh[2][2] = {}, sl[2][2] = {};
  load(0);
  for (int64_t r0 = 0; ch.r0 + r0 < ch.r1; r0 += TN_ROWS) {
    bool nz = false;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = cg + 8 * i;
      float2 v;
      df::split(va[i], v.x, v.y);
      As[rr][c] = v;
      df::split(vb[i], v.x, v.y);
      Bs[rr][c] = v;
      nz |= !(v.x == 0.f);
    }
    load(r0 + TN_ROWS);
    if (__syncthreads_or(nz)) {
      const int rows = (int)min((int64_t)TN_ROWS, ch.r1 - ch.r0 - r0);
#pragma unroll 4
      for (int q = 0; q < rows; ++q) {
        float2 a[2], b[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) a[i] = As[q][ti + 16 * i];
#pragma unroll
        for (int j = 0; j < 2; ++j) b[j] = Bs[q][tj + 16 * j];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const float p = a[i].x * b[j].x;
            const float e = fmaf(a[i].x, b[j].x, -p);               // hi hi - p, exact
            const float t = fmaf(a[i].x, b[j].y, fmaf(a[i].y, b[j].x, e));
            const float s = sh[i][j] + p;                            // TwoSum(sh, p)
            const float z = s - sh[i][j];
            const float err = (sh[i][j] - (s - z)) + (p - z);
            sh[i][j] = s;
            sl[i][j] += err + t;
          }
      }
    }
    __syncthreads();
  }
  double* out = partial + (int64_t)blockIdx.x * ka * kb;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int ii = a0 + ti + 16 * i, jj = b0 + tj + 16 * j;
      if (ii < a1 && jj < b1) out[ii + jj * ka] = df::join(sh[i][j], sl[i][j]);
    }
}

// out[node] = sum of the node's chunk partials, in chunk order (deterministic).
template <typename T>
__global__ void k_seg_tn_reduce(const double* __restrict__ partial,
                                const int32_t* __restrict__ chunk_begin, int ka, int kb,
                                T* __restrict__ out) {
  const int node = blockIdx.y;
  const int c0 = chunk_begin[node], c1 = chunk_begin[node + 1];
  const int m = ka * kb;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m; e += gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int c = c0; c < c1; ++c) s += partial[(int64_t)c * m + e];
    out[(int64_t)node * m + e] = (T)s;
  }
}

constexpr int NN_ROWS = 64;
constexpr int NN_MAX = 128;

// One chunk of <= 64 rows.  Warp w owns output columns [16w, 16w + 16); lane
// owns rows lane and lane + 32.  P is staged before any write (in-place safe).
template <typename T>
__global__ __launch_bounds__(256) void k_seg_nn(
    const Chunk* __restrict__ chunks, int node0, const T* P, int64_t ldp, int poff_e,
    int poff_o, int kin, const T* __restrict__ C, int64_t cstride, int cld, int cflip, T* Y,
    int64_t ldy, int yoff_e, int yoff_o, int kout, T alpha, T beta) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* Ps = reinterpret_cast<T*>(smem_raw);   // [NN_MAX][NN_ROWS]
  T* Cs = Ps + NN_MAX * NN_ROWS;             // [NN_MAX][NN_MAX]
  const Chunk ch = chunks[blockIdx.x];
  const int rows = (int)(ch.r1 - ch.r0);
  const int poff = (ch.node & 1) ? poff_o : poff_e;
  const int yoff = (ch.node & 1) ? yoff_o : yoff_e;
  const T* Cn = C + (int64_t)((ch.node ^ cflip) - node0) * cstride;
  const int tid = threadIdx.x;
  for (int idx = tid; idx < kin * NN_ROWS; idx += 256) {
    const int rr = idx % NN_ROWS, k = idx / NN_ROWS;
    Ps[k * NN_ROWS + rr] = (rr < rows) ? P[ch.r0 + rr + (int64_t)(poff + k) * ldp] : (T)0;
  }
  for (int idx = tid; idx < kin * NN_MAX; idx += 256) {
    const int j = idx % NN_MAX, k = idx / NN_MAX;
    Cs[k * NN_MAX + j] = (j < kout) ? Cn[k + (int64_t)j * cld] : (T)0;
  }
  __syncthreads();
  const int lane = tid & 31, w = tid >> 5;
  double acc[2][16];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 16; ++j) acc[i][j] = 0.0;
  for (int k0 = 0; k0 < kin && w * 16 < kout; k0 += 16) {
    const int k1 = (k0 + 16 < kin) ? k0 + 16 : kin;
    T tmp[2][16];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 16; ++j) tmp[i][j] = 0;
    for (int k = k0; k < k1; ++k) {
      const T a0 = Ps[k * NN_ROWS + lane], a1 = Ps[k * NN_ROWS + lane + 32];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const T c = Cs[k * NN_MAX + w * 16 + j];
        tmp[0][j] = fma(a0, c, tmp[0][j]);
        tmp[1][j] = fma(a1, c, tmp[1][j]);
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 16; ++j) acc[i][j] += (double)tmp[i][j];
  }
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int col = w * 16 + j;
    if (col >= kout) continue;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int rr = lane + 32 * i;
      if (rr >= rows) continue;
      T* yp = Y + ch.r0 + rr + (int64_t)(yoff + col) * ldy;
      const double v = (double)alpha * acc[i][j];
      *yp = (beta == (T)0) ? (T)v : (T)(v + (double)beta * (double)(*yp));
    }
  }
}

// The FP64 expansion.  Bound by the FP64 pipe, as k_seg_tn_partial64: a block takes
// one chunk (<= 64 rows) and every gridDim.y-th tile of CT columns, its four warps
// the (row half, column group) pairs that exist, so that no FMA is issued for a
// column past kout or a row half past the chunk (the form with 16 columns a warp
// issued 128 columns whatever kout: 308 us for N = 16384, 60 x 37, this 85).  CT = 4
// where CT = 8 would leave schedulers without a block.  P aliasing Y: one block has
// all the tiles (P is staged whole before any write).
template <int CT>
__global__ __launch_bounds__(128) void k_seg_nn64(
    const Chunk* __restrict__ chunks, int node0, const double* P, int64_t ldp, int poff_e,
    int poff_o, int kin, const double* __restrict__ C, int64_t cstride, int cld, int cflip,
    double* Y, int64_t ldy, int yoff_e, int yoff_o, int kout, double alpha, double beta) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* Ps = reinterpret_cast<double*>(smem_raw);  // [kin][NN_ROWS]
  double* Cs = Ps + kin * NN_ROWS;                   // [CT][kin]
  const Chunk ch = chunks[blockIdx.x];
  const int rows = (int)(ch.r1 - ch.r0);
  const int poff = (ch.node & 1) ? poff_o : poff_e;
  const int yoff = (ch.node & 1) ? yoff_o : yoff_e;
  const double* Cn = C + (int64_t)((ch.node ^ cflip) - node0) * cstride;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  for (int idx = tid; idx < kin * NN_ROWS; idx += 128) {
    const int rr = idx % NN_ROWS, k = idx / NN_ROWS;
    Ps[idx] = (rr < rows) ? P[ch.r0 + rr + (int64_t)(poff + k) * ldp] : 0.0;
  }
  const int nh = rows > 32 ? 2 : 1, ng = 4 / nh;  // row halves, column groups
  const int rr = (nh == 2 ? (w & 1) * 32 : 0) + lane, g = w / nh;
  for (int c0 = blockIdx.y * CT; c0 < kout; c0 += gridDim.y * CT) {
    const int nc = min(CT, kout - c0);
    for (int idx = tid; idx < nc * kin; idx += 128) {
      const int k = idx % kin, j = idx / kin;
      Cs[idx] = Cn[k + (int64_t)(c0 + j) * cld];
    }
    __syncthreads();
    // this warp's columns g, g + ng, .. of the tile (at most CT / 2)
    const int nj = g < nc ? (nc - g + ng - 1) / ng : 0;
    double acc[CT / 2] = {};
    if (nj > 0)
      with_count<CT / 2>(nj, [&](auto cols) {
        for (int k0 = 0; k0 < kin; k0 += SUM64) {
          const int k1 = min(kin, k0 + SUM64);
          double t[cols] = {};
#pragma unroll 4
          for (int k = k0; k < k1; ++k) {
            const double a = Ps[k * NN_ROWS + rr];
#pragma unroll
            for (int j = 0; j < cols; ++j) t[j] = fma(a, Cs[(g + ng * j) * kin + k], t[j]);
          }
#pragma unroll
          for (int j = 0; j < cols; ++j) acc[j] += t[j];
        }
      });
#pragma unroll
    for (int j = 0; j < CT / 2; ++j) {
      if (j >= nj || rr >= rows) continue;
      double* yp = Y + ch.r0 + rr + (int64_t)(yoff + c0 + g + ng * j) * ldy;
      double v = acc[j];
      if (alpha == -1.0) v = -v;
      else if (alpha != 1.0) v *= alpha;
      *yp = (beta == 0.0) ? v : fma(beta, *yp, v);
    }
    __syncthreads();
  }
}

// The FP64 expansion in double-float arithmetic (HM_A32), as k_seg_tn_partial_df:
// inputs cut to hi + lo floats when staged, products by TwoProduct, sums by TwoSum.
// A block takes one chunk (<= 64 rows) and every gridDim.y-th 32-column tile of the
// output; warp w owns four of the columns, a lane rows lane and lane + 32.  Only
// what kin and 32 columns need is staged, so that four blocks share an SM where the
// full-width staging (196 KB) left one.  With P aliasing Y the launch gives one
// block all the tiles (P is staged whole before any write).  N = 16384, kin = 60,
// 120 columns: 126 -> 99 us; 60 columns: 67 -> 49.
__global__ __launch_bounds__(256) void k_seg_nn_df(
    const Chunk* __restrict__ chunks, int node0, const double* P, int64_t ldp, int poff_e,
    int poff_o, int kin, const double* __restrict__ C, int64_t cstride, int cld, int cflip,
    double* Y, int64_t ldy, int yoff_e, int yoff_o, int kout, double alpha, double beta) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int kp = kin | 1;                            // row pitch of Cs
  float2* Ps = reinterpret_cast<float2*>(smem_raw);  // [kin][NN_ROWS]
  float2* Cs = Ps + kin * NN_ROWS;                   // [DT][kp]
  const Chunk ch = chunks[blockIdx.x];
  const int rows = (int)(ch.r1 - ch.r0);
  const int poff = (ch.node & 1) ? poff_o : poff_e;
  const int yoff = (ch.node & 1) ? yoff_o : yoff_e;
  const double* Cn = C + (int64_t)((ch.node ^ cflip) - node0) * cstride;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  for (int idx = tid; idx < kin * NN_ROWS; idx += 256) {
    const int rr = idx % NN_ROWS, k = idx / NN_ROWS;
    float2 v;
    df::split((rr < rows) ? P[ch.r0 + rr + (int64_t)(poff + k) * ldp] : 0.0, v.x, v.y);
    Ps[idx] = v;
  }
  for (int c0 = blockIdx.y * DT; c0 < kout; c0 += gridDim.y * DT) {
    const int nc = min(DT, kout - c0);
    for (int j = w; j < DT; j += 8)
      for (int k = lane; k < kin; k += 32) {
        float2 v;
        df::split((j < nc) ? Cn[k + (int64_t)(c0 + j) * cld] : 0.0, v.x, v.y);
        Cs[j * kp + k] = v;
      }
    __syncthreads();
    float sh[2][4] = {}, sl[2][4] = {};
    if (4 * w < nc) {
#pragma unroll 2
      for (int k = 0; k < kin; ++k) {
        const float2 a[2] = {Ps[k * NN_ROWS + lane], Ps[k * NN_ROWS + lane + 32]};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 cj = Cs[(4 * w + j) * kp + k];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const float p = a[i].x * cj.x;
            const float e = fmaf(a[i].x, cj.x, -p);
            const float t = fmaf(a[i].x, cj.y, fmaf(a[i].y, cj.x, e));
            const float s = sh[i][j] + p;
            const float z = s - sh[i][j];
            const float err = (sh[i][j] - (s - z)) + (p - z);
            sh[i][j] = s;
            sl[i][j] += err + t;
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (4 * w + j >= nc) continue;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int rr = lane + 32 * i;
          if (rr >= rows) continue;
          double* yp = Y + ch.r0 + rr + (int64_t)(yoff + c0 + 4 * w + j) * ldy;
          double v = df::join(sh[i][j], sl[i][j]);
          if (alpha == -1.0) v = -v;  // (an FP64 product costs as much as the join's sum)
          else if (alpha != 1.0) v *= alpha;
          *yp = (beta == 0.0) ? v : fma(beta, *yp, v);
        }
      }
    }
    __syncthreads();
  }
}

}  // namespace

template <typename T, int TI, int TJ>
void seg_tn_partial_tiled(const Chunk* chunks, int nchunks, const T* A, int64_t lda,
                          int aoff_even, int aoff_odd, int ka, const T* B, int64_t ldb,
                          int boff_even, int boff_odd, int kb, double* partial, cudaStream_t st) {
  constexpr int LDA = 16 * TI + 1, LDB = 16 * TJ + 1;
    const size_t smem = TN_ROWS * (LDA + LDB) * sizeof(T);
    static std::atomic<uint32_t> done{0};
    raise_smem_limit((const void*)k_seg_tn_partial<T, TI, TJ>, done);
    k_seg_tn_partial<T, TI, TJ><<<nchunks, 256, smem, st>>>(
        chunks, A, lda, aoff_even, aoff_odd, ka, B, ldb, boff_even, boff_odd, kb, partial);
}

template <typename T, int TI>
void seg_tn_partial_pick_j(const Chunk* chunks, int nchunks, const T* A, int64_t lda,
                           int aoff_even, int aoff_odd, int ka, const T* B, int64_t ldb,
                           int boff_even, int boff_odd, int kb, double* partial, cudaStream_t st) {
  switch (tn_tile(kb)) {
    case 2:
      seg_tn_partial_tiled<T, TI, 2>(chunks, nchunks, A, lda, aoff_even, aoff_odd, ka, B, ldb,
                                     boff_even, boff_odd, kb, partial, st);
      break;
    case 4:
      seg_tn_partial_tiled<T, TI, 4>(chunks, nchunks, A, lda, aoff_even, aoff_odd, ka, B, ldb,
                                     boff_even, boff_odd, kb, partial, st);
      break;
    default:
      seg_tn_partial_tiled<T, TI, 8>(chunks, nchunks, A, lda, aoff_even, aoff_odd, ka, B, ldb,
                                     boff_even, boff_odd, kb, partial, st);
  }
}

// FP64 TN: outputs per thread (4, 2 or 1) so that the blocks of 4 warps cover the 608
// schedulers several times over (a block's time is set by its FMAs); below two warps of
// outputs a scheduler, the form that splits the rows.
static void seg_tn64(const Chunk* chunks, int nchunks, const double* A, int64_t lda, int aoff_even,
                     int aoff_odd, int ka, const double* B, int64_t ldb, int boff_even,
                     int boff_odd, int kb, double* partial, cudaStream_t st) {
  auto run = [&](auto kern, int m) {
    const int nb = std::min(kb, (128 * m - 1) / ka + 2);
    const size_t smem = (size_t)TN_ROWS * ((ka | 1) + (nb | 1)) * sizeof(double);
    const dim3 grid((unsigned)nchunks, (unsigned)((ka * kb + 128 * m - 1) / (128 * m)));
    kern<<<grid, 128, smem, st>>>(chunks, A, lda, aoff_even, aoff_odd, ka, B, ldb, boff_even,
                                  boff_odd, kb, partial);
  };
  static std::atomic<uint32_t> d0{0}, d1{0}, d2{0}, d4{0};
  const int64_t warps = (int64_t)nchunks * ((ka * kb + 31) / 32);  // one output a lane
  if (warps < 2 * 608) {
    const int nb = std::min(kb, 31 / ka + 2);
    raise_smem_limit((const void*)k_seg_tn_partial64_split, d0);
    const dim3 grid((unsigned)nchunks, (unsigned)((ka * kb + 31) / 32));
    k_seg_tn_partial64_split<<<grid, 256, (size_t)256 * (33 + (nb | 1)) * sizeof(double), st>>>(
        chunks, A, lda, aoff_even, aoff_odd, ka, B, ldb, boff_even, boff_odd, kb, partial);
  } else if (warps >= 16 * 608) {
    raise_smem_limit((const void*)k_seg_tn_partial64<4>, d4);
    run(k_seg_tn_partial64<4>, 4);
  } else if (warps >= 8 * 608) {
    raise_smem_limit((const void*)k_seg_tn_partial64<2>, d2);
    run(k_seg_tn_partial64<2>, 2);
  } else {
    raise_smem_limit((const void*)k_seg_tn_partial64<1>, d1);
    run(k_seg_tn_partial64<1>, 1);
  }
}

template <typename T>
void launch_seg_tn(const Chunk* chunks, int nchunks, const int32_t* chunk_begin, int nnodes,
                   int node0, const T* A, int64_t lda, int aoff_even, int aoff_odd, int ka,
                   const T* B, int64_t ldb, int boff_even, int boff_odd, int kb, double* partial,
                   T* out, cudaStream_t st, bool df, int half) {
  count_launches(2);
  (void)node0;
  if constexpr (sizeof(T) == 8) {
    if (df) {
      const int h = half > 0 ? half : kb;
      const dim3 grid((unsigned)nchunks, (unsigned)((ka + DT - 1) / DT),
                      (unsigned)(((h + DT - 1) / DT) * ((kb + h - 1) / h)));
      k_seg_tn_partial_df<<<grid, 256, 0, st>>>(chunks, A, lda, aoff_even, aoff_odd, ka, B, ldb,
                                                boff_even, boff_odd, kb, h, partial);
    } else {
      seg_tn64(chunks, nchunks, A, lda, aoff_even, aoff_odd, ka, B, ldb, boff_even, boff_odd, kb,
               partial, st);
    }
  } else {
    switch (tn_tile(ka)) {
      case 2:
        seg_tn_partial_pick_j<T, 2>(chunks, nchunks, A, lda, aoff_even, aoff_odd, ka, B, ldb,
                                    boff_even, boff_odd, kb, partial, st);
        break;
      case 4:
        seg_tn_partial_pick_j<T, 4>(chunks, nchunks, A, lda, aoff_even, aoff_odd, ka, B, ldb,
                                    boff_even, boff_odd, kb, partial, st);
        break;
      default:
        seg_tn_partial_pick_j<T, 8>(chunks, nchunks, A, lda, aoff_even, aoff_odd, ka, B, ldb,
                                    boff_even, boff_odd, kb, partial, st);
    }
  }
  const int m = ka * kb;
  dim3 grid((unsigned)((m + 255) / 256), (unsigned)nnodes);
  k_seg_tn_reduce<T><<<grid, 256, 0, st>>>(partial, chunk_begin, ka, kb, out);
}

template <typename T>
void launch_seg_nn(const Chunk* chunks, int nchunks, int node0, const T* P, int64_t ldp,
                   int poff_even, int poff_odd, int kin, const T* C, int64_t cstride, int cld,
                   int cflip, T* Y, int64_t ldy, int yoff_even, int yoff_odd, int kout, T alpha,
                   T beta, cudaStream_t st, bool df) {
  count_launches(1);
  if constexpr (sizeof(T) == 8) {
    const bool alias = (const void*)P == (const void*)Y;
    auto run = [&](auto kern, int threads, int ct, size_t smem) {
      const dim3 grid((unsigned)nchunks, alias ? 1u : (unsigned)((kout + ct - 1) / ct));
      kern<<<grid, threads, smem, st>>>(chunks, node0, P, ldp, poff_even, poff_odd, kin, C, cstride,
                                        cld, cflip, Y, ldy, yoff_even, yoff_odd, kout, alpha, beta);
    };
    static std::atomic<uint32_t> ddf{0}, d4{0}, d8{0};
    if (df) {
      raise_smem_limit((const void*)k_seg_nn_df, ddf);
      run(k_seg_nn_df, 256, DT, (size_t)(kin * NN_ROWS + DT * (kin | 1)) * sizeof(float2));
    } else if (alias || (int64_t)nchunks * ((kout + 7) / 8) >= 304) {  // two blocks per SM
      raise_smem_limit((const void*)k_seg_nn64<8>, d8);
      run(k_seg_nn64<8>, 128, 8, (size_t)kin * (NN_ROWS + 8) * sizeof(double));
    } else {
      raise_smem_limit((const void*)k_seg_nn64<4>, d4);
      run(k_seg_nn64<4>, 128, 4, (size_t)kin * (NN_ROWS + 4) * sizeof(double));
    }
  } else {
    const size_t smem = (size_t)(NN_MAX * NN_ROWS + NN_MAX * NN_MAX) * sizeof(T);
    static std::atomic<uint32_t> done{0};
    raise_smem_limit((const void*)k_seg_nn<T>, done);
    k_seg_nn<T><<<nchunks, 256, smem, st>>>(chunks, node0, P, ldp, poff_even, poff_odd, kin, C,
                                            cstride, cld, cflip, Y, ldy, yoff_even, yoff_odd, kout,
                                            alpha, beta);
  }
}

template void launch_seg_tn<float>(const Chunk*, int, const int32_t*, int, int, const float*,
                                   int64_t, int, int, int, const float*, int64_t, int, int, int,
                                   double*, float*, cudaStream_t, bool, int);
template void launch_seg_tn<double>(const Chunk*, int, const int32_t*, int, int, const double*,
                                    int64_t, int, int, int, const double*, int64_t, int, int,
                                    int, double*, double*, cudaStream_t, bool, int);
template void launch_seg_nn<float>(const Chunk*, int, int, const float*, int64_t, int, int, int,
                                   const float*, int64_t, int, int, float*, int64_t, int, int,
                                   int, float, float, cudaStream_t, bool);
template void launch_seg_nn<double>(const Chunk*, int, int, const double*, int64_t, int, int,
                                    int, const double*, int64_t, int, int, double*, int64_t, int,
                                    int, int, double, double, cudaStream_t, bool);

}  // namespace hm
