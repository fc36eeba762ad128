// Factored HODLR apply y = H x (the O(k N log N) product of Sec. 2.8 with
// sibling matrices B = I) and its hand-written adjoint (vector-Jacobian product
// for x, U, V, D; with r = H x - b and scale 2, the gradients of ||H x - b||^2).
//
// All are HBM-streaming.  Pass 1 reduces t_node = V(I_node)^T x(I_node) (and s_node =
// U(I_node)^T res(I_node) for the adjoint) over 256-row chunks of all levels; pass 2
// reduces the chunk partials per node in a fixed order; pass 3 runs one block per tile
// of a leaf's rows: every row gathers the contributions of its L ancestors' siblings
// (ancestor of leaf l on level j = l >> (L - j)) and of the leaf block D, and, for
// the adjoint, writes the gradient rows.  The fused step (loss_grad) forms the tile's
// share of s and of D^T res and the gradient of D in the forward's block too, from the
// tile's rows of U in shared memory and its rows of D in L2, so that U and D are read
// from HBM once.
#include <algorithm>
#include <atomic>
#include <string>

#include "hm_internal.h"

namespace hm {
namespace {

constexpr int kMaxK = 64;

// partial[chunk][0:k] = V_j(rows)^T x(rows); with second operand pair for the
// adjoint: partial[chunk][k:2k] = U_j(rows)^T res(rows).  Thread t loads row t's k
// factor entries at once (independent, coalesced loads), the products go to
// shared memory (row-major, stride k + 1: conflict-free both ways), thread
// (col, part) sums its 32-row part of a column, and the 8 parts are added.
// N = 262144, k = 32: 70 us for one operand (335 MB, 4.8 TB/s), 126 for two.  A form with
// a warp a column and no shared memory measured 67 for one operand but 241 for two (177
// with the operands in separate blocks, which cost 93 for one).
__global__ __launch_bounds__(256) void k_fact_partial(const FactChunk* __restrict__ ch,
                                                      int64_t n, int k,
                                                      const float* __restrict__ A0,
                                                      const float* __restrict__ v0,
                                                      const float* __restrict__ A1,
                                                      const float* __restrict__ v1,
                                                      float* __restrict__ partial) {
  extern __shared__ float prod[];  // [256][k + 1]
  __shared__ float red[8][2 * kMaxK];
  const FactChunk c = ch[blockIdx.x];
  const int tid = threadIdx.x;
  const int ldp = k + 1;
  const int64_t row = c.r0 + tid;
  const bool live = row < c.r1;
  const int npair = A1 ? 2 : 1;
  const int cl = tid & 31, part = tid >> 5;
  for (int p = 0; p < npair; ++p) {
    const float* A = (p == 0 ? A0 : A1) + (int64_t)(c.level - 1) * n * k;
    const float xv = live ? (p == 0 ? v0 : v1)[row] : 0.f;
#pragma unroll 8
    for (int col = 0; col < k; ++col)
      prod[tid * ldp + col] = live ? A[row + (int64_t)col * n] * xv : 0.f;
    __syncthreads();
    for (int col = cl; col < k; col += 32) {
      float s = 0.f;
#pragma unroll
      for (int i = 0; i < 32; ++i) s += prod[(part * 32 + i) * ldp + col];
      red[part][p * k + col] = s;
    }
    __syncthreads();
  }
  for (int e = tid; e < npair * k; e += 256) {
    float s = 0.f;
    for (int w = 0; w < 8; ++w) s += red[w][e];
    partial[(int64_t)blockIdx.x * npair * k + e] = s;
  }
}

// out[node][e] = sum over the node's chunks (heap ids 2 .. 2^(L+1)-1): chunks
// begin[node] .. begin[node + 1] at partial[chunk * width + e].  The threads form
// RED_C / width groups; group q sums chunks q, q + groups, ... and the group sums are
// added in group order (deterministic).  width <= 128.
constexpr int RED_T = 1024, RED_C = 256;
__global__ __launch_bounds__(RED_C) void k_fact_reduce(const float* __restrict__ partial,
                                                       const int32_t* __restrict__ fbegin,
                                                       int width, float* __restrict__ out) {
  __shared__ float sred[RED_C];
  const int node = 2 + blockIdx.x;
  const int c0 = fbegin[node], c1 = fbegin[node + 1];
  const int groups = RED_C / width;
  const int t = threadIdx.x, e = t % width, q = t / width;
  float s = 0.f;
  if (q < groups) {
#pragma unroll 8
    for (int c = c0 + q; c < c1; c += groups) s += partial[(int64_t)c * width + e];
  }
  sred[t] = s;
  __syncthreads();
  if (t < width) {
    float tot = 0.f;
    for (int g = 0; g < groups; ++g) tot += sred[g * width + t];
    out[(int64_t)node * width + t] = tot;
  }
}

// The same over the row tiles (`tiles` a leaf, L rows of k per tile) of a node's leaves:
// thousands for a node of level 1, where the chain of a thread's loads takes the time, one
// or two for most nodes, where the blocks do.  A block's RED_T / k groups are dealt out to
// as many nodes of one level as they serve with two tiles each.  N = 262144, k = 32: 16 us
// with a block a node, 14 so; the fused step at N = 70000, leaves of 69, k = 4: 90 and 75,
// at N = 131073, leaves of 9, k = 4: 702 and 440.
struct TileReduce {
  int k, L, tiles, blocks;
  int first[32], gpn[32];  // of a level: its first block, a node's groups
  TileReduce(int k_, int L_, int tiles_) : k(k_), L(L_), tiles(tiles_), blocks(0) {
    const int groups = RED_T / k;
    for (int j = 1; j <= L; ++j) {
      first[j] = blocks;
      gpn[j] = (int)std::min<int64_t>(groups, (((int64_t)tiles << (L - j)) + 1) / 2);
      const int npb = groups / gpn[j];
      blocks += ((1 << j) + npb - 1) / npb;
    }
  }
};
__global__ __launch_bounds__(RED_T, 2) void k_fact_reduce_tiles(const __grid_constant__ TileReduce r,
                                                             const float* __restrict__ partial,
                                                             float* __restrict__ out) {
  __shared__ float sred[RED_T];
  int j = 1;
  while (j < r.L && (int)blockIdx.x >= r.first[j + 1]) ++j;
  const int k = r.k, gpn = r.gpn[j], npb = RED_T / k / gpn;
  const int t = threadIdx.x, e = t % k, q = t / k, local = q / gpn, p = q - local * gpn;
  const int64_t x = (int64_t)(blockIdx.x - r.first[j]) * npb + local;  // node of the level
  const bool on = local < npb && x < (1 << j);
  float s = 0.f;
  if (on) {
    const int T = r.tiles << (r.L - j);
    const int64_t step = (int64_t)gpn * r.L * k;
    const float* a = partial + ((x * T + p) * r.L + j - 1) * k + e;
#pragma unroll 8
    for (int c = p; c < T; c += gpn, a += step) s += *a;
  }
  sred[t] = s;
  __syncthreads();
  if (on && p == 0) {
    float tot = 0.f;
    for (int g = 0; g < gpn; ++g) tot += sred[t + g * k];
    out[((1 << j) + x) * k + e] = tot;
  }
}

// The leaf kernels: a block takes a tile of `rt` rows of a leaf (a power of two), a
// thread a row and every LEAF_T / rt-th column (group g), eight loads in flight; the
// groups' row sums meet in shared memory.  The leaf's x is staged LEAF_X at a time.
constexpr int LEAF_T = 512, LEAF_X = 1024;

// Leaf and tile of a block (see tile_order): a leaf's tiles next to each other, or (tiles
// negative) every leaf's first tile before any second one.
__device__ __forceinline__ int2 leaf_tile(int L, int tiles) {
  const int b = blockIdx.x;
  if (tiles < 0) return make_int2(b & ((1 << L) - 1), b >> L);
  return make_int2(b / tiles, b % tiles);
}

// acc + sum over columns e = g, g + G, .. < m of a[e * ld] c[e]
constexpr int ROWB = 8;
__device__ __forceinline__ float row_dot(const float* a, int64_t ld, const float* c, int g, int G,
                                         int m, float acc) {
  for (int e0 = g; e0 < m; e0 += ROWB * G) {
    float v[ROWB];
#pragma unroll
    for (int q = 0; q < ROWB; ++q) {
      const int e = e0 + q * G;
      v[q] = e < m ? a[(int64_t)e * ld] : 0.f;
    }
#pragma unroll
    for (int q = 0; q < ROWB; ++q) {
      const int e = e0 + q * G;
      if (e < m) acc = fmaf(v[q], c[e], acc);
    }
  }
  return acc;
}
__device__ __forceinline__ float warp_total(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// y(I_leaf) = sum_j Uex_j(I_leaf) coef[sib(anc_j)] + op(D_leaf) x(I_leaf) for the block's
// rows.
__global__ __launch_bounds__(LEAF_T) void k_fact_expand(
    const int64_t* __restrict__ start, const int64_t* __restrict__ size, int L, int64_t n, int k,
    int nmax, int rt, const float* __restrict__ Uex, const float* __restrict__ coef,
    const float* __restrict__ D, int trans, const float* __restrict__ x, float* __restrict__ y) {
  extern __shared__ float sm[];
  const int ncol = L * k;          // column e of level 1 + e / k starts at Uex + e n
  float* cs = sm;                  // ncol coefficients
  float* xs = cs + ncol;           // LEAF_X entries of the leaf's x
  float* part = xs + LEAF_X;       // the groups' row sums
  float* rs = part + LEAF_T;       // rt rows of D^T x (trans)
  const int leaf = (1 << L) + blockIdx.x;
  const int64_t s0 = start[leaf];
  const int ns = (int)size[leaf];
  const int i0 = blockIdx.y * rt;
  if (i0 >= ns) return;  // uniform over the block
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = LEAF_T / rt, g = tid / rt, i = i0 + (tid & (rt - 1));
  for (int e = tid; e < ncol; e += LEAF_T) {
    const int j = 1 + e / k, col = e % k;
    const int anc = leaf >> (L - j);
    cs[e] = coef[(int64_t)(anc ^ 1) * k + col];
  }
  const float* Dl = D + (int64_t)blockIdx.x * nmax * nmax;
  if (trans)
    for (int q = warp; q < rt; q += LEAF_T / 32) {
      float v = 0.f;
      if (i0 + q < ns)
#pragma unroll 8
        for (int m = lane; m < ns; m += 32) v += Dl[m + (int64_t)(i0 + q) * nmax] * x[s0 + m];
      v = warp_total(v);
      if (lane == 0) rs[q] = v;
    }
  __syncthreads();
  const bool live = i < ns;
  float acc = 0.f;
  if (live) acc = row_dot(Uex + s0 + i, n, cs, g, G, ncol, acc);
  if (!trans)
    for (int m0 = 0; m0 < ns; m0 += LEAF_X) {
      const int mn = min(LEAF_X, ns - m0);
      __syncthreads();
      for (int m = tid; m < mn; m += LEAF_T) xs[m] = x[s0 + m0 + m];
      __syncthreads();
      if (live) acc = row_dot(Dl + i + (int64_t)m0 * nmax, nmax, xs, g, G, mn, acc);
    }
  part[tid] = acc;
  __syncthreads();
  if (g == 0 && live) {
    for (int q = 1; q < G; ++q) acc += part[q * rt + tid];
    if (trans) acc += rs[tid];
    y[s0 + i] = acc;
  }
}

// The same by whole leaves: a block of 256 threads holds the leaf's x (and D^T x) in shared
// memory, a thread takes a row.  For y in x's place (the tiles above read x over the whole
// leaf while other tiles write), and where the leaves alone fill the chip and the factors
// come from HBM (leaf_form_apply): N = 262144, k = 32, 604 MB: 100 us, the tiles 113-128
// (shorter runs of each column).
// IN_PLACE: x is y (the same address) and is read through y: a block reads its leaf before
// its first barrier, writes it after, and touches no other.  Plain loops over qualified
// pointers (the whole apply 181 us at k = 32; 189 with batches of eight conditional loads,
// 235 with the same loops unqualified; more loads in flight cost up to 1.6 times, N = 65536,
// k = 8 or 180001, k = 32: a block's warps then leave the column that they share).  Sums by
// level and by 32 columns of D: one chain over all of them rounds 2.5 times as much.
template <bool IN_PLACE>
__global__ __launch_bounds__(256) void k_fact_expand_leaf(
    const int64_t* __restrict__ start, const int64_t* __restrict__ size, int L, int64_t n, int k,
    int nmax, const float* __restrict__ Uex, const float* __restrict__ coef,
    const float* __restrict__ D, int trans, const float* __restrict__ x, float* __restrict__ y) {
  extern __shared__ float sm[];
  const int ncol = L * k;
  float* cs = sm;          // ncol coefficients
  float* xs = cs + ncol;   // the leaf's x
  float* dt = xs + nmax;   // D^T x (trans)
  const int leaf = (1 << L) + blockIdx.x;
  const int64_t s0 = start[leaf];
  const int ns = (int)size[leaf];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int e = tid; e < ncol; e += 256)
    cs[e] = coef[(int64_t)((leaf >> (L - 1 - e / k)) ^ 1) * k + e % k];
  for (int m = tid; m < ns; m += 256) xs[m] = (IN_PLACE ? y : x)[s0 + m];
  __syncthreads();
  const float* Dl = D + (int64_t)blockIdx.x * nmax * nmax;
  if (trans) {
    for (int i = warp; i < ns; i += 8) {
      float v = 0.f;
      for (int m = lane; m < ns; m += 32) v += Dl[m + (int64_t)i * nmax] * xs[m];
      v = warp_total(v);
      if (lane == 0) dt[i] = v;
    }
    __syncthreads();
  }
  for (int i = tid; i < ns; i += 256) {
    const float* u = Uex + s0 + i;
    float acc = 0.f;
    for (int j = 0; j < L; ++j) {
      float t = 0.f;
      for (int c = 0; c < k; ++c) t = fmaf(u[(int64_t)(j * k + c) * n], cs[j * k + c], t);
      acc += t;
    }
    if (trans) {
      acc += dt[i];
    } else {
      float t = 0.f;
      for (int m = 0; m < ns; ++m) {
        t = fmaf(Dl[i + (int64_t)m * nmax], xs[m], t);
        if ((m & 31) == 31) { acc += t; t = 0.f; }
      }
      acc += t;
    }
    y[s0 + i] = acc;
  }
}

// The forward of the fused step for one tile of rows: y = H x, res = y - b, the tile's
// share of every ancestor's s_node = U^T res (sp[leaf][tile][level][k]) and of D^T res
// (dtr[tile][row]), and its rows of the gradient of D.  The tile's rows of U and, where
// they fit (DS), of D are brought into shared memory by asynchronous copies (4 bytes:
// rows may start anywhere) that are all in flight at once, so that both products read
// them from there and HBM once; two blocks an SM overlap copies and arithmetic.
// N = 262144, k = 32, 870 MB: 227 us, bound by the copies' and the products'
// instructions; 340 us through registers with U and D read again from L2, 274 us with
// one block an SM walking the tiles, the next tile's copies in flight.
__device__ __forceinline__ void copy_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
template <int DS, int rt>
__global__ __launch_bounds__(LEAF_T) void k_fact_forward(
    const int64_t* __restrict__ start, const int64_t* __restrict__ size, int L, int64_t n, int k,
    int nmax, int tiles, const float* __restrict__ U, const float* __restrict__ coef,
    const float* __restrict__ D, const float* __restrict__ x, float* __restrict__ y,
    const float* __restrict__ b, float* __restrict__ res, float scale, float* __restrict__ sp,
    float* __restrict__ dtr, float* __restrict__ gD) {
  extern __shared__ float sm[];
  constexpr int pt = rt + 1, G = LEAF_T / rt;
  const int ncol = L * k;
  float* cs = sm;                  // ncol coefficients
  float* xs = cs + ncol;           // the leaf's x (DS), else LEAF_X entries of it
  float* part = xs + (DS ? nmax : LEAF_X);
  float* rs = part + LEAF_T;       // rt rows of res
  float* us = rs + rt;             // the tile's rows of U, [ncol][pt]
  float* ds = us + ncol * pt;      // DS: its rows of D, [nmax][pt]
  const int2 lt = leaf_tile(L, tiles);
  const int li = lt.x, tile = lt.y, leaf = (1 << L) + li;
  const int64_t s0 = start[leaf];
  const int ns = (int)size[leaf];
  const int i0 = tile * rt;
  const int tid = threadIdx.x;
  const int g = tid / rt, ti = tid & (rt - 1), i = i0 + ti;
  const bool live = i < ns;
  const float* Dl = D + (int64_t)li * nmax * nmax;
  if (live) {
    const float* u = U + s0 + i + (int64_t)g * n;
    float* d = us + g * pt + ti;
#pragma unroll 4
    for (int e = g; e < ncol; e += G, u += G * n, d += G * pt) copy_async4(d, u);
    if (DS) {
      u = Dl + i + (int64_t)g * nmax;
      d = ds + g * pt + ti;
#pragma unroll 4
      for (int m = g; m < ns; m += G, u += G * nmax, d += G * pt) copy_async4(d, u);
    }
  } else {
    for (int e = g; e < ncol; e += G) us[e * pt + ti] = 0.f;
    if (DS)
      for (int m = g; m < ns; m += G) ds[m * pt + ti] = 0.f;
  }
  for (int e = tid; e < ncol; e += LEAF_T) {
    const int j = 1 + e / k, col = e % k;
    const int anc = leaf >> (L - j);
    cs[e] = coef[(int64_t)(anc ^ 1) * k + col];
  }
  if (DS)
    for (int m = tid; m < ns; m += LEAF_T) xs[m] = x[s0 + m];
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  float acc = 0.f;
#pragma unroll 4
  for (int e = g; e < ncol; e += G) acc = fmaf(us[e * pt + ti], cs[e], acc);
  if (DS) {
#pragma unroll 4
    for (int m = g; m < ns; m += G) acc = fmaf(ds[m * pt + ti], xs[m], acc);
  } else {
    for (int m0 = 0; m0 < ns; m0 += LEAF_X) {
      const int mn = min(LEAF_X, ns - m0);
      __syncthreads();
      for (int m = tid; m < mn; m += LEAF_T) xs[m] = x[s0 + m0 + m];
      __syncthreads();
      if (live) acc = row_dot(Dl + i + (int64_t)m0 * nmax, nmax, xs, g, G, mn, acc);
    }
  }
  part[tid] = acc;
  __syncthreads();
  if (g == 0) {
#pragma unroll
    for (int q = 1; q < G; ++q) acc += part[q * rt + tid];
    float r = 0.f;
    if (live) {
      r = acc - b[s0 + i];
      y[s0 + i] = acc;
      res[s0 + i] = r;
    }
    rs[ti] = r;
  }
  __syncthreads();
  // a thread a column: D^T res, then U^T res over the tile's rows
  float* spt = sp + ((int64_t)li * abs(tiles) + tile) * ncol;
  float* dt = dtr + (int64_t)tile * n + s0;
  const int nd = DS ? ns : 0;
  for (int e = tid; e < nd + ncol; e += LEAF_T) {
    const float* c = e < nd ? ds + e * pt : us + (e - nd) * pt;
    float v = 0.f;
#pragma unroll
    for (int q = 0; q < rt; ++q) v = fmaf(c[q], rs[q], v);
    if (e < nd) dt[e] = v;
    else spt[e - nd] = v;
  }
  if (!DS) {
    const int lane = tid & 31, nr = max(0, min(rt, ns - i0));
    for (int m = tid >> 5; m < ns; m += LEAF_T / 32) {
      float v = 0.f;
      for (int q = lane; q < nr; q += 32) v = fmaf(Dl[i0 + q + (int64_t)m * nmax], rs[q], v);
      v = warp_total(v);
      if (lane == 0) dt[m] = v;
    }
  }
  if (gD && i < nmax) {
    // (zero past the leaf's size, in rows and columns)
    const float sr = scale * rs[ti];
    float* o = gD + (int64_t)li * nmax * nmax + i + (int64_t)g * nmax;
#pragma unroll 4
    for (int m = g; m < nmax; m += G, o += G * nmax)
      __stcs(o, live && m < ns ? sr * (DS ? xs[m] : x[s0 + m]) : 0.f);
  }
}

// Adjoint rows of one tile of a leaf.  Per node, coef_t holds t_node = V_j(I_node)^T x
// and coef_s holds s_node = U_j(I_node)^T res, at node * cw (+ the k entries).  dtr: the
// tiles' shares of D^T res where the forward has formed them (and written gD), else null.
__global__ __launch_bounds__(LEAF_T) void k_fact_adjoint(
    const int64_t* __restrict__ start, const int64_t* __restrict__ size, int L, int64_t n, int k,
    int nmax, int rt, int tiles, const float* __restrict__ V, const float* __restrict__ D,
    const float* __restrict__ coef_t, const float* __restrict__ coef_s, int cw,
    const float* __restrict__ x, const float* __restrict__ res, float scale,
    const float* __restrict__ dtr, int dtiles, float* __restrict__ gx, float* __restrict__ gU,
    float* __restrict__ gV, float* __restrict__ gD) {
  extern __shared__ float sm[];
  const int ncol = L * k;
  float* ts = sm;                  // t of the sibling per level
  float* ss = ts + ncol;           // s of the sibling per level
  float* part = ss + ncol;         // the groups' row sums
  float* dt = part + LEAF_T;       // D^T res of the tile's rows
  const int2 lt = leaf_tile(L, tiles);
  const int li = lt.x, leaf = (1 << L) + li;
  const int64_t s0 = start[leaf];
  const int ns = (int)size[leaf];
  const int i0 = lt.y * rt;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = LEAF_T / rt, g = tid / rt, i = i0 + (tid & (rt - 1));
  for (int e = tid; e < ncol; e += LEAF_T) {
    const int j = 1 + e / k, col = e % k;
    const int sib = (leaf >> (L - j)) ^ 1;
    ts[e] = coef_t[(int64_t)sib * cw + col];
    ss[e] = coef_s[(int64_t)sib * cw + col];
  }
  if (gx && !dtr) {
    const float* Dl = D + (int64_t)li * nmax * nmax;
    for (int q = warp; q < rt; q += LEAF_T / 32) {
      float v = 0.f;
      if (i0 + q < ns)
#pragma unroll 8
        for (int m = lane; m < ns; m += 32) v += Dl[m + (int64_t)(i0 + q) * nmax] * res[s0 + m];
      v = warp_total(v);
      if (lane == 0) dt[q] = v;
    }
  }
  __syncthreads();
  const bool live = i < ns;
  const float xi = live ? x[s0 + i] : 0.f, ri = live ? res[s0 + i] : 0.f;
  float acc = 0.f;
  if (live) {
    const float sx = scale * xi, sr = scale * ri;
    const int64_t row = s0 + i;
    for (int e0 = g; e0 < ncol; e0 += 8 * G) {
      float v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int e = e0 + q * G;
        v[q] = (gx && e < ncol) ? V[row + (int64_t)e * n] : 0.f;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int e = e0 + q * G;
        if (e < ncol) {
          const int64_t off = row + (int64_t)e * n;
          acc = fmaf(v[q], ss[e], acc);
          if (gU) __stcs(gU + off, sr * ts[e]);
          if (gV) __stcs(gV + off, sx * ss[e]);
        }
      }
    }
  }
  if (gx) {
    part[tid] = acc;
    __syncthreads();
    if (g == 0 && live) {
      for (int q = 1; q < G; ++q) acc += part[q * rt + tid];
      float d = 0.f;
      if (dtr) for (int q = 0; q < dtiles; ++q) d += dtr[(int64_t)q * n + s0 + i];
      else d = dt[tid];
      gx[s0 + i] = scale * (acc + d);
    }
  }
  if (gD && !dtr && i < nmax) {
    // (zero past the leaf's size, in rows and columns)
    float* gDl = gD + (int64_t)li * nmax * nmax + i;
    const float sr = scale * ri;
#pragma unroll 4
    for (int m = g; m < nmax; m += G)
      __stcs(gDl + (int64_t)m * nmax, live && m < ns ? sr * x[s0 + m] : 0.f);
  }
}

// The same by whole leaves (leaf_form_adjoint), coefficients of t and s in one array: a
// thread a row of the leaf, x, res and D^T res in shared memory.  N = 262144, leaves of 256:
// 276 us at k = 32 (the tiles 301); the whole adjoint at k = 8 208 us (231).  A thread's sum
// over all columns is compensated (its own rounding would be 1.8 times the tiles'); sums by
// groups of columns cost up to a fifth of the time.
__global__ __launch_bounds__(256) void k_fact_adjoint_leaf(
    const int64_t* __restrict__ start, const int64_t* __restrict__ size, int L, int64_t n, int k,
    int nmax, const float* __restrict__ V, const float* __restrict__ D,
    const float* __restrict__ coef, const float* __restrict__ x, const float* __restrict__ res,
    float scale, float* __restrict__ gx, float* __restrict__ gU, float* __restrict__ gV,
    float* __restrict__ gD) {
  extern __shared__ float sm[];
  const int ncol = L * k;
  float* ts = sm;           // t of the sibling per level
  float* ss = ts + ncol;    // s of the sibling per level
  float* xs = ss + ncol;
  float* rs = xs + nmax;
  float* dt = rs + nmax;    // D^T res
  const int leaf = (1 << L) + blockIdx.x;
  const int64_t s0 = start[leaf];
  const int ns = (int)size[leaf];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int e = tid; e < ncol; e += 256) {
    const float* c = coef + (int64_t)((leaf >> (L - 1 - e / k)) ^ 1) * 2 * k + e % k;
    ts[e] = c[0];
    ss[e] = c[k];
  }
  for (int m = tid; m < ns; m += 256) {
    xs[m] = x[s0 + m];
    rs[m] = res[s0 + m];
  }
  __syncthreads();
  if (gx) {
    const float* Dl = D + (int64_t)blockIdx.x * nmax * nmax;
    for (int i = warp; i < ns; i += 8) {
      float v = 0.f;
      for (int m = lane; m < ns; m += 32) v += Dl[m + (int64_t)i * nmax] * rs[m];
      v = warp_total(v);
      if (lane == 0) dt[i] = v;
    }
    __syncthreads();
  }
  float* gDl = gD + (int64_t)blockIdx.x * nmax * nmax;
  for (int i = tid; i < ns; i += 256) {
    const int64_t row = s0 + i;
    const float xr = xs[i], rr = rs[i];
    float acc = 0.f, err = 0.f;
    for (int e = 0; e < ncol; ++e) {
      const int64_t off = row + (int64_t)e * n;
      if (gx) {
        const float v = V[off], s = fmaf(v, ss[e], acc);
        err += fmaf(v, ss[e], acc - s);  // what the sum has just lost
        acc = s;
      }
      if (gU) gU[off] = scale * rr * ts[e];
      if (gV) gV[off] = scale * xr * ss[e];
    }
    // (a sum that overflowed has lost NaN; it stays infinite)
    if (gx) gx[row] = scale * (acc + (isnan(err) ? 0.f : err) + dt[i]);
    if (gD)
      for (int m = 0; m < nmax; ++m) gDl[i + (int64_t)m * nmax] = m < ns ? scale * rr * xs[m] : 0.f;
  }
  if (gD && ns < nmax) {  // rows past the leaf's size
    const int pad = nmax - ns;
    for (int e = tid; e < pad * nmax; e += 256)
      gDl[ns + e % pad + (int64_t)(e / pad) * nmax] = 0.f;
  }
}

}  // namespace

// Leaves are taken up to this much shared memory for a whole leaf's slices of x (and
// res, D^T res) beside the coefficients: the limit of hm_hodlr_factored_apply and its
// adjoint, kept although the kernels' tiles need less.
static size_t fact_leaf_smem(const hm_tree* t, bool adjoint) {
  const size_t nmax = (size_t)t->nmax, L = (size_t)t->L;
  return adjoint ? sizeof(float) * (2 * L * kMaxK + 3 * nmax)
                 : sizeof(float) * (L * kMaxK + 2 * nmax);
}

// dynamic shared memory of k_fact_partial (66.5 KB at k = 64: limit raised once)
static size_t fact_partial_smem(int k) {
  static std::atomic<uint32_t> done{0};
  raise_smem_limit((const void*)k_fact_partial, done);
  return sizeof(float) * 256 * (size_t)(k + 1);
}

// Whole leaves where they fill the chip and long runs of each column count more than the
// number of blocks: leaves enough, and few columns beside a leaf's own (its D is most of
// what is read), or a large n.  Measured on 400 trees of 512 to 262144 points, us by
// leaves / by tiles: apply N = 70000, leaves of 137, k = 8 24 / 40, N = 200001, 196, 32
// 137 / 179, N = 50000, 196, 4 (256 leaves) 21 / 27; the other side N = 65536, 128, 64
// 113 / 95, N = 131072, 64, 32 131 / 113, N = 65536, 512, 4 101 / 51.  (The transposed
// product's tiles read D along its columns and hold out longer: N = 131072, 256, 4 74 / 65.)
static bool leaf_form_apply(const hm_tree* t, int k, int trans) {
  const int64_t leaves = (int64_t)1 << t->L, ncol = (int64_t)t->L * k;
  if (!trans && leaves >= 256 && ncol <= 96) return true;
  if (leaves >= 608 && 4 * t->n * (ncol + t->nmax) >= (trans ? 128ll : 256ll) << 20) return true;
  if (trans && (t->n < 57000 || (leaves < 1024 && t->nmax > 200))) return false;
  return leaves >= 512 &&
         (ncol <= std::max<int64_t>(t->nmax, 160) || (t->n >= 100000 && t->nmax >= 70));
}
// The adjoint writes as much as it reads: N = 131072, leaves of 256, k = 8 102 / 128,
// N = 262144, 256, 32 420 / 433; the other side N = 262144, 128, 32 514 / 432, N = 30001, 15,
// 64 488 / 244.
static bool leaf_form_adjoint(const hm_tree* t, int k) {
  const int64_t leaves = (int64_t)1 << t->L, ncol = (int64_t)t->L * k;
  return leaves >= 512 && 2 * ncol <= 3 * t->nmax && (t->nmax >= 100 || 5 * ncol <= 3 * t->nmax);
}
// Rows of a block's tile: 64, or 32 where 64 would leave SMs without two blocks
// (N = 4096 in leaves of 256: 64 blocks of 64 rows, 128 of 32).
static int leaf_rows(const hm_tree* t) {
  const int64_t leaves = (int64_t)1 << t->L;
  return leaves * ((t->nmax + 63) / 64) >= 304 ? 64 : 32;
}
// The fused forward keeps its tile's L k columns of U and, where two blocks an SM then
// still fit, its rows of D in shared memory: 32 rows, 16 where L k is above 797 (13 levels
// at k = 64; at the most, L = 24 and k = 64, one block an SM).
static size_t forward_smem(const hm_tree* t, int k, int rt, bool ds) {
  const size_t ncol = (size_t)t->L * k, nmax = (size_t)t->nmax;
  return sizeof(float) * (ncol * (rt + 2) + LEAF_T + rt + (ds ? nmax * (rt + 2) : LEAF_X));
}
constexpr size_t kForwardSmem = 112 * 1024;
static int forward_rows(const hm_tree* t, int k) {
  return forward_smem(t, k, 32, false) <= kForwardSmem ? 32 : 16;
}
static bool forward_ds(const hm_tree* t, int k) {
  return forward_smem(t, k, forward_rows(t, k), true) <= kForwardSmem;
}
static size_t expand_smem(const hm_tree* t, int k, int rt) {
  return sizeof(float) * ((size_t)t->L * k + LEAF_X + LEAF_T + rt);
}
static size_t adjoint_smem(const hm_tree* t, int k, int rt) {
  return sizeof(float) * (2 * (size_t)t->L * k + LEAF_T + rt);
}
static size_t dsize(const hm_tree* t) { return ((size_t)1 << t->L) * t->nmax * t->nmax; }

// An output that shares memory with an input: the tiles of a leaf read its whole slices of
// x, res and D while others write, and the kernels' pointers are qualified as disjoint, so
// such calls take a copy or launches of their own.
bool factored_overlap(const float* a, size_t na, const float* b, size_t nb) {
  return a < b + nb && b < a + na;
}

// V is read for gx by the launch that writes gU and gV.  (U is not.)
static bool v_in_place(const hm_tree* t, int k, const float* V, const float* gU, const float* gV) {
  const size_t m = (size_t)t->n * t->L * k;
  return (gU && factored_overlap(gU, m, V, m)) || (gV && factored_overlap(gV, m, V, m));
}

static int leaf_tiles(const hm_tree* t, int rt) { return (int)((t->nmax + rt - 1) / rt); }
static unsigned leaf_grid(const hm_tree* t, int rt) {
  return (1u << t->L) * (unsigned)leaf_tiles(t, rt);
}
// The order of the tiles in the kernels that write gradients.  Two tiles of a leaf share
// memory sectors (rows may start anywhere).  With every leaf's first tile before any second
// one the two parts of a gradient's sector went to HBM apart: fused step, k = 32, N = 262143
// 763 us (571 with a leaf's tiles next to each other; N = 262144 525 and 513), N = 200001
// 666 (467).  While the gradients fit L2 they meet there in any order, and the leaves' last
// tiles, which may be short, are better last (adjoint, N = 20000, leaves of 157, k = 64: 69
// us, 74 by neighbours); so they are in the apply, which writes no columns.
static int tile_order(const hm_tree* t, int k, int rt) {
  const int64_t written = 4 * t->n * (2 * (int64_t)t->L * k + t->nmax);
  return written < (96ll << 20) ? -leaf_tiles(t, rt) : leaf_tiles(t, rt);
}

hm_status factored_check(const hm_tree* t, bool adjoint) {
  int dev = 0, optin = 0;
  HM_CUDA_TRY(cudaGetDevice(&dev));
  HM_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  const size_t need = fact_leaf_smem(t, adjoint);
  if (need > (size_t)optin) {
    set_error(std::string(adjoint ? "hm_hodlr_factored_adjoint" : "hm_hodlr_factored_apply") +
              ": leaves of " + std::to_string(t->nmax) + " points need " + std::to_string(need) +
              " bytes of shared memory per block; the device allows " + std::to_string(optin));
    return HM_EINVAL;
  }
  static std::atomic<uint32_t> done_e{0}, done_i{0}, done_p{0}, done_a{0}, done_l{0};
  raise_smem_limit((const void*)k_fact_expand, done_e);
  raise_smem_limit((const void*)k_fact_expand_leaf<false>, done_i);
  raise_smem_limit((const void*)k_fact_expand_leaf<true>, done_p);
  if (adjoint) {
    raise_smem_limit((const void*)k_fact_adjoint, done_a);
    raise_smem_limit((const void*)k_fact_adjoint_leaf, done_l);
  }
  return HM_OK;
}

size_t factored_scratch_bytes(const hm_tree* t, int k) {
  const size_t nodes = (size_t)1 << (t->L + 1);
  return sizeof(float) * ((size_t)t->n_fchunks * 2 * k + nodes * 2 * k) + 256;
}

// x and y: one vector (x == y) or disjoint ones (other overlaps: the callers copy x).
void launch_factored_apply(const hm_tree* t, int k, const float* U, const float* V,
                           const float* D, int trans, const float* x, float* y, float* scratch,
                           cudaStream_t st) {
  count_launches(3);
  const int L = t->L;
  const int nodes = 1 << (L + 1), rt = leaf_rows(t);
  float* partial = scratch;
  float* coef = scratch + (size_t)t->n_fchunks * k;
  // t_node = Proj(I_node)^T x with Proj = V (H x) or U (H^T x)
  k_fact_partial<<<t->n_fchunks, 256, fact_partial_smem(k), st>>>(
      t->d_fchunks, t->n, k, trans ? U : V, x, nullptr, nullptr, partial);
  k_fact_reduce<<<nodes - 2, RED_C, 0, st>>>(partial, t->d_fbegin, k, coef);
  const size_t leaf_smem = sizeof(float) * ((size_t)L * k + 2 * t->nmax);
  if (x == y)
    k_fact_expand_leaf<true><<<1u << L, 256, leaf_smem, st>>>(
        t->d_start, t->d_size, L, t->n, k, (int)t->nmax, trans ? V : U, coef, D, trans, nullptr, y);
  else if (leaf_form_apply(t, k, trans))
    k_fact_expand_leaf<false><<<1u << L, 256, leaf_smem, st>>>(
        t->d_start, t->d_size, L, t->n, k, (int)t->nmax, trans ? V : U, coef, D, trans, x, y);
  else
    k_fact_expand<<<dim3(1u << L, leaf_tiles(t, rt)), LEAF_T, expand_smem(t, k, rt), st>>>(
        t->d_start, t->d_size, L, t->n, k, (int)t->nmax, rt, trans ? V : U, coef, D, trans, x, y);
}

// gU and gV may share memory with U and V, gD with D; gx shares none with the inputs.
void launch_factored_adjoint(const hm_tree* t, int k, const float* U, const float* V,
                             const float* D, const float* x, const float* res, float scale,
                             float* gx, float* gU, float* gV, float* gD, float* scratch,
                             cudaStream_t st) {
  count_launches(3);
  const int L = t->L;
  const int nodes = 1 << (L + 1), rt = leaf_rows(t);
  float* partial = scratch;
  float* coef = scratch + (size_t)t->n_fchunks * 2 * k;
  k_fact_partial<<<t->n_fchunks, 256, fact_partial_smem(k), st>>>(t->d_fchunks, t->n, k, V, x, U,
                                                                  res, partial);
  k_fact_reduce<<<nodes - 2, RED_C, 0, st>>>(partial, t->d_fbegin, 2 * k, coef);
  const bool d_in_place = gD && factored_overlap(gD, dsize(t), D, dsize(t));
  auto run = [&](float* ox, float* oU, float* oV, float* oD) {
    if (leaf_form_adjoint(t, k))
      k_fact_adjoint_leaf<<<1u << L, 256, sizeof(float) * (2 * (size_t)L * k + 3 * t->nmax), st>>>(
          t->d_start, t->d_size, L, t->n, k, (int)t->nmax, V, D, coef, x, res, scale, ox, oU, oV,
          oD);
    else
      k_fact_adjoint<<<leaf_grid(t, rt), LEAF_T, adjoint_smem(t, k, rt), st>>>(
          t->d_start, t->d_size, L, t->n, k, (int)t->nmax, rt, tile_order(t, k, rt), V, D, coef,
          coef + k, 2 * k, x, res, scale, nullptr, 0, ox, oU, oV, oD);
  };
  if (gx && v_in_place(t, k, V, gU, gV)) {
    run(gx, nullptr, nullptr, d_in_place ? nullptr : gD);
    count_launches(1);
    run(nullptr, gU, gV, nullptr);  // once every row of V has been read
  } else {
    run(gx, gU, gV, d_in_place ? nullptr : gD);
  }
  if (d_in_place) {  // once every tile has read D
    count_launches(1);
    run(nullptr, nullptr, nullptr, gD);
  }
}

size_t factored_loss_grad_scratch_bytes(const hm_tree* t, int k) {
  const size_t nodes = (size_t)1 << (t->L + 1);
  const size_t tiles = leaf_tiles(t, forward_rows(t, k));
  return sizeof(float) * ((size_t)t->n_fchunks * k + (nodes / 2) * tiles * t->L * k +
                          2 * nodes * k + (2 + tiles) * (size_t)t->n) + 512;
}

// y = H x, res = y - b and the adjoint at res: the forward's projections t = V^T x are
// the adjoint's too, the forward's blocks also form s = U^T res (per tile of rows;
// reduced per node), D^T res and the gradient of D, and the adjoint's pass reads V once
// more and writes gx, gU, gV.  y and res share no memory with x and b, gx none with x; gU
// and gV may with U and V, gD with D, gx with res.  N = 262144, k = 32 (2.2 GB instead of
// 2.8): 557 -> 502 us.
void launch_factored_loss_grad(const hm_tree* t, int k, const float* U, const float* V,
                               const float* D, const float* x, const float* b, float scale,
                               float* y, float* res, float* gx, float* gU, float* gV, float* gD,
                               float* scratch, cudaStream_t st) {
  count_launches(5);
  const int L = t->L;
  const int nodes = 1 << (L + 1);
  const int nmax = (int)t->nmax;
  const int rf = forward_rows(t, k), rt = leaf_rows(t);
  const int tiles = leaf_tiles(t, rf), order = tile_order(t, k, rt);
  float* partial = scratch;
  float* sp = partial + (size_t)t->n_fchunks * k;
  float* coef_t = sp + (size_t)(nodes / 2) * tiles * L * k;
  float* coef_s = coef_t + (size_t)nodes * k;
  float* tmp = coef_s + (size_t)nodes * k;
  float* yy = y ? y : tmp;
  float* rr = res ? res : tmp + t->n;
  float* dtr = tmp + 2 * t->n;
  k_fact_partial<<<t->n_fchunks, 256, fact_partial_smem(k), st>>>(t->d_fchunks, t->n, k, V, x,
                                                                  nullptr, nullptr, partial);
  k_fact_reduce<<<nodes - 2, RED_C, 0, st>>>(partial, t->d_fbegin, k, coef_t);
  const bool ds = forward_ds(t, k);
  const bool d_in_place = gD && factored_overlap(gD, dsize(t), D, dsize(t));
  auto forward = [&](auto kern, std::atomic<uint32_t>& done) {
    raise_smem_limit((const void*)kern, done);
    kern<<<leaf_grid(t, rf), LEAF_T, forward_smem(t, k, rf, ds), st>>>(
        t->d_start, t->d_size, L, t->n, k, nmax, tile_order(t, k, rf), U, coef_t, D, x, yy, b, rr,
        scale, sp, dtr, d_in_place ? nullptr : gD);
  };
  static std::atomic<uint32_t> done[4] = {{0}, {0}, {0}, {0}};
  if (rf == 32 && ds) forward(k_fact_forward<1, 32>, done[0]);
  else if (rf == 32) forward(k_fact_forward<0, 32>, done[1]);
  else if (ds) forward(k_fact_forward<1, 16>, done[2]);
  else forward(k_fact_forward<0, 16>, done[3]);
  const TileReduce tr(k, L, tiles);
  k_fact_reduce_tiles<<<tr.blocks, RED_T, 0, st>>>(tr, sp, coef_s);
  if (d_in_place) {  // once every tile has read D
    count_launches(1);
    k_fact_adjoint<<<leaf_grid(t, rt), LEAF_T, adjoint_smem(t, k, rt), st>>>(
        t->d_start, t->d_size, L, t->n, k, nmax, rt, order, V, D, coef_t, coef_s, k, x, rr, scale,
        nullptr, 0, nullptr, nullptr, nullptr, gD);
  }
  if (res && gx && factored_overlap(gx, t->n, res, t->n)) {
    launch_copy_cols<float>(res, t->n, tmp + t->n, t->n, t->n, 1, st);
    rr = tmp + t->n;
  }
  auto adjoint = [&](float* ox, float* oU, float* oV) {
    k_fact_adjoint<<<leaf_grid(t, rt), LEAF_T, adjoint_smem(t, k, rt), st>>>(
        t->d_start, t->d_size, L, t->n, k, nmax, rt, order, V, D, coef_t, coef_s, k, x, rr, scale,
        dtr, tiles, ox, oU, oV, nullptr);
  };
  if (gx && v_in_place(t, k, V, gU, gV)) {
    adjoint(gx, nullptr, nullptr);
    count_launches(1);
    adjoint(nullptr, gU, gV);  // once every row of V has been read
  } else if (gx || gU || gV) {
    adjoint(gx, gU, gV);
  }
}

}  // namespace hm
