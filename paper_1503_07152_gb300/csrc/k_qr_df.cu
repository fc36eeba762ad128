// FP64-accurate SVD of the panels' R factors in double-float arithmetic
// (HM_A32): the phases of k_jacobi_mp (k_qr.cu) with every bulk FP64 operation
// carried by float pairs on the FP32 pipe, which GB300 runs at many times its
// FP64 rate.  Inputs and outputs stay FP64.
#include <atomic>

#include "df.cuh"
#include "hm_internal.h"

namespace hm {
namespace {

// (xh, xl) <- c x - s y and (yh, yl) <- s x + c y for DF c, s, x, y: the leading
// products exactly by TwoProduct, the cross terms in FP32, one TwoSum and a
// renormalization per output.
__device__ __forceinline__ void rot_df(float ch, float cl, float sh, float sl, float& xh, float& xl,
                                       float& yh, float& yl) {
  const float x0 = xh, x1 = xl, y0 = yh, y1 = yl;
  {
    const float p1 = ch * x0, p2 = sh * y0;
    const float e1 = fmaf(ch, x0, -p1), e2 = fmaf(sh, y0, -p2);
    float r, e3;
    df::two_sum(p1, -p2, r, e3);
    float lo = (e1 - e2) + e3;
    lo = fmaf(ch, x1, fmaf(cl, x0, lo));
    lo = fmaf(-sh, y1, fmaf(-sl, y0, lo));
    df::fast_two_sum(r, lo, xh, xl);
  }
  {
    const float p1 = sh * x0, p2 = ch * y0;
    const float e1 = fmaf(sh, x0, -p1), e2 = fmaf(ch, y0, -p2);
    float r, e3;
    df::two_sum(p1, p2, r, e3);
    float lo = (e1 + e2) + e3;
    lo = fmaf(sh, x1, fmaf(sl, x0, lo));
    lo = fmaf(ch, y1, fmaf(cl, y0, lo));
    df::fast_two_sum(r, lo, yh, yl);
  }
}

// Rotation of one FP32 Jacobi pair (phase B below): ga = a_p . a_q, al and be
// the squared norms.  Flags a correlation above big2 (another sweep is due) and
// returns false when the pair is already orthogonal to tol; otherwise (tc, ts)
// = (cos, sin) of the angle that zeroes ga (the smaller root of the standard
// two-sided formula).
__device__ __forceinline__ bool jacobi_angle32(float ga, float al, float be, float tol,
                                               float big2, int gl, int& large, float& tc,
                                               float& ts) {
  if (gl == 0 && al > 0.f && be > 0.f && (ga / al) * (ga / be) > big2) large = 1;
  if (!(ga != 0.f && fabsf(ga) > tol * sqrtf(al) * sqrtf(be))) return false;
  const float zeta = (be - al) / (2.f * ga);
  const float t = (zeta >= 0.f ? 1.f : -1.f) / (fabsf(zeta) + sqrtf(1.f + zeta * zeta));
  tc = 1.f / sqrtf(1.f + t * t);
  ts = tc * t;
  return true;
}
// The rotation of an FP32 pair with its roundings spelled out: left to the compiler, the
// contraction of the two products can differ between instantiations of the kernel, and
// a node's result must not depend on the widths it shares a launch with.
__device__ __forceinline__ float rot_c(float tc, float ts, float x, float y) {
  return fmaf(tc, x, -__fmul_rn(ts, y));
}
__device__ __forceinline__ float rot_s(float tc, float ts, float x, float y) {
  return fmaf(ts, x, __fmul_rn(tc, y));
}
// the pair's squared norms after the rotation (c^2 al - 2cs ga + s^2 be and
// s^2 al + 2cs ga + c^2 be, clamped at 0)
__device__ __forceinline__ void jacobi_norms32(float tc, float ts, float ga, float& np,
                                               float& nq) {
  const float al = np, be = nq;
  const float cs2 = 2.f * tc * ts, c2 = tc * tc, s2 = ts * ts;
  np = fmaxf(fmaf(c2, al, fmaf(-cs2, ga, s2 * be)), 0.f);
  nq = fmaxf(fmaf(s2, al, fmaf(cs2, ga, c2 * be)), 0.f);
}

// SVD of R (c x c, c <= 128) to about 2^-46 relative accuracy for HM_A32, the
// phases of k_jacobi_mp with every bulk FP64 operation in double-float:
//   A. column-pivoted Householder QR R P = Q2 R2 (Businger-Golub; DF entries,
//      column norms and reflector scalars in FP64); X = R2^T (graded columns)
//      parked in the node's W slot;
//   B. one-sided Jacobi on float(X), rotations accumulated into V32 (FP32);
//   C. Q = classical Gram-Schmidt of V32 in DF;
//   D. X1 = X Q in DF: the left singular vectors of X, columns orthogonal to
//      FP32 precision;
//   E. one-sided Jacobi sweeps on X1 in DF until every pair's correlation is
//      below the DF rounding level (angles from FP32 ratios of DF quantities:
//      small-angle series for |t| < 2^-11, FP64 formulas otherwise; the
//      rotations themselves in DF, orthogonal to DF rounding);
//   F. sigma_j = |X1_j|, W = P U_x from the normalized columns, sorted
//      descending, the sign convention of k_jacobi_mp.
// R is scaled by a power of two (exact) so that its largest entry lies in
// [1, 2): squared column norms then stay inside the float range.
template <int NB>
__global__ __launch_bounds__(512, 1) void k_jacobi_df(const int32_t* __restrict__ node_slot,
                                                      const double* __restrict__ R, int c,
                                                      double* __restrict__ W,
                                                      double* __restrict__ sigma,
                                                      const NodeJob* __restrict__ jobs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const double* Rs;
  double *Wn, *sig;
  if (jobs) {  // a level-wide launch over several operators' nodes
    const NodeJob& jb = jobs[blockIdx.x];
    c = jb.c;
    Rs = jb.R;
    Wn = jb.W;
    sig = jb.sigma;
  } else {
    Rs = R + (int64_t)node_slot[blockIdx.x] * c * c;
    Wn = W + (int64_t)blockIdx.x * c * c;
    sig = sigma + (int64_t)blockIdx.x * c;
  }
  // Columns are LD apart and their rows padded with zeros to 32 NB >= c, so that every
  // element loop has a fixed count and no condition (a condition per element kept the
  // loads of a loop from overlapping); LD = 8 mod 32 puts the columns that the four
  // groups of a warp work on in different banks.
  constexpr int LD = 32 * NB + 8, NE = 4 * NB;  // NE: an 8-lane group's elements per lane
  const int cc = c * c;
  float* reg0 = reinterpret_cast<float*>(smem_raw);
  float* reg1 = reg0 + c * LD;
  float* reg2 = reg1 + c * LD;
  float* Mh = reg0;   // A: R, then R2 (column-major)
  float* Ml = reg1;
  float* V32 = reg0;  // B, C
  float* X32 = reg1;  // B
  float* Qh = reg1;   // C - F
  float* Ql = reg2;
  __shared__ int rotated, large;
  __shared__ double sv[128], hb[128];
  __shared__ float cnh[128], cnl[128], hbh[128], hbl[128];
  __shared__ float psh[4][128], psl[4][128];
  __shared__ int perm[128], order[128];
  __shared__ signed char sgn[128];
  __shared__ double red_v[16];
  __shared__ int red_i[16];
  __shared__ float pnh[128], pnl[128], ph0[128];  // A: pivoting norms
  __shared__ float sh_ah, sh_al, sh_sh, sh_sl, sh_vh, sh_vl;
  __shared__ int sh_exp;
  __shared__ float2 vb[32 * NB];  // A: the reflector, zero outside its rows
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int nthr = blockDim.x;
  const int pg = tid >> 3, gl = tid & 7;
  // ------------------------------------------------------------- scale
  {
    double mx = 0.0;
    for (int idx = tid; idx < cc; idx += nthr) mx = fmax(mx, fabs(Rs[idx]));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) red_v[warp] = mx;
    __syncthreads();
    if (tid == 0) {
      double m2 = 0.0;
      for (int w = 0; w < nwarps; ++w) m2 = fmax(m2, red_v[w]);
      int e = 0;
      if (m2 > 0.0 && isfinite(m2)) frexp(m2, &e);  // m2 in [2^(e-1), 2^e)
      sh_exp = e - 1;
    }
    __syncthreads();
  }
  const int ex = sh_exp;
  // ---------------------------------------------------------------- A
  for (int idx = tid; idx < cc; idx += nthr) {
    const int rr = idx / c, col = idx % c;
    df::split(ldexp(Rs[idx], -ex), Mh[col * LD + rr], Ml[col * LD + rr]);
  }
  for (int idx = tid; idx < c * (LD - c); idx += nthr) {
    const int o = idx / (LD - c) * LD + c + idx % (LD - c);
    Mh[o] = 0.f;
    Ml[o] = 0.f;
  }
  for (int j = tid; j < c; j += nthr) perm[j] = j;
  __syncthreads();
  // Squared column norms for the pivoting, kept as double-float pairs (pnh, pnl)
  // and downdated per step; ph0 holds the value at the last exact recompute.
  // Every scalar of this phase is double-float: a dependent chain of FP64
  // instructions (a square root, a division) is very long on GB300's FP64 pipe.
  for (int k = warp; k < c; k += nwarps) {
    float sh = 0.f, sl = 0.f;
    for (int i = lane; i < c; i += 32) df::dot_acc(Mh[k * LD + i], Ml[k * LD + i], Mh[k * LD + i], Ml[k * LD + i], sh, sl);
    df::warp_sum(sh, sl);
    if (lane == 0) { df::fast_two_sum(sh, sl, pnh[k], pnl[k]); ph0[k] = pnh[k]; }
  }
  __syncthreads();
  for (int j = 0; j < c; ++j) {
    // recompute the norms that downdating has left with few correct digits
    for (int k = j + warp; k < c; k += nwarps) {
      if (!(pnh[k] > 5.9604644775390625e-08f * ph0[k])) {
        float sh = 0.f, sl = 0.f;
        for (int i = j + lane; i < c; i += 32)
          df::dot_acc(Mh[k * LD + i], Ml[k * LD + i], Mh[k * LD + i], Ml[k * LD + i], sh, sl);
        df::warp_sum(sh, sl);
        if (lane == 0) { df::fast_two_sum(sh, sl, pnh[k], pnl[k]); ph0[k] = pnh[k]; }
      }
    }
    __syncthreads();
    if (warp == 0) {  // the largest remaining norm, the first on ties
      float bh = -1.f, bl = 0.f;
      int bi = c;
      for (int k = j + lane; k < c; k += 32)
        if (pnh[k] > bh || (pnh[k] == bh && pnl[k] > bl)) { bh = pnh[k]; bl = pnl[k]; bi = k; }
      for (int o = 16; o > 0; o >>= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, bh, o);
        const float ol = __shfl_xor_sync(0xffffffffu, bl, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (oh > bh || (oh == bh && (ol > bl || (ol == bl && oi < bi)))) { bh = oh; bl = ol; bi = oi; }
      }
      if (lane == 0) red_i[0] = bi;
    }
    __syncthreads();
    const int p = red_i[0];
    if (p != j && p < c) {
      for (int i = tid; i < c; i += nthr) {
        float t = Mh[j * LD + i]; Mh[j * LD + i] = Mh[p * LD + i]; Mh[p * LD + i] = t;
        t = Ml[j * LD + i]; Ml[j * LD + i] = Ml[p * LD + i]; Ml[p * LD + i] = t;
      }
      if (tid == 0) {
        const int t = perm[j]; perm[j] = perm[p]; perm[p] = t;
        float u = pnh[j]; pnh[j] = pnh[p]; pnh[p] = u;
        u = pnl[j]; pnl[j] = pnl[p]; pnl[p] = u;
        u = ph0[j]; ph0[j] = ph0[p]; ph0[p] = u;
      }
    }
    __syncthreads();
    float* mjh = Mh + j * LD;
    float* mjl = Ml + j * LD;
    if (warp == 0) {  // the reflector needs the pivot column's exact norm
      float sh = 0.f, sl = 0.f;
      for (int i = j + lane; i < c; i += 32) df::dot_acc(mjh[i], mjl[i], mjh[i], mjl[i], sh, sl);
      df::warp_sum(sh, sl);
      if (lane == 0) {
        // x0 and the reflector scale sqrt(2 / v^T v), v^T v = 2 nrm (nrm + |x0|)
        const float xh = mjh[j], xl = mjl[j];
        float nh, nl;
        df::sqrt_df(sh, sl, nh, nl);
        const float ah = (xh > 0.f) ? -nh : nh, al = (xh > 0.f) ? -nl : nl;
        float vh, vl, wh = nh, wl = nl, qh, ql, sch = 0.f, scl = 0.f;
        df::sub(xh, xl, ah, al, vh, vl);                        // v0 = x0 - alpha
        df::add_to(wh, wl, fabsf(xh), xh < 0.f ? -xl : xl);      // nrm + |x0|
        df::mul(nh, nl, wh, wl, qh, ql);                         // v^T v / 2
        if (qh > 0.f) {
          float ih, il;
          df::div_df(1.f, 0.f, qh, ql, ih, il);
          df::sqrt_df(ih, il, sch, scl);
        }
        sh_ah = ah;
        sh_al = al;
        sh_sh = sch;
        sh_sl = scl;
        df::mul(vh, vl, sch, scl, sh_vh, sh_vl);
      }
    }
    __syncthreads();
    const float sch = sh_sh, scl = sh_sl;
    if (tid < 32 * NB) {
      float2 v = make_float2(0.f, 0.f);
      if (tid == j) v = make_float2(sh_vh, sh_vl);
      else if (tid > j) df::mul(sch, scl, mjh[tid], mjl[tid], v.x, v.y);
      vb[tid] = v;
    }
    __syncthreads();
    if (sch != 0.f) {
      // One 8-lane group per trailing column; lane gl holds rows 8 q + gl (the group sum
      // does not see by how many lanes the rows are rotated: k_tsqr_df), four slices of
      // rows at a time
      for (int k0 = j + 1; k0 < c; k0 += 64) {
        const int k = k0 + pg;
        const bool on = k < c;
        float* mkh = Mh + (on ? k : j) * LD + gl;
        float* mkl = Ml + (on ? k : j) * LD + gl;
        float dh = 0.f, dl = 0.f;
        if (on) {
#pragma unroll
          for (int q0 = 0; q0 < NE; q0 += 4) {
            if (8 * q0 + 31 < j) continue;
            float2 v[4], m[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              v[q] = vb[8 * (q0 + q) + gl];
              m[q] = make_float2(mkh[8 * (q0 + q)], mkl[8 * (q0 + q)]);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) df::dot_acc(v[q].x, v[q].y, m[q].x, m[q].y, dh, dl);
          }
        }
        df::group8_sum(dh, dl);
        if (on) {
          float fh, fl;
          df::fast_two_sum(dh, dl, fh, fl);
#pragma unroll
          for (int q0 = 0; q0 < NE; q0 += 4) {
            if (8 * q0 + 31 < j) continue;
            float2 v[4], m[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              v[q] = vb[8 * (q0 + q) + gl];
              m[q] = make_float2(mkh[8 * (q0 + q)], mkl[8 * (q0 + q)]);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              df::axpy_neg(fh, fl, v[q].x, v[q].y, m[q].x, m[q].y);
              mkh[8 * (q0 + q)] = m[q].x;
              mkl[8 * (q0 + q)] = m[q].y;
            }
          }
        }
      }
    }
    __syncthreads();
    if (tid == 0) {  // R2(j, j)
      mjh[j] = sch != 0.f ? sh_ah : 0.f;
      mjl[j] = sch != 0.f ? sh_al : 0.f;
    }
    for (int k = j + 1 + tid; k < c; k += nthr) {  // downdate: |col k|^2 -= R(j, k)^2
      float rh, rl;
      df::mul(Mh[k * LD + j], Ml[k * LD + j], Mh[k * LD + j], Ml[k * LD + j], rh, rl);
      df::sub(pnh[k], pnl[k], rh, rl, pnh[k], pnl[k]);
    }
    __syncthreads();
  }
  // X = R2^T, column-major, parked in the W slot as float pairs (hi parts, then
  // lo parts: the c x c doubles of the slot hold both), so that phase D reads it
  // without conversions
  float* Xph = reinterpret_cast<float*>(Wn);
  float* Xpl = Xph + cc;
  for (int idx = tid; idx < cc; idx += nthr) {
    const int col = idx / c, row = idx % c;  // X(row, col) = R2(col, row), zero above
    const bool low = row >= col;
    Xph[idx] = low ? Mh[row * LD + col] : 0.f;
    Xpl[idx] = low ? Ml[row * LD + col] : 0.f;
  }
  __syncthreads();
  // ---------------------------------------------------------------- B
  for (int idx = tid; idx < c * LD; idx += nthr) {
    const int col = idx / LD, row = idx - col * LD;
    X32[idx] = row < c ? Xph[col * c + row] : 0.f;
    V32[idx] = col == row ? 1.f : 0.f;
  }
  __syncthreads();
  const int cp = (c + 1) & ~1;
  float* cn32 = cnh;  // FP32 squared column norms of X32 (cnh is free until E)
  for (int j = warp; j < c; j += nwarps) {
    float s2 = 0.f;
    for (int i = lane; i < c; i += 32) s2 = fmaf(X32[j * LD + i], X32[j * LD + i], s2);
    for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    if (lane == 0) cn32[j] = s2;
  }
  __syncthreads();
  {
    const float tol = (float)(5.960464477539063e-08 * sqrt((double)c));
    const float big2 = tol;
    const bool vec = (c & 3) == 0;
    for (int sweep = 0; sweep < 40; ++sweep) {
      if (tid == 0) { rotated = 0; large = 0; }
      __syncthreads();
      for (int step = 0; step < cp - 1; ++step) {
        int p = c, q = c;
        if (pg < cp / 2) {
          const int a = pg, b = cp - 1 - pg;
          // round-robin pairing: a - 1 + step < 2 (cp - 1) and b - 1 + step < 2 (cp - 1)
          int va = a - 1 + step, vb = b - 1 + step;
          if (va >= cp - 1) va -= cp - 1;
          if (vb >= cp - 1) vb -= cp - 1;
          p = (a == 0) ? 0 : va + 1;
          q = vb + 1;
        }
        const bool valid = p < c && q < c;
        float* ap = X32 + (valid ? p : 0) * LD;
        float* aq = X32 + (valid ? q : 0) * LD;
        if (vec) {
          // c a multiple of 4: lane gl holds the 16-byte chunks gl, gl + 8, ..
          // of both columns in registers (one 128-byte row of shared memory per
          // group and load: no bank conflicts) for the dot product and the
          // rotation
          float4 xa[NB], xb[NB];
          float ga = 0.f;
#pragma unroll
          for (int k = 0; k < NB; ++k) {
            xa[k] = reinterpret_cast<const float4*>(ap)[gl + 8 * k];
            xb[k] = reinterpret_cast<const float4*>(aq)[gl + 8 * k];
          }
#pragma unroll
          for (int k = 0; k < NB; ++k) {
            ga = fmaf(xa[k].x, xb[k].x, ga);
            ga = fmaf(xa[k].y, xb[k].y, ga);
            ga = fmaf(xa[k].z, xb[k].z, ga);
            ga = fmaf(xa[k].w, xb[k].w, ga);
          }
          ga += __shfl_xor_sync(0xffffffffu, ga, 4);
          ga += __shfl_xor_sync(0xffffffffu, ga, 2);
          ga += __shfl_xor_sync(0xffffffffu, ga, 1);
          float tc, ts;
          if (valid && jacobi_angle32(ga, cn32[p], cn32[q], tol, big2, gl, large, tc, ts)) {
            float4* vp = reinterpret_cast<float4*>(V32 + p * LD);
            float4* vq = reinterpret_cast<float4*>(V32 + q * LD);
            float4 u[NB], w[NB];
#pragma unroll
            for (int k = 0; k < NB; ++k) {
              u[k] = vp[gl + 8 * k];
              w[k] = vq[gl + 8 * k];
            }
#pragma unroll
            for (int k = 0; k < NB; ++k) {
              const int ch = gl + 8 * k;
              const float4 x = xa[k], y = xb[k];
              reinterpret_cast<float4*>(ap)[ch] =
                  make_float4(rot_c(tc, ts, x.x, y.x), rot_c(tc, ts, x.y, y.y), rot_c(tc, ts, x.z, y.z),
                              rot_c(tc, ts, x.w, y.w));
              reinterpret_cast<float4*>(aq)[ch] =
                  make_float4(rot_s(tc, ts, x.x, y.x), rot_s(tc, ts, x.y, y.y), rot_s(tc, ts, x.z, y.z),
                              rot_s(tc, ts, x.w, y.w));
              vp[ch] = make_float4(rot_c(tc, ts, u[k].x, w[k].x), rot_c(tc, ts, u[k].y, w[k].y),
                                   rot_c(tc, ts, u[k].z, w[k].z), rot_c(tc, ts, u[k].w, w[k].w));
              vq[ch] = make_float4(rot_s(tc, ts, u[k].x, w[k].x), rot_s(tc, ts, u[k].y, w[k].y),
                                   rot_s(tc, ts, u[k].z, w[k].z), rot_s(tc, ts, u[k].w, w[k].w));
            }
            __syncwarp(0xffu << (8 * (lane >> 3)));  // the group's reads of the norms first
            if (gl == 0) {
              jacobi_norms32(tc, ts, ga, cn32[p], cn32[q]);
              rotated = 1;
            }
          }
        } else {
          float ga = 0;
#pragma unroll
          for (int ii = 0; ii < NE; ++ii) ga = fmaf(ap[gl + 8 * ii], aq[gl + 8 * ii], ga);
          ga += __shfl_xor_sync(0xffffffffu, ga, 4);
          ga += __shfl_xor_sync(0xffffffffu, ga, 2);
          ga += __shfl_xor_sync(0xffffffffu, ga, 1);
          float tc, ts;
          if (valid && jacobi_angle32(ga, cn32[p], cn32[q], tol, big2, gl, large, tc, ts)) {
            float* vp = V32 + p * LD;
            float* vq = V32 + q * LD;
#pragma unroll
            for (int ii = 0; ii < NE; ++ii) {
              const int i = gl + 8 * ii;
              const float x = ap[i], y = aq[i];
              ap[i] = rot_c(tc, ts, x, y);
              aq[i] = rot_s(tc, ts, x, y);
            }
#pragma unroll
            for (int ii = 0; ii < NE; ++ii) {
              const int i = gl + 8 * ii;
              const float x = vp[i], y = vq[i];
              vp[i] = rot_c(tc, ts, x, y);
              vq[i] = rot_s(tc, ts, x, y);
            }
            __syncwarp(0xffu << (8 * (lane >> 3)));  // the group's reads of the norms first
            if (gl == 0) {
              jacobi_norms32(tc, ts, ga, cn32[p], cn32[q]);
              rotated = 1;
            }
          }
        }
        __syncthreads();
      }
      const int any = rotated && large;
      __syncthreads();
      if (!any) break;
    }
  }
  // ---------------------------------------------------------------- C
  // (X32 is dead; Q overlays it and the third region)
  for (int j = 0; j < c; ++j) {
    float* qjh = Qh + j * LD;
    float* qjl = Ql + j * LD;
    for (int i = tid; i < LD; i += nthr) { qjh[i] = V32[j * LD + i]; qjl[i] = 0.f; }
    __syncthreads();
    for (int i0 = 0; i0 < j; i0 += 64) {  // one 8-lane group per earlier column
      const int i = i0 + pg;
      const bool on = i < j;
      const float* qih = Qh + (on ? i : 0) * LD + gl;
      const float* qil = Ql + (on ? i : 0) * LD + gl;
      float sh = 0.f, sl = 0.f;
      if (on) {
#pragma unroll
        for (int e0 = 0; e0 < NE; e0 += 4) {
          float xh[4], xl[4], yh[4], yl[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int o = 8 * (e0 + e);
            xh[e] = qih[o]; xl[e] = qil[o]; yh[e] = qjh[gl + o]; yl[e] = qjl[gl + o];
          }
#pragma unroll
          for (int e = 0; e < 4; ++e) df::dot_acc(xh[e], xl[e], yh[e], yl[e], sh, sl);
        }
      }
      df::group8_sum(sh, sl);
      if (on && gl == 0) { hbh[i] = sh; hbl[i] = sl; }
    }
    __syncthreads();
    {  // q_j -= sum_i hb[i] Q_i in four partial sums over quarters of i
      const int e = tid & 127, part = tid >> 7;
      const int i0 = (j * part) >> 2, i1 = (j * (part + 1)) >> 2;
      float sh = 0.f, sl = 0.f;
      if (e < c) {
#pragma unroll 4
        for (int i = i0; i < i1; ++i) df::dot_acc(hbh[i], hbl[i], Qh[i * LD + e], Ql[i * LD + e], sh, sl);
      }
      df::add_to(sh, sl, 0.f, 0.f);
      psh[part][e] = sh;
      psl[part][e] = sl;
    }
    __syncthreads();
    for (int e = tid; e < c; e += nthr) {
      float sh = psh[0][e], sl = psl[0][e];
      df::add_to(sh, sl, psh[1][e], psl[1][e]);
      df::add_to(sh, sl, psh[2][e], psl[2][e]);
      df::add_to(sh, sl, psh[3][e], psl[3][e]);
      df::add_to(qjh[e], qjl[e], -sh, -sl);
    }
    __syncthreads();
    if (warp == 0) {
      float sh = 0.f, sl = 0.f;
      for (int e = lane; e < c; e += 32) df::dot_acc(qjh[e], qjl[e], qjh[e], qjl[e], sh, sl);
      df::warp_sum(sh, sl);
      if (lane == 0) {
        const double s = df::join(sh, sl);
        df::split((s > 0.0) ? 1.0 / sqrt(s) : 0.0, sh_sh, sh_sl);
      }
    }
    __syncthreads();
    const float ih = sh_sh, il = sh_sl;
    for (int e = tid; e < c; e += nthr) df::mul(ih, il, qjh[e], qjl[e], qjh[e], qjl[e]);
    __syncthreads();
  }
  // ---------------------------------------------------------------- D
  for (int j = warp; j < c; j += nwarps) {
    float ah[NB] = {}, alo[NB] = {};
#pragma unroll 4
    for (int k = 0; k < c; ++k) {
      const float qh = Qh[j * LD + k], ql = Ql[j * LD + k];
      const float* xkh = Xph + k * c;
      const float* xkl = Xpl + k * c;
#pragma unroll
      for (int rr = 0; rr < NB; ++rr) {
        const int row = lane + 32 * rr;
        const float xh = row < c ? xkh[row] : 0.f, xl = row < c ? xkl[row] : 0.f;
        df::dot_acc(xh, xl, qh, ql, ah[rr], alo[rr]);
      }
    }
    __syncwarp();
#pragma unroll
    for (int rr = 0; rr < NB; ++rr) {  // (zero in the padding)
      const int row = lane + 32 * rr;
      df::fast_two_sum(ah[rr], alo[rr], Qh[j * LD + row], Ql[j * LD + row]);
    }
  }
  __syncthreads();
  // ---------------------------------------------------------------- E
  for (int j = warp; j < c; j += nwarps) {
    float sh = 0.f, sl = 0.f;
    for (int i = lane; i < c; i += 32) df::dot_acc(Qh[j * LD + i], Ql[j * LD + i], Qh[j * LD + i], Ql[j * LD + i], sh, sl);
    df::warp_sum(sh, sl);
    if (lane == 0) df::fast_two_sum(sh, sl, cnh[j], cnl[j]);
  }
  __syncthreads();
  {
    // a pair is rotated while its correlation exceeds the DF rounding level of
    // the length-c dot products that measure it
    const float tol = (float)(3.552713678800501e-15 * sqrt((double)c));  // 2^-48 sqrt(c)
    const float tol2 = tol * tol, big2 = tol;
    for (int sweep = 0; sweep < 12; ++sweep) {
      if (tid == 0) { rotated = 0; large = 0; }
      __syncthreads();
      for (int step = 0; step < cp - 1; ++step) {
        int p = c, q = c;
        if (pg < cp / 2) {
          const int a = pg, b = cp - 1 - pg;
          int va = a - 1 + step, vb = b - 1 + step;
          if (va >= cp - 1) va -= cp - 1;
          if (vb >= cp - 1) vb -= cp - 1;
          p = (a == 0) ? 0 : va + 1;
          q = vb + 1;
        }
        const bool valid = p < c && q < c;
        float* aph = Qh + (valid ? p : 0) * LD + gl;
        float* apl = Ql + (valid ? p : 0) * LD + gl;
        float* aqh = Qh + (valid ? q : 0) * LD + gl;
        float* aql = Ql + (valid ? q : 0) * LD + gl;
        float gh = 0.f, glo = 0.f;
        if (valid) {
#pragma unroll
          for (int e0 = 0; e0 < NE; e0 += 4) {
            float xh[4], xl[4], yh[4], yl[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int o = 8 * (e0 + e);
              xh[e] = aph[o]; xl[e] = apl[o]; yh[e] = aqh[o]; yl[e] = aql[o];
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) df::dot_acc(xh[e], xl[e], yh[e], yl[e], gh, glo);
          }
        }
        df::group8_sum(gh, glo);
        df::fast_two_sum(gh, glo, gh, glo);
        if (valid) {
          const float al = cnh[p], be = cnh[q];
          const bool live = al > 0.f && be > 0.f && gh != 0.f;
          const float r2 = live ? (gh / al) * (gh / be) : 0.f;  // correlation squared
          if (gl == 0 && r2 > big2) large = 1;
          if (r2 > tol2) {
            const float d = (be - al) + (cnl[q] - cnl[p]);
            float ch, cl, sh, sl;
            if (fabsf(gh) < 0.00048828125f * fabsf(d)) {  // |t| < 2^-11
              const float u = gh / d;                       // 1 / (2 zeta)
              const float t = fmaf(-u * u, u, u);           // tan(theta) = u - u^3 + ...
              const float t2 = t * t;
              ch = 1.f;
              cl = t2 * fmaf(t2, 0.375f, -0.5f);            // cos - 1 = -t^2/2 + 3t^4/8
              sh = t;
              sl = t * cl;                                  // sin = t cos
            } else {  // |zeta| <= 2^10 here: zeta^2 stays in float range
              float zh, zl, th, tl, uh, ul;
              df::sub(be, cnl[q], al, cnl[p], uh, ul);             // |a_q|^2 - |a_p|^2
              df::div_df(uh, ul, 2.f * gh, 2.f * glo, zh, zl);     // zeta
              df::mul(zh, zl, zh, zl, th, tl);
              df::add_to(th, tl, 1.f, 0.f);
              df::sqrt_df(th, tl, uh, ul);                         // sqrt(1 + zeta^2)
              df::add_to(uh, ul, fabsf(zh), zh < 0.f ? -zl : zl);
              df::div_df(zh >= 0.f ? 1.f : -1.f, 0.f, uh, ul, th, tl);  // t = tan(theta)
              df::mul(th, tl, th, tl, uh, ul);
              df::add_to(uh, ul, 1.f, 0.f);
              float rh, rl;
              df::sqrt_df(uh, ul, rh, rl);
              df::div_df(1.f, 0.f, rh, rl, ch, cl);               // cos = 1 / sqrt(1 + t^2)
              df::mul(ch, cl, th, tl, sh, sl);                     // sin = t cos
            }
#pragma unroll
            for (int e0 = 0; e0 < NE; e0 += 4) {
              float xh[4], xl[4], yh[4], yl[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const int o = 8 * (e0 + e);
                xh[e] = aph[o]; xl[e] = apl[o]; yh[e] = aqh[o]; yl[e] = aql[o];
              }
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const int o = 8 * (e0 + e);
                rot_df(ch, cl, sh, sl, xh[e], xl[e], yh[e], yl[e]);
                aph[o] = xh[e]; apl[o] = xl[e]; aqh[o] = yh[e]; aql[o] = yl[e];
              }
            }
            __syncwarp(0xffu << (8 * (lane >> 3)));  // the group's reads of the norms first
            if (gl == 0) {
              // norms after the rotation: c^2 al - 2cs ga + s^2 be, s^2 al + 2cs ga + c^2 be
              float c2h, c2l, s2h, s2l, csh, csl, th, tl;
              df::mul(ch, cl, ch, cl, c2h, c2l);
              df::mul(sh, sl, sh, sl, s2h, s2l);
              df::mul(ch, cl, sh, sl, csh, csl);
              csh *= 2.f;
              csl *= 2.f;
              const float alh = cnh[p], all = cnl[p], beh = cnh[q], bel = cnl[q];
              float ph = 0.f, pl = 0.f, qh = 0.f, ql = 0.f;
              df::mul(c2h, c2l, alh, all, ph, pl);
              df::mul(csh, csl, gh, glo, th, tl);
              df::add_to(ph, pl, -th, -tl);
              df::mul(s2h, s2l, beh, bel, th, tl);
              df::add_to(ph, pl, th, tl);
              df::mul(s2h, s2l, alh, all, qh, ql);
              df::mul(csh, csl, gh, glo, th, tl);
              df::add_to(qh, ql, th, tl);
              df::mul(c2h, c2l, beh, bel, th, tl);
              df::add_to(qh, ql, th, tl);
              cnh[p] = ph; cnl[p] = pl;
              cnh[q] = qh; cnl[q] = ql;
              rotated = 1;
            }
          }
        }
        __syncthreads();
      }
      const int any = rotated && large;
      __syncthreads();
      if (!any) break;
    }
  }
  // ---------------------------------------------------------------- F
  for (int j = warp; j < c; j += nwarps) {
    float sh = 0.f, sl = 0.f;
    for (int i = lane; i < c; i += 32) df::dot_acc(Qh[j * LD + i], Ql[j * LD + i], Qh[j * LD + i], Ql[j * LD + i], sh, sl);
    df::warp_sum(sh, sl);
    if (lane == 0) {
      const double s = df::join(sh, sl);
      sv[j] = isfinite(s) ? sqrt(s) : -1.0;
    }
  }
  __syncthreads();
  for (int j = tid; j < c; j += nthr) {
    int rk = 0;
    for (int i = 0; i < c; ++i) rk += (sv[i] > sv[j]) || (sv[i] == sv[j] && i < j);
    order[rk] = j;
  }
  __syncthreads();
  for (int j = warp; j < c; j += nwarps) {
    const float* xh = Qh + order[j] * LD;
    const float* xl = Ql + order[j] * LD;
    double best = -1.0, bv = 0.0;
    int bi = c;
    for (int i = lane; i < c; i += 32) {
      const double x = df::join(xh[i], xl[i]);
      const double a = fabs(x);
      const int row = perm[i];
      if (a > best || (a == best && row < bi)) { best = a; bi = row; bv = x; }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
      if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; bv = ov; }
    }
    if (lane == 0) {
      sgn[j] = (bv < 0.0) ? -1 : 1;
      hb[j] = (sv[order[j]] > 0.0) ? 1.0 / sv[order[j]] : 0.0;
    }
  }
  __syncthreads();
  for (int idx = tid; idx < cc; idx += nthr) {
    const int i = idx % c, col = idx / c;
    const int j = order[col];
    const double u = df::join(Qh[j * LD + i], Ql[j * LD + i]) * hb[col];
    Wn[perm[i] + col * c] = sgn[col] < 0 ? -u : u;
  }
  for (int j = tid; j < c; j += nthr)
    sig[j] = sv[order[j]] > 0.0 ? ldexp(sv[order[j]], ex) : 0.0;
}


constexpr int TQ_THREADS = 512;  // threads of the double-float TSQR kernels
constexpr int TQ_G = TQ_THREADS / 8;  // 8-lane groups: group p holds columns p, p + TQ_G
constexpr int TQ_Q = kTsqrRows / 8;   // a lane's rows of a column: 8 q + lane

// The trailing columns' update of step j of a double-float Householder QR held in
// registers: column k = grp + TQ_G s of the block has row 8 q + gl in (mh, ml)[s][q] of
// lane gl of group grp.  v (smem): the reflector, zero outside its rows, which lie in
// the eight-row slices qa .. qb (taken four slices at a time: a branch per slice kept the
// loads from overlapping).  d[s] = v^T column s over the group, in two chains (even and
// odd slices) for latency.
//
// The lane of a row is fixed (row mod 8) where the shared-memory form gave it to
// lane (row - j) mod 8: lanes are only rotated by j, which neither the lanes' sums (a
// lane's rows are the same set in the same order; the two chains trade places) nor the
// group sum (xor 4, 2, 1 pairs classes mod 8, 4, 2) sees, so the results are the same
// bit for bit.
template <int NC>
__device__ __forceinline__ void hh_dots(const float2* v, int qa, int qb, int gl,
                                        const float (&mh)[NC][TQ_Q], const float (&ml)[NC][TQ_Q],
                                        float (&dh)[NC], float (&dl)[NC]) {
  float eh[NC], el[NC];
#pragma unroll
  for (int s = 0; s < NC; ++s) dh[s] = dl[s] = eh[s] = el[s] = 0.f;
#pragma unroll
  for (int q0 = 0; q0 < TQ_Q; q0 += 4) {
    if (q0 + 3 < qa || q0 > qb) continue;  // uniform over the block
    float2 x[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) x[q] = v[8 * (q0 + q) + gl];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int s = 0; s < NC; ++s) {
        if (q & 1) df::dot_acc(x[q].x, x[q].y, mh[s][q0 + q], ml[s][q0 + q], eh[s], el[s]);
        else df::dot_acc(x[q].x, x[q].y, mh[s][q0 + q], ml[s][q0 + q], dh[s], dl[s]);
      }
  }
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    df::add_to(dh[s], dl[s], eh[s], el[s]);
    df::group8_sum(dh[s], dl[s]);
  }
}
template <int NC>
__device__ __forceinline__ void hh_axpy(const float2* v, int qa, int qb, int gl,
                                        float (&mh)[NC][TQ_Q], float (&ml)[NC][TQ_Q],
                                        const bool (&on)[NC], const float (&fh)[NC],
                                        const float (&fl)[NC]) {
#pragma unroll
  for (int q0 = 0; q0 < TQ_Q; q0 += 4) {
    if (q0 + 3 < qa || q0 > qb) continue;
    float2 x[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) x[q] = v[8 * (q0 + q) + gl];
#pragma unroll
    for (int s = 0; s < NC; ++s)
      if (on[s])
#pragma unroll
        for (int q = 0; q < 4; ++q)
          df::axpy_neg(fh[s], fl[s], x[q].x, x[q].y, mh[s][q0 + q], ml[s][q0 + q]);
  }
}

// |x|^2 of v[first .. last] (at most 128 entries), one warp: each lane's entries of
// every 32-row piece summed over the warp, the pieces in order
__device__ __forceinline__ void hh_norm2(const float2* v, int first, int last, int lane, float& th,
                                         float& tl) {
  float sh[TQ_Q / 4], sl[TQ_Q / 4];
#pragma unroll
  for (int w = 0; w < TQ_Q / 4; ++w) {
    sh[w] = sl[w] = 0.f;
    const int i = first + 32 * w + lane;
    if (i <= last) df::dot_acc(v[i].x, v[i].y, v[i].x, v[i].y, sh[w], sl[w]);
  }
  // (an empty piece's sum is zero, and adding zero renormalizes th, tl once: below)
  if (last - first < 32) {
    df::warp_sum(sh[0], sl[0]);
    th = sh[0];
    tl = sl[0];
  } else if (last - first < 64) {
#pragma unroll
    for (int w = 0; w < 2; ++w) df::warp_sum(sh[w], sl[w]);
    th = sh[0];
    tl = sl[0];
    df::add_to(th, tl, sh[1], sl[1]);
  } else {
#pragma unroll
    for (int w = 0; w < TQ_Q / 4; ++w) df::warp_sum(sh[w], sl[w]);
    th = sh[0];
    tl = sl[0];
#pragma unroll
    for (int w = 1; w < TQ_Q / 4; ++w) df::add_to(th, tl, sh[w], sl[w]);
  }
  df::add_to(th, tl, 0.f, 0.f);
}

// Householder QR of one row block of a panel (the first TSQR round, <= 128 rows,
// FP64 data) in double-float: the steps of k_tsqr with every operation (the
// norms, the reflector's scalars, the dot products and updates of the trailing
// columns) carried by float pairs on the FP32 pipe.  v^T v is formed as
// 2 nrm (nrm + |x0|), the cancellation-free form of |x|^2 - x0^2 + v0^2.
// Writes the c x c R (row-major, upper triangle) in FP64.
//
// The block is held in registers (an 8-lane group per column, NC columns a group); only
// the reflector passes through shared memory, written with its norm and scalars by the
// warp that owns the column, so a step has one barrier (the reflector is double-
// buffered) and its updates no shared-memory stores.  Bound by the step's chain (norm,
// square root, division: ~1300 cycles) and by the updates' FP32 instructions.  N = 16384,
// 60 columns: 181 -> 139 us; N = 20001, 120 columns: 672 -> 567 us (before: six barriers a
// step and the block in shared memory).
template <int NC>
__global__ __launch_bounds__(TQ_THREADS) void k_tsqr_df(const TsqrTask* __restrict__ tasks,
                                                 const double* __restrict__ P, int64_t ldp,
                                                 int c, double* __restrict__ R,
                                                 const NodeJob* __restrict__ jobs) {
  const TsqrTask* tkp = tasks + blockIdx.x;
  if (jobs) {  // a level-wide launch over several operators' nodes
    const NodeJob& jb = jobs[blockIdx.x];
    tkp = jb.task;
    P = jb.P;
    ldp = jb.ldp;
    c = jb.c;
    R = jb.R;
  }
  __shared__ float2 vbuf[2][kTsqrRows];
  __shared__ float4 scal[2];  // beta, alpha
  const int64_t r0 = tkp->r0[0];
  const int m = (int)(tkp->r1[0] - r0);
  const int tid = threadIdx.x, lane = tid & 31, gl = tid & 7, grp = tid >> 3;
  float mh[NC][TQ_Q], ml[NC][TQ_Q];
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    const int k = grp + TQ_G * s;
#pragma unroll
    for (int q = 0; q < TQ_Q; ++q) {
      const int i = 8 * q + gl;
      df::split((k < c && i < m) ? P[r0 + i + (int64_t)k * ldp] : 0.0, mh[s][q], ml[s][q]);
    }
  }
  const int steps = m < c ? m : c;
  const int qb = (m - 1) >> 3;
  for (int j = 0; j < steps; ++j) {
    float2* v = vbuf[j & 1];
    const int og = j % TQ_G, os = j / TQ_G;
    if ((tid >> 5) == (og >> 2)) {  // the warp that holds column j
      if (grp == og) {
#pragma unroll
        for (int s = 0; s < NC; ++s)
          if (s == os)
#pragma unroll
            for (int q = 0; q < TQ_Q; ++q) {
              const bool in = 8 * q + gl >= j;
              v[8 * q + gl] = make_float2(in ? mh[s][q] : 0.f, in ? ml[s][q] : 0.f);
            }
      }
      __syncwarp();
      float th, tl;
      hh_norm2(v, j, m - 1, lane, th, tl);
      const float xh = v[j].x, xl = v[j].y;
      float nh, nl;
      df::sqrt_df(th, tl, nh, nl);
      const float ah = (xh > 0.f) ? -nh : nh, al = (xh > 0.f) ? -nl : nl;
      float vh, vl, wh = nh, wl = nl, qh, ql, bh = 0.f, bl = 0.f;
      df::sub(xh, xl, ah, al, vh, vl);                                 // v0 = x0 - alpha
      df::add_to(wh, wl, fabsf(xh), xh < 0.f ? -xl : xl);               // nrm + |x0|
      df::mul(nh, nl, wh, wl, qh, ql);                                  // v^T v / 2
      if (qh > 0.f) df::div_df(1.f, 0.f, qh, ql, bh, bl);               // beta = 2 / v^T v
      __syncwarp();
      if (lane == 0) {
        v[j] = make_float2(vh, vl);
        scal[j & 1] = make_float4(bh, bl, ah, al);
      }
    }
    __syncthreads();
    const float4 sc = scal[j & 1];
    bool on[NC], any = false;
#pragma unroll
    for (int s = 0; s < NC; ++s) {
      const int k = grp + TQ_G * s;
      on[s] = k > j && k < c;
      any |= on[s];
    }
    if (sc.x != 0.f && __any_sync(0xffffffffu, any)) {
      float dh[NC], dl[NC], fh[NC], fl[NC];
      hh_dots<NC>(v, j >> 3, qb, gl, mh, ml, dh, dl);
#pragma unroll
      for (int s = 0; s < NC; ++s) {
        df::fast_two_sum(dh[s], dl[s], dh[s], dl[s]);
        df::mul(sc.x, sc.y, dh[s], dl[s], fh[s], fl[s]);
      }
      hh_axpy<NC>(v, j >> 3, qb, gl, mh, ml, on, fh, fl);
    }
    if (grp == og) {  // R(j, j) = alpha
#pragma unroll
      for (int s = 0; s < NC; ++s)
        if (s == os)
#pragma unroll
          for (int q = 0; q < TQ_Q; ++q)
            if (8 * q + gl == j) { mh[s][q] = sc.z; ml[s][q] = sc.w; }
    }
  }
  double* Ro = R + (int64_t)tkp->out_slot * c * c;
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    const int k = grp + TQ_G * s;
#pragma unroll
    for (int q = 0; q < TQ_Q; ++q) {
      const int i = 8 * q + gl;
      if (k < c && i < c)
        Ro[i * c + k] = (i <= k && i < steps) ? df::join(mh[s][q], ml[s][q]) : 0.0;
    }
  }
}

// The merge of two c x c triangles R = qr([R1; R2]) of k_tsqr_merge (packed
// triangles, the j-th reflector touching row j of R1 and rows 0..j of R2) in
// double-float; FP64 in and out.  R2 is held in registers as in k_tsqr_df, R1 (one row
// a step) in shared memory, packed.  120 columns: 433 -> 293 us a round; 60 columns: 148
// -> 100.
template <int NC>
__global__ __launch_bounds__(TQ_THREADS) void k_tsqr_merge_df(const TsqrTask* __restrict__ tasks,
                                                              int c, double* __restrict__ R,
                                                              const NodeJob* __restrict__ jobs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const TsqrTask* tkp = tasks + blockIdx.x;
  if (jobs) {  // a level-wide launch over several operators' nodes
    const NodeJob& jb = jobs[blockIdx.x];
    tkp = jb.task;
    c = jb.c;
    R = jb.R;
  }
  float2* A = reinterpret_cast<float2*>(smem_raw);  // R1, packed upper: column k at k(k+1)/2
  __shared__ float2 vbuf[2][kTsqrRows];
  __shared__ float4 scal[2], vtop[2];  // beta, alpha; v0 (the reflector's entry in R1)
  const int tid = threadIdx.x, lane = tid & 31, gl = tid & 7, grp = tid >> 3;
  const double* R1 = R + (int64_t)tkp->slot[0] * c * c;
  const double* R2 = R + (int64_t)tkp->slot[1] * c * c;
  for (int idx = tid; idx < c * c; idx += TQ_THREADS) {
    const int rr = idx / c, col = idx % c;
    if (rr <= col) {
      float2 x;
      df::split(R1[idx], x.x, x.y);
      A[col * (col + 1) / 2 + rr] = x;
    }
  }
  float mh[NC][TQ_Q], ml[NC][TQ_Q];
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    const int k = grp + TQ_G * s;
#pragma unroll
    for (int q = 0; q < TQ_Q; ++q) {
      const int i = 8 * q + gl;
      df::split((k < c && i <= k) ? R2[i * c + k] : 0.0, mh[s][q], ml[s][q]);
    }
  }
  __syncthreads();
  for (int j = 0; j < c; ++j) {
    float2* v = vbuf[j & 1];
    const int og = j % TQ_G, os = j / TQ_G;
    if ((tid >> 5) == (og >> 2)) {  // the warp that holds column j of R2
      if (grp == og) {
#pragma unroll
        for (int s = 0; s < NC; ++s)
          if (s == os)
#pragma unroll
            for (int q = 0; q < TQ_Q; ++q) {
              const bool in = 8 * q + gl <= j;
              v[8 * q + gl] = make_float2(in ? mh[s][q] : 0.f, in ? ml[s][q] : 0.f);
            }
      }
      __syncwarp();
      float th, tl;
      hh_norm2(v, 0, j, lane, th, tl);
      const float2 x0 = A[j * (j + 1) / 2 + j];
      const float xh = x0.x, xl = x0.y;
      float sh2, sl2, nh, nl;
      df::mul(xh, xl, xh, xl, sh2, sl2);
      df::add_to(sh2, sl2, th, tl);                                     // x0^2 + tail
      df::sqrt_df(sh2, sl2, nh, nl);
      const float ah = (xh > 0.f) ? -nh : nh, al = (xh > 0.f) ? -nl : nl;
      float vh, vl, wh = nh, wl = nl, qh, ql, bh = 0.f, bl = 0.f;
      df::sub(xh, xl, ah, al, vh, vl);                                 // v0 = x0 - alpha
      df::add_to(wh, wl, fabsf(xh), xh < 0.f ? -xl : xl);               // nrm + |x0|
      df::mul(nh, nl, wh, wl, qh, ql);                                  // v^T v / 2
      if (qh > 0.f) df::div_df(1.f, 0.f, qh, ql, bh, bl);               // beta = 2 / v^T v
      __syncwarp();
      if (lane == 0) {
        scal[j & 1] = make_float4(bh, bl, ah, al);
        vtop[j & 1] = make_float4(vh, vl, 0.f, 0.f);
        if (bh != 0.f) A[j * (j + 1) / 2 + j] = make_float2(ah, al);
      }
    }
    __syncthreads();
    const float4 sc = scal[j & 1], v0 = vtop[j & 1];
    bool on[NC], any = false;
#pragma unroll
    for (int s = 0; s < NC; ++s) {
      const int k = grp + TQ_G * s;
      on[s] = k > j && k < c;
      any |= on[s];
    }
    if (sc.x != 0.f && __any_sync(0xffffffffu, any)) {
      float dh[NC], dl[NC], fh[NC], fl[NC];
      hh_dots<NC>(v, 0, j >> 3, gl, mh, ml, dh, dl);
#pragma unroll
      for (int s = 0; s < NC; ++s) {
        const int k = grp + TQ_G * s;
        float2* a = A + k * (k + 1) / 2 + j;
        const float2 x = on[s] ? *a : make_float2(0.f, 0.f);
        // f = beta (dot + v0 A(j, k))
        df::dot_acc(v0.x, v0.y, x.x, x.y, dh[s], dl[s]);
        df::fast_two_sum(dh[s], dl[s], dh[s], dl[s]);
        df::mul(sc.x, sc.y, dh[s], dl[s], fh[s], fl[s]);
        __syncwarp();
        if (on[s] && gl == 0) {
          float2 y = x;
          df::axpy_neg(fh[s], fl[s], v0.x, v0.y, y.x, y.y);
          *a = y;
        }
      }
      hh_axpy<NC>(v, 0, j >> 3, gl, mh, ml, on, fh, fl);
    }
  }
  __syncthreads();
  double* Ro = R + (int64_t)tkp->out_slot * c * c;
  for (int idx = tid; idx < c * c; idx += TQ_THREADS) {
    const int rr = idx / c, col = idx % c;
    const float2 x = (rr <= col) ? A[col * (col + 1) / 2 + rr] : make_float2(0.f, 0.f);
    Ro[idx] = (rr <= col) ? df::join(x.x, x.y) : 0.0;
  }
}
}  // namespace

template <int NB>
static void jacobi_df_run(const int32_t* node_slot, int nblocks, const double* R, int c, double* W,
                          double* sigma, const NodeJob* jobs, cudaStream_t st) {
  const size_t smem = (size_t)3 * c * (32 * NB + 8) * sizeof(float);
  static std::atomic<uint32_t> done{0};
  raise_smem_limit((const void*)k_jacobi_df<NB>, done);
  k_jacobi_df<NB><<<nblocks, 512, smem, st>>>(node_slot, R, c, W, sigma, jobs);
}
// rows padded to the next multiple of 32
static void jacobi_df_launch(const int32_t* node_slot, int nblocks, const double* R, int c,
                             double* W, double* sigma, const NodeJob* jobs, cudaStream_t st) {
  count_launches(1);
  if (c <= 32) jacobi_df_run<1>(node_slot, nblocks, R, c, W, sigma, jobs, st);
  else if (c <= 64) jacobi_df_run<2>(node_slot, nblocks, R, c, W, sigma, jobs, st);
  else if (c <= 96) jacobi_df_run<3>(node_slot, nblocks, R, c, W, sigma, jobs, st);
  else jacobi_df_run<4>(node_slot, nblocks, R, c, W, sigma, jobs, st);
}

void launch_jacobi_df(const int32_t* node_slot, int nnodes, const double* R, int c, double* W,
                      double* sigma, cudaStream_t st) {
  jacobi_df_launch(node_slot, nnodes, R, c, W, sigma, nullptr, st);
}

void launch_jacobi_df_jobs(const NodeJob* jobs, int njobs, int cmax, cudaStream_t st) {
  if (njobs <= 0) return;
  jacobi_df_launch(nullptr, njobs, nullptr, cmax, nullptr, nullptr, jobs, st);
}

// One column a group up to 64 columns (two blocks an SM), two above.
static void tsqr_df_launch(const TsqrTask* tasks, int ntasks, int merge, const double* P,
                           int64_t ldp, int c, int cmax, double* R, const NodeJob* jobs,
                           cudaStream_t st) {
  count_launches(1);
  if (!merge) {
    if (cmax <= TQ_G) k_tsqr_df<1><<<ntasks, TQ_THREADS, 0, st>>>(tasks, P, ldp, c, R, jobs);
    else k_tsqr_df<2><<<ntasks, TQ_THREADS, 0, st>>>(tasks, P, ldp, c, R, jobs);
    return;
  }
  const size_t smem = (size_t)cmax * (cmax + 1) / 2 * sizeof(float2);
  static std::atomic<uint32_t> d1{0}, d2{0};
  if (cmax <= TQ_G) {
    raise_smem_limit((const void*)k_tsqr_merge_df<1>, d1);
    k_tsqr_merge_df<1><<<ntasks, TQ_THREADS, smem, st>>>(tasks, c, R, jobs);
  } else {
    raise_smem_limit((const void*)k_tsqr_merge_df<2>, d2);
    k_tsqr_merge_df<2><<<ntasks, TQ_THREADS, smem, st>>>(tasks, c, R, jobs);
  }
}

void launch_tsqr_df(const TsqrTask* tasks, int ntasks, int merge, const double* P, int64_t ldp,
                    int c, double* R, cudaStream_t st) {
  tsqr_df_launch(tasks, ntasks, merge, P, ldp, c, c, R, nullptr, st);
}

void launch_tsqr_df_jobs(const NodeJob* jobs, int njobs, int merge, int cmax, cudaStream_t st) {
  if (njobs <= 0) return;
  tsqr_df_launch(nullptr, njobs, merge, nullptr, 0, cmax, cmax, nullptr, jobs, st);
}

}  // namespace hm
