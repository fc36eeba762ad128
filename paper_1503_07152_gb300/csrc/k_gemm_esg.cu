// Sampling GEMM of the FP32 dense operator with FP64 samples (HM_A32) on the
// 5th-generation tensor cores: Y = op(A) X, A FP32, X and Y FP64, to about
// 2^-32 of (max slice)^2 relative per product term (the FP64 black-box products
// A Omega / A^* Omega of the compression figures, without FP64 arithmetic in
// the contraction).
//
// Exact-accumulation split: every row of op(A) and every column of X inside a
// window of 256 K values (the A exponents are recorded once per operator) is
// scaled by a power of two so that its largest entry lies in [64, 128), and cut
// into four 8-bit integer slices
// (a = sum_s a_s 2^(-8(s-1)) up to the scale, |a_s| <= 128, each exact in BF16).
// A BF16 x BF16 product of slices is an integer of magnitude <= 2^14, and the
// products of one order d = s + t (d = 2..5, at most four of them) summed over
// a window of 256 K values stay within 2^24, so the FP32 accumulators in TMEM
// hold them EXACTLY whatever the tensor cores' rounding.  Orders above 5 are
// not formed.  Per window and output element the drain adds
//     2^(e_A + e_X - 14) (L + 2^-8 M + 2^-16 C + 2^-24 D)
// (L, M, C, D: the exact sums of orders 2..5) into an FP32 double-float
// (hi, lo), every term through an error-free TwoSum.  Y = hi + lo in FP64.
//
// MMA form: a stage holds the four A slices and the X slices stacked as five
// 64-row blocks [0 x1 x2 x3 x4] (the zero block written once).  A pair of
// neighbouring blocks times an A slice s is an N = 128 product that lands in two
// neighbouring orders: x1 x2 and x3 x4 for slice 1, 0 x1 and x2 x3 for slice 2,
// x1 x2 for slice 3, 0 x1 for slice 4 give the ten products of orders 2..5 in six
// MMAs per 16 K values (twelve per tile), all of one shape and in two accumulator
// halves, so that they are ordered by the tensor pipe without waits.
//
// What bounds it and what was measured (dense A^T X, N = 32768, 60 columns, every
// tile active, the pre-cut of X included): 2.40 -> 1.64 ms; per 32-wide tile and
// block 2430 -> ~1600 cycles, of which the twelve MMAs take 768, the FP32 pipe ~640
// (cuts and drain) and shared memory ~1400 (operands read by the MMAs, slices
// written, raw tile and X copied in).  A clock of every role showed where the rest
// went: the tile search in each role (TileIter now), 256 arrivals a barrier (one per
// warp now), one X-copying thread that searched three tiles ahead, and one cutter
// group whose cycle (two waits, loads, cuts, the proxy fence: ~2000 cycles, mostly
// latency) the MMAs waited for (three groups now, one per stage).  Eight N = 256
// products a tile over three zero blocks (the earlier form) cost 1024 cycles of MMAs
// and 8 KB more a stage; a fourth raw buffer measured the same as three.
//
// Block: 128 rows of op(A) x 64 columns of X, 32 warps:
//   warp 0: allocates 512 TMEM columns (two windows x four orders x 64 columns);
//     one elected lane issues the MMAs;
//   warp 1 (one lane): TMA loads of the FP32 tiles of A (128 x 32), one raw buffer
//     per cutter group;
//   warp 2 (one lane): bulk copies of the pre-cut X slices;
//   warps 4-15, three groups: move a raw tile to registers (releasing its buffer),
//     scale, and cut the slices into the group's operand stage (K-major, 64-byte
//     swizzle).  An entry that does not fit its recorded row scale (the operator
//     changed after the scales were taken) aborts the block, whose outputs are
//     then NaN;
//   warps 16-31: drain once per window (four warps per TMEM lane quarter, 16
//     columns each) and write Y.
// Every waiter on an mbarrier here waits for each of its phases in turn: a parity
// says nothing about a phase further away.
// All-zero K tiles of X are skipped; the four X slices of an active tile are
// always loaded (a zero slice contributes zeros).  Every mbarrier wait is bounded
// (the pipeline waits by the limit the host sets, hm_set_wait_limit); on timeout
// the block raises the error flag, writes NaN, lets its own TMA copies land and
// its issued MMAs complete (waits of the full limit) and leaves; TMEM is
// released unless even the full-limit wait for its MMAs ran out.
#include <algorithm>
#include <cstring>
#include <atomic>

#include "tc_util.cuh"

namespace hm {
namespace {

using namespace tc;

constexpr int TM = 128, TN = 64, TK = 32;  // TK: the K extent of a stage
constexpr int NSL = 4;                  // slices of A and of X
constexpr int A_SLICE = TM * TK * 2;    // 8 KB: 128 rows x 64 bytes
constexpr int XB = TN * TK * 2;         // 4 KB: one X slice, 64 rows x 64 bytes
constexpr int XZ = 1;                   // zero blocks before x1
constexpr int X_BYTES = (XZ + NSL) * XB;                 // 20 KB
constexpr int STAGE_BYTES = NSL * A_SLICE + X_BYTES;     // 52 KB
constexpr int SSTAGES = 3;
constexpr int RAW_BYTES = TM * TK * 4;  // 16 KB
constexpr int RSTAGES = SSTAGES;  // one raw tile per cutter group
constexpr int RAW_REGION = RSTAGES * RAW_BYTES;          // 48 KB
constexpr int LAYOUT_BYTES = RAW_REGION + SSTAGES * STAGE_BYTES;  // 204 KB
// Warps: 0 MMA, 1 TMA of A, 2 copies of X, 3 idle; then three groups of four
// cutter warps (group g cuts the tiles of stage g), then sixteen drain warps.
constexpr int GT = 128, NG = SSTAGES;    // threads of a group, groups
constexpr int NDRAIN = 512, NTHREADS = 128 + NG * GT + NDRAIN;
constexpr int W_MMA = 0, W_TMA = 1, W_XTMA = 2, W_CUT0 = 4, W_DRAIN0 = W_CUT0 + NG * GT / 32;
constexpr int DC = TN * TM / NDRAIN;     // columns of a drain thread: 16
static_assert(NTHREADS <= 1024, "one block");
constexpr uint32_t TMEM_COLS = 512;  // 2 buffers x 4 orders x 64 columns
constexpr int WIN_ROWS = 256;        // K values per exact accumulation window
constexpr int WIN_TILES = WIN_ROWS / TK;
constexpr int KPAD = 64;             // K padding of the pre-cut X (k_split_x64's rows)
constexpr int MAX_KT = 16384;        // K tiles a call may have (n <= 524288)

static_assert(STAGE_BYTES % 1024 == 0 && RAW_BYTES % 1024 == 0, "1 KB aligned stages");

// Shared-memory matrix descriptor: K-major, 64-byte swizzle (16-byte chunk c of
// row r at chunk c ^ ((r >> 1) & 3)), 8-row groups 512 bytes apart; start
// address and offsets in 16-byte units.
__device__ __forceinline__ uint64_t sw64_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)1 << 16;            // leading byte offset (unused for this layout)
  d |= (uint64_t)(512 >> 4) << 32;   // stride byte offset between 8-row groups
  d |= (uint64_t)1 << 46;            // descriptor version
  d |= (uint64_t)4 << 61;            // 64-byte swizzle
  return d;
}
// byte offset of 16-byte chunk q (0..3) of row m in a 64-byte-swizzled K-major tile
__device__ __forceinline__ uint32_t sw64_off(int m, int q) {
  return (uint32_t)((m >> 3) * 512 + (m & 7) * 64 + ((q ^ ((m >> 1) & 3)) << 4));
}

__device__ __forceinline__ float pow2f(int k) {  // 2^k for k in [-126, 127]
  return __int_as_float((k + 127) << 23);
}

// exponent e with |x| < 2^e for x = the largest magnitude (0 for x == 0)
__device__ __forceinline__ int exp_above(float x) {
  if (!(x > 0.f)) return 0;
  int e;
  frexpf(x, &e);
  return e;
}

// Two FP32 values as one operand of the packed FP32 instructions: one issue slot
// for two lanes' worth of adds, at the scalar instructions' FP32 rate.  The
// cutter and drain warps share four schedulers with the MMA-issuing warp, so
// the issue slots are what they save (both results round as the scalar forms).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float x, float y) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// a - b as b * (-1) + a: one rounding, the same one, in one instruction (the
// packed add takes no negated operand: negating by xor costs two more)
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(b), "l"(0xbf800000bf800000ull), "l"(a));
  return r;
}
// the largest magnitude of three, NaN if one is (the range check of the cutters)
__device__ __forceinline__ float max_abs(float a, float b, float c) {
  float r;
  asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Cut v (|v| < 128) into four digits, digit t a multiple of 2^(-8 (t - 1)) with at
// most eight significant bits: v rounded to a multiple of 2^-24.  Each digit is
// rounded (ties to even) by adding 1.5 * 2^(23 - 8 (t - 1)), which lands where
// the FP32 spacing is the digit's unit, and taking the constant off again
// (exact); two adds on the FMA pipe instead of an instruction of the slower
// conversion pipe.  The digits keep their scale 2^(-8 (t - 1)): the X slices carry
// theirs too, so every product of order d = s + t has the weight 2^(-8 (d - 2)) in
// its accumulator and the drain needs no factor per order.  The compiler does not
// reassociate the adds (no fast-math).
__device__ __forceinline__ void cut4(f32x2 v, f32x2& s1, f32x2& s2, f32x2& s3, f32x2& s4) {
  constexpr float C1 = 12582912.f, C2 = 49152.f, C3 = 192.f, C4 = 0.75f;
  const f32x2 c1 = pack2(C1, C1), c2 = pack2(C2, C2), c3 = pack2(C3, C3), c4 = pack2(C4, C4);
  const f32x2 m1 = pack2(-C1, -C1), m2 = pack2(-C2, -C2), m3 = pack2(-C3, -C3),
              m4 = pack2(-C4, -C4);
  s1 = add2(add2(v, c1), m1);
  v = sub2(v, s1);
  s2 = add2(add2(v, c2), m2);
  v = sub2(v, s2);
  s3 = add2(add2(v, c3), m3);
  v = sub2(v, s3);
  s4 = add2(add2(v, c4), m4);
}

// Two digits as a BF16 pair (the first in the low half).  A digit has at most 8
// significant bits, so its FP32 pattern ends in 16 zero bits and its BF16 pattern
// is the FP32 pattern's upper half: one byte permute, no rounding.
__device__ __forceinline__ uint32_t pack_bf16(f32x2 d) {
  return __byte_perm((uint32_t)d, (uint32_t)(d >> 32), 0x7632);
}

// Exponents of A per row and window of 256 columns: e_row[i * nw + w] = e with
// max over the window of |A(i, j)| < 2^e (clamped to >= -120).  One warp per
// row, eight entries per lane and window.
__global__ __launch_bounds__(256) void k_row_exp(const float* __restrict__ A, int64_t lda,
                                                 int64_t n, int nw, int* __restrict__ e_row) {
  const int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= n) return;
  const float* a = A + row * lda;
  for (int w = 0; w < nw; ++w) {
    float mx = 0.f;
    for (int64_t j = (int64_t)w * WIN_ROWS + lane; j < n && j < (int64_t)(w + 1) * WIN_ROWS;
         j += 32)
      mx = fmaxf(mx, fabsf(a[j]));
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) e_row[row * nw + w] = max(exp_above(mx), -120);
  }
}

// The same per column and window of 256 rows (the rows of op(A) = A^T): a block takes one
// window of 256 columns, a thread a column, eight rows in flight.  Bound by HBM (A read
// once); with one block walking all the windows of its columns n = 16384 had 64 blocks on
// 152 SMs: 2909 us, 159 now.
__global__ __launch_bounds__(256) void k_col_exp(const float* __restrict__ A, int64_t lda,
                                                 int64_t n, int nw, int* __restrict__ e_col) {
  const int64_t col = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (col >= n) return;
  const int w = blockIdx.y;
  float mx = 0.f;
  const int64_t i1 = (n < (int64_t)(w + 1) * WIN_ROWS) ? n : (int64_t)(w + 1) * WIN_ROWS;
#pragma unroll 8
  for (int64_t i = (int64_t)w * WIN_ROWS; i < i1; ++i) mx = fmaxf(mx, fabsf(A[i * lda + col]));
  e_col[col * nw + w] = max(exp_above(mx), -120);
}

// X (FP64, column-major n x ncols) -> per (window, column) exponents and four
// BF16 digit slices, laid out as the GEMM's shared memory wants them: per
// (column tile ct, K tile kt) one contiguous 16 KB block of 256 rows
// (row t * 64 + c: slice t of column c) x 32 K values, each row's four 16-byte
// chunks in 64-byte-swizzle order, so one 1-D bulk copy lands a tile in place.
// Flags of (kt, ct) nonzero when that K tile has a nonzero digit.  Block: one
// window (256 rows) x 64 columns; a warp takes two columns, lanes along the rows.
//
// Digit t is v = X 2^(7 - e) rounded (ties to even) to a multiple of 2^(-8 t) after
// the digits before it are taken off, as in cut4.  Formed on the integer pipe from
// v in fixed point (54 fraction bits, what lies below as a sticky bit): the FP64
// form (ldexp, four rint / subtract / scale steps) held the FP64 units for ~1100
// cycles per warp and 32 entries and, with its strided loads, took ~115 us at any
// size up to n = 32768 x 60; this form 13-14 us.
constexpr int SPLIT_THREADS = 1024;
__global__ __launch_bounds__(SPLIT_THREADS) void k_split_x64(
    const double* __restrict__ X, int64_t ldx, int64_t n, int64_t ncols, int64_t kpad, int nct,
    __nv_bfloat16* __restrict__ Xs, int* __restrict__ ex, uint8_t* __restrict__ flags) {
  const int win = blockIdx.x, ct = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ int fl[WIN_TILES];
  if (threadIdx.x < WIN_TILES) fl[threadIdx.x] = 0;
  __syncthreads();
  for (int c = warp; c < TN; c += SPLIT_THREADS / 32) {
    const int64_t col = (int64_t)ct * TN + c;
    long long x[WIN_TILES];  // the bits of rows 32 i + lane of the window
    long long mx = 0;        // the largest finite magnitude's bits
#pragma unroll
    for (int i = 0; i < WIN_TILES; ++i) {
      const int64_t row = (int64_t)win * WIN_ROWS + i * 32 + lane;
      x[i] = (row < n && col < ncols) ? __double_as_longlong(X[row + col * ldx]) : 0ll;
      const long long a = x[i] & 0x7fffffffffffffffll;
      if (a < 0x7ff0000000000000ll) mx = a > mx ? a : mx;
    }
    for (int o = 16; o > 0; o >>= 1) {
      const long long y = __shfl_xor_sync(0xffffffffu, mx, o);
      mx = y > mx ? y : mx;
    }
    int e = 0;  // 2^(e - 1) <= largest magnitude < 2^e
    if (mx > 0) {
      e = (int)(mx >> 52) - 1022;
      if (e == -1022) e = -1010 - __clzll(mx);  // subnormal: the leading bit's place
    }
    if (lane == 0) ex[((int64_t)win * nct + ct) * TN + c] = e;
#pragma unroll
    for (int i = 0; i < WIN_TILES; ++i) {
      const int64_t kt = (int64_t)win * WIN_TILES + i;
      if (kt * TK >= kpad) break;
      const int be = (int)(x[i] >> 52) & 0x7ff;
      unsigned d[4];  // the digits' BF16 patterns (upper half of the FP32 ones)
      if (be == 0x7ff) {
        d[0] = d[1] = d[2] = d[3] = 0x7fc00000u;  // NaN or infinity: NaN products
      } else {
        unsigned long long m = (unsigned long long)x[i] & 0xfffffffffffffull;
        if (be > 0) m |= 1ull << 52;
        // |v| 2^54 = m 2^s with s <= 8
        const int s = (be > 0 ? be : 1) - 1014 - e;
        long long f;
        if (s >= 0) f = (long long)(m << s);
        else if (s > -60) f = (long long)((m >> -s) | ((m << (64 + s)) != 0ull ? 1ull : 0ull));
        else f = m != 0ull ? 1ll : 0ll;
        if (x[i] < 0) f = -f;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int b = 54 - 8 * t;  // the digit's unit is bit b
          const long long q = (f + ((1ll << (b - 1)) - 1) + ((f >> b) & 1ll)) >> b;
          f -= q << b;
          d[t] = __float_as_uint(pow2f(-8 * t) * (float)(int)q);
        }
      }
      const bool any = ((d[0] | d[1] | d[2] | d[3]) << 1) != 0u;
      if (__any_sync(0xffffffffu, any) && lane == 0) fl[i] = 1;
      const int64_t tile = (int64_t)ct * (kpad / TK) + kt;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int rr = t * TN + c;
        const unsigned up = __shfl_down_sync(0xffffffffu, d[t], 1);
        if (!(lane & 1)) {  // rows lane, lane + 1 of the tile
          const int off = (((lane >> 3) ^ ((rr >> 1) & 3)) << 3) + (lane & 7);
          *reinterpret_cast<unsigned*>(Xs + (tile * (NSL * TN) + rr) * TK + off) =
              __byte_perm(d[t], up, 0x7632);
        }
      }
    }
  }
  __syncthreads();
  if (threadIdx.x < WIN_TILES) {
    const int64_t kt = (int64_t)win * WIN_TILES + threadIdx.x;
    if (kt * TK < kpad) flags[kt * nct + ct] = (uint8_t)fl[threadIdx.x];
  }
}

// Named barrier 1 + g of the 128 threads of cutter group g, and its AND-reduction
// form: the generating cutters (GEN) stage their group's table windows in shared
// memory and must leave their loop together.
__device__ __forceinline__ void group_sync(int g) {
  asm volatile("bar.sync %0, 128;" ::"r"(g + 1) : "memory");
}
__device__ __forceinline__ bool group_all(int g, bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, %2, 128, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}\n"
      : "=r"(r)
      : "r"((uint32_t)v), "r"(g + 1)
      : "memory");
  return r != 0;
}
// Walk over a block's active K tiles: the bits of the current word stay in a
// register, so a step is a handful of instructions (a search from shared memory at
// every step took each role 150-450 cycles a tile).
struct TileIter {
  const uint32_t* bits;
  int nwords, end, wd;
  uint32_t b;
  __device__ __forceinline__ int next() {  // the next active tile, `end` past the last
    while (!b) {
      if (++wd >= nwords) { wd = nwords; return end; }
      b = bits[wd];
    }
    const int kt = (wd << 5) + __ffs((int)b) - 1;
    b &= b - 1u;
    return kt;
  }
};

// GEN = 1: the operator is the matrix-free log kernel of the ellipse (see
// launch_gemm_esg_gen): the cutters generate each tile's entries from two
// tables instead of reading a TMA tile of A (no A bytes from HBM); the
// operator is symmetric, so only TRANS = 0 is instantiated.
template <int TRANS, int GEN>
__global__ __launch_bounds__(NTHREADS, 1) void k_gemm_esg(
    const __grid_constant__ CUtensorMap tmA, const __nv_bfloat16* __restrict__ Xs, int64_t n,
    int64_t ncols, const uint8_t* __restrict__ flags, const int* __restrict__ ex,
    const int* __restrict__ e_rows, double* __restrict__ Y, int64_t ldy, int* __restrict__ err,
    long long poll_limit, const float* __restrict__ tabS, const float* __restrict__ tabP) {
  extern __shared__ unsigned char smem_raw[];
  // st_full: one arrival per cutter warp (not per thread) and the X copy's bytes
  __shared__ __align__(8) uint64_t raw_full[RSTAGES], raw_empty[RSTAGES], st_full[SSTAGES],
      st_empty[SSTAGES], acc_full[2], acc_empty[2], bar_final;
  __shared__ uint32_t tmem_base_slot;
  __shared__ volatile int abort_flag;
  __shared__ int win_lo, win_hi;  // this block's share of the windows (split over K)
  __shared__ uint32_t act_bits[MAX_KT / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ct = blockIdx.x, mt = blockIdx.y, nct = gridDim.x;
  const int64_t m0 = (int64_t)mt * TM;
  const int nkt = (int)((n + TK - 1) / TK);
  const int nwin = (nkt + WIN_TILES - 1) / WIN_TILES;
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sbase = smem_raw + (base - raw);
  const uint32_t raw_addr = base, stage_addr0 = base + RAW_REGION;
  // 2^(7 - e), e the exponent of row m of this block in window w (1 past n)
  auto row_scale = [&](int m, int w) -> float {
    return pow2f(7 - ((m0 + m < n) ? e_rows[(m0 + m) * nwin + w] : 0));
  };

  if (tid == 0) {
    abort_flag = 0;
    for (int i = 0; i < RSTAGES; ++i) {
      mbar_init(smem_u32(&raw_full[i]), 1);
      mbar_init(smem_u32(&raw_empty[i]), GT / 32);
    }
    for (int i = 0; i < SSTAGES; ++i) {
      mbar_init(smem_u32(&st_full[i]), GT / 32 + 1);
      mbar_init(smem_u32(&st_empty[i]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&acc_full[b]), 1);
      mbar_init(smem_u32(&acc_empty[b]), NDRAIN / 32);
    }
    mbar_init(smem_u32(&bar_final), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the zero blocks in front of each stage's X slices, written once; the MMAs
  // read them through the async proxy
  for (int i = tid; i < SSTAGES * XZ * XB / 16; i += NTHREADS) {
    const int sidx = i / (XZ * XB / 16), o = i % (XZ * XB / 16);
    *reinterpret_cast<uint4*>(sbase + RAW_REGION + sidx * STAGE_BYTES + NSL * A_SLICE + o * 16) =
        make_uint4(0u, 0u, 0u, 0u);
  }
  fence_proxy_async();
  if (warp == W_TMA) {
    // blocks z = 0 .. gridDim.z - 1 of a row block share its active windows
    // (those with a nonzero K tile of X) in equal counts, in window order
    const int ks = (int)gridDim.z, z = (int)blockIdx.z;
    int lo = 0, hi = nwin;
    if (ks > 1) {
      auto win_active = [&](int w) -> bool {
        bool a = false;
        for (int t = 0; t < WIN_TILES; ++t) {
          const int kt = w * WIN_TILES + t;
          if (kt < nkt && flags[(int64_t)kt * nct + ct]) a = true;
        }
        return a;
      };
      int total = 0;
      for (int w0 = 0; w0 < nwin; w0 += 32) {
        const int w = w0 + lane;
        total += __popc(__ballot_sync(0xffffffffu, w < nwin && win_active(w)));
      }
      const int r0 = (int)((int64_t)z * total / ks), r1 = (int)((int64_t)(z + 1) * total / ks);
      int seen = 0, clo = nwin, chi = nwin;
      for (int w0 = 0; w0 < nwin; w0 += 32) {
        const int w = w0 + lane;
        const bool a = w < nwin && win_active(w);
        const unsigned b = __ballot_sync(0xffffffffu, a);
        const int rank = seen + __popc(b & ((1u << lane) - 1u));
        if (a && rank == r0) clo = w;
        if (a && rank == r1) chi = w;
        seen += __popc(b);
      }
      for (int o = 16; o > 0; o >>= 1) {
        clo = min(clo, __shfl_xor_sync(0xffffffffu, clo, o));
        chi = min(chi, __shfl_xor_sync(0xffffffffu, chi, o));
      }
      lo = clo;
      hi = (r1 >= total) ? nwin : chi;
    }
    if (lane == 0) { win_lo = lo; win_hi = hi; }
  }
  if (warp == W_MMA) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_base_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_slot;
  const int wlo = win_lo, whi = win_hi;
  // one bit per K tile: nonzero X and inside this block's share of the windows
  // (every role walks the tiles; a shared-memory bit instead of a global load
  // per tile and role)
  for (int wd = tid; wd < (nkt + 31) / 32; wd += NTHREADS) {
    uint32_t b = 0;
    for (int i = 0; i < 32; ++i) {
      const int kt = wd * 32 + i, w = kt / WIN_TILES;
      if (kt < nkt && w >= wlo && w < whi && flags[(int64_t)kt * nct + ct]) b |= 1u << i;
    }
    act_bits[wd] = b;
  }
  __syncthreads();
  const int nwords = (nkt + 31) / 32;
  const auto tiles = [&]() { return TileIter{act_bits, nwords, nkt, -1, 0u}; };

  // A cutter warp that gives up still arrives once more on its group's stage: the
  // X copy of the tile it did not cut may be in flight, and the copying thread's
  // wait for it on the way out then ends with the copy
  auto leave_stage = [&](int g) {
    if (lane == 0) mbar_arrive(smem_u32(&st_full[g]));
  };

  if (warp < W_CUT0) {
    if (warp == W_TMA) {
      // -------------------------------------------------------- TMA of A
      if (!GEN && lane == 0) {
        int it = 0;
        const uint64_t pol = l2_policy_evict_first();  // A is read once per call
        TileIter ti = tiles();
        for (int kt = ti.next(); kt < nkt; kt = ti.next()) {
          const int r = it % RSTAGES;
          if (!mbar_wait(smem_u32(&raw_empty[r]), ((it / RSTAGES) & 1) ^ 1, &abort_flag,
                         poll_limit))
            break;
          mbar_arrive_tx(smem_u32(&raw_full[r]), RAW_BYTES);
          if (!TRANS)
            tma_load_2d_hint(raw_addr + r * RAW_BYTES, &tmA, kt * TK, (int)m0,
                             smem_u32(&raw_full[r]), pol);
          else
            tma_load_2d_hint(raw_addr + r * RAW_BYTES, &tmA, (int)m0, kt * TK,
                             smem_u32(&raw_full[r]), pol);
          ++it;
        }
        // the copies in flight land before the block's shared memory is given up
        for (int j = (it > RSTAGES ? it - RSTAGES : 0); j < it; ++j)
          mbar_wait_drain(smem_u32(&raw_full[j % RSTAGES]), (j / RSTAGES) & 1);
      }
    } else if (warp == W_XTMA) {
      // -------------------------------------------------------- bulk copies of the X slices
      // the four pre-cut slices of a K tile are one contiguous 16 KB block of Xs,
      // already in the stage's swizzled order
      if (lane == 0) {
        const int64_t nkt_pad = 2 * ((n + KPAD - 1) / KPAD);  // K tiles of the padded Xs
        int it = 0;
        const uint64_t pol = l2_policy_evict_last();  // every row block re-reads X
        TileIter ti = tiles(), tp = tiles();
        int kp = 0;  // the tile to prefetch, SSTAGES active ones ahead
        for (int i = 0; i <= SSTAGES; ++i) kp = tp.next();
        for (int kt = ti.next(); kt < nkt; kt = ti.next()) {
          const int s = it % SSTAGES;
          if (!mbar_wait(smem_u32(&st_empty[s]), ((it / SSTAGES) & 1) ^ 1, &abort_flag, poll_limit))
            break;
          const uint32_t st = stage_addr0 + (uint32_t)s * STAGE_BYTES;
          mbar_arrive_tx(smem_u32(&st_full[s]), (uint32_t)(NSL * XB));
          const int64_t tile = (int64_t)ct * nkt_pad + kt;
          bulk_load_hint(st + NSL * A_SLICE + XZ * XB, Xs + tile * (NSL * TN * TK),
                         (uint32_t)(NSL * XB), smem_u32(&st_full[s]), pol);
          // the tile SSTAGES active tiles ahead, into L2 while this stage turns over
          if (kp < nkt) {
            bulk_prefetch_l2(Xs + ((int64_t)ct * nkt_pad + kp) * (NSL * TN * TK),
                             (uint32_t)(NSL * XB));
            kp = tp.next();
          }
          ++it;
        }
        for (int j = (it > SSTAGES ? it - SSTAGES : 0); j < it; ++j)
          mbar_wait_drain(smem_u32(&st_full[j % SSTAGES]), (j / SSTAGES) & 1);
      }
    } else if (warp == W_MMA) {
      // -------------------------------------------------------- MMA issue
      // The whole warp walks the tiles and one elected lane issues.  Loop control goes
      // through votes, so that the stage, window and descriptor values are uniform
      // over the warp and can live in uniform registers, which is what the MMA takes
      // its operands from.
      // The look at the next tile's barrier (~250 cycles) comes after the first eight
      // of a tile's MMAs, so that it runs beside them.
      constexpr uint32_t kAll = 0xffffffffu;
      const bool leader = elect_one();
      uint32_t s = 0, ph = 0, ab = 0, aph = 1;  // stage and phase; accumulator buffer and phase
      uint32_t started = 0;
      bool ready = false, fresh = true, ok = true;
      const uint32_t id = idesc_bf16_f32_n(2 * TN);  // M = 128, N = 128
      TileIter ti = tiles();
      int kt = ti.next();
      while (__any_sync(kAll, kt < nkt)) {
        if (fresh) {
          ok = __all_sync(kAll, mbar_wait(smem_u32(&acc_empty[ab]), aph, &abort_flag, poll_limit));
          started = 0;
        }
        if (ok && !ready)
          ok = __all_sync(kAll, mbar_wait(smem_u32(&st_full[s]), ph, &abort_flag, poll_limit));
        if (!ok) break;
        tc_fence_after();
        const uint32_t dbase = tmem + ab * (4 * TN);
        // descriptors of the stage's operands: the address field holds addr / 16
        // (the stage lies below 256 KB, so offsets add without carry)
        const uint64_t d0 = sw64_desc(stage_addr0 + s * STAGE_BYTES);
        const uint32_t sn = s + 1 == SSTAGES ? 0 : s + 1, phn = s + 1 == SSTAGES ? ph ^ 1 : ph;
        // the six products [A slice sl + 1] x [X blocks b, b + 1] of the tile: orders
        // 2, 3 (accumulator half 0) take x1 x2 for slice 1 and 0 x1 for slice 2;
        // orders 4, 5 (half 1) take x3 x4, x2 x3, x1 x2, 0 x1 for slices 1 to 4
        auto product = [&](int sl, int half, int blk, uint32_t accum) {
          const uint64_t ad = d0 + (uint64_t)((sl * A_SLICE) >> 4);
          const uint64_t bd = d0 + (uint64_t)((NSL * A_SLICE + blk * XB) >> 4);
          const uint32_t dt = dbase + (uint32_t)(half * 2 * TN);
          mma_bf16(dt, ad, bd, id, accum);
          mma_bf16(dt, ad + 2, bd + 2, id, 1);  // the second K step is 32 bytes on
        };
        if (leader) {
          product(0, 0, 1, started);
          product(0, 1, 3, started);
          product(1, 0, 0, 1);
          product(1, 1, 2, 1);
        }
        const int ktn = ti.next();
        ready = __all_sync(kAll, ktn < nkt && mbar_test(smem_u32(&st_full[sn]), phn));
        fresh = __any_sync(kAll, ktn >= nkt || ktn / WIN_TILES != kt / WIN_TILES);
        if (leader) {
          product(2, 1, 1, 1);
          product(3, 1, 0, 1);
          mma_commit(smem_u32(&st_empty[s]));
          if (fresh) mma_commit(smem_u32(&acc_full[ab]));  // the window's last tile
        }
        started = 1;
        if (fresh) {
          ab ^= 1;
          aph ^= ab ^ 1;  // the phase turns when buffer 0 comes round again
        }
        kt = ktn;
        s = sn;
        ph = phn;
      }
      // every MMA issued by this warp completes before TMEM is released: this wait
      // ignores the other roles' abort and takes the full limit; only if even that
      // runs out is TMEM left allocated (the error flag reports it)
      if (leader) {
        mma_commit(smem_u32(&bar_final));
        if (!mbar_wait_drain(smem_u32(&bar_final), 0)) abort_flag = 2;
      }
      __syncwarp();
    }
  } else if (warp < W_DRAIN0) {
    if (GEN) {
      // -------------------------------------------------------- generate A and cut
      // A(i, j) = (S[|i - j|] + P[i + j]) in float pairs: fl((Sh + Ph) + (Sl + Pl)),
      // 1 on the diagonal, 0 outside [0, n).  A tile's entries use TM + TK - 1
      // values of each table, staged in the (unused) raw region: window entry e
      // holds S[|d|] for i - j = d = m0 - k0 - (TK - 1) + e, and P[m0 + k0 + e].
      const int g = (warp - W_CUT0) >> 2, t = threadIdx.x - W_CUT0 * 32 - g * GT;
      // Four shifted copies of each window (copy q holds window entry x + q at x),
      // so that every thread reads its four consecutive entries of a table as one
      // aligned float4: for row m the P entries start at m + 4 k4 and the S entries
      // (descending) at m - 4 k4 + TK - 4, both congruent to m mod 4.
      constexpr int WC = 164;  // floats per copy (16-byte multiple, covers index 161)
      static_assert(NG * 16 * WC * 4 <= RAW_REGION, "a group's windows in the raw region");
      float* win = reinterpret_cast<float*>(sbase) + g * (16 * WC);  // [Sh, Sl, Ph, Pl][q][WC]
      // Thread t owns window entries t and t + 128 (< TM + TK - 1).  The group's next
      // tile's entries are loaded from the (L2-resident) tables one tile ahead, so
      // the load latency hides behind the current tile's cut.
      float pv[2][4];
      auto load_win = [&](int ktn) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          pv[i][0] = pv[i][1] = pv[i][2] = pv[i][3] = 0.f;
          const int e = t + i * GT;
          if (e < TM + TK - 1) {
            const int64_t kn = (int64_t)ktn * TK;
            const int64_t d = m0 - kn - (TK - 1) + e, ad = d < 0 ? -d : d, sidx = m0 + kn + e;
            if (ad > 0 && ad < n) { pv[i][0] = tabS[ad]; pv[i][1] = tabS[n + ad]; }
            if (sidx < 2 * n - 1) { pv[i][2] = tabP[sidx]; pv[i][3] = tabP[2 * n - 1 + sidx]; }
          }
        }
      };
      // the group's tiles: every NG-th active one, from the g-th
      TileIter ti = tiles();
      int kt = ti.next();
      for (int i = 0; i < g; ++i) kt = ti.next();
      if (kt < nkt) load_win(kt);
      constexpr int NP = TM * TK / 4 / GT;  // 8 passes: rows 16 p + t / 8
      float scs[NP];                        // this thread's row scales in window scw
      int scw = -1;
      uint32_t ph = 1;
      while (kt < nkt) {
        const bool ok = !abort_flag &&
                        mbar_wait(smem_u32(&st_empty[g]), ph, &abort_flag, poll_limit);
        ph ^= 1;
        // the group leaves together (it shares the table windows); the barrier also
        // orders the previous tile's window reads before the new writes
        if (!group_all(g, ok)) { leave_stage(g); break; }
        const int64_t k0 = (int64_t)kt * TK;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int x = t + i * GT - q;
            if (x >= 0 && x < WC)
#pragma unroll
              for (int a = 0; a < 4; ++a) win[(a * 4 + q) * WC + x] = pv[i][a];
          }
        int ktn = ti.next();
#pragma unroll
        for (int i = 1; i < NG; ++i) ktn = ti.next();
        if (ktn < nkt) load_win(ktn);
        group_sync(g);
        // tiles that hold a diagonal entry or reach past n take the per-entry fixes
        const bool fix = (m0 + TM > n) || (k0 + TK > n) || (m0 < k0 + TK && k0 < m0 + TM);
        const int dk = (int)(fix ? k0 - m0 : 0);  // i == j  <=>  m - (4 k4 + e) == dk
        const int mrow = (int)(n - m0 < TM ? n - m0 : TM), kcol = (int)(n - k0 < TK ? n - k0 : TK);
        unsigned char* sp = sbase + RAW_REGION + g * STAGE_BYTES;
        float mx = 0.f;
        if (kt / WIN_TILES != scw) {
          scw = kt / WIN_TILES;
#pragma unroll
          for (int p = 0; p < NP; ++p) scs[p] = row_scale((p * GT + t) >> 3, scw);
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          const int f = p * GT + t, m = f >> 3, k4 = f & 7;
          const float sc = scs[p];
          const int q = m & 3, ps = m + 4 * k4 - q, ds = m - 4 * k4 + (TK - 4) - q;
          const float4 sh4 = *reinterpret_cast<const float4*>(win + (0 * 4 + q) * WC + ds);
          const float4 sl4 = *reinterpret_cast<const float4*>(win + (1 * 4 + q) * WC + ds);
          const float4 ph4 = *reinterpret_cast<const float4*>(win + (2 * 4 + q) * WC + ps);
          const float4 pl4 = *reinterpret_cast<const float4*>(win + (3 * 4 + q) * WC + ps);
          // entry e: S at window index m - 4 k4 + TK - 1 - e (component 3 - e of the
          // S float4), P at m + 4 k4 + e (component e)
          const float shv[4] = {sh4.w, sh4.z, sh4.y, sh4.x}, slv[4] = {sl4.w, sl4.z, sl4.y, sl4.x};
          const float phv[4] = {ph4.x, ph4.y, ph4.z, ph4.w}, plv[4] = {pl4.x, pl4.y, pl4.z, pl4.w};
          float a[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float v = (shv[e] + phv[e]) + (slv[e] + plv[e]);
            if (fix) {
              const int kk = 4 * k4 + e;
              if (m - kk == dk) v = 1.f;
              if (m >= mrow || kk >= kcol) v = 0.f;
            }
            a[e] = v * sc;
          }
          mx = max_abs(max_abs(mx, a[0], a[1]), a[2], a[3]);
          f32x2 sl[4][2];
#pragma unroll
          for (int e = 0; e < 2; ++e)
            cut4(pack2(a[2 * e], a[2 * e + 1]), sl[0][e], sl[1][e], sl[2][e], sl[3][e]);
          const uint32_t off = sw64_off(m, k4 >> 1) + (uint32_t)((k4 & 1) * 8);
#pragma unroll
          for (int t4 = 0; t4 < NSL; ++t4)
            *reinterpret_cast<uint2*>(sp + t4 * A_SLICE + off) =
                make_uint2(pack_bf16(sl[t4][0]), pack_bf16(sl[t4][1]));
        }
        if (!(mx < 128.f)) abort_flag = 3;
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&st_full[g]));
        kt = ktn;
      }
    } else {
      // -------------------------------------------------------- cut A
      const int g = (warp - W_CUT0) >> 2, t = threadIdx.x - W_CUT0 * 32 - g * GT;
      constexpr int NP = TM * TK / 4 / GT;  // 8 passes: rows 16 p + t / 8 (not TRANS)
      float scs[NP];                        // this thread's row scales in window scw
      int scw = -1;
      unsigned char* sp = sbase + RAW_REGION + g * STAGE_BYTES;
      float v[TK];  // the thread's 32 entries of its tile
      // the group's tiles: every NG-th active one, from the g-th
      TileIter ti = tiles();
      int kt = ti.next();
      for (int i = 0; i < g; ++i) kt = ti.next();
      uint32_t ph = 1;
      while (kt < nkt) {
        if (kt / WIN_TILES != scw) {  // (issued before the waits: the loads overlap them)
          scw = kt / WIN_TILES;
          if (!TRANS) {
#pragma unroll
            for (int p = 0; p < NP; ++p) scs[p] = row_scale((p * GT + t) >> 3, scw);
          } else {
            scs[0] = row_scale(t, scw);
          }
        }
        // The warp's lanes leave together: one of them arrives for all.  The raw tile
        // is waited for and read before the stage is free: safe because raw buffer g
        // is this group's alone, so its phases cannot run ahead of the group (with
        // buffers shared between groups, a group could meet the phase before the
        // one it waits for, whose parity reads as complete).
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&raw_full[g]), ph ^ 1, &abort_flag,
                                               poll_limit))) {
          leave_stage(g);
          break;
        }
        // the raw tile into registers first (the wait for the stage follows), so that
        // the raw buffer is free again early
        const unsigned char* rw = sbase + g * RAW_BYTES;
        if (!TRANS) {
          // raw [128 rows][32 k]; pass p: rows 16 p .. 16 p + 15, 8 threads per row
#pragma unroll
          for (int p = 0; p < NP; ++p) {
            const int f = p * GT + t, m = f >> 3, k4 = f & 7;
            const float4 x = *reinterpret_cast<const float4*>(rw + m * (TK * 4) + k4 * 16);
            v[4 * p] = x.x; v[4 * p + 1] = x.y; v[4 * p + 2] = x.z; v[4 * p + 3] = x.w;
          }
        } else {
          // raw [32 k][128 m]; thread m = t takes all 32 k
#pragma unroll
          for (int i = 0; i < TK; ++i) v[i] = *reinterpret_cast<const float*>(rw + (i * TM + t) * 4);
        }
        // the next TMA write (async proxy) must follow these generic reads
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&raw_empty[g]));
        if (!__all_sync(0xffffffffu,
                        mbar_wait(smem_u32(&st_empty[g]), ph, &abort_flag, poll_limit))) {
          leave_stage(g);
          break;
        }
        ph ^= 1;
        float mx = 0.f;
        if (!TRANS) {
#pragma unroll
          for (int p = 0; p < NP; ++p) {
            const int f = p * GT + t, m = f >> 3, k4 = f & 7;
            const float sc = scs[p];
            f32x2 sl[4][2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const float a = v[4 * p + 2 * i] * sc, b = v[4 * p + 2 * i + 1] * sc;
              mx = max_abs(mx, a, b);
              cut4(pack2(a, b), sl[0][i], sl[1][i], sl[2][i], sl[3][i]);
            }
            const uint32_t off = sw64_off(m, k4 >> 1) + (uint32_t)((k4 & 1) * 8);
#pragma unroll
            for (int t4 = 0; t4 < NSL; ++t4)
              *reinterpret_cast<uint2*>(sp + t4 * A_SLICE + off) =
                  make_uint2(pack_bf16(sl[t4][0]), pack_bf16(sl[t4][1]));
          }
        } else {
          const float sc = scs[0];
#pragma unroll
          for (int q = 0; q < 4; ++q) {  // 16-byte chunk q: k = 8 q ..
            f32x2 sl[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float a = v[q * 8 + 2 * i] * sc, b = v[q * 8 + 2 * i + 1] * sc;
              mx = max_abs(mx, a, b);
              cut4(pack2(a, b), sl[0][i], sl[1][i], sl[2][i], sl[3][i]);
            }
            const uint32_t off = sw64_off(t, q);
#pragma unroll
            for (int t4 = 0; t4 < NSL; ++t4)
              *reinterpret_cast<uint4*>(sp + t4 * A_SLICE + off) =
                  make_uint4(pack_bf16(sl[t4][0]), pack_bf16(sl[t4][1]), pack_bf16(sl[t4][2]),
                             pack_bf16(sl[t4][3]));
          }
        }
        if (!(mx < 128.f)) abort_flag = 3;  // an entry outgrew its recorded row scale
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&st_full[g]));
#pragma unroll
        for (int i = 0; i < NG; ++i) kt = ti.next();
      }
    }
  } else {
    // ---------------------------------------------------------- drain / epilogue
    const int dw = warp - W_DRAIN0;  // 0 .. 15
    const int q4 = warp & 3;         // TMEM lane quarter
    const int c0 = (dw >> 2) * DC;   // columns c0 .. c0 + 15 of the tile
    const int r = q4 * 32 + lane;
    f32x2 hi[DC / 2], lo[DC / 2];  // columns 2 j, 2 j + 1 of them
#pragma unroll
    for (int j = 0; j < DC / 2; ++j) { hi[j] = 0ull; lo[j] = 0ull; }
    int wc = 0;
    for (int w = 0; w < nwin; ++w) {
      // the window's eight K tiles are one byte of the activity mask
      if (!((act_bits[w >> 2] >> ((w & 3) * 8)) & 0xffu)) continue;
      const int b = wc & 1;
      const int exl = ex[((int64_t)w * nct + ct) * TN + c0 + (lane & 15)];  // column lane
      const int ea = (m0 + r < n) ? e_rows[(m0 + r) * nwin + w] : 0;      // row, window
      // every scale 2^(ea + exl - 14) of the warp in the normal range: its bits are a sum
      const int emin = __reduce_min_sync(0xffffffffu, exl), emax = __reduce_max_sync(0xffffffffu, exl);
      const bool normal = __all_sync(0xffffffffu, ea + emin - 14 >= -126 && ea + emax - 14 <= 127);
      if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&acc_full[b]), (wc >> 1) & 1, &abort_flag,
                                             poll_limit)))
        break;
      tc_fence_after();
      const uint32_t tl = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(b * 4 * TN + c0);
#pragma unroll
      for (int g = 0; g < DC / 8; ++g) {
        float sc[8];
        if (normal) {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            sc[j] = __int_as_float(((ea + 113) << 23) + __shfl_sync(0xffffffffu, exl << 23, g * 8 + j));
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            sc[j] = ldexpf(1.f, ea + __shfl_sync(0xffffffffu, exl, g * 8 + j) - 14);
        }
        // orders 2..5: exact sums (integers times 2^(-8 (d - 2))) times an exact power
        // of two, each added into (hi, lo) through TwoSum, so that lo only gathers
        // rounding residues (the lower orders are not small: their digits run up
        // to 128 against a leading digit that may be much smaller)
#pragma unroll
        for (int d = 0; d < 4; ++d) {
          float v[8];
          tmem_ld8(tl + (uint32_t)(d * TN + g * 8), v);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int jj = g * 4 + j;
            const f32x2 t = mul2(pack2(v[2 * j], v[2 * j + 1]), pack2(sc[2 * j], sc[2 * j + 1]));
            const f32x2 sum = add2(hi[jj], t);
            const f32x2 bp = sub2(sum, hi[jj]);
            lo[jj] = add2(lo[jj], add2(sub2(hi[jj], sub2(sum, bp)), sub2(t, bp)));
            hi[jj] = sum;
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&acc_empty[b]));
      ++wc;
    }
    const int64_t grow = m0 + r;
    const bool bad = abort_flag != 0;
    if (grow < n) {
#pragma unroll
      for (int j = 0; j < DC; ++j) {
        const int64_t col = (int64_t)ct * TN + c0 + j;
        if (col < ncols) {
          float h[2], l[2];
          unpack2(hi[j >> 1], h[0], h[1]);
          unpack2(lo[j >> 1], l[0], l[1]);
          const double v = bad ? __longlong_as_double(0x7ff8000000000000ll)
                               : (double)h[j & 1] + (double)l[j & 1];
          // split over K: Y was zeroed and every block adds its share
          if (gridDim.z > 1) atomicAdd(&Y[grow + col * ldy], v);
          else Y[grow + col * ldy] = v;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (abort_flag && tid == 0) atomicExch(err, 1);
  if (warp == W_MMA && abort_flag != 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TMEM_COLS)
                 : "memory");
  }
}

}  // namespace

size_t gemm_esg_smem_bytes() { return (size_t)LAYOUT_BYTES + 1024; }

// bytes of the pre-cut X workspace: four BF16 slices per padded column tile,
// then one int exponent per (window, column) (sized per K tile, which is more)
int64_t gemm_esg_work_bytes(int64_t n, int64_t ncols) {
  const int64_t kpad = ((n + KPAD - 1) / KPAD) * KPAD;
  const int64_t nct = (ncols + TN - 1) / TN;
  const int64_t xs = nct * NSL * TN * kpad * 2;
  return ((xs + 255) / 256) * 256 + (kpad / TK) * nct * TN * 4;
}

int64_t gemm_esg_exp_count(int64_t n) { return n * ((n + WIN_ROWS - 1) / WIN_ROWS); }

void launch_esg_scales(const float* A, int64_t lda, int64_t n, int* aexp, cudaStream_t st) {
  count_launches(2);
  const int nw = (int)((n + WIN_ROWS - 1) / WIN_ROWS);
  k_row_exp<<<(unsigned)((n + 7) / 8), 256, 0, st>>>(A, lda, n, nw, aexp);
  k_col_exp<<<dim3((unsigned)((n + 255) / 256), (unsigned)nw), 256, 0, st>>>(A, lda, n, nw, aexp + gemm_esg_exp_count(n));
}

int launch_gemm_esg(const float* A, int64_t lda, int trans, int64_t n, int64_t ncols,
                    const double* X, int64_t ldx, double* Y, int64_t ldy, void* work,
                    const int* aexp, uint8_t* flags, int* err, cudaStream_t st) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = tc::encode_fn();
  if (!enc || !gemm_tc_supported(A, lda, n)) return 1;
  const int64_t kpad = ((n + KPAD - 1) / KPAD) * KPAD;
  const int nct = (int)((ncols + TN - 1) / TN);
  const int nkt = (int)(kpad / TK);
  if (nkt > MAX_KT) return 1;
  __nv_bfloat16* Xs = (__nv_bfloat16*)work;
  const int64_t xs_bytes = (int64_t)nct * NSL * TN * kpad * 2;
  int* ex = (int*)((unsigned char*)work + ((xs_bytes + 255) / 256) * 256);
  CUtensorMap tmA;
  const cuuint64_t adim[2] = {(cuuint64_t)n, (cuuint64_t)n};
  const cuuint64_t astr[1] = {(cuuint64_t)lda * 4};
  const cuuint32_t abox[2] = {trans ? (cuuint32_t)TM : (cuuint32_t)TK,
                              trans ? (cuuint32_t)TK : (cuuint32_t)TM};
  const cuuint32_t one[2] = {1, 1};
  if (enc(&tmA, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, (void*)A, adim, astr, abox, one,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return 2;
  count_launches(2);
  const int nwin = (nkt + WIN_TILES - 1) / WIN_TILES;
  k_split_x64<<<dim3(nwin, nct), SPLIT_THREADS, 0, st>>>(X, ldx, n, ncols, kpad, nct, Xs, ex, flags);
  const int* e_rows = trans ? aexp + gemm_esg_exp_count(n) : aexp;
  const size_t smem = gemm_esg_smem_bytes();
  static std::atomic<uint32_t> done[2] = {{0}, {0}};
  // Split over K when the row blocks alone leave the last wave of blocks
  // (one per SM) markedly short: two blocks per row block share its windows,
  // each keeping >= 16 windows of the (typically half active) K range.  At most
  // two: two FP64 partials added into a zeroed Y give the same sum in either
  // order, so the results stay reproducible.
  const int nrb = (int)((n + TM - 1) / TM);
  int nsm = 0, dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm < 1)
    nsm = 1;
  auto eff = [&](int k) {
    const int64_t c = (int64_t)nct * nrb * k;
    return (double)c / ((double)nsm * (double)((c + nsm - 1) / nsm));
  };
  int ks = 1;
  const int ks_max = std::max(1, std::min(2, nwin / 16));
  for (int k = 2; k <= ks_max; ++k)
    if (eff(k) > eff(ks) + 0.05) ks = k;
  if (ks > 1 &&
      cudaMemset2DAsync(Y, (size_t)ldy * sizeof(double), 0, (size_t)n * sizeof(double),
                        (size_t)ncols, st) != cudaSuccess)
    return 2;
  dim3 grid((unsigned)nct, (unsigned)nrb, (unsigned)ks);
  if (trans) {
    raise_smem_limit((const void*)k_gemm_esg<1, 0>, done[1]);
    k_gemm_esg<1, 0><<<grid, NTHREADS, smem, st>>>(tmA, Xs, n, ncols, flags, ex, e_rows, Y, ldy,
                                                   err, wait_limit(), nullptr, nullptr);
  } else {
    raise_smem_limit((const void*)k_gemm_esg<0, 0>, done[0]);
    k_gemm_esg<0, 0><<<grid, NTHREADS, smem, st>>>(tmA, Xs, n, ncols, flags, ex, e_rows, Y, ldy,
                                                   err, wait_limit(), nullptr, nullptr);
  }
  return 0;
}

}  // namespace hm

namespace hm {
namespace {

// The tables hold float pairs: S[0 .. n) high parts then S[n .. 2n) low parts,
// P[0 .. 2n - 1) high parts then P[2n - 1 .. 4n - 2) low parts.
// Exponents of the matrix-free log kernel per row and window of 256 columns: e
// with max |A(i, j)| < 2^e over the window (clamped to >= -120), the entries
// formed exactly as the generating cutters form them.  One warp per row.  The
// operator is symmetric: these are also the column exponents.
__global__ __launch_bounds__(256) void k_row_exp_logtab(const float* __restrict__ S,
                                                        const float* __restrict__ P, int64_t n,
                                                        int nw, int* __restrict__ e_row) {
  const int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= n) return;
  for (int w = 0; w < nw; ++w) {
    float mx = 0.f;
    for (int64_t j = (int64_t)w * WIN_ROWS + lane; j < n && j < (int64_t)(w + 1) * WIN_ROWS;
         j += 32) {
      const int64_t d = row > j ? row - j : j - row;
      const float v = (d == 0) ? 1.f : (S[d] + P[row + j]) + (S[n + d] + P[2 * n - 1 + row + j]);
      mx = fmaxf(mx, fabsf(v));
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) e_row[row * nw + w] = max(exp_above(mx), -120);
  }
}

// out[(i - r0) * ld + (j - c0)] = A(i, j) of the matrix-free log kernel.
__global__ void k_logtab_block(const float* __restrict__ S, const float* __restrict__ P,
                               int64_t n, int64_t r0, int64_t r1, int64_t c0, int64_t c1,
                               float* __restrict__ out, int64_t ld) {
  for (int64_t i = r0 + blockIdx.y; i < r1; i += gridDim.y)
    for (int64_t j = c0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < c1;
         j += (int64_t)gridDim.x * blockDim.x) {
      const int64_t d = i > j ? i - j : j - i;
      out[(i - r0) * ld + (j - c0)] =
          (d == 0) ? 1.f : (S[d] + P[i + j]) + (S[n + d] + P[2 * n - 1 + i + j]);
    }
}

}  // namespace

void launch_logtab_rowexp(const float* S, const float* P, int64_t n, int* e_row, cudaStream_t st) {
  count_launches(1);
  k_row_exp_logtab<<<(unsigned)((n + 7) / 8), 256, 0, st>>>(
      S, P, n, (int)((n + WIN_ROWS - 1) / WIN_ROWS), e_row);
}

void launch_logtab_block(const float* S, const float* P, int64_t n, int64_t r0, int64_t r1,
                         int64_t c0, int64_t c1, float* out, int64_t ld, cudaStream_t st) {
  count_launches(1);
  const int64_t w = c1 - c0, h = r1 - r0;
  dim3 grid((unsigned)std::min<int64_t>((w + 255) / 256, 1024),
            (unsigned)std::min<int64_t>(h, 65535));
  k_logtab_block<<<grid, 256, 0, st>>>(S, P, n, r0, r1, c0, c1, out, ld);
}

// Y = A X for the matrix-free log kernel (symmetric, so either product), FP64
// X and Y, with the exact-accumulation split of launch_gemm_esg; the entries of
// A are formed in the cutter warps from the tables S and P and never stored.
int launch_gemm_esg_gen(const float* S, const float* P, const int* rowexp, int64_t n,
                        int64_t ncols, const double* X, int64_t ldx, double* Y, int64_t ldy,
                        void* work, uint8_t* flags, int* err, cudaStream_t st) {
  const int64_t kpad = ((n + KPAD - 1) / KPAD) * KPAD;
  const int nct = (int)((ncols + TN - 1) / TN);
  const int nkt = (int)(kpad / TK);
  if (nkt > MAX_KT) return 1;
  __nv_bfloat16* Xs = (__nv_bfloat16*)work;
  const int64_t xs_bytes = (int64_t)nct * NSL * TN * kpad * 2;
  int* ex = (int*)((unsigned char*)work + ((xs_bytes + 255) / 256) * 256);
  // the kernel takes no TMA map of A in this form: a zeroed map fills the slot
  CUtensorMap tm0;
  memset(&tm0, 0, sizeof(tm0));
  count_launches(2);
  const int nwin = (nkt + WIN_TILES - 1) / WIN_TILES;
  k_split_x64<<<dim3(nwin, nct), SPLIT_THREADS, 0, st>>>(X, ldx, n, ncols, kpad, nct, Xs, ex, flags);
  const size_t smem = gemm_esg_smem_bytes();
  static std::atomic<uint32_t> done{0};
  // the same K split as the dense engine: two blocks share a row block's windows
  // when the grid's last wave is short
  const int nrb = (int)((n + TM - 1) / TM);
  int nsm = 0, dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm < 1)
    nsm = 1;
  auto eff = [&](int k) {
    const int64_t c = (int64_t)nct * nrb * k;
    return (double)c / ((double)nsm * (double)((c + nsm - 1) / nsm));
  };
  int ks = 1;
  const int ks_max = std::max(1, std::min(2, nwin / 16));
  for (int k = 2; k <= ks_max; ++k)
    if (eff(k) > eff(ks) + 0.05) ks = k;
  if (ks > 1 &&
      cudaMemset2DAsync(Y, (size_t)ldy * sizeof(double), 0, (size_t)n * sizeof(double),
                        (size_t)ncols, st) != cudaSuccess)
    return 2;
  dim3 grid((unsigned)nct, (unsigned)nrb, (unsigned)ks);
  raise_smem_limit((const void*)k_gemm_esg<0, 1>, done);
  k_gemm_esg<0, 1><<<grid, NTHREADS, smem, st>>>(tm0, Xs, n, ncols, flags, ex, rowexp, Y, ldy,
                                                 err, wait_limit(), S, P);
  return 0;
}

}  // namespace hm
