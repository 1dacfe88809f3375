// gram_tc.cu -- the contractions with W on the tensor cores.
//
//   partial[s m + a] = sum over the points r of tile T of A[a][r] W[list(T)[s]][r]
//
// (s a slot of tile T's W list); the per-orbital sums of M = Phi^T W and of
// W^T psi add these partials afterwards in FP64.
//
// Precision: FP64 operands, FP16 tensor-core products by exact splitting (the
// Ozaki scheme).  Each row segment x (the 64 points of one half tile, 8 x 4 x 2,
// of an A row or a W row) shares one exponent E (|x| < 2^E); x 2^-E is taken to
// an integer X on a 2^-47 grid and written in S = 6 base-256 digits (W's
// balanced, |d_k| <= 128, A's the bytes of |x| on a 2^-48 grid with x's sign),
// each exactly an FP16 value.  For a pair of segments,
//   sum_r x_r w_r ~ 2^(Ex+Ew) sum_{d=0}^{S-1} 2^(-15-8d) D_d,
//   D_d = sum_{k+l=d} sum_r dx_k(r) dw_l(r),
// where every D_d is a sum of at most 6 x 64 products of magnitude < 2^15,
// hence an integer below 2^24: the tensor core's FP32 accumulation of it is
// exact.  The epilogue combines the D_d exactly in 64-bit integers, aligns the
// two halves' integers on the larger scale (the other truncated at its unit,
// 2^-55 of that segment's scale) and truncates once to FP64, with no FP64
// instruction.  Error: the truncation of X (2^-47 and 2^-48 of the segment's
// power of two) and the dropped diagonals d >= S (below 2^-45.7 of max|x| max|w|
// times the segment length).
//
// The plain form (DIG = 7) has seven digits per operand and eight diagonals
// (each still below 2^24): W rounded to 55 bits, A's bytes to 56, both against
// their segment's power of two 2^E, the diagonals d >= 8 dropped (2^-61 a point),
// the two halves' sums to 2^-55 of the larger scale, one rounding.  So a product
// errs by at most 2^-56 (|x| 2^Ew + |w| 2^Ex): an absolute bound per segment, not
// one relative to the product as an FP64 multiply-add has it.  Values within a
// factor of 8 (A) or 4 (W) of 2^E are kept whole; where large x meets small w
// throughout a segment the sum keeps fewer digits than an FP64 chain (rms error
// of a partial against one's: values of one size 0.25, W falling by 2^4 where A
// rises by as much 1.1, 2^8 17, 2^14 900), which matters to sums that are as
// small against the operands.  The expansion holds W against the largest value at each point
// (k_wx_digits).  Errors of V^ACE psi against extended precision, relative to its
// norm, 16 to 256 orbitals, 27^3 to 101^3: 3.3 to 6.0e-16, with FP64 multiply-adds
// 3.9 to 6.3e-16 (with the seven diagonals, W truncated and the tile's scale in
// the expansion 4.3 to 6.6e-16).  The FP64 unit took 3.68 ms per contraction (256
// rows, 96^3) and 3.51 ms for the expansion.  Segments with a non-finite value
// give NaN.
//
// Kernel shape: persistent CTAs (one per SM) take tiles from a queue and
// walk units (W block of up to 32 slots, A block of 128 rows, half tile).
// Per unit the A digits go to shared memory in the tensor core's K-major
// layout without swizzle (8 x 16-byte core matrices; row groups 128 B
// apart, x-runs of 8 points one row-group stack apart).  W's digit planes
// of the block are stacked along N (plane l at rows l P, P = 16 or 32 the
// padded block width) and the accumulator of diagonal d sits at
// tensor-memory columns d P, so one MMA of A plane k against the stacked W
// planes 0..5-k (N = (6 - k) P) adds every product of plane k to the
// diagonals k..5 at once: 24 tcgen05.mma instructions (M = 128, K = 16) per
// unit (28 with seven digits, N = (8 - k) P).  After the second half tile the converting warps read the
// accumulators back with tcgen05.ld for the epilogue (k_gram_tc).  A few rows
// take k_gram_few, whose partials are the same bits.
// Every wait on a completion barrier is bounded: on expiry the kernel sets
// SEA_FLAG_WAIT, waits once more (bounded) for work in flight, frees its
// tensor memory and ends.
#include <cuda.h>

#include <climits>
#include <cstring>

#include "cg_fixed.cuh"
#include "sea_internal.cuh"
#include "tcgen05.cuh"

namespace sea {
namespace {

// DIG digits per operand: 6 in the mixed form, 7 in the plain form
constexpr int KH = 64;                          // points per half tile
constexpr int MBLK = 128;                       // A rows per block
constexpr uint32_t CORE_SBO = 128;              // row-group-adjacent core matrices
constexpr uint32_t TMEM_COLS = 512;
// Diagonals d = k + l of the digit planes' products that are formed.  Seven digits
// keep an eighth: the products of diagonal 7, 2^-56.3 of max|x| max|w| a point
// (rms), were the largest error of a partial, 3.5 times the digits' own.  B then
// has an eighth plane of zeros, so that every diagonal's accumulator is set by
// the first MMA.
constexpr int diagonals(int digits) { return digits == 7 ? 8 : 6; }
template <int DIG>
struct GramSizes {
  // W rows per block: seven digit planes of A beside the raw rows leave room
  // for 16 (all but 92 of the 6912 tiles of 256 orbitals on 96^3 have no more)
  static constexpr int NBLK = DIG == 6 ? 32 : 16;
  static constexpr int ND = diagonals(DIG);
  static constexpr uint32_t W_HALF = ND * NBLK * KH * 2;  // bytes of W digits per half tile
  static constexpr uint32_t SMEM_W = 2 * W_HALF;          // 48 KB (both halves)
  static constexpr uint32_t TMEM_HALF = ND * NBLK;        // accumulator columns per half tile
};
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
               "r"(valid ? 16 : 0));
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// x 2^-E on the 2^-(8 DIG - 1) grid, E = emax - 1022 for the segment's largest
// biased exponent emax: a signed integer below 2^(8 DIG - 1), truncated toward
// zero with six digits, rounded with seven.  Integer operations only.
template <int DIG>
__device__ __forceinline__ long long fixed_bal(double v, int emax) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int e = (int)((b >> 52) & 0x7FF);
  unsigned long long X;
  if (DIG == 6) {
    const int sh = emax - e + 6;
    if (e == 0 || sh > 60) return 0;
    X = ((b & 0xFFFFFFFFFFFFFULL) | (1ULL << 52)) >> sh;
  } else {
    if (e == 0) return 0;
    X = (shr64c(((b & 0xFFFFFFFFFFFFFULL) | (1ULL << 52)) << 3, (unsigned)(emax - e)) + 1) >> 1;
  }
  return (b >> 63) ? -(long long)X : (long long)X;
}

// Balanced base-256 digits of X: with Y = X + 128 (256^0 + ... +
// 256^(DIG-2)), digit DIG - 1 - i = byte i of Y minus 128 (i < DIG - 1) and
// digit 0 = Y >> 8 (DIG - 1), so X = sum_k d_k 256^(DIG-1-k), d_1.. in [-128,
// 127], |d_0| <= 128.  Each digit as an FP32 value (exact), from the bit
// pattern 0x4B4000bb = 2^23 + 2^22 + b.
template <int DIG>
__device__ __forceinline__ void digit_floats(long long X, float* f) {
  const long long Y = X + (DIG == 6 ? 0x8080808080LL : 0x808080808080LL);
  const unsigned lo = (unsigned)Y, hi = (unsigned)(Y >> 32);
  const float m = 12582912.0f + 128.0f;
  f[DIG - 1] = __uint_as_float(__byte_perm(lo, 0x4B400000u, 0x7650)) - m;
  f[DIG - 2] = __uint_as_float(__byte_perm(lo, 0x4B400000u, 0x7651)) - m;
  f[DIG - 3] = __uint_as_float(__byte_perm(lo, 0x4B400000u, 0x7652)) - m;
  f[DIG - 4] = __uint_as_float(__byte_perm(lo, 0x4B400000u, 0x7653)) - m;
  f[DIG - 5] = __uint_as_float(__byte_perm(hi, 0x4B400000u, 0x7650)) - m;
  if (DIG == 7) f[1] = __uint_as_float(__byte_perm(hi, 0x4B400000u, 0x7651)) - m;
  f[0] = __int_as_float(0x4B400000 + (int)(Y >> (8 * (DIG - 1)))) - 12582912.0f;
}

// FP16 bit patterns of two small integer-valued floats (|v| <= 2048, exact),
// packed low/high.
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// Digits of one row group (8 rows) of a block, half h of tile T, held in
// registers: the warp's lane l takes row l % 8 and the x-runs u = l / 8 and
// l / 8 + 4 (run u: y = u % 4, z = 2h + u / 4, 8 points along x).  Row
// pointer rp (nullptr: zero row).
template <int DIG>
struct GroupDigits {
  uint32_t w[2][DIG][4];  // [run][digit plane][pair of points]
  int emax;               // the row's largest biased exponent
};

template <int DIG>
__device__ __forceinline__ void make_digits(const double* __restrict__ rp, const TileGeom& G,
                                            int T, int h, GroupDigits<DIG>& o) {
  const int lane = threadIdx.x & 31;
  const int txi = T % G.ntx, tyi = (T / G.ntx) % G.nty, tzi = T / (G.ntx * G.nty);
  const int gx0 = txi * TX;
  double v[2][8];
  int em = 0;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int u = (lane >> 3) + 4 * q;
    const int gy = tyi * TY + (u & 3), gz = tzi * TZ + 2 * h + (u >> 2);
    const bool in = rp && gy < G.ny && gz < G.nz;
    const double* src = in ? rp + ((size_t)gz * G.ny + gy) * G.nx + gx0 : rp;
    if (in && gx0 + 8 <= G.nx && (((uintptr_t)src) & 15) == 0) {
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const double2 t = __ldg(reinterpret_cast<const double2*>(src) + p);
        v[q][2 * p] = t.x;
        v[q][2 * p + 1] = t.y;
      }
    } else {
#pragma unroll
      for (int x = 0; x < 8; ++x) v[q][x] = (in && gx0 + x < G.nx) ? src[x] : 0.0;
    }
#pragma unroll
    for (int x = 0; x < 8; ++x)
      em = max(em, (int)((__double_as_longlong(v[q][x]) >> 52) & 0x7FF));
  }
  em = max(em, __shfl_xor_sync(0xffffffffu, em, 8));
  em = max(em, __shfl_xor_sync(0xffffffffu, em, 16));
  o.emax = em;
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      float f0[DIG], f1[DIG];
      digit_floats<DIG>(fixed_bal<DIG>(v[q][2 * p], em), f0);
      digit_floats<DIG>(fixed_bal<DIG>(v[q][2 * p + 1], em), f1);
#pragma unroll
      for (int k = 0; k < DIG; ++k) o.w[q][k][p] = pack_f16(f0[k], f1[k]);
    }
}

// Integer value of an integer-valued FP32 number at most 2^22 in magnitude:
// adding 1.5 2^23 puts it in the low mantissa bits.
__device__ __forceinline__ int small_float_int(uint32_t f) {
  return __float_as_int(__uint_as_float(f) + 12582912.0f) - 0x4B400000;
}

// v 2^e2 truncated toward zero to FP64, 0 below the normal range, with the
// 64-bit truncating conversion done by the
// conversion instruction (on the FP64 pipe, which the integer epilogues
// otherwise leave idle) and the scaling by 2^e2 added to the exponent field.
__device__ __forceinline__ double scaled_i64_rz_cvt(long long v, int e2) {
  const long long b = __double_as_longlong(__ll2double_rz(v));
  const int ex = (int)((b >> 52) & 0x7FF) + e2;  // biased exponent of the result
  return (v == 0 || ex <= 0) ? 0.0 : __longlong_as_double(b + ((long long)e2 << 52));
}

// Eight diagonal sums (integer-valued floats, |D_0|, |D_1| < 2^22, the others
// below 2^24) as the integer sum_d D_d 256^(6-d) rounded at its lowest DROP bits,
// so that 64 bits hold it.
template <int DROP>
__device__ __forceinline__ long long combine7(const uint32_t* f) {
  auto big = [](uint32_t x) { return __float2int_rz(__uint_as_float(x)); };
  const long long hi = (long long)(small_float_int(f[0]) * 256 + small_float_int(f[1])) * 4096 +
                       (long long)big(f[2]) * 16;
  // D_7 to D_6's unit, half a unit of the result for the rounding
  const int last = big(f[6]) + (big(f[7]) >> 8) + (1 << (DROP - 1));
  const long long lo = (long long)big(f[3]) * 16777216 + (long long)big(f[4]) * 65536 +
                       (long long)big(f[5]) * 256 + (long long)last;
  return (hi << (28 - DROP)) + (lo >> DROP);
}
// v 2^e2 rounded to nearest: the conversion instruction (on the FP64 pipe that
// the integer epilogues leave idle), the scaling added to the exponent field;
// 0 below the normal range, infinite above it.
__device__ __forceinline__ double scaled_i64_rn_cvt(long long v, int e2) {
  const long long b = __double_as_longlong(__ll2double_rn(v));
  const int ex = (int)((b >> 52) & 0x7FF) + e2;  // biased exponent of the result
  if (v == 0 || ex <= 0) return 0.0;
  if (ex >= 0x7FF) return __longlong_as_double((b & (1LL << 63)) | 0x7FF0000000000000LL);
  return __longlong_as_double(b + ((long long)e2 << 52));
}
// Two half tiles' sums (combine7<8>: below 2^61, units 2^e0 and 2^e1) on the
// larger scale, one rounding; NaN if `bad`.
__device__ __forceinline__ double join7(long long a0, int e0, long long a1, int e1, bool bad) {
  const bool b0 = e0 >= e1;
  const int sh = min(b0 ? e0 - e1 : e1 - e0, 63);
  const double y = scaled_i64_rn_cvt((b0 ? a0 : a1) + ((b0 ? a1 : a0) >> sh), b0 ? e0 : e1);
  return bad ? __longlong_as_double(0x7FF8000000000000LL) : y;
}
__device__ __forceinline__ double quiet_nan() { return __longlong_as_double(0x7FF8000000000000LL); }
constexpr int EXP_NONFINITE = 0x7FF;

// W digits, once per W: for every slot s of every tile list and half h,
// wdig[((s * 2 + h) * DIG + k) * 8 + u] = the 8 FP16 digits (16 bytes) of
// plane k, x-run u of W row list[s] on that half tile, and wexp[2 s + h]
// the row segment's largest biased exponent, s counted from slot s0, for the
// n_tiles tiles from t0.  Warp per (tile, half, group of 8 slots).  Four CTAs per SM: the warps wait on their row loads, so
// occupancy is what hides the latency.
template <int DIG>
__global__ void __launch_bounds__(256, DIG == 6 ? 4 : 3)
    k_w_digits(const double* __restrict__ W, TileGeom G, size_t ng, int t0, int n_tiles, int s0,
               int ngroups, const int* __restrict__ tptr, const int* __restrict__ tlist,
               uint4* __restrict__ wdig, int* __restrict__ wexp) {
  const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (gw >= (long long)n_tiles * 2 * ngroups) return;  // warp-uniform
  const int g = (int)(gw % ngroups), h = (int)((gw / ngroups) % 2),
            T = t0 + (int)(gw / (2 * ngroups));
  const int j0 = tptr[T], nJ = tptr[T + 1] - j0;
  if (8 * g >= nJ) return;  // warp-uniform
  const int lane = threadIdx.x & 31, r = lane & 7, s = 8 * g + r;
  const double* rp = s < nJ ? W + (size_t)tlist[j0 + s] * ng : nullptr;
  GroupDigits<DIG> d;
  make_digits(rp, G, T, h, d);
  if (s < nJ) {
    uint4* dst = wdig + ((size_t)(j0 + s - s0) * 2 + h) * DIG * 8;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int u = (lane >> 3) + 4 * q;
#pragma unroll
      for (int k = 0; k < DIG; ++k) dst[k * 8 + u] = make_uint4(d.w[q][k][0], d.w[q][k][1], d.w[q][k][2], d.w[q][k][3]);
    }
    if (lane < 8) wexp[(size_t)(j0 + s - s0) * 2 + h] = d.emax;
  }
}

// A unit of work: half h of A block mb against W block jb of tile T, whose W
// exponents are in buffer wb.
struct Unit {
  int T, j0, nJ, jb, mb, h, wb;
  int ab;  // parity of the A block in processing order (its exponent buffer)
};

// ---------------------------------------------------------------------------
// The contraction's kernel.  A's rows come in by the tensor memory accelerator
// or, where the rows are not 16-byte strided (odd nx) or A is unaligned (TMA =
// false), by 8-byte asynchronous copies of every warp's own rows into the same
// places.  Per unit two 4D boxes (x 8, y 4, z 1, rows 128): the two
// z-planes of the half tile (K halves 0 and 1) for the whole A block, 32 KB
// each, written with the 64-byte swizzle so that the reads below are free
// of bank conflicts.  Thread t takes row t / 4 and the x-run y = t % 4 of
// both planes (16 values; the row's exponent from a 4-lane maximum), forms
// the digits in registers and stores one 16-byte core-matrix row per digit
// plane.  The MMAs of K half 0 (committed to barrier 0) run while K half 1
// is converted; those of K half 1 (barrier 1) run while the next unit's
// rows are read and converted.  Both raw buffers are refilled for the next
// unit as soon as their values are in registers.  Points outside the grid
// and rows beyond m read the box's zero fill.  One W buffer: a new W block
// is loaded after every MMA of the previous block completed.
// ---------------------------------------------------------------------------
constexpr int GT2_CONV = 512;                        // converting threads: 4 per A row
constexpr int GT2_THREADS = GT2_CONV + 32;           // and one MMA-issuing warp
constexpr uint32_t A2_LBO = (MBLK / 8) * 128 + 32;   // 2080: x-runs 8 banks apart
constexpr uint32_t A2_PLANE = 8 * A2_LBO;            // 8 runs of 8 points
constexpr uint32_t RAW_KHALF = MBLK * (KH / 2) * 8;  // 32 KB: 128 rows x 32 points
template <int DIG>
struct GramTmaSizes {
  static constexpr uint32_t SMEM_A2 = DIG * A2_PLANE;  // 99,840 with six digits
  static constexpr size_t SMEM = 1024 + 2 * RAW_KHALF + SMEM_A2 + GramSizes<DIG>::SMEM_W;
};

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1,
                                            int c2, int c3, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
      : "memory");
}

// L2 prefetch of bytes (a multiple of 16) at p (16-byte aligned).
__device__ __forceinline__ void bulk_prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// A's digits in the TMA kernel: unsigned bytes of |x| on the segment's
// 2^-48 grid, each carrying the sign of x.  With E = emax - 1022 (|x| <
// 2^E), X = floor(|x| 2^(48 - E)) = m >> (emax - e + 5) for the 53-bit
// significand m and biased exponent e of x, so X < 2^48 and
//   x ~ s 2^(E - 48) sum_k b_k 256^(5 - k),  b_k = byte 5 - k of X,
// with an error below 2^(E - 48).  b_k in [0, 255] is exact in FP16; the
// FP16 pattern 0x6400 | b is 1024 + b, so one packed FMA (1024 + b) s -
// 1024 s gives the signed digit s b for two points at once.  Against W's
// balanced digits (|d| <= 128) every product is below 2^15 and a diagonal
// sum of at most 6 x 64 of them stays below 2^24, exact in the FP32
// accumulator.  em_sh = (emax + 5) << 20; segments whose largest value is
// below 2^-959 (emax < 64) are taken as zero (em_sh = 0xF0000000 makes
// every shift reach 64).  Integer work per value: the exponent field, the
// shift count, the significand word, one 64-bit shift; per pair of values
// nine byte permutations and the sign word.

__device__ __forceinline__ uint32_t hfma2_u(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t r;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}

// With seven digits X = floor(|x| 2^(56 - E)) = 8 m >> (emax - e) < 2^56
// (truncated: rounding it costs the converting warps two 64-bit operations a
// value and W's error is twice as large), the bytes 6 - k; em_sh = emax << 20, nothing but zeros and subnormals (taken
// as zero) when emax is 0.

// X of one value: the significand of v (bits h, l) shifted onto the grid.
template <int DIG>
__device__ __forceinline__ unsigned long long fixed_uns(uint32_t h, uint32_t l, uint32_t em_sh) {
  const uint32_t sh = (em_sh - (h & 0x7FF00000u)) >> 20;
  const unsigned long long m = ((unsigned long long)((h & 0xFFFFFu) | 0x100000u) << 32) | l;
  if (DIG == 6) return shr64c(m, sh);
  return (h & 0x7FF00000u) ? shr64c(m << 3, sh) : 0ULL;
}

// The digit planes of a pair of values from their integers X0, X1 and high
// words (signs): d(k) receives plane k's two signed FP16 digits.
template <int DIG, class Put>
__device__ __forceinline__ void digit_pair_u(unsigned long long X0, unsigned long long X1,
                                             uint32_t h0, uint32_t h1, Put&& put) {
  constexpr uint32_t K64 = 0x64646464u;
  const uint32_t x0h = (uint32_t)(X0 >> 32), x0l = (uint32_t)X0;
  const uint32_t x1h = (uint32_t)(X1 >> 32), x1l = (uint32_t)X1;
  // bytes of the two points interleaved: [p0 b, p1 b, p0 b', p1 b']
  const uint32_t tH = __byte_perm(x0h, x1h, 0x5140);  // bytes 4, 5 of X
  const uint32_t tB = __byte_perm(x0l, x1l, 0x7362);  // bytes 2, 3
  const uint32_t tA = __byte_perm(x0l, x1l, 0x5140);  // bytes 0, 1
  // sign word: FP16 pair (s0, s1) = +-1, and -1024 (s0, s1)
  const uint32_t S = (__byte_perm(h0, h1, 0x7030) & 0x80008000u) | 0x3C003C00u;
  const uint32_t C = S ^ 0xD800D800u;
  // plane k = byte DIG - 1 - k: FP16 1024 + b from the pattern 0x64bb
  if (DIG == 7) {
    const uint32_t tT = __byte_perm(x0h, x1h, 0x7362);  // byte 6 (and 7, zero)
    put(0, hfma2_u(__byte_perm(tT, K64, 0x4140), S, C));
  }
  put(DIG - 6, hfma2_u(__byte_perm(tH, K64, 0x4342), S, C));
  put(DIG - 5, hfma2_u(__byte_perm(tH, K64, 0x4140), S, C));
  put(DIG - 4, hfma2_u(__byte_perm(tB, K64, 0x4342), S, C));
  put(DIG - 3, hfma2_u(__byte_perm(tB, K64, 0x4140), S, C));
  put(DIG - 2, hfma2_u(__byte_perm(tA, K64, 0x4342), S, C));
  put(DIG - 1, hfma2_u(__byte_perm(tA, K64, 0x4140), S, C));
}

// The FP16 digit planes of 8 consecutive points: d[k] = their 8 signed
// digits of plane k (points 2i, 2i + 1 in word i, low half first).
template <int DIG>
__device__ __forceinline__ void digits8_u(const double (&v)[8], uint32_t em_sh, uint4 (&d)[DIG]) {
  uint32_t w[DIG][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const unsigned long long b0 = (unsigned long long)__double_as_longlong(v[2 * i]);
    const unsigned long long b1 = (unsigned long long)__double_as_longlong(v[2 * i + 1]);
    const uint32_t h0 = (uint32_t)(b0 >> 32), h1 = (uint32_t)(b1 >> 32);
    digit_pair_u<DIG>(fixed_uns<DIG>(h0, (uint32_t)b0, em_sh), fixed_uns<DIG>(h1, (uint32_t)b1, em_sh),
                      h0, h1, [&](int k, uint32_t x) { w[k][i] = x; });
  }
#pragma unroll
  for (int k = 0; k < DIG; ++k) d[k] = make_uint4(w[k][0], w[k][1], w[k][2], w[k][3]);
}

// The same unsigned-byte FP16 digits for a pair of values with exponents of
// their own (the expansion's H(j, v) 2^E_j against E_v): emax0, emax1 are
// the largest biased exponents the two values are measured against (six
// digits, below 64: the value counts as zero).  pk[k][e] = the pair's digits
// of plane k.
template <int DIG>
__device__ __forceinline__ void digits2_u(double v0, double v1, int emax0, int emax1,
                                          uint32_t (&pk)[DIG][2], int e) {
  const unsigned long long b0 = (unsigned long long)__double_as_longlong(v0);
  const unsigned long long b1 = (unsigned long long)__double_as_longlong(v1);
  const uint32_t h0 = (uint32_t)(b0 >> 32), h1 = (uint32_t)(b1 >> 32);
  unsigned long long X0, X1;
  if (DIG == 6) {
    X0 = fixed_uns<6>(h0, (uint32_t)b0, emax0 >= 64 ? (uint32_t)(emax0 + 5) << 20 : 0xF0000000u);
    X1 = fixed_uns<6>(h1, (uint32_t)b1, emax1 >= 64 ? (uint32_t)(emax1 + 5) << 20 : 0xF0000000u);
  } else {
    // exponents may leave the FP64 range here: plain integer shift counts
    auto fixed = [](uint32_t h, uint32_t l, int emax) -> unsigned long long {
      const int ex = (int)((h >> 20) & 0x7FFu);
      const unsigned long long m = ((unsigned long long)((h & 0xFFFFFu) | 0x100000u) << 32) | l;
      return ex ? (shr64c(m << 4, (unsigned)max(emax - ex, 0)) + 1) >> 1 : 0ULL;
    };
    X0 = fixed(h0, (uint32_t)b0, emax0);
    X1 = fixed(h1, (uint32_t)b1, emax1);
  }
  digit_pair_u<DIG>(X0, X1, h0, h1, [&](int k, uint32_t x) { pk[k][e] = x; });
}

// Converting warps 0..15 (named barrier 1) and the issuing warp 16.  Per
// unit the converting warps post the unit's block width and half to a
// two-entry ring and arrive on ready[0] once K half 0's digits are in place,
// on ready[1] once K half 1's are; the issuing thread waits on each,
// issues that K half's MMAs and commits them to mma[0] / mma[1].  A unit
// with width 0 ends the issuing loop.
__device__ __forceinline__ void conv_sync() { asm volatile("bar.sync 1, 512;" ::: "memory"); }
// The same barrier returning whether v held in any converting thread (the
// same value in all of them).
__device__ __forceinline__ bool conv_sync_or(bool v) {
  uint32_t r;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.or.pred q, 1, 512, p;\n"
      "selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)v)
      : "memory");
  return r != 0;
}

template <int DIG, bool TMA>
__global__ void __launch_bounds__(GT2_THREADS, 1)
    k_gram_tc(const __grid_constant__ CUtensorMap tmA, const double* __restrict__ A, size_t ng, int m,
              TileGeom G, int t0, int n_tiles,  // tiles [t0, n_tiles)
              const int* __restrict__ tptr, const uint4* __restrict__ wdig, int slot0,
              const int* __restrict__ wexp, double* __restrict__ partial, int* __restrict__ queue,
              unsigned* __restrict__ status) {
  using Z = GramSizes<DIG>;
  constexpr int NBLK = Z::NBLK, ND = Z::ND;
  constexpr uint32_t W_HALF = Z::W_HALF, TMEM_HALF = Z::TMEM_HALF,
                     SMEM_A2 = GramTmaSizes<DIG>::SMEM_A2;
  extern __shared__ unsigned char gt_raw[];
  unsigned char* sR = gt_raw + ((1024 - (smem_addr(gt_raw) & 1023)) & 1023);  // two K halves
  unsigned char* sA = sR + 2 * RAW_KHALF;
  unsigned char* sW = sA + SMEM_A2;
  __shared__ int Aexp[2][2][MBLK], Wexp[2][2][NBLK];  // [A block parity][half][row],
                                                     // [W block parity][half][slot]
  __shared__ __align__(8) unsigned long long mbar[2], tbar[2], rbar[2];
  __shared__ int u_ring[2][2];  // per posted unit: W block width (0: end), half
  __shared__ uint32_t tmem_base;
  __shared__ int s_tile, s_j[2], s_fail, s_ifail;  // claimed tile, its list bounds; failures
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t mb[2] = {smem_addr(&mbar[0]), smem_addr(&mbar[1])};
  const uint32_t tb[2] = {smem_addr(&tbar[0]), smem_addr(&tbar[1])};
  const uint32_t rb[2] = {smem_addr(&rbar[0]), smem_addr(&rbar[1])};

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(&tmem_base)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int q = 0; q < 2; ++q) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb[q]));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tb[q]));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(rb[q]));
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
    if (TMA)
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
    s_fail = 0;
    s_ifail = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  const uint32_t a_base = smem_addr(sA), w_base = smem_addr(sW), r_base = smem_addr(sR);

  if (warp == GT2_CONV / 32) {
    // ---- the issuing warp ----
    if (lane == 0) {
      uint32_t rph[2] = {0, 0};
      for (int seq = 0;; ++seq) {
        if (!mbar_wait(rb[0], rph[0])) {
          s_ifail = 1;
          break;
        }
        rph[0] ^= 1;
        const int nj = u_ring[seq & 1][0], h = u_ring[seq & 1][1];
        if (nj == 0) break;
        const int P = nj <= 16 ? 16 : 32;
        const uint32_t lbo = ND * P * 16;
        const uint64_t a0 = sdesc(a_base, A2_LBO, CORE_SBO);
        const uint64_t w0 = sdesc(w_base + h * W_HALF, lbo, CORE_SBO);
        const uint32_t dcol = tmem + (uint32_t)(h * TMEM_HALF);
        for (int kh = 0; kh < 2; ++kh) {
          if (kh == 1) {
            if (!mbar_wait(rb[1], rph[1])) {
              s_ifail = 1;
              break;
            }
            rph[1] ^= 1;
          }
          tc_fence_after();
#pragma unroll
          for (int qq = 0; qq < 2; ++qq) {
            const int q = 2 * kh + qq;
#pragma unroll
            for (int k = 0; k < DIG; ++k)
              mma_kf16(dcol + (uint32_t)(k * P), a0 + ((k * A2_PLANE + q * 2 * A2_LBO) >> 4),
                       w0 + ((q * 2 * lbo) >> 4), idesc_kf16((ND - k) * P, MBLK, false),
                       (k > 0 || q > 0) ? 1u : 0u);
          }
          asm volatile(
              "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                  mb[kh])
              : "memory");
        }
        if (s_ifail) break;
      }
    }
    __syncwarp();
  } else {
    // ---- the converting warps ----
    const int nmb = (m + MBLK - 1) / MBLK;
    // the thread that issues the A rows' TMA loads (lane 0 of the last
    // converting warp: thread 0 already claims the tiles)
    constexpr int TMA_TID = GT2_CONV - 32;
    bool tma_pending[2] = {false, false};  // meaningful in TMA_TID
    // this thread's row and x-run, and the swizzled offset of its run
    const int row = tid >> 2, run = tid & 3;
    const uint32_t r_off = (uint32_t)(row * 256 + run * 64);
    const uint32_t r_swz = (uint32_t)((((row & 1) << 1) | (run >> 1)) << 4);
    // Thread 0 claims tiles one ahead: the next index is taken from the
    // queue when the current tile is published, and over the following units
    // its bounds are read (q_stage 1 -> 2), empty tiles skipped and its first
    // W block prefetched to L2 (2 -> 3), so a claim seldom waits on memory.
    int q_t = 0, q_j0 = 0, q_j1 = 0, q_stage = 0;  // 1 index taken, 2 bounds read, 3 resolved
    auto q_step = [&]() {
      if (q_stage == 1) {
        if (q_t < n_tiles) {
          q_j0 = __ldg(tptr + q_t);
          q_j1 = __ldg(tptr + q_t + 1);
          q_stage = 2;
        } else {
          q_stage = 3;
        }
      } else if (q_stage == 2) {
        if (q_j1 == q_j0) {
          q_t = t0 + atomicAdd(queue, 1);
          q_stage = 1;
        } else {
          bulk_prefetch_l2(wdig + (size_t)(q_j0 - slot0) * 2 * DIG * 8,
                           (uint32_t)min(q_j1 - q_j0, NBLK) * 2 * DIG * 8 * 16);
          q_stage = 3;
        }
      }
    };
    auto claim = [&](Unit& u) -> bool {
      conv_sync();
      if (tid == 0) {
        if (q_stage == 0) {
          q_t = t0 + atomicAdd(queue, 1);
          q_stage = 1;
        }
        while (q_stage != 3) q_step();
        s_tile = q_t;
        s_j[0] = q_j0;
        s_j[1] = q_j1;
        if (q_t < n_tiles) {
          q_t = t0 + atomicAdd(queue, 1);
          q_stage = 1;
        }
      }
      conv_sync();
      const int T = s_tile;
      if (T >= n_tiles) return false;
      u.T = T;
      u.j0 = s_j[0];
      u.nJ = s_j[1] - u.j0;
      u.jb = 0;
      u.mb = 0;
      u.h = 0;
      return true;
    };
    auto advance = [&](Unit& u, bool* new_block) -> bool {
      *new_block = false;
      if (u.h == 0) {
        u.h = 1;
        return true;
      }
      u.h = 0;
      u.ab ^= 1;
      if (++u.mb < nmb) return true;
      u.mb = 0;
      *new_block = true;
      u.wb ^= 1;
      u.jb += NBLK;
      if (u.jb < u.nJ) return true;
      return claim(u);
    };
    // the same without the accelerator: every warp copies its own eight rows
    // (a row's 4 x 8 points of a plane per instruction; zeros outside the grid
    // and beyond m), in flight until cp_async_wait_all and a warp barrier
    auto raw_copy = [&](const Unit& u) {
      const int txi = u.T % G.ntx, tyi = (u.T / G.ntx) % G.nty, tzi = u.T / (G.ntx * G.nty);
      const int rn = lane >> 3, x = lane & 7, gx = txi * TX + x, gy = tyi * TY + rn;
      const uint32_t dx = (uint32_t)(rn * 64 + 8 * (x & 1));
      __syncwarp();  // the lanes have read the values that are replaced
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int z = tzi * TZ + 2 * u.h + q;
        const bool in = gx < G.nx && gy < G.ny && z < G.nz;
        const double* src = A + (in ? ((size_t)z * G.ny + gy) * G.nx + gx : 0);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int r = 8 * warp + i, a = u.mb * MBLK + r;
          const uint32_t swz = (uint32_t)((((r & 1) << 1) | (rn >> 1)) << 4);
          const bool ok = in && a < m;
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(
                           r_base + q * RAW_KHALF + r * 256 + dx + (((uint32_t)(x >> 1) << 4) ^ swz)),
                       "l"(ok ? src + (size_t)a * ng : A), "r"(ok ? 8 : 0)
                       : "memory");
        }
      }
    };
    // K half q (z-plane 2 h + q of the half tile) of unit u's A block (thread 0)
    auto tma_issue = [&](const Unit& u, int q) {
      const int txi = u.T % G.ntx, tyi = (u.T / G.ntx) % G.nty, tzi = u.T / (G.ntx * G.nty);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_expect_tx(tb[q], RAW_KHALF);
      tma_load_4d(r_base + q * RAW_KHALF, &tmA, txi * TX, tyi * TY, tzi * TZ + 2 * u.h + q,
                  u.mb * MBLK, tb[q]);
      tma_pending[q] = true;
    };
    auto load_w = [&](const Unit& u) {
      const int nj = min(NBLK, u.nJ - u.jb), P = nj <= 16 ? 16 : 32;
      const uint32_t lbo = ND * P * 16;
      for (int p = tid; p < P * 2 * DIG * 8; p += GT2_CONV) {
        const int rn = p & 7, k = (p >> 3) % DIG, h = (p / (8 * DIG)) & 1, sl = p / (16 * DIG);
        const bool ok = sl < nj;
        const uint4* src =
            ok ? wdig + ((size_t)(u.j0 - slot0 + u.jb + sl) * 2 + h) * DIG * 8 + k * 8 + rn : wdig;
        const int r = k * P + sl;
        cp_async16(w_base + h * W_HALF + (r >> 3) * CORE_SBO + rn * lbo + (r & 7) * 16, src, ok);
      }
      if (tid < 2 * NBLK) {
        const int h = tid / NBLK, sl = tid % NBLK;
        Wexp[u.wb][h][sl] = sl < nj ? wexp[(size_t)(u.j0 - slot0 + u.jb + sl) * 2 + h] : 0;
      }
    };
    // bounded waits; false on expiry
    uint32_t tphase[2] = {0, 0}, mphase[2] = {0, 0};
    bool mma_pend[2] = {false, false};
    auto wait_raw = [&](int q) -> bool {
      const bool ok = mbar_wait(tb[q], tphase[q]);
      tphase[q] ^= 1;
      if (tid == TMA_TID) tma_pending[q] = false;
      return ok;
    };
    auto wait_mma = [&](int q) -> bool {
      if (!mma_pend[q]) return true;
      if (!mbar_wait(mb[q], mphase[q])) return false;
      mphase[q] ^= 1;
      mma_pend[q] = false;
      return true;
    };
    // digits of K half q (x-run run + 4 q of the half tile) to shared memory
    auto store_digits = [&](const uint4 (&d)[DIG], int q) {
      unsigned char* dst = sA + (row >> 3) * CORE_SBO + (run + 4 * q) * A2_LBO + (row & 7) * 16;
#pragma unroll
      for (int k = 0; k < DIG; ++k) *reinterpret_cast<uint4*>(dst + k * A2_PLANE) = d[k];
    };
    auto epilogue = [&](const Unit& u) {
      const int nj = min(NBLK, u.nJ - u.jb), P = nj <= 16 ? 16 : 32;
      const int quarter = warp & 3, g = warp >> 2, ng4 = GT2_CONV / 128;
      const int a = u.mb * MBLK + 32 * quarter + lane;
      const uint32_t lane_addr = tmem + ((uint32_t)(32 * quarter) << 16);
      const int ea0 = Aexp[u.ab][0][32 * quarter + lane] - 1022,
                ea1 = Aexp[u.ab][1][32 * quarter + lane] - 1022;
      // column pairs (c0, c0 + 1), c0 = 2 g, 2 g + 8, ...: one two-column
      // tensor-memory load per diagonal and half
#pragma unroll 1
      for (int c0 = 2 * g; c0 < nj; c0 += 2 * ng4) {
        // |D_d| < (d + 1) 2^21 (A digits up to 255, W digits up to 128 in
        // magnitude, 64 points): D_0, D_1 (< 2^22) by the 2^22 conversion on
        // the FP32 pipe, the others by the conversion unit (exact: integer
        // values below 2^24); D_0 256 + D_1 and D_2 256 + D_3 stay below 2^31
        if constexpr (DIG == 7) {
          long long s7[2][2];  // [half][column]
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t f[2][ND];
#pragma unroll
            for (int d = 0; d < ND; ++d) {
              uint32_t t[2];
              tmem_ld2(lane_addr + (uint32_t)(h * TMEM_HALF + d * P + c0), t);
              f[0][d] = t[0];
              f[1][d] = t[1];
            }
            tmem_wait_ld();
            s7[h][0] = combine7<8>(f[0]);
            s7[h][1] = combine7<8>(f[1]);
          }
          // sum_r x w = 2^(E_x + E_w - 63 + 8) s7
#pragma unroll
          for (int cc = 0; cc < 2; ++cc) {
            const int c = c0 + cc;
            if (c < nj && a < m) {
              const int w0 = Wexp[u.wb][0][c], w1 = Wexp[u.wb][1][c];
              const bool bad = ea0 + 1022 == EXP_NONFINITE || ea1 + 1022 == EXP_NONFINITE ||
                               w0 == EXP_NONFINITE || w1 == EXP_NONFINITE;
              partial[(size_t)(u.j0 + u.jb + c) * m + a] =
                  join7(s7[0][cc], ea0 + w0 - 1022 - 55, s7[1][cc], ea1 + w1 - 1022 - 55, bad);
            }
          }
        } else {
          long long acc[2][2];  // [half][column]
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t f[DIG][2];
#pragma unroll
            for (int d = 0; d < DIG; ++d)
              tmem_ld2(lane_addr + (uint32_t)(h * TMEM_HALF + d * P + c0), f[d]);
            tmem_wait_ld();
#pragma unroll
            for (int cc = 0; cc < 2; ++cc) {
              const int t01 = small_float_int(f[0][cc]) * 256 + small_float_int(f[1][cc]);
              const int t23 = __float2int_rz(__uint_as_float(f[2][cc])) * 256 +
                              __float2int_rz(__uint_as_float(f[3][cc]));
              acc[h][cc] = ((long long)t01 << 32) + ((long long)t23 << 16) +
                           ((long long)__float2int_rz(__uint_as_float(f[4][cc])) << 8) +
                           (long long)__float2int_rz(__uint_as_float(f[5][cc]));
            }
          }
          // sum_r x w = 2^(E_x + E_w - 55) acc; the two halves on the larger
          // scale (the other truncated at its unit, 2^-55 of that segment's
          // scale), one truncation
#pragma unroll
          for (int cc = 0; cc < 2; ++cc) {
            const int c = c0 + cc;
            if (c < nj) {
              const int e0 = ea0 + Wexp[u.wb][0][c] - 1022 - 55, e1 = ea1 + Wexp[u.wb][1][c] - 1022 - 55;
              const bool b0 = e0 >= e1;
              const int sh = min(b0 ? e0 - e1 : e1 - e0, 63);
              const long long s2 = (b0 ? acc[0][cc] : acc[1][cc]) + ((b0 ? acc[1][cc] : acc[0][cc]) >> sh);
              if (a < m) partial[(size_t)(u.j0 + u.jb + c) * m + a] = scaled_i64_rz_cvt(s2, b0 ? e0 : e1);
            }
          }
        }
      }
    };

    // post unit u (or the end, nj = 0) to the issuing thread: ring entry
    // seq & 1, then ready[0] (thread 0, after a converting-warp barrier)
    auto post = [&](int seq, int nj, int h) {
      if (tid == 0) {
        u_ring[seq & 1][0] = nj;
        u_ring[seq & 1][1] = h;
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(rb[0]) : "memory");
      }
    };

    if (ND > DIG) {  // the zero plane of both halves (blocks of NBLK = 16 alone)
      static_assert(ND == DIG || NBLK == 16, "one layout of the stack");
      for (int p = tid; p < 2 * 8 * NBLK; p += GT2_CONV) {
        const int r = DIG * NBLK + p % NBLK, rn = (p / NBLK) & 7, h = p / (8 * NBLK);
        *reinterpret_cast<uint4*>(sW + h * W_HALF + (r >> 3) * CORE_SBO + rn * (ND * NBLK * 16) +
                                  (r & 7) * 16) = make_uint4(0, 0, 0, 0);
      }
    }
    Unit cur;
    cur.wb = 0;
    cur.ab = 0;
    bool have_prev = false, fail = false;  // fail: uniform over the converting threads
    Unit prev = cur;
    int seq = 0;
    // Per unit two barriers of the converting warps: B1 once every thread
    // holds its values (the raw buffers may be refilled), B2 once the digits
    // of both K halves, a new W block and the exponents are in place (both K
    // halves are then posted).  The digit buffers are guarded per thread by
    // the MMA completion barriers, the A exponents double-buffered by A block.
    if (claim(cur)) {
      load_w(cur);
      if (!TMA) {
        raw_copy(cur);
      } else if (tid == TMA_TID) {
        tma_issue(cur, 0);
        tma_issue(cur, 1);
      }
      bool need_w = false;
      for (;;) {
        // both K halves of cur to registers; the row's exponent
        bool ok = true;
        if (TMA) {
          ok = wait_raw(0);
          ok = wait_raw(1) && ok;
        } else {
          cp_async_wait_all();
          __syncwarp();
        }
        double v[2][8];
        uint32_t emf = 0;  // largest exponent field (high-word bits 20..30) of the row segment
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            const double2 t = *reinterpret_cast<const double2*>(
                sR + q * RAW_KHALF + r_off + (((uint32_t)p << 4) ^ r_swz));
            v[q][2 * p] = t.x;
            v[q][2 * p + 1] = t.y;
            emf = max(emf, (uint32_t)__double2hiint(t.x) & 0x7FF00000u);
            emf = max(emf, (uint32_t)__double2hiint(t.y) & 0x7FF00000u);
          }
        emf = max(emf, __shfl_xor_sync(0xffffffffu, emf, 1));
        emf = max(emf, __shfl_xor_sync(0xffffffffu, emf, 2));
        const int em = (int)(emf >> 20);
        const uint32_t em_sh = DIG == 6 ? (em < 64 ? 0xF0000000u : emf + (5u << 20)) : emf;
        if (tid == 0) q_step();
        if (TMA && conv_sync_or(!ok)) {  // B1: both raw buffers consumed
          fail = true;
          break;
        }
        Unit next = cur;
        bool new_block = false;
        const bool has_next = advance(next, &new_block);  // may claim (uniform, syncs)
        if (!TMA) {
          if (has_next) raw_copy(next);
        } else if (tid == TMA_TID && has_next) {
          tma_issue(next, 0);
          tma_issue(next, 1);
        }
        // each K half's digits replace those prev's MMAs of that half read
        uint4 d[DIG];
        ok = wait_mma(0);
        digits8_u<DIG>(v[0], em_sh, d);
        store_digits(d, 0);
        ok = wait_mma(1) && ok;
        digits8_u<DIG>(v[1], em_sh, d);
        store_digits(d, 1);
        tc_fence_after();
        if (have_prev && prev.h == 1) epilogue(prev);  // all of prev's MMAs are done
        // a new W block: the MMAs that read the old one are done (waited
        // above) and its exponents sit in the other buffer
        if (need_w) load_w(cur);
        if (run == 0) Aexp[cur.ab][cur.h][row] = em;
        if (TMA || need_w || !have_prev) cp_async_wait_all();  // W's digits
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        if (conv_sync_or(!ok)) {  // B2: digits, W and exponents in place
          fail = true;
          break;
        }
        post(seq, min(NBLK, cur.nJ - cur.jb), cur.h);
        if (tid == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(rb[1]) : "memory");
        ++seq;
        mma_pend[0] = mma_pend[1] = true;
        prev = cur;
        have_prev = true;
        if (!has_next) break;
        need_w = new_block;
        cur = next;
      }
    }
    // the last unit's MMAs (bounded waits; the issuing thread has then taken
    // every posted unit), the end of the issuing loop, the last epilogue
    if (!fail) {
      bool ok = wait_mma(0);
      ok = wait_mma(1) && ok;
      fail = conv_sync_or(!ok);
    }
    post(seq, 0, 0);
    if (!fail) {
      tc_fence_after();
      if (have_prev && prev.h == 1) epilogue(prev);
    } else {
      // once more, bounded, before the tensor memory is freed
      for (int q = 0; q < 2; ++q)
        if (mma_pend[q]) mbar_wait(mb[q], mphase[q]);
      // loads still in flight land before the CTA's shared memory is released
      if (tid == TMA_TID)
        for (int q = 0; q < 2; ++q)
          if (tma_pending[q]) mbar_wait(tb[q], tphase[q]);
    }
    cp_async_wait_all();
    if (fail && tid == 0) s_fail = 1;
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && (s_fail || s_ifail)) atomicOr(status, SEA_FLAG_WAIT);
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TMEM_COLS));
  }
}

// ---------------------------------------------------------------------------
// A few rows of A (an operator applied to one or a handful of vectors): the
// kernel above works on 128 rows per unit whatever their number, so up to
// GRAM_FEW rows each warp takes 16 list entries of a tile against eight rows
// with the warp-wide mma.sync.m16n8k16 (FP16 operands, FP32 accumulators): W's
// digits straight from their global image as the A fragments, the rows'
// digits formed in registers as the B fragments.  The contraction index is
// permuted so that a thread's four fragment words are one 16-byte piece of
// the image.  Digits, diagonals and the final combination are those of
// k_gram_tc, every D_d the same exact integer, so the partials are the same
// bits.  Bound by the latency of its loads and conversions; 8 rows of 75^3
// against 128 orbitals 320 -> 35 us.  Three CTAs an SM (168 registers, 80 in
// k_expand_few; four spill, the registers left alone allow two) and the digits of
// one z-plane at a time: apply of 8 vectors on 75^3 141 -> 118 us mixed, 208 -> 162
// us plain.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                          uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// acc of the six diagonals (k_gram_tc's epilogue): sum_d D_d 256^(5-d)
__device__ __forceinline__ long long combine6(const uint32_t* f) {
  const int t01 = small_float_int(f[0]) * 256 + small_float_int(f[1]);
  const int t23 =
      __float2int_rz(__uint_as_float(f[2])) * 256 + __float2int_rz(__uint_as_float(f[3]));
  return ((long long)t01 << 32) + ((long long)t23 << 16) +
         ((long long)__float2int_rz(__uint_as_float(f[4])) << 8) +
         (long long)__float2int_rz(__uint_as_float(f[5]));
}
// two half tiles' sums on the larger scale, one truncation
__device__ __forceinline__ double join6(long long a0, int e0, long long a1, int e1) {
  const bool b0 = e0 >= e1;
  const int sh = min(b0 ? e0 - e1 : e1 - e0, 63);
  return scaled_i64_rz_cvt((b0 ? a0 : a1) + ((b0 ? a1 : a0) >> sh), b0 ? e0 : e1);
}

constexpr int FEW_WARPS = 4;
// Rows (GRAM_FEW) and vectors (EXPAND_FEW) up to which the warp-wide kernels are
// the faster ones.  Measured with six digits (seven): contraction of 8 and 32 rows
// of 75^3 against 128 orbitals 35 and 90 us (45, 129), of 33 rows of 76^3 on the
// other 177 (217); of 32 and 33 rows of 96^3 against 256 orbitals 211 and 323 (260,
// 397); expansion of 8 vectors 43 us (66), of 9 to 16 as much again, against 84 (91).
constexpr int GRAM_FEW = 32, EXPAND_FEW = 8;
template <int DIG>
__global__ void __launch_bounds__(32 * FEW_WARPS, 3)
    k_gram_few(const double* __restrict__ A, int m, TileGeom G, size_t ng, int t0, int n_tiles,
               const int* __restrict__ tptr, const uint4* __restrict__ wdig, int slot0,
               const int* __restrict__ wexp, double* __restrict__ partial) {
  constexpr int ND = GramSizes<DIG>::ND;
  const int T = t0 + blockIdx.x * FEW_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (T >= n_tiles) return;  // warp-uniform
  const int j0 = tptr[T], nJ = tptr[T + 1] - j0;
  if (nJ == 0) return;
  const int a0 = blockIdx.y * 8, g = lane >> 2, q = lane & 3;
  const int txi = T % G.ntx, tyi = (T / G.ntx) % G.nty, tzi = T / (G.ntx * G.nty);
  const int x0 = txi * TX, y = tyi * TY + q;
  long long acc0[4];  // the first half's integers, units and non-finite marks
  int e0[4];
  bool bad0[4];
  for (int s0 = 0; s0 < nJ; s0 += 16) {
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      // row a0 + g: x-runs y = q of the planes 2h, 2h + 1
      double v[2][8];
      uint32_t emf = 0;
#pragma unroll
      for (int qq = 0; qq < 2; ++qq) {
        const int z = tzi * TZ + 2 * h + qq;
        const bool in = a0 + g < m && y < G.ny && z < G.nz;
        const double* src = A + (in ? (size_t)(a0 + g) * ng + ((size_t)z * G.ny + y) * G.nx + x0 : 0);
#pragma unroll
        for (int x = 0; x < 8; ++x) {
          v[qq][x] = (in && x0 + x < G.nx) ? src[x] : 0.0;
          emf = max(emf, (uint32_t)__double2hiint(v[qq][x]) & 0x7FF00000u);
        }
      }
      emf = max(emf, __shfl_xor_sync(0xffffffffu, emf, 1));
      emf = max(emf, __shfl_xor_sync(0xffffffffu, emf, 2));
      const int em = (int)(emf >> 20);
      const uint32_t em_sh = DIG == 6 ? (em < 64 ? 0xF0000000u : emf + (5u << 20)) : emf;
      float c[ND][4];
#pragma unroll
      for (int k = 0; k < ND; ++k) c[k][0] = c[k][1] = c[k][2] = c[k][3] = 0.f;
      // entries s0 + g and s0 + g + 8 (zeros beyond the list)
      const bool in0 = s0 + g < nJ, in1 = s0 + g + 8 < nJ;
      const uint4* ws = wdig + ((size_t)(j0 - slot0 + s0) * 2 + h) * DIG * 8 + q;
      const uint4* w0 = ws + (in0 ? g : 0) * 2 * DIG * 8;
      const uint4* w1 = ws + (in1 ? g + 8 : 0) * 2 * DIG * 8;
#pragma unroll
      for (int qq = 0; qq < 2; ++qq) {  // the planes in turn: one's digits in registers
        uint4 d[DIG];
        digits8_u<DIG>(v[qq], em_sh, d);
        const uint4 z4 = make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int l = 0; l < DIG; ++l) {
          const uint4 u0 = in0 ? w0[l * 8 + 4 * qq] : z4, u1 = in1 ? w1[l * 8 + 4 * qq] : z4;
#pragma unroll
          for (int k = 0; k < DIG && k + l < ND; ++k) {
            mma_16816(c[k + l], u0.x, u1.x, u0.y, u1.y, d[k].x, d[k].y);
            mma_16816(c[k + l], u0.z, u1.z, u0.w, u1.w, d[k].z, d[k].w);
          }
        }
      }
      // c[d][i]: entry s0 + g + 8 (i / 2), row a0 + 2 q + (i & 1)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int s = s0 + g + 8 * (i >> 1), a = a0 + 2 * q + (i & 1);
        const int ea = __shfl_sync(0xffffffffu, em, 8 * q + 4 * (i & 1));
        const int ew = s < nJ ? wexp[(size_t)(j0 - slot0 + s) * 2 + h] : 0;
        uint32_t f[ND];
#pragma unroll
        for (int k = 0; k < ND; ++k) f[k] = __float_as_uint(c[k][i]);
        long long ac;
        if constexpr (DIG == 7)
          ac = combine7<8>(f);
        else
          ac = combine6(f);
        const int e = ea - 1022 + ew - 1022 - 55;
        const bool bad = ea == EXP_NONFINITE || ew == EXP_NONFINITE;
        if (h == 0) {
          acc0[i] = ac;
          e0[i] = e;
          bad0[i] = bad;
        }
        const double y0 = DIG == 7 ? join7(acc0[i], e0[i], ac, e, bad || bad0[i])
                                   : join6(acc0[i], e0[i], ac, e);
        if (h == 1 && s < nJ && a < m) partial[(size_t)(j0 + s) * m + a] = y0;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// The expansion y[v][r] = sign sum_j W[list(j)][r] H(j, v) on the tensor cores,
// per tile (M = the tile's 128 points, N = vectors, K = the tile's W list, at
// most XJ = 32 entries; longer lists go to the general kernels of ace.cu).  With
// six digits (mixed form; seven as in k_wx_digits):  scales: W's digits are taken per (tile, list entry j) with the
// exponent E_j of that W row on the tile (six balanced FP16 digits a_k,
// |a_k| <= 128, on the 2^-47 grid); H(j, v) is scaled exactly by 2^E_j and
// measured against one exponent E_v per (tile, vector v) over the list, its
// digits the unsigned bytes b_l of |H| 2^(E_j - E_v) on the 2^-48 grid with
// H's sign (as A's in the contraction), so
//   y = 2^(E_v) sum_d 2^(-15-8d) D_d,  D_d = sum_j sum_{k+l=d} a_k(j) b_l(j),
// E_j cancels and every D_d (at most 32 x 6 products of magnitude < 2^15)
// is an integer below 2^23, exact in the FP32 accumulator.  W's digits are
// formed once per W into a per-tile image in the K-major layout (two K steps
// of 16 list entries, six planes, 4 KB each); H's digits per chunk of 32
// vectors into a slot of a shared-memory ring with the six planes stacked
// along N, so one MMA of A plane k against planes 0..5-k adds plane k's
// products to diagonals k..5 (TMEM columns 32 d).  Two accumulator buffers
// of 192 columns: the MMAs of chunk c + 1 run while chunk c's epilogue reads
// its buffer back, and the digits of the following chunks are formed
// meanwhile by warps of their own.
// ---------------------------------------------------------------------------
constexpr int XJ = SEA_XJ, XKS = SEA_XKS, XN = 32;
constexpr uint32_t XA_BLOCK = MBLK * XKS * 2;          // 4 KB: one plane, one K step
constexpr uint32_t XA_LBO = (MBLK / 8) * 128;          // 2048
constexpr int XR = 4;                                  // ring slots (chunks of XN vectors)
template <int DIG>
struct ExpandSizes {  // with six digits
  static constexpr uint32_t XA_STEP = DIG * XA_BLOCK;       // 24 KB
  static constexpr uint32_t XA_TILE = 2 * XA_STEP;          // 48 KB
  static constexpr int ND = diagonals(DIG);
  static constexpr uint32_t XB_LBO = (ND * XN / 8) * 128;   // 3072
  static constexpr uint32_t XB_CHUNK = 2 * XB_LBO;          // 6 KB: 192 rows x 16 K
  static constexpr uint32_t XT_COLS = ND * XN;              // 192
  static constexpr uint32_t XS_SLOT = 2 * XB_CHUNK;         // 12 KB: both K steps of one chunk
  static constexpr size_t XE_SMEM = 2 * XA_TILE + XR * XS_SLOT + 128;
};

// W's digit image: CTA per tile (thread = point p), for tiles whose list has
// 1..XJ entries; only the K steps in use are stored, tile T's from step xoff[T]
// on (a step of every tile would be 448 bytes a grid point in the plain form,
// 60 GB at 512^3).  wx[step xoff[T]][(q 6 + k) 4096 + (p / 8) 128 + (jq / 8) 2048 +
// (p % 8) 16 + (jq % 8) 2] = digit k of W[list(16 q + jq)] at point p (zero
// outside the entry's sub-box and beyond the list), wxexp[slot] = E_j + 1022.
// Seven digits: the digits are those of W 2^(-E_j - e_p), e_p = wxpe[step][p] <= 0
// the point's largest exponent of W 2^(-E_j) over the list, so that points where
// all of W is small against the tile (an orbital's tail falls by 2^20 and more
// across a tile) keep their digits; exact, and e_p goes into the output's
// exponent.
template <int DIG>
__global__ void __launch_bounds__(MBLK)
    k_wx_digits(const double* __restrict__ W, TileGeom G, size_t ng, int n_tiles,
                const int* __restrict__ tptr, const int* __restrict__ tlist,
                const int* __restrict__ tsub, const int* __restrict__ xoff,
                uint4* __restrict__ wx, int* __restrict__ wxexp, int* __restrict__ wxpe) {
  constexpr uint32_t XA_STEP = ExpandSizes<DIG>::XA_STEP;
  const int T = blockIdx.x;
  const int j0 = tptr[T], nJ = tptr[T + 1] - j0;
  if (nJ == 0 || nJ > XJ) return;  // uniform
  __shared__ int emx[XJ];
  const int p = threadIdx.x;
  if (p < XJ) emx[p] = 0;
  const long long g = tile_point(G, T, p);
  const int pz = p / (TX * TY), py = (p / TX) % TY, px = p % TX;
  auto wval = [&](int jl) -> double {
    if (jl >= nJ || g < 0) return 0.0;
    const int sb = tsub[j0 + jl];
    const bool in = px >= (sb & 15) && px < ((sb >> 4) & 15) && py >= ((sb >> 8) & 15) &&
                    py < ((sb >> 12) & 15) && pz >= ((sb >> 16) & 15) && pz < ((sb >> 20) & 15);
    return in ? W[(size_t)tlist[j0 + jl] * ng + g] : 0.0;
  };
  __syncthreads();
  for (int jl = 0; jl < nJ; ++jl)
    atomicMax(&emx[jl], (int)((__double_as_longlong(wval(jl)) >> 52) & 0x7FF));
  __syncthreads();
  if (p < nJ) wxexp[j0 + p] = emx[p];
  int ep = 0;
  if (DIG == 7) {
    ep = INT_MIN;
    for (int jl = 0; jl < nJ; ++jl) {
      const int e = (int)((__double_as_longlong(wval(jl)) >> 52) & 0x7FF);
      if (e) ep = max(ep, e - emx[jl]);
    }
    if (ep == INT_MIN) ep = 0;  // no value
    wxpe[(size_t)xoff[T] * MBLK + p] = ep;
  }
  const int nq = (nJ + XKS - 1) / XKS;
  unsigned char* base = reinterpret_cast<unsigned char*>(wx) + (size_t)xoff[T] * XA_STEP;
  for (int grp = 0; grp < 2 * nq; ++grp) {  // 8 list entries at a time
    uint32_t pk[DIG][4];
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
      const int jl = 8 * grp + e;
      float f0[DIG], f1[DIG];
      digit_floats<DIG>(jl < nJ ? fixed_bal<DIG>(wval(jl), emx[jl] + ep) : 0, f0);
      digit_floats<DIG>(jl + 1 < nJ ? fixed_bal<DIG>(wval(jl + 1), emx[jl + 1] + ep) : 0, f1);
#pragma unroll
      for (int k = 0; k < DIG; ++k) pk[k][e / 2] = pack_f16(f0[k], f1[k]);
    }
    const int q = grp >> 1, jj = grp & 1;
#pragma unroll
    for (int k = 0; k < DIG; ++k)
      *reinterpret_cast<uint4*>(base + (q * DIG + k) * XA_BLOCK + (p >> 3) * 128 + jj * XA_LBO +
                                (p & 7) * 16) = make_uint4(pk[k][0], pk[k][1], pk[k][2], pk[k][3]);
  }
}

// E_v of the expansion for every (tile, vector): the largest biased
// exponent of H(j, v) 2^(E_j) over the tile's list (0 where all are zero);
// thread = vector, grid x = tile (grid y ends at 65535, a 204^3 grid has more
// tiles).  Tiles with an empty list or more than XJ entries are skipped (not
// read).  STRICT: EV_NONFINITE where a factor is not
// finite.
constexpr int EV_NONFINITE = 1 << 20;
template <bool STRICT>
__global__ void __launch_bounds__(128)
    k_expand_ev(const int* __restrict__ tptr, const int* __restrict__ tlist,
                const int* __restrict__ wxexp, const double* __restrict__ H, long long hj,
                long long hv, int m, int* __restrict__ ev) {
  const int T = blockIdx.x, v = blockIdx.y * 128 + threadIdx.x;
  const int j0 = tptr[T], nJ = tptr[T + 1] - j0;
  if (v >= m || nJ == 0 || nJ > XJ) return;
  int em = 0;
  for (int jl = 0; jl < nJ; ++jl) {
    const int e =
        (int)((__double_as_longlong(H[(long long)tlist[j0 + jl] * hj + (long long)v * hv]) >> 52) &
              0x7FF);
    if (e) em = max(em, e + wxexp[j0 + jl] - 1022);
    if (STRICT && (e == EXP_NONFINITE || wxexp[j0 + jl] == EXP_NONFINITE)) em = EV_NONFINITE;
  }
  ev[(size_t)T * m + v] = em;
}

constexpr int XE_WARPS = 16;                 // epilogue warps (tensor-memory read-back, stores)
constexpr int XP_WARPS = 8;                  // H-digit warps
constexpr int XE_ISSUER = XE_WARPS + XP_WARPS;           // the MMA-issuing warp
constexpr int XE_THREADS = 32 * (XE_ISSUER + 1);         // 800
constexpr int XF_FIRST = 1, XF_LAST = 2, XF_END = 4;    // slot flags

// Persistent CTAs (one per SM) over the tiles whose list has at most XJ
// entries, in three roles that run side by side.
//  * H-digit warps (XP_WARPS): claim the tiles, bring each tile's W digit
//    image in (bulk copy, two buffers), and for every chunk of XN = 32
//    vectors of the tile form E_v and H's digits into the next slot of a
//    ring of XR chunks, with the chunk's tile, first vector and E_v beside
//    it; a slot is refilled once its MMAs are done and the epilogue warps
//    have read its E_v.
//  * The issuing warp: per chunk, once its slot is full (and, at a tile's
//    first chunk, the tile's W image is in) and the accumulator buffer it
//    takes is free, the chunk's MMAs into one of two buffers of 192
//    tensor-memory columns, committed to that buffer's barrier, to the
//    slot's and, at a tile's last chunk, to the W image's.
//  * Epilogue warps (16): warp w reads tensor-memory lanes 32 (w % 4) back
//    for vectors 8 (w / 4) .. + 7 of each chunk, combines the diagonal sums
//    and stores the FP64 outputs; zero tiles (empty list) are stored as
//    zeros without MMAs.
// So the digits of the next chunks and the MMAs of the next chunk run while
// a chunk's outputs are being converted and stored.  H(j, v) = H[j hj + v
// hv]; out[v ng + r].  Every wait is bounded; on expiry the role stops, the
// others see s_fail (or expire themselves) and the kernel reports
// SEA_FLAG_WAIT after the MMAs and copies in flight are done.
template <int DIG>
__global__ void __launch_bounds__(XE_THREADS, 1)
    k_expand_tc(const uint4* __restrict__ wx, const int* __restrict__ wxexp,
                const int* __restrict__ wxpe, TileGeom G, size_t ng, int n_tiles, const int* __restrict__ tptr, const int* __restrict__ tlist,
                const int* __restrict__ xoff, const double* __restrict__ H, long long hj,
                long long hv, int m, int negate, double* __restrict__ out,
                const int* __restrict__ evp, int* __restrict__ queue,
                unsigned* __restrict__ status) {
  using Z = ExpandSizes<DIG>;
  constexpr int ND = Z::ND;
  static_assert(2 * Z::XT_COLS <= TMEM_COLS, "two accumulator buffers");
  constexpr uint32_t XA_STEP = Z::XA_STEP, XA_TILE = Z::XA_TILE, XB_LBO = Z::XB_LBO,
                     XB_CHUNK = Z::XB_CHUNK, XT_COLS = Z::XT_COLS, XS_SLOT = Z::XS_SLOT;
  extern __shared__ unsigned char xe_raw[];
  unsigned char* sA = xe_raw + ((128 - (smem_addr(xe_raw) & 127)) & 127);  // two tile images
  unsigned char* sS = sA + 2 * XA_TILE;                                     // XR chunk slots
  __shared__ int s_T[XR], s_nJ[XR], s_v0[XR], s_fl[XR], s_ab[XR], s_xo[XR];
  __shared__ __align__(16) int s_ev[XR][XN];
  __shared__ int p_lj[XJ], p_shj[XJ], p_tile;
  __shared__ __align__(8) unsigned long long bar_full[XR], bar_free[XR], bar_md[2], bar_tf[2],
      bar_a[2], bar_af[2], bar_fin;
  __shared__ uint32_t tmem_base;
  __shared__ volatile int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(&tmem_base)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int q = 0; q < XR; ++q) {
      mbar_init(smem_addr(&bar_full[q]), XP_WARPS);
      mbar_init(smem_addr(&bar_free[q]), 1 + XE_WARPS);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(smem_addr(&bar_md[q]), 1);
      mbar_init(smem_addr(&bar_tf[q]), XE_WARPS);
      mbar_init(smem_addr(&bar_a[q]), 1);
      mbar_init(smem_addr(&bar_af[q]), 1);
    }
    mbar_init(smem_addr(&bar_fin), 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
    s_fail = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  const uint32_t a_base = smem_addr(sA), s_base = smem_addr(sS);
  const int nch = (m + XN - 1) / XN;  // chunks per tile

  if (warp >= XE_WARPS && warp < XE_ISSUER) {
    // ---- H-digit warps: lane = vector of the chunk, warp pw = list entries
    // jp pw .. jp pw + jp - 1 with jp = 2 nq (so every warp has work) ----
    const int pw = warp - XE_WARPS, ptid = tid - 32 * XE_WARPS;
    auto pbar = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(32 * XP_WARPS) : "memory"); };
    auto pbar_or = [&](bool v) -> bool {
      uint32_t r;
      asm volatile(
          "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.or.pred q, 1, %2, p;\n"
          "selp.u32 %0, 1, 0, q;\n}\n"
          : "=r"(r)
          : "r"((uint32_t)v), "n"(32 * XP_WARPS)
          : "memory");
      return r != 0;
    };
    if (ND > DIG)  // the zero plane of every slot and K step: 32 rows of two core matrices
      for (int z = ptid; z < XR * 2 * 2 * XN; z += 32 * XP_WARPS) {
        const int row = DIG * XN + z % XN, jj = (z / XN) & 1, st = z / (2 * XN);
        *reinterpret_cast<uint4*>(sS + st * XB_CHUNK + jj * XB_LBO + (row >> 3) * 128 +
                                  (row & 7) * 16) = make_uint4(0, 0, 0, 0);
      }
    int pseq = 0, tseq = 0;               // chunks published; tiles whose W image was loaded
    uint32_t a_pend = 0, a_par = 0;       // ptid 0, bit b: a load into image buffer b was
                                          // issued; the parity of its completion
    bool fail = false;
    for (;;) {
      if (ptid == 0) {
        int t;
        do {
          t = atomicAdd(queue, 1);
        } while (t < n_tiles && tptr[t + 1] - tptr[t] > XJ);
        p_tile = t;
      }
      pbar();
      const int T = p_tile;
      const bool end = T >= n_tiles;
      const int j0 = end ? 0 : tptr[T], nJ = end ? 0 : tptr[T + 1] - j0;
      const int nq = (nJ + XKS - 1) / XKS, ab = tseq & 1, jp = 2 * nq, jb = jp * pw;
      const int xo = nJ > 0 ? xoff[T] : 0;
      if (ptid < nJ) {
        p_lj[ptid] = tlist[j0 + ptid];
        p_shj[ptid] = wxexp[j0 + ptid] - 1022;
      }
      bool ok = true;
      if (ptid == 0 && nJ > 0) {
        // the image buffer is free once the MMAs of the tile two back are done
        if (tseq >= 2) ok = mbar_wait(smem_addr(&bar_af[ab]), (uint32_t)(((tseq - 2) >> 1) & 1));
        if (ok) {
          const uint32_t bytes = (uint32_t)nq * XA_STEP;
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          mbar_expect_tx(smem_addr(&bar_a[ab]), bytes);
          bulk_load(a_base + ab * XA_TILE,
                    reinterpret_cast<const unsigned char*>(wx) + (size_t)xo * XA_STEP, bytes,
                    smem_addr(&bar_a[ab]));
          a_pend |= 1u << ab;
          a_par = (a_par & ~(1u << ab)) | ((uint32_t)((tseq >> 1) & 1) << ab);
        }
      }
      if (pbar_or(!ok || s_fail)) {  // p_lj, p_shj visible
        fail = true;
        break;
      }
      // H(j, v) of this thread's entries for chunk c (sign folded in), zero
      // beyond the list and the vectors, and E_v of the chunk's vector
      auto load_h = [&](int c, double (&h)[4], int& ev) {
        const int v = c * XN + lane;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int jl = jb + i;
          h[i] = (i < jp && v < m && jl < nJ) ? H[(long long)p_lj[jl] * hj + (long long)v * hv] : 0.0;
          if (negate)  // the sign of y folded into H's digits (sign bit, exact)
            h[i] = __longlong_as_double(__double_as_longlong(h[i]) ^ (long long)0x8000000000000000ULL);
        }
        ev = v < m ? evp[(size_t)T * m + v] : 0;
      };
      // chunk c from the values in h (the next chunk's values are loaded into
      // hn meanwhile: two register sets used in turn, so nothing waits on
      // those loads before the next chunk).  The warps of this role do not
      // wait on one another here: each waits for the slot itself and
      // arrives on its full barrier; a warp whose wait expired (wfail) skips
      // the rest of the tile's chunks and the role stops at the tile's end.
      bool wfail = false;
      auto chunk = [&](int c, double (&h)[4], int ev, double (&hn)[4], int& evn) {
        const int slot = pseq % XR, use = pseq / XR;
        ++pseq;
        if (wfail) return;
        // the slot is free once its previous chunk's MMAs are done and its
        // E_v was read
        bool ok = true;
        if (lane == 0) {
          if (use >= 1) ok = mbar_wait(smem_addr(&bar_free[slot]), (uint32_t)((use - 1) & 1));
          ok = ok && !s_fail;
        }
        if (!__shfl_sync(0xffffffffu, ok, 0)) {  // the same decision in every lane
          wfail = true;
          return;
        }
        if (nJ > 0) {
          if (c + 1 < nch) load_h(c + 1, hn, evn);
          if (pw == 0) s_ev[slot][lane] = ev;
          uint32_t pk[DIG][2];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int jl = jb + 2 * e;
            digits2_u<DIG>(h[2 * e], h[2 * e + 1], jl < nJ ? ev - p_shj[jl] : 0,
                           jl + 1 < nJ ? ev - p_shj[jl + 1] : 0, pk, e);
          }
          // entries jb.. of K step jb / 16: core matrix (jb / 8) % 2, bytes
          // (jb % 8) 2 of its 16-byte rows
          unsigned char* dst = sS + slot * XS_SLOT + (jb >> 4) * XB_CHUNK +
                               ((jb >> 3) & 1) * XB_LBO + (jb & 7) * 2;
#pragma unroll
          for (int l = 0; l < DIG; ++l) {
            const int row = l * XN + lane;
            unsigned char* q = dst + (row >> 3) * 128 + (row & 7) * 16;
            if (jp == 4)
              *reinterpret_cast<uint2*>(q) = make_uint2(pk[l][0], pk[l][1]);
            else
              *reinterpret_cast<uint32_t*>(q) = pk[l][0];
          }
        }
        if (ptid == 0) {
          s_T[slot] = T;
          s_nJ[slot] = nJ;
          s_v0[slot] = c * XN;
          s_fl[slot] = end ? XF_END : ((c == 0 ? XF_FIRST : 0) | (c == nch - 1 ? XF_LAST : 0));
          s_ab[slot] = ab;
          if (DIG == 7) s_xo[slot] = xo;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // digits -> tensor core
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&bar_full[slot])) : "memory");
      };
      double hA[4], hB[4];
      int eA = 0, eB = 0;
      if (nJ > 0) load_h(0, hA, eA);
      const int nc = end ? 1 : nch;
      for (int c = 0; c < nc; c += 2) {
        chunk(c, hA, eA, hB, eB);
        if (c + 1 < nc) chunk(c + 1, hB, eB, hA, eA);
      }
      fail = pbar_or(wfail);  // every thread is done with this tile's lists
      if (fail || end) break;
      if (nJ > 0) ++tseq;
    }
    // image loads in flight land before the shared memory is released
    if (ptid == 0)
      for (int b = 0; b < 2; ++b)
        if ((a_pend >> b) & 1u) mbar_wait(smem_addr(&bar_a[b]), (a_par >> b) & 1u);
    if (fail) s_fail = 1;
  } else if (warp == XE_ISSUER) {
    // ---- the issuing warp ----
    if (lane == 0) {
      bool fail = false;
      long long cgm = 0;  // chunks with MMAs so far
      int tcount = 0;     // tiles with MMAs started
      for (int seq = 0;; ++seq) {
        const int slot = seq % XR, use = seq / XR;
        if (s_fail || !mbar_wait(smem_addr(&bar_full[slot]), (uint32_t)(use & 1))) {
          fail = true;
          break;
        }
        const int fl = s_fl[slot], nJ = s_nJ[slot], ab = s_ab[slot];
        if (fl & XF_END) break;
        if (nJ == 0) {
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&bar_free[slot])) : "memory");
          continue;
        }
        if (fl & XF_FIRST) {
          if (!mbar_wait(smem_addr(&bar_a[ab]), (uint32_t)((tcount >> 1) & 1))) {
            fail = true;
            break;
          }
          ++tcount;
        }
        const int tb = (int)(cgm & 1);
        const long long u = cgm >> 1;
        if (u >= 1 && !mbar_wait(smem_addr(&bar_tf[tb]), (uint32_t)((u - 1) & 1))) {
          fail = true;
          break;
        }
        tc_fence_after();
        const int nq = (nJ + XKS - 1) / XKS;
        const uint32_t dcol = tmem + (uint32_t)(tb * XT_COLS);
        for (int qq = 0; qq < nq; ++qq)
#pragma unroll
          for (int k = 0; k < DIG; ++k) {
            const uint64_t a = sdesc(a_base + ab * XA_TILE + qq * XA_STEP + k * XA_BLOCK, XA_LBO, 128);
            const uint64_t b = sdesc(s_base + slot * XS_SLOT + qq * XB_CHUNK, XB_LBO, 128);
            mma_kf16(dcol + (uint32_t)(k * XN), a, b, idesc_kf16((ND - k) * XN, MBLK, false),
                     (k > 0 || qq > 0) ? 1u : 0u);
          }
        mma_commit(smem_addr(&bar_md[tb]));
        mma_commit(smem_addr(&bar_free[slot]));
        if (fl & XF_LAST) mma_commit(smem_addr(&bar_af[ab]));
        ++cgm;
      }
      // every MMA issued is done before the tensor memory is freed
      mma_commit(smem_addr(&bar_fin));
      mbar_wait(smem_addr(&bar_fin), 0);
      if (fail) s_fail = 1;
    }
    __syncwarp();
  } else {
    // ---- epilogue warps ----
    const int p = 32 * (warp & 3) + lane;  // tensor-memory lane = point of the tile
    const int vv0 = 8 * (warp >> 2);
    const uint32_t lane_q = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)vv0;
    long long cgm = 0, g = -1;
    int lastT = -1, ep = 0;  // seven digits: the point's exponent
    bool fail = false;
    for (int seq = 0;; ++seq) {
      const int slot = seq % XR, use = seq / XR;
      bool ok = !s_fail && mbar_wait(smem_addr(&bar_full[slot]), (uint32_t)(use & 1));
      if (!__all_sync(0xffffffffu, ok)) {
        fail = true;
        break;
      }
      const int fl = s_fl[slot], nJ = s_nJ[slot], T = s_T[slot], v0 = s_v0[slot];
      const int4 e4[2] = {*reinterpret_cast<const int4*>(&s_ev[slot][vv0]),
                          *reinterpret_cast<const int4*>(&s_ev[slot][vv0 + 4])};
      const int xo = DIG == 7 ? s_xo[slot] : 0;
      __syncwarp();
      if (fl & XF_END) break;
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&bar_free[slot])) : "memory");
      if (T != lastT) {
        g = tile_point(G, T, p);
        lastT = T;
        if (DIG == 7) ep = nJ > 0 ? wxpe[(size_t)xo * MBLK + p] : 0;
      }
      const int vbase = v0 + vv0;  // this warp's first vector of the chunk
      double* o = out + (size_t)vbase * ng + (g >= 0 ? g : 0);
      const bool full = vbase + 8 <= m;
      if (nJ > 0) {
        const int tb = (int)(cgm & 1);
        ok = mbar_wait(smem_addr(&bar_md[tb]), (uint32_t)((cgm >> 1) & 1));
        if (!__all_sync(0xffffffffu, ok)) {
          fail = true;
          break;
        }
        ++cgm;
        tc_fence_after();
        const uint32_t la = lane_q + (uint32_t)(tb * XT_COLS);
        const int ev[8] = {e4[0].x, e4[0].y, e4[0].z, e4[0].w, e4[1].x, e4[1].y, e4[1].z, e4[1].w};
        const bool wide = nJ > XKS;
        // four vectors at a time: six diagonal sums each
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          uint32_t f[ND][4];
#pragma unroll
          for (int d = 0; d < ND; ++d) tmem_ld4(la + (uint32_t)(d * XN + 4 * hh), f[d]);
          tmem_wait_ld();
          if (hh == 1) {  // the buffer is read: the next MMAs may overwrite it
            tc_fence_before();
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&bar_tf[tb])) : "memory");
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            double val;
            if constexpr (DIG == 7) {
              uint32_t fd[ND];
#pragma unroll
              for (int d = 0; d < ND; ++d) fd[d] = f[d][u];
              const int e = ev[4 * hh + u];
              val = e >= EV_NONFINITE ? quiet_nan()
                                      : scaled_i64_rn_cvt(combine7<6>(fd), e + ep - 1022 - 63 + 6);
            } else {
              // sum_d D_d 256^(5 - d) in three 32-bit pairs; |D_d| < 2^22 except
              // D_4 and D_5 of lists longer than 16 (below 2^23): those by the
              // conversion instruction
              const int t01 = small_float_int(f[0][u]) * 256 + small_float_int(f[1][u]);
              const int t23 = small_float_int(f[2][u]) * 256 + small_float_int(f[3][u]);
              const int d4 = wide ? __float2int_rz(__uint_as_float(f[4][u])) : small_float_int(f[4][u]);
              const int d5 = wide ? __float2int_rz(__uint_as_float(f[5][u])) : small_float_int(f[5][u]);
              const int t45 = d4 * 256 + d5;
              const long long base = ((long long)t01 << 32) + (long long)t45;
              const long long acc = base + (long long)t23 * 65536LL;
              val = scaled_i64_rz_cvt(acc, ev[4 * hh + u] - 1022 - 55);
            }
            if (g >= 0 && (full || vbase + 4 * hh + u < m)) o[(size_t)(4 * hh + u) * ng] = val;
          }
        }
      } else if (g >= 0) {
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (full || vbase + u < m) o[(size_t)u * ng] = 0.0;
      }
    }
    if (fail && lane == 0) s_fail = 1;
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && s_fail) atomicOr(status, SEA_FLAG_WAIT);
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TMEM_COLS));
  }
}

// The expansion for a few vectors, the counterpart of k_gram_few: CTA per
// tile, warp w the points 16 w .. + 15 against eight vectors, W's image as the
// A fragments, H's digits formed in registers as the B fragments, E_v over the
// tile's list by the warp itself.  The outputs are k_expand_tc's bits.
template <int DIG>
__global__ void __launch_bounds__(256, 3)
    k_expand_few(const uint4* __restrict__ wx, const int* __restrict__ wxexp,
                 const int* __restrict__ wxpe, TileGeom G, size_t ng, const int* __restrict__ tptr, const int* __restrict__ tlist,
                 const int* __restrict__ xoff, const double* __restrict__ H, long long hj,
                 long long hv, int m, int negate, double* __restrict__ out) {
  constexpr uint32_t XA_STEP = ExpandSizes<DIG>::XA_STEP;
  constexpr int ND = ExpandSizes<DIG>::ND;
  const int T = blockIdx.x, v0 = blockIdx.y * 8;
  const int j0 = tptr[T], nJ = tptr[T + 1] - j0, x0 = xoff[T];
  if (nJ > XJ) return;  // uniform: the long-list kernel's
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3, p0 = 16 * (threadIdx.x >> 5);
  const long long o0 = tile_point(G, T, p0 + g), o1 = tile_point(G, T, p0 + g + 8);
  int ep[2] = {0, 0};  // the points' exponents
  if (DIG == 7 && nJ > 0)
    for (int i = 0; i < 2; ++i) ep[i] = wxpe[(size_t)x0 * MBLK + p0 + g + 8 * i];
  float c[ND][4];
#pragma unroll
  for (int k = 0; k < ND; ++k) c[k][0] = c[k][1] = c[k][2] = c[k][3] = 0.f;
  // entries j = 16 s + {2q, 2q + 1, 8 + 2q, 9 + 2q} of vector v0 + g
  double hval[2][4];
  int sh[2][4], em = 0;
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int j = 16 * s + 2 * q + (i & 1) + 8 * (i >> 1);
      const bool in = j < nJ && v0 + g < m;
      double h = in ? H[(long long)tlist[j0 + j] * hj + (long long)(v0 + g) * hv] : 0.0;
      const int e = (__double2hiint(h) >> 20) & 0x7FF, w = j < nJ ? wxexp[j0 + j] : 0;
      if (e) em = max(em, e + w - 1022);
      if (DIG == 7 && in && (e == EXP_NONFINITE || w == EXP_NONFINITE)) em = EV_NONFINITE;
      if (negate) h = __longlong_as_double(__double_as_longlong(h) ^ (long long)0x8000000000000000ULL);
      hval[s][i] = h;
      sh[s][i] = j < nJ ? w - 1022 : INT_MIN;
    }
  em = max(em, __shfl_xor_sync(0xffffffffu, em, 1));
  em = max(em, __shfl_xor_sync(0xffffffffu, em, 2));
  const unsigned char* base = reinterpret_cast<const unsigned char*>(wx) + (size_t)x0 * XA_STEP;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    if (16 * s >= nJ) break;  // uniform
    uint32_t pk[DIG][2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int s0 = sh[s][2 * e], s1 = sh[s][2 * e + 1];
      digits2_u<DIG>(hval[s][2 * e], hval[s][2 * e + 1], s0 != INT_MIN ? em - s0 : 0,
                     s1 != INT_MIN ? em - s1 : 0, pk, e);
    }
#pragma unroll
    for (int k = 0; k < DIG; ++k) {
      const unsigned char* a = base + (s * DIG + k) * XA_BLOCK + (p0 >> 3) * 128 + g * 16 + q * 4;
      auto word = [&](uint32_t off) { return __ldg(reinterpret_cast<const uint32_t*>(a + off)); };
      const uint32_t a0 = word(0), a1 = word(128), a2 = word(XA_LBO), a3 = word(XA_LBO + 128);
#pragma unroll
      for (int l = 0; l < DIG && k + l < ND; ++l)
        mma_16816(c[k + l], a0, a1, a2, a3, pk[l][0], pk[l][1]);
    }
  }
  // c[d][i]: point p0 + g + 8 (i / 2), vector v0 + 2 q + (i & 1)
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int v = v0 + 2 * q + (i & 1);
    const long long o = i < 2 ? o0 : o1;
    const int ev = __shfl_sync(0xffffffffu, em, 8 * q + 4 * (i & 1));
    uint32_t f[ND];
#pragma unroll
    for (int k = 0; k < ND; ++k) f[k] = __float_as_uint(c[k][i]);
    double val;
    if constexpr (DIG == 7)
      val = ev >= EV_NONFINITE
                ? quiet_nan()
                : scaled_i64_rn_cvt(combine7<6>(f), ev + ep[i >> 1] - 1022 - 63 + 6);
    else
      val = scaled_i64_rz_cvt(combine6(f), ev - 1022 - 55);
    if (nJ == 0) val = 0.0;
    if (o >= 0 && v < m) out[(size_t)v * ng + o] = val;
  }
}

}  // namespace


size_t w_digits_bytes(long long slots, int digits) {
  return (size_t)std::max(slots, 1LL) * 2 * digits * 8 * sizeof(uint4) +
         (size_t)std::max(slots, 1LL) * 2 * sizeof(int);
}
static int* w_digits_exp(const void* wbuf, long long slots, int digits) {
  return (int*)((uint4*)wbuf + (size_t)std::max(slots, 1LL) * 2 * digits * 8);
}

cudaError_t launch_w_digits(cudaStream_t st, const double* W, const TileGeom& G, size_t ng,
                            int2 a, int2 b, int max_list, const int* tptr, const int* tlist,
                            void* wbuf, int digits) {
  if (b.x <= a.x || max_list <= 0) return cudaSuccess;
  const int ngroups = (max_list + 7) / 8;
  const long long warps = (long long)(b.x - a.x) * 2 * ngroups;
  (digits == 7 ? k_w_digits<7> : k_w_digits<6>)<<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(
      W, G, ng, a.x, b.x - a.x, a.y, ngroups, tptr, tlist, (uint4*)wbuf,
      w_digits_exp(wbuf, b.y - a.y, digits));
  return cudaGetLastError();
}

// cuTensorMapEncodeTiled from the driver, looked up once through the
// runtime (no link-time dependence on the driver library).
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}

// The 4D view (x, y, z, row) of A for the tensor-memory-accelerator path;
// false where it does not apply (odd nx: rows not 16-byte strided; A not
// 16-byte aligned; no driver entry point).
static bool make_a_map(const double* A, int m, const TileGeom& G, CUtensorMap* map) {
  if ((G.nx & 1) || (((uintptr_t)A) & 15)) return false;
  EncodeTiledFn fn = encode_tiled();
  if (!fn) return false;
  const cuuint64_t dim[4] = {(cuuint64_t)G.nx, (cuuint64_t)G.ny, (cuuint64_t)G.nz, (cuuint64_t)m};
  const cuuint64_t stride[3] = {(cuuint64_t)G.nx * 8, (cuuint64_t)G.nx * G.ny * 8,
                                (cuuint64_t)G.nx * G.ny * G.nz * 8};
  const cuuint32_t box[4] = {TX, TY, 1, MBLK};
  const cuuint32_t estride[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 4, (void*)A, dim, stride, box, estride,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static size_t xa_step(int digits) {
  return digits == 7 ? ExpandSizes<7>::XA_STEP : ExpandSizes<6>::XA_STEP;
}
// Images, the list entries' exponents and the points' (per K step, seven digits).
size_t wx_digits_bytes(long long steps, long long slots, int digits) {
  return (size_t)steps * xa_step(digits) +
         ((size_t)std::max(slots, 1LL) + (digits == 7 ? (size_t)steps * MBLK : 0)) * sizeof(int);
}
static int* wx_exp(const void* wxbuf, long long steps, int digits) {
  return (int*)((unsigned char*)wxbuf + (size_t)steps * xa_step(digits));
}

cudaError_t launch_wx_digits(cudaStream_t st, const double* W, const TileGeom& G, size_t ng,
                             int n_tiles, const int* tptr, const int* tlist, const int* tsub,
                             const int* xoff, long long steps, long long slots, void* wxbuf,
                             int digits) {
  if (n_tiles <= 0) return cudaSuccess;
  int* wxexp = wx_exp(wxbuf, steps, digits);
  (digits == 7 ? k_wx_digits<7> : k_wx_digits<6>)<<<n_tiles, MBLK, 0, st>>>(
      W, G, ng, n_tiles, tptr, tlist, tsub, xoff, (uint4*)wxbuf, wxexp,
      wxexp + std::max(slots, 1LL));
  return cudaGetLastError();
}

template <int DIG>
static cudaError_t expand_tc(cudaStream_t st, int device, const void* wxbuf, const TileGeom& G,
                             size_t ng, int n_tiles, const int* tptr, const int* tlist,
                             const int* xoff, long long steps, long long slots, const double* H,
                             long long hj, long long hv, int m, bool negate, double* out, int* evbuf,
                             int* queue, unsigned* status) {
  constexpr size_t smem = ExpandSizes<DIG>::XE_SMEM;
  cudaError_t e =
      cudaFuncSetAttribute(k_expand_tc<DIG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (n_tiles <= 0 || m <= 0) return cudaSuccess;
  const uint4* wx = (const uint4*)wxbuf;
  const int* wxexp = wx_exp(wxbuf, steps, DIG);
  const int* wxpe = wxexp + std::max(slots, 1LL);
  if (m <= EXPAND_FEW) {
    k_expand_few<DIG><<<dim3(n_tiles, (m + 7) / 8), 256, 0, st>>>(wx, wxexp, wxpe, G, ng, tptr, tlist,
                                                                  xoff, H, hj, hv, m, negate ? 1 : 0, out);
    return cudaGetLastError();
  }
  int nsm = 0;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, device);
  e = cudaMemsetAsync(queue, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  k_expand_ev<DIG == 7><<<dim3(n_tiles, (m + 127) / 128), 128, 0, st>>>(tptr, tlist, wxexp, H, hj,
                                                                       hv, m, evbuf);
  k_expand_tc<DIG><<<std::min(nsm, n_tiles), XE_THREADS, smem, st>>>(
      wx, wxexp, wxpe, G, ng, n_tiles, tptr, tlist, xoff, H, hj, hv, m, negate ? 1 : 0, out, evbuf,
      queue, status);
  return cudaGetLastError();
}

cudaError_t launch_expand_tc(cudaStream_t st, int device, const void* wxbuf, const TileGeom& G,
                             size_t ng, int n_tiles, const int* tptr, const int* tlist,
                             const int* xoff, long long steps, long long slots, const double* H,
                             long long hj, long long hv, int m, bool negate, double* out, int* evbuf,
                             int* queue, unsigned* status, int digits) {
  return (digits == 7 ? expand_tc<7> : expand_tc<6>)(st, device, wxbuf, G, ng, n_tiles, tptr, tlist,
                                                     xoff, steps, slots, H, hj, hv, m, negate, out, evbuf,
                                                     queue, status);
}

template <int DIG>
static cudaError_t gram_tc(cudaStream_t st, int device, const double* A, int m, const TileGeom& G,
                           size_t ng, int2 a, int2 b, const int* tptr, const void* wbuf,
                           double* partial, int* queue, unsigned* status) {
  constexpr size_t smem = GramTmaSizes<DIG>::SMEM;
  static_assert(smem <= 232448 - 4096, "shared memory of an SM");
  const uint4* wdig = (const uint4*)wbuf;
  const int* wexp = w_digits_exp(wbuf, b.y - a.y, DIG);
  const int n_tiles = b.x - a.x;
  if (n_tiles <= 0) return cudaSuccess;
  if (m <= GRAM_FEW) {
    k_gram_few<DIG><<<dim3((n_tiles + FEW_WARPS - 1) / FEW_WARPS, (m + 7) / 8), 32 * FEW_WARPS, 0, st>>>(
        A, m, G, ng, a.x, b.x, tptr, wdig, a.y, wexp, partial);
    return cudaGetLastError();
  }
  int nsm = 0;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, device);
  alignas(64) CUtensorMap map;
  memset(&map, 0, sizeof(map));
  const bool tma = make_a_map(A, m, G, &map);
  auto kern = tma ? k_gram_tc<DIG, true> : k_gram_tc<DIG, false>;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) e = cudaMemsetAsync(queue, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  kern<<<std::min(nsm, n_tiles), GT2_THREADS, smem, st>>>(
      map, A, ng, m, G, a.x, b.x, tptr, wdig, a.y, wexp, partial, queue, status);
  return cudaGetLastError();
}

cudaError_t launch_gram_tc(cudaStream_t st, int device, const double* A, int m, const TileGeom& G,
                           size_t ng, int2 a, int2 b, const int* tptr, const void* wbuf,
                           double* partial, int* queue, unsigned* status, int digits) {
  return (digits == 7 ? gram_tc<7> : gram_tc<6>)(st, device, A, m, G, ng, a, b, tptr, wbuf, partial,
                                                 queue, status);
}

}  // namespace sea
