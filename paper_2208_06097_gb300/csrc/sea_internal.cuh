// sea_internal.cuh -- device helpers and the context of the GB300 exx engine.
//
// Everything here belongs to the CUDA library (libsea.so).  It is written
// from the paper's equations; nothing is shared with the CPU oracle.
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>

#include <algorithm>
#include <cstddef>
#include <map>
#include <mutex>
#include <utility>
#include <vector>

#include "../../include/sea.h"

#define SEA_LMAX 6
#define SEA_NQ ((SEA_LMAX + 1) * (SEA_LMAX + 1))
// monomials x^a y^b z^c with a + b + c <= SEA_LMAX
#define SEA_NMONO ((SEA_LMAX + 1) * (SEA_LMAX + 2) * (SEA_LMAX + 3) / 6)
// per pair: the moments Qs (SEA_NQ), then the multipole potential's
// coefficients in the Kelvin-inverted variables (SEA_NMONO)
#define SEA_QSTRIDE (SEA_NQ + SEA_NMONO)
#define SEA_FDP 6  // stencil half width: O(h^12) second difference (App. C)

// Status bits written by kernels (device word, read back by the host).
#define SEA_FLAG_CG_CAP 1u
#define SEA_FLAG_NOT_PD 2u
#define SEA_FLAG_BOUNDS 4u
#define SEA_FLAG_NONFINITE 8u
#define SEA_FLAG_WAIT 16u  // a bounded wait on a tensor-core completion expired
#define SEA_FLAG_TIMEOUT 32u  // the CG's time budget (sea_params.timeout_ms) was spent
#define SEA_FLAG_NORM 64u     // an orbital's norm is off 1 by more than orth_tol

// Slot (in doubles) of E_xx^ACE in the context's exx_dev buffer (the first
// five hold sea_apply_vxx's E_xx and CG statistics).
#define SEA_EXX_ACE_SLOT 6

// At most this many chunks per pipelined host-buffer call.
#define SEA_XCHUNKS_MAX 64

namespace sea {

// NVTX ranges of an entry point and its stages, for timeline tools (Nsight
// Systems, or ncu's --nvtx filters); without an attached tool each push and
// pop is a test of one function pointer.  The ranges mark where the host
// enqueues each stage's launches; the stage times on the device are the
// CUDA-event times in sea_stats.  stage() closes the previous stage's range
// and opens the next; the destructor closes the open stage and the call.
struct Trace {
  explicit Trace(const char* call) { nvtxRangePushA(call); }
  void stage(const char* name) {
    if (open) nvtxRangePop();
    nvtxRangePushA(name);
    open = true;
  }
  ~Trace() {
    if (open) nvtxRangePop();
    nvtxRangePop();
  }
  Trace(const Trace&) = delete;
  Trace& operator=(const Trace&) = delete;
  bool open = false;
};

__host__ __device__ inline int wrapi(int x, int n) {
  int r = x % n;
  return r < 0 ? r + n : r;
}

__host__ __device__ inline int lmi(int l, int m) { return l * l + l + m; }

// Position of x^a y^b z^c among the SEA_NMONO monomials (a-major, then b,
// then c), the layout of the potential's coefficients.
__host__ __device__ constexpr int mono_k(int a, int b, int c) {
  int k = 0;
  for (int i = 0; i < a; ++i) k += (SEA_LMAX - i + 1) * (SEA_LMAX - i + 2) / 2;
  for (int j = 0; j < b; ++j) k += SEA_LMAX - a - j + 1;
  return k + c;
}

// Real solid harmonics in a rescaled basis D_lm = C_lm / kappa_lm, where
// C_lm are the Racah-normalized real regular solid harmonics
// (C_l0 = r^l P_l(cos theta)).  The scaling is chosen so that the
// recurrences carry no per-term normalization:
//   D_00 = 1, D_11 = x, D_1-1 = y,
//   D_{l+1,l+1} = x D_ll - y D_l,-l,   D_{l+1,-(l+1)} = y D_ll + x D_l,-l,
//   D_{l+1,m} = z D_lm - gam_lm r^2 D_{l-1,m}   (|m| <= l; no second term
//                                                 when |m| = l).
// With Q_lm = sum rho C_lm dV the multipole potential of Eq. me is
//   v(r) = sum_lm Q_lm C_lm(r) / r^(2l+1)
// (the orthonormal form 4 pi Q Y / ((2l+1) r^(l+1)), the (2l+1)/(4 pi)
// normalization folded into C).  Kelvin inversion, u = r / r^2, gives
// C_lm(r) / r^(2l+1) = C_lm(u) / r, so
//   v(r) = (1/r) sum_lm Qs_lm D_lm(u),   Qs_lm = kappa_lm^2 sum rho D_lm dV,
// the D_lm(u) from the same recurrence with r^2 replaced by |u|^2 = 1/r^2.
struct HarmCoef {
  double gam[SEA_LMAX][2 * SEA_LMAX + 1];
  double kap2[SEA_NQ];
  // D_lm as a homogeneous polynomial of degree l:
  //   D_lm(x, y, z) = sum_{a + b <= l} cart[lm][a][b] x^a y^b z^(l - a - b)
  // (the recurrence above carried out on coefficient arrays)
  double cart[SEA_NQ][SEA_LMAX + 1][SEA_LMAX + 1];
};
// Each translation unit that evaluates harmonics holds its own copy (the
// library is built without relocatable device code) and uploads it through
// its own upload_harmonics_<unit>() at context creation.
static __constant__ HarmCoef c_harm;

HarmCoef make_harmonic_coefficients();
static inline cudaError_t upload_harmonics_here() {
  const HarmCoef h = make_harmonic_coefficients();
  return cudaMemcpyToSymbol(c_harm, &h, sizeof(h));
}

// v 2^e2 rounded to the nearest FP64 value (ties to even); 0 if below the
// normal range.  Integer operations only.
__device__ __forceinline__ double scaled_i64(long long v, int e2) {
  if (v == 0) return 0.0;
  const unsigned long long sgn = (unsigned long long)v & 0x8000000000000000ULL;
  unsigned long long a = v < 0 ? 0ULL - (unsigned long long)v : (unsigned long long)v;
  const int lz = __clzll((long long)a);
  a <<= lz;
  unsigned long long mnt = a >> 11;
  const unsigned rem = (unsigned)(a & 0x7FF);
  if (rem > 0x400u || (rem == 0x400u && (mnt & 1ULL))) ++mnt;
  int ex = 63 - lz + e2 + 1023;
  if (mnt >> 53) {
    mnt >>= 1;
    ++ex;
  }
  if (ex <= 0) return 0.0;
  return __longlong_as_double(
      (long long)(sgn | ((unsigned long long)ex << 52) | (mnt & 0xFFFFFFFFFFFFFULL)));
}

// ---------------------------------------------------------------------------
// Double-float arithmetic (a value is hi + lo, |lo| <= ulp(hi) / 2): Knuth's
// two-sum and the fused-multiply-add two-product (Dekker's method), about 48
// significant bits from FP32 operations only.  The mixed form evaluates the
// multipole potential with it: on this part an FP64 instruction of a warp
// costs the issue time of 64 FP32 ones.
// ---------------------------------------------------------------------------
struct DF {
  float hi, lo;
};

__device__ __forceinline__ DF df_fast_two_sum(float a, float b) {  // |a| >= |b|
  const float s = a + b;
  return DF{s, b - (s - a)};
}
__device__ __forceinline__ DF df_add(DF a, DF b) {
  const float s = a.hi + b.hi;
  const float v = s - a.hi;
  const float e = (a.hi - (s - v)) + (b.hi - v);
  return df_fast_two_sum(s, e + (a.lo + b.lo));
}
__device__ __forceinline__ DF df_neg(DF a) { return DF{-a.hi, -a.lo}; }
__device__ __forceinline__ DF df_mul(DF a, DF b) {
  const float p = a.hi * b.hi;
  const float e = fmaf(a.hi, b.hi, -p);
  return df_fast_two_sum(p, fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e)));
}
__device__ __forceinline__ DF df_mul_f(float a, DF b) {  // a exact in FP32
  const float p = a * b.hi;
  const float e = fmaf(a, b.hi, -p);
  return df_fast_two_sum(p, fmaf(a, b.lo, e));
}
// a b + c with one normalisation: the product's high part and c.hi by an
// exact two-sum, every low-order term added to its error, then one fast
// two-sum (15 FP32 operations instead of 17 for df_add(df_mul(a, b), c)).
__device__ __forceinline__ DF df_fma(DF a, DF b, DF c) {
  const float p = a.hi * b.hi;
  const float pe = fmaf(a.hi, b.hi, -p);
  const float s = p + c.hi;
  const float v = s - p;
  const float e = (p - (s - v)) + (c.hi - v);
  return df_fast_two_sum(s, (fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, pe)) + c.lo) + e);
}
// a b + c d with one normalisation: the two products' high parts by an
// exact two-sum, their errors and cross terms added to its error (19 FP32
// operations instead of 22).  For a b - c d pass df_neg(c).
__device__ __forceinline__ DF df_dot2(DF a, DF b, DF c, DF d) {
  const float p = a.hi * b.hi, q = c.hi * d.hi;
  const float pe = fmaf(a.hi, b.hi, -p), qe = fmaf(c.hi, d.hi, -q);
  const float s = p + q;
  const float v = s - p;
  const float e = (p - (s - v)) + (q - v);
  const float lo = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, pe)) + fmaf(c.hi, d.lo, fmaf(c.lo, d.hi, qe));
  return df_fast_two_sum(s, lo + e);
}
// 1 / a: FP32 reciprocal, one Newton step in double-float
__device__ __forceinline__ DF df_rcp(DF a) {
  const float y = 1.0f / a.hi;
  const DF t = df_mul_f(y, a);  // a y = 1 - e
  const float e = (1.0f - t.hi) - t.lo;
  return df_fast_two_sum(y, y * e);
}
// sqrt(a): FP32 square root, one Newton step in double-float
__device__ __forceinline__ DF df_sqrt(DF a) {
  const float s = sqrtf(a.hi);
  const float p = s * s;
  const float pe = fmaf(s, s, -p);
  const float d = ((a.hi - p) - pe) + a.lo;  // a - s^2
  return df_fast_two_sum(s, d * (0.5f / s));
}
// An int |v| < 2^22 as FP32, exactly, without a conversion instruction:
// added to the bit pattern of 1.5 2^23 it lands in the low mantissa bits.
__device__ __forceinline__ float i2f_exact(int v) {
  return __int_as_float(0x4B400000 + v) - 12582912.0f;
}
// hi + lo as FP64 with integer operations only: both terms as fixed-point
// integers on the larger one's exponent (bits more than 2^-62 below it
// dropped), one rounding to nearest.  FP32 subnormals count as zero.
__device__ __forceinline__ double df_to_double(DF a) {
  const unsigned bh = __float_as_uint(a.hi), bl = __float_as_uint(a.lo);
  const int eh = (int)((bh >> 23) & 0xFF), el = (int)((bl >> 23) & 0xFF);
  const int E = max(eh, el);
  if (E == 0) return 0.0;
  auto fixed = [&](unsigned b, int e) -> long long {
    if (e == 0) return 0;
    const int sh = E - e;
    if (sh > 62) return 0;
    const long long v = ((long long)((b & 0x7FFFFFu) | 0x800000u) << 38) >> sh;
    return (b >> 31) ? -v : v;
  };
  return scaled_i64(fixed(bh, eh) + fixed(bl, el), E - 150 - 38);
}

// v = hi + lo with integer operations only (no FP64 instruction): hi keeps
// the sign, the exponent and the top 23 mantissa bits (truncation), lo the
// remaining 29 bits, rounded to an FP32 value of the same sign.  |v| below
// the FP32 normal range (2^-126) is flushed to (0, 0).  Relative error of
// hi + lo: <= 2^-47.
__device__ __forceinline__ float2 split64(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned sign = (unsigned)(b >> 63) << 31;
  const int e = (int)((b >> 52) & 0x7FF);
  if (e - 1023 + 127 <= 0) return make_float2(0.f, 0.f);
  const unsigned long long m = b & 0xFFFFFFFFFFFFFULL;
  const float hi = __uint_as_float(sign | ((unsigned)(e - 1023 + 127) << 23) | (unsigned)(m >> 29));
  // lo = (m mod 2^29) 2^(e - 1075) = ((m mod 2^29) 2^-64) 2^(e - 1011); e > 896 keeps
  // the second factor a normal FP32 power of two
  const float l = ((float)(unsigned)(m & 0x1FFFFFFFULL) * 5.421010862427522e-20f) *
                  __uint_as_float((unsigned)(e - 884) << 23);
  return make_float2(hi, __uint_as_float(__float_as_uint(l) | sign));
}

// An FP64 value as a double-float pair, by split64 (no FP64 instruction:
// on this part a warp's FP64 conversion or add holds the FP64 pipe for
// about 64 cycles).
__device__ __forceinline__ DF df_from_double(double x) {
  const float2 s = split64(x);
  return DF{s.x, s.y};
}

// The multipole potential of Eq. me along grid lines.  With u = r / r^2,
// sum_lm Qs_lm D_lm(u) = sum_abc P_abc ux^a uy^b uz^c, P_abc = sum_m Qs_lm
// cart[lm][a][b] (l = a + b + c; formed once per pair by k_pair_moments,
// layout mono_k), so with w = 1/r^2
//   v(r) = (1/r) sum_l w^l S_l(r),  S_l = sum_{a+b+c=l} P_abc x^a y^b z^c.
// On a line along axis AX the other two coordinates are fixed and S_l is a
// polynomial of degree l in the third: its 28 coefficients take 112
// operations once per line, a point then 21 + 6 multiply-adds instead of the
// 84 of the full three-variable Horner form.  The evaluation is bound by the
// FP64 unit (plain form) or by dependent FP32 chains (double-float, mixed
// form), and a line of a window or face has 12 to 30 points.
struct MeF64 {
  typedef double T;
  static __device__ __forceinline__ T mul(T a, T b) { return a * b; }
  static __device__ __forceinline__ T fma_(T a, T b, T c) { return fma(a, b, c); }
  // (1/r, 1/r^2) from r^2
  static __device__ __forceinline__ void inv(T r2, T* ir, T* ir2) {
    *ir = rsqrt(r2);
    *ir2 = *ir * *ir;
  }
};
struct MeDF {
  typedef DF T;
  static __device__ __forceinline__ T mul(T a, T b) { return df_mul(a, b); }
  static __device__ __forceinline__ T fma_(T a, T b, T c) { return df_fma(a, b, c); }
  static __device__ __forceinline__ void inv(T r2, T* ir, T* ir2) {
    *ir2 = df_rcp(r2);
    *ir = df_sqrt(*ir2);
  }
};
constexpr int ME_LINE = (SEA_LMAX + 1) * (SEA_LMAX + 2) / 2;  // coefficients: degree l, power k <= l
// The index of P for power k along axis AX and i, j along the other two.
template <int AX>
__device__ __forceinline__ constexpr int me_line_mono(int k, int i, int j) {
  return AX == 0 ? mono_k(k, i, j) : AX == 1 ? mono_k(i, k, j) : mono_k(i, j, k);
}
// c[l (l + 1) / 2 + k] for the line with coordinates s, t on the other axes
// (in axis order); P: the pair's coefficients (shared memory).
template <class R, int AX>
__device__ __forceinline__ void me_line(const typename R::T* __restrict__ P, typename R::T s,
                                        typename R::T t, typename R::T (&c)[ME_LINE]) {
  typedef typename R::T T;
  T m[SEA_LMAX + 1];  // m[i] = s^i t^(d-i)
#pragma unroll
  for (int d = 0; d <= SEA_LMAX; ++d) {
    if (d > 0) {
      m[d] = d == 1 ? s : R::mul(m[d - 1], s);
#pragma unroll
      for (int i = d - 1; i >= 0; --i) m[i] = d == 1 ? t : R::mul(m[i], t);
    }
#pragma unroll
    for (int k = 0; k + d <= SEA_LMAX; ++k) {
      const int l = k + d;
      T a = P[me_line_mono<AX>(k, 0, d)];
      if (d > 0) {
        a = R::mul(a, m[0]);
#pragma unroll
        for (int i = 1; i <= d; ++i) a = R::fma_(P[me_line_mono<AX>(k, i, d - i)], m[i], a);
      }
      c[l * (l + 1) / 2 + k] = a;
    }
  }
}
// v at coordinate x of the line, q = s^2 + t^2.
template <class R>
__device__ __forceinline__ typename R::T me_line_at(const typename R::T (&c)[ME_LINE],
                                                    typename R::T x, typename R::T q) {
  typedef typename R::T T;
  T ir, w;
  R::inv(R::fma_(x, x, q), &ir, &w);
  T v = c[0];
#pragma unroll
  for (int l = SEA_LMAX; l >= 0; --l) {
    T s = c[l * (l + 1) / 2 + l];
#pragma unroll
    for (int k = l - 1; k >= 0; --k) s = R::fma_(s, x, c[l * (l + 1) / 2 + k]);
    v = l == SEA_LMAX ? s : R::fma_(v, w, s);
  }
  return R::mul(v, ir);
}

// Exclusive scan over the CTA of one 64-bit integer per thread (blockDim.x
// a multiple of 32, at most 1024): warp shuffles, then the warp totals by
// the first warp.  Returns this thread's exclusive prefix; *total = the
// CTA's sum in every thread.  `ws` holds 32 values of shared memory.
// Integer sums, so the results equal a serial scan's.
__device__ __forceinline__ long long block_exscan_ll(long long v, long long* ws, long long* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  long long x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  if (w == 0) {
    long long t = lane < nw ? ws[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    ws[lane] = t;
  }
  __syncthreads();
  const long long before = (w ? ws[w - 1] : 0) + x - v;
  *total = ws[nw - 1];
  __syncthreads();  // ws may be reused
  return before;
}
// Maximum over the CTA of one 64-bit integer per thread (same shape rules).
__device__ __forceinline__ long long block_max_ll(long long v, long long* ws) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long y = __shfl_xor_sync(0xffffffffu, v, o);
    v = y > v ? y : v;
  }
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if ((threadIdx.x & 31) == 0) ws[w] = v;
  __syncthreads();
  long long m = ws[0];
  for (int k = 1; k < nw; ++k) m = ws[k] > m ? ws[k] : m;
  __syncthreads();
  return m;
}

// Sum over the block of one double; every thread gets the same total, added
// in a fixed order (lane tree, then warps in index order).  `slots` holds
// 32 doubles of shared memory, reused only after the next __syncthreads.
__device__ __forceinline__ double block_sum(double v, double* slots) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  if ((threadIdx.x & 31) == 0) slots[w] = v;
  __syncthreads();
  double s = 0.0;
  for (int k = 0; k < nw; ++k) s += slots[k];
  return s;
}

}  // namespace sea

// ---------------------------------------------------------------------------
// Context
// ---------------------------------------------------------------------------

struct SeaBuf {
  void* p = nullptr;
  size_t bytes = 0;
};

namespace sea {

// Grid tiles of the ACE contractions: 8 x 4 x 4 points, point r of a tile
// at x = r % 8, y = (r / 8) % 4, z = r / 32 inside it.
#define TX 8
#define TY 4
#define TZ 4
#define TP (TX * TY * TZ)

struct TileGeom {
  int nx, ny, nz, ntx, nty, ntz;
};

// Flat grid index of point r of tile T (-1 outside the grid).
__device__ __forceinline__ long long tile_point(const TileGeom& G, int T, int r) {
  const int txi = T % G.ntx, tyi = (T / G.ntx) % G.nty, tzi = T / (G.ntx * G.nty);
  const int x = txi * TX + (r % TX), y = tyi * TY + (r / TX) % TY, z = tzi * TZ + r / (TX * TY);
  if (x >= G.nx || y >= G.ny || z >= G.nz) return -1;
  return ((long long)z * G.ny + y) * G.nx + x;
}

inline TileGeom make_tile_geom(const int N[3]) {
  TileGeom G;
  G.nx = N[0];
  G.ny = N[1];
  G.nz = N[2];
  G.ntx = (G.nx + TX - 1) / TX;
  G.nty = (G.ny + TY - 1) / TY;
  G.ntz = (G.nz + TZ - 1) / TZ;
  return G;
}

}  // namespace sea

// A launch sequence recorded into a CUDA graph: the executable graph, the
// signature (sizes, parameters, buffer addresses) it was recorded with, and
// the number of kernels in it.
struct LaunchGraph {
  cudaGraphExec_t exec = nullptr;
  std::vector<uintptr_t> sig;
  long long launches = 0;
};

// A stream that runs a second kernel beside one on the context stream, and the
// events that fork and join it.
struct CgAux {
  cudaStream_t stream = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
};

struct sea_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  double cell[3] = {0, 0, 0};
  int N[3] = {0, 0, 0};
  double h[3] = {0, 0, 0};
  double dV = 0;
  size_t ng = 0;
  sea_params prm{};
  double w_ax[3][SEA_FDP + 1];  // -c_k / h_a^2 (negated second-difference weights)
  double w_center = 0;          // -sum_a c_0 / h_a^2

  bool poisoned = false;
  char err[256] = {0};

  int n_orb = 0;
  bool have_phi = false, have_vxx = false, have_ace = false, apply_timed = false;
  bool ace_eigen = false, w_dense = false;
  void* batch_cache = nullptr;  // CUDA graph of sea_apply_vxx_batch (batch.cu)
  SeaBuf bdesc, bitems;

  // plan sizes (host copies)
  int P = 0, Pproto = 0, E = 0;
  long long U = 0, WC = 0, max_window = 0;
  int cg_pad_max = 0;  // largest padded pair box (points), for the CG
  int n_large = 0;     // pairs of the CG's large class

  sea_stats stats{};

  // device buffers
  SeaBuf phi, vxx_dev, psi_dev, out_dev;
  SeaBuf rowsum, colsum, marg, box;
  bool sums_ready = false;  // rowsum and colsum are those of phi (formed as it was read)
  SeaBuf cand_flag, cand_geom, list_a, list_b, cand_S, counts;
  SeaBuf pinfo, pS, psize, voff, order, Q, epair, iters;
  SeaBuf vbuf, bbuf, rbuf, pbuf, qbuf;
  SeaBuf eptr, eent, ewin, coff, cbuf;
  SeaBuf status, exx_dev, queue;
  SeaBuf onorm;  // per-orbital partial sums of phi^2 (input check of sea_set_orbitals)
  // ACE
  SeaBuf wdig;  // W's digits (tensor-core contraction)
  SeaBuf wx;    // W's per-tile digit images (tensor-core expansion)
  // (tile, slot) bounds of the parts of W whose digits fit wdig at a time: one
  // part, formed once per build, where device memory allows it; empty: not
  // planned for the present W
  std::vector<int2> wparts;
  int wx_steps = 0;       // K steps of all images
  bool wx_ready = false;  // the images are those of the present W
  SeaBuf xevb;  // the expansion's H exponents per (tile, vector)
  SeaBuf gbuf;  // ghost (boundary) values of the pair boxes, 36 voff per pair
  SeaBuf flowbuf;  // the mixed form's one-launch Cholesky chain: DF blocks and task flags
  SeaBuf scdm_u, scdm_c;  // SCDM rotation and pivots
  SeaBuf scdm_s, scdm_a;  // SCDM step state; candidates' rows and coefficients
  SeaBuf rot;             // digit images of the SCDM rotation
  SeaBuf tmask, tptr_o, tlist_o, tslot_o, tptr_t, tlist_t, partial, Mbuf, Abuf, Lbuf, Linv,
      Gbuf, Hbuf, Hbuf2;
  int n_tiles = 0, tile_inc = 0, max_tile_list = 0;
  long long list_cap = 1;    // entries per list array (the second array's offset)
  bool lists_ready = false;  // the tile lists of the last plan's W support are formed
                             // and their counts on the host

  long long launches = 0;
  cudaEvent_t ev[16] = {};
  // host-buffer transfers: copy streams (host to device, device to host) and
  // per-chunk events, created with the context
  cudaStream_t xfer[2] = {};
  CgAux aux;  // the CG's second class of pairs
  std::vector<int> h_eptr;  // entry offsets per orbital, host copy (last plan)
  struct sea_unet* unet = nullptr;  // learned warm start (attached model, not owned)
  bool cg_warm = false;             // the next CG starts from the guess in vbuf
  LaunchGraph g_chol;  // the Cholesky / L^-1 / E_xx^ACE chain
  LaunchGraph g_plan;  // the plan (boxes, pairs, accumulation entries)
  bool far_side = false;            // the contributions outside the pair boxes were
                                    // launched on xfer[0] (done at xev[1])
  cudaEvent_t xev[2 * SEA_XCHUNKS_MAX + 2] = {};
};
// enqueue() issues a fixed launch sequence on c->stream.  On a stream that
// can be captured it is recorded once into gc (again whenever sig changes)
// and the graph is replayed, which removes most of the gaps between short
// dependent launches; on the legacy stream it runs directly.  enqueue()
// must not allocate or synchronise.
template <class F>
inline cudaError_t run_graph(sea_ctx* c, LaunchGraph& gc, const std::vector<uintptr_t>& sig,
                             F enqueue) {
  if (!c->stream) return enqueue();
  if (!gc.exec || gc.sig != sig) {
    if (gc.exec) {
      cudaGraphExecDestroy(gc.exec);
      gc.exec = nullptr;
    }
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return e;
    const long long l0 = c->launches;
    e = enqueue();
    const cudaError_t e2 = cudaStreamEndCapture(c->stream, &g);
    if (e != cudaSuccess) {
      if (g) cudaGraphDestroy(g);
      return e;
    }
    if (e2 != cudaSuccess) return e2;
    e = cudaGraphInstantiate(&gc.exec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return e;
    gc.launches = c->launches - l0;
    c->launches = l0;
    gc.sig = sig;
  }
  c->launches += gc.launches;
  return cudaGraphLaunch(gc.exec, c->stream);
}


// Whether a kernel on `device` may read memory of these attributes where it
// lies: memory of the device itself.  Memory of another GPU (which needs peer
// access) or of the host goes through a copy by the runtime.
inline bool sea_reads_in_place(const cudaPointerAttributes& a, int device) {
  return a.type == cudaMemoryTypeDevice && a.device == device;
}

// Lets `kernel` take `bytes` of dynamic shared memory on the current device.  The
// attribute is the process's, and calls of other contexts and threads need other
// sizes: it only ever grows, so that no launch finds it below its own size.
inline cudaError_t sea_allow_smem(const void* kernel, size_t bytes) {
  static std::mutex mutex;
  static std::map<std::pair<int, const void*>, size_t> most;
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mutex);
  size_t& m = most[{dev, kernel}];
  const size_t want = std::max(m, bytes);
  const cudaError_t e2 =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)want);
  if (e2 == cudaSuccess) m = want;
  return e2;
}

// Host-side helpers implemented in api.cu.
sea_status sea_fail(sea_ctx* c, sea_status s, const char* msg);
void sea_batch_cache_free(sea_ctx* c);
bool sea_ensure(sea_ctx* c, SeaBuf& b, size_t bytes);

// Pair record (device), one per selected pair, in (i, j) order.
struct PairInfo {
  int i, j;
  int lo[3], ext[3], k[3];
  int n;  // ext[0]*ext[1]*ext[2]
};

// Accumulation entry (Eq. tDxx): orbital o receives v_pair * phi_partner on
// the window [ws, ws + wl) (unwrapped grid coordinates, pair frame).
struct Entry {
  int pair, o, partner;
  int ws[3], wl[3];
};

namespace sea {
// q = floor(a / d) and *r = a - q d for 0 <= a < 2^24, 1 <= d < 2^24: the
// FP32 product a (1/d) is within (a/d) 2^-23 < 1 of a/d, so its truncation
// is q or q +- 1, corrected once by the sign and size of the remainder.
__host__ __device__ __forceinline__ int divmod_small(int a, int d, int* r) {
  int q = (int)((float)a * (1.0f / (float)d));
  int rr = a - q * d;
  if (rr < 0) {
    --q;
    rr += d;
  } else if (rr >= d) {
    ++q;
    rr -= d;
  }
  *r = rr;
  return q;
}

// The pair box in the coordinates of an entry's window, clipped to it:
// [b0[a], b1[a]) per axis, n_in points inside and n_out outside.  An empty
// intersection is kept as the empty box [0, 0)^3, so that every window point
// falls in the "z above" part of window_outside_point.
struct WinSplit {
  int b0[3], b1[3];
  int n_in, n_out;
};
__host__ __device__ __forceinline__ WinSplit window_split(const Entry& e, const PairInfo& P) {
  WinSplit s;
  bool empty = false;
  for (int a = 0; a < 3; ++a) {
    const int lo = P.lo[a] - e.ws[a], hi = lo + P.ext[a];
    s.b0[a] = lo < 0 ? 0 : (lo > e.wl[a] ? e.wl[a] : lo);
    s.b1[a] = hi < 0 ? 0 : (hi > e.wl[a] ? e.wl[a] : hi);
    empty = empty || s.b0[a] >= s.b1[a];
  }
  if (empty)
    for (int a = 0; a < 3; ++a) s.b0[a] = s.b1[a] = 0;
  s.n_in = (s.b1[0] - s.b0[0]) * (s.b1[1] - s.b0[1]) * (s.b1[2] - s.b0[2]);
  s.n_out = e.wl[0] * e.wl[1] * e.wl[2] - s.n_in;
  return s;
}

// The lines along x of a window that hold points outside the pair box, in
// window coordinates: first the whole lines (n_whole: the planes below and
// above the box's z range, then within that range the rows below and above
// its y range), then the n_cut lines that cross the box, whose points outside
// are [0, b0[0]) and [b1[0], wl[0]).
struct WinLines {
  int n_whole, n_cut;
};
__host__ __device__ __forceinline__ WinLines window_lines(const WinSplit& s, const int wl[3]) {
  WinLines n;
  n.n_cut = (s.b1[1] - s.b0[1]) * (s.b1[2] - s.b0[2]);
  n.n_whole = wl[1] * wl[2] - n.n_cut;
  if (s.b1[0] - s.b0[0] == wl[0]) n.n_cut = 0;  // those lines lie inside
  return n;
}
// (ty, tz) of line i < n_whole + n_cut (fewer than 2^24 lines: windows have
// at most 1024 points per axis).
__host__ __device__ __forceinline__ void window_outside_line(const WinSplit& s, const int wl[3],
                                                             int i, int* ty, int* tz) {
  const int wy = wl[1], zb = s.b1[2] - s.b0[2], yb = s.b1[1] - s.b0[1];
  const int n1 = s.b0[2] * wy, n2 = (wl[2] - s.b1[2]) * wy;
  const int n3 = zb * s.b0[1], n4 = zb * (wy - s.b1[1]);
  int oy = 0, oz = 0, by = wy;
  if (i < n1) {
  } else if ((i -= n1) < n2) {
    oz = s.b1[2];
  } else {
    i -= n2;
    oz = s.b0[2];
    if (i < n3) {
      by = s.b0[1];
    } else if ((i -= n3) < n4) {
      oy = s.b1[1];
      by = wy - s.b1[1];
    } else {
      i -= n4;
      oy = s.b0[1];
      by = yb;
    }
  }
  int ry;
  *tz = oz + divmod_small(i, by, &ry);
  *ty = oy + ry;
}

// The points outside the box of a piece [x0, x1) of a line in the order above
// (cut: a line that crosses the box): the first one is window_piece_first, the
// one after tx window_piece_next, while they are below x1.
__host__ __device__ __forceinline__ int window_piece_first(const WinSplit& s, bool cut, int x0) {
  return cut && x0 >= s.b0[0] && x0 < s.b1[0] ? s.b1[0] : x0;
}
__host__ __device__ __forceinline__ int window_piece_next(const WinSplit& s, bool cut, int tx) {
  ++tx;
  return cut && tx == s.b0[0] ? s.b1[0] : tx;
}

// Window coordinates of point u (0 <= u < n_out, n_out < 2^24) of the window
// points outside the pair box, line after line in the order above, on the
// cut lines first all points left of the box, then all right of it (the kernels
// go by lines and pieces; tests check the numbering).
__host__ __device__ __forceinline__ void window_outside_point(const WinSplit& s, const int wl[3],
                                                              int u, int* tx, int* ty, int* tz) {
  const WinLines n = window_lines(s, wl);
  const int left = s.b0[0], right = wl[0] - s.b1[0];
  int line, rx, x0 = 0;
  if (u < n.n_whole * wl[0]) {
    line = divmod_small(u, wl[0], &rx);
  } else if ((u -= n.n_whole * wl[0]) < n.n_cut * left) {
    line = n.n_whole + divmod_small(u, left, &rx);
  } else {
    line = n.n_whole + divmod_small(u - n.n_cut * left, right, &rx);
    x0 = s.b1[0];
  }
  window_outside_line(s, wl, line, ty, tz);
  *tx = x0 + rx;
}

// Shared-memory layout of a CG vector on a pair box: the planes of ex x ey
// points stored row after row (so consecutive points of a warp sit in
// consecutive banks), each plane followed by F = SEA_FDP zero rows, which
// serve as the y halo on both sides, and F zero planes before and after the
// box for the z halo.  Box point t = (z ey + y) ex + x sits at
// F ex (ey + F) + t + z F ex.  Neighbours along y and z outside the box read
// zeros; along x they are masked.  Points of the layout of one of `team` CTAs
// that share the box's points (cg_share; INT_MAX above that):
__host__ __device__ __forceinline__ int sea_min(int a, int b) { return a < b ? a : b; }
__host__ __device__ __forceinline__ int cg_share(int n, int team) { return (n + team - 1) / team; }
__host__ __device__ __forceinline__ int cg_pad_volume(int ex, int ey, int ez, int team) {
  const int area = ex * ey;
  const int nz = team == 1 ? ez : sea_min(ez, (cg_share(area * ez, team) + area - 1) / area + 1);
  const long long v = (long long)ex * (ey + SEA_FDP) * (nz + 2 * SEA_FDP);
  return v > 2147483647LL ? 2147483647 : (int)v;
}

// The pairs of a launch in two classes, each a kernel of its own (the class is
// the pair's alone, so a pair is solved by the same CTA size, hence with the
// same bits, in every launch).  Boxes of at most SEA_CG_SPLIT points: CTAs of
// 512 threads, two per SM, where one fills the other's waits at the step's
// barriers.  Larger boxes: CTAs of 1024 threads, one per SM: a step of a large
// box takes several rounds of its CTA's points, a launch seldom has two of
// them per SM, and one may hold a padded box twice as large in shared memory.
// (H2O)16 on 81^3, most boxes large: FP64 CG 26.7 -> 3.05 ms, since the padded
// boxes no longer miss the fixed-point stencil.  With the
// line at 3072 or 2048 points the 96^3 workloads, whose boxes lie below it,
// lose 0 to 0.4 and 0.2 to 0.75 ms.
#define SEA_CG_SPLIT 4096
// In the mixed form the line is at SEA_CG_SINGLE padded points, where its inner
// solve changes its arrangement: its FP32 sums depend on the CTA size, so each
// arrangement keeps one.
#define SEA_CG_SINGLE 13824
__host__ __device__ __forceinline__ bool cg_large(const int* ext, bool mixed) {
  return mixed ? cg_pad_volume(ext[0], ext[1], ext[2], 1) > SEA_CG_SINGLE
               : ext[0] * ext[1] * ext[2] > SEA_CG_SPLIT;
}

__host__ __device__ constexpr int cg_threads(bool large) { return large ? 1024 : 512; }
// Padded points of a box that fit shared memory, 8 bytes (plain form) or 4
// (mixed form) each.
__host__ __device__ constexpr int cg_pad_limit(bool mixed, bool large, bool team = false) {
  return mixed ? (large ? 56000 : SEA_CG_SINGLE) : (large ? (team ? 27000 : 28000) : 13824);
}

// Points of a team's CTA in registers: the largest of cg_fix_team's forms.
#define SEA_CG_TEAM_NP 4

// CTAs (a cluster, at most SEA_CG_TEAM_MAX) that share a box of a bare batch of
// n_box boxes on a GPU of nsm SMs.
#define SEA_CG_TEAM_MAX 8
// The rule: as many CTAs a box (8 at most, the portable cluster size) as fill two
// places per SM, fewer where a box that one CTA solves in fixed point would not
// fit the team's registers and shared memory.  Time of a call with teams of 1, 2,
// 4 and 8, us, boxes of 9 to 16 points an edge: 16 boxes 1019, 873, 770, 689; 48
// boxes 1376, 1045, 933, 1055; 100 boxes 1335, 1337, 1136, 1721; 150 boxes 1450,
// 1412, 1659, 2480; 450 boxes 1884, 2185, 3500, 6410 (there the teams' barriers
// only delay SMs that have other boxes to work on).  A box's sums, hence its last
// bits, depend on its team, so on the other boxes of the call (sea.h says so); the
// pairs of sea_apply_vxx stay on single CTAs, since batched and single calls give
// the same bits.
// A box that not even the team solves in fixed point (over the shared memory of
// one CTA and the team's registers) is left to the team's first CTA: not more
// teams' places than SMs then, since boxes of the large class take an SM a CTA
// (152 boxes of 25^3 44.8 -> 22.6 ms, 64 of 40^3 262 -> 135 ms).
inline int cg_team_rule(int n_box, const int* ext, int nsm) {
  int team = SEA_CG_TEAM_MAX;
  while (team > 1 && (long long)team * n_box > 2LL * nsm) team /= 2;
  // fits(b): the team solves box b in fixed point
  auto fits = [&](const int* e, bool large) {
    return cg_share(e[0] * e[1] * e[2], team) <= SEA_CG_TEAM_NP * cg_threads(large) &&
           cg_pad_volume(e[0], e[1], e[2], team) <= cg_pad_limit(false, large, true);
  };
  long long n_large = 0;
  for (int b = 0; b < n_box; ++b) {
    const int* e = ext + 3 * b;
    const bool large = e[0] * e[1] * e[2] > SEA_CG_SPLIT;
    n_large += large;
    if (cg_pad_volume(e[0], e[1], e[2], 1) > cg_pad_limit(false, large)) continue;
    while (team > 1 && !fits(e, large)) team /= 2;
  }
  auto one_left = [&] {
    for (int b = 0; b < n_box; ++b) {
      const int* e = ext + 3 * b;
      if (e[0] * e[1] * e[2] > SEA_CG_SPLIT && !fits(e, true)) return true;
    }
    return false;
  };
  while (team > 1 && n_large * team > nsm && one_left()) team /= 2;
  return team;
}
int cg_box_team(int n_box, const int* ext);  // on the current device

// Launch wrappers (each file implements its own).
// Rows that the plan's sums are formed of in registers.
#define SEA_SUMS_REG_MAX 256
cudaError_t launch_row_col_sums(sea_ctx* c, const double* phi, int o0, int o1, double* dst,
                                double* part);
cudaError_t launch_plan_boxes(sea_ctx* c);
cudaError_t launch_plan_pairs(sea_ctx* c);
cudaError_t launch_pair_setup(sea_ctx* c);
cudaError_t launch_cg(sea_ctx* c);
cudaError_t launch_contrib_far(sea_ctx* c, cudaEvent_t setup_done);
// chol_flow.cu: the mixed form's Cholesky of -Mbar, L^-1 and E_xx^ACE in one
// cooperative launch (scratch of chol_flow_bytes(n) bytes).
size_t chol_flow_bytes(int n);
cudaError_t launch_chol_flow(cudaStream_t st, int device, const double* M, int n, double* L,
                             double* Linv, void* scratch, unsigned* status, double* exx);
void make_batch_desc(sea_ctx* c, void* out);
size_t batch_desc_bytes();
// The persistent batched CG: ctas_per_sm CTAs per SM for the smaller boxes (0
// or above the occupancy limit: the limit); queue: two counters; pad_max: the
// largest padded pair box.
cudaError_t launch_cg_batch(cudaStream_t st, const CgAux* aux, const void* descs, const int2* items,
                            int total, int n_large, int* queue, int pad_max, bool mixed,
                            int ctas_per_sm);
int cg_batch_max_ctas_per_sm(int pad_max, bool mixed);
cudaError_t launch_entries(sea_ctx* c);
// V_xx phi into out (the context's W) and, when out2 is not null, also into
// out2 (the caller's device buffer), both written by the same stores.
cudaError_t launch_accumulate(sea_ctx* c, double* out, double* out2 = nullptr,
                              bool with_exx = true);
cudaError_t launch_accumulate_range(sea_ctx* c, double* out, int o_begin, int o_end, int e_begin,
                                    int e_end, double* out2 = nullptr);
cudaError_t launch_exx(sea_ctx* c, cudaStream_t st);
// Learned warm start (unet.cu): x0 of every pair's CG from the attached model.
cudaError_t launch_warm_start(sea_ctx* c);
// SCDM localization of the orbitals in c->vxx_dev (scdm.cu): U and the pivots
// on the device; the localized orbitals go to c->phi.
cudaError_t launch_scdm(sea_ctx* c, double* U_dev, long long* C_dev);
// out[i][r] = sum_j U[j][i] phi[j][r] on the tensor cores (rotate_tc.cu).
cudaError_t launch_rotate(sea_ctx* c, const double* phi, int n, size_t N, const double* U,
                          double* out);
// Damped Jacobi sweeps on every pair's starting vector (pair.cu).
cudaError_t launch_smooth(sea_ctx* c, int sweeps, double omega);
// The contraction with W on the tensor cores.  launch_w_digits splits W's rows
// on the lists of tiles [a.x, b.x), slots [a.y, b.y), into wbuf
// (w_digits_bytes(b.y - a.y)); launch_gram_tc then forms partial[slot m + a]
// of those slots for A's m rows.  *queue is reset on the stream.
// digits: 6 (mixed form) or 7 (plain form).
size_t w_digits_bytes(long long slots, int digits);
cudaError_t launch_w_digits(cudaStream_t st, const double* W, const TileGeom& G, size_t ng,
                            int2 a, int2 b, int max_list, const int* tptr, const int* tlist,
                            void* wbuf, int digits);
// The expansion's images: SEA_XKS list entries a K step, for tiles of 1 to
// SEA_XJ entries; tile T's first step is xoff[T], `steps` in all, `slots` the
// total list length.
#define SEA_XJ 32
#define SEA_XKS 16
__host__ __device__ __forceinline__ int wx_tile_steps(int list) {
  return list > SEA_XJ ? 0 : (list + SEA_XKS - 1) / SEA_XKS;
}
size_t wx_digits_bytes(long long steps, long long slots, int digits);
cudaError_t launch_wx_digits(cudaStream_t st, const double* W, const TileGeom& G, size_t ng,
                             int n_tiles, const int* tptr, const int* tlist, const int* tsub,
                             const int* xoff, long long steps, long long slots, void* wxbuf,
                             int digits);
cudaError_t launch_expand_tc(cudaStream_t st, int device, const void* wxbuf, const TileGeom& G,
                             size_t ng, int n_tiles, const int* tptr, const int* tlist,
                             const int* xoff, long long steps, long long slots, const double* H,
                             long long hj, long long hv, int m, bool negate, double* out, int* evbuf,
                             int* queue, unsigned* status, int digits);
cudaError_t launch_gram_tc(cudaStream_t st, int device, const double* A, int m, const TileGeom& G,
                           size_t ng, int2 a, int2 b, const int* tptr, const void* wbuf,
                           double* partial, int* queue, unsigned* status, int digits);
// sea_ensure; where memory is short the digits and images of W are given up
// first (they are formed again, or done without).
bool sea_ensure_first(sea_ctx* c, SeaBuf& b, size_t bytes);
cudaError_t launch_ace_lists(sea_ctx* c, cudaStream_t st);
cudaError_t launch_ace_build(sea_ctx* c);
cudaError_t launch_ace_eigen(sea_ctx* c);
cudaError_t launch_ace_apply(sea_ctx* c, const double* psi, int n_vec, double* out);
cudaError_t launch_ace_vectors(sea_ctx* c, double* xi);
cudaError_t upload_harmonics_pair();
void fornberg_weights(double* w);
cudaError_t launch_cg_boxes(cudaStream_t stream, const double h[3], int nbox,
                            const PairInfo* boxes, const long long* voff, const int* order,
                            const double* rhs, double* x, double* r, double* p, double* q,
                            int* iters, unsigned* status, int* queue, double tol, int tol_mode,
                            int max_iter, int team, int pad_max, int n_large);
}  // namespace sea
