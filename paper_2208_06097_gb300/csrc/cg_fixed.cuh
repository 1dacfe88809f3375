// cg_fixed.cuh -- the plain form's pair solve with the stencil in fixed point.
//
// The FP64 unit of this part issues 2 multiply-adds per clock and SM, 1/32 of
// its integer rate, and the 37-point operator is 37 of the 42 FP64
// instructions that a CG step spends per unknown.  The stencil's weights are
// rational: times 831600 they are integers below 2^22.  So the search
// direction p is kept in shared memory as 57-bit integers on one power of two
// per step (2^(E-56) with |p| < 2^E), and -Lap_h p is formed exactly in
// integer arithmetic and rounded once to FP64: more exact than the FP64 sum of
// 37 rounded products whenever p's largest value is what the sum's rounding is
// measured against (quantization 2^-57 of it against 2^-53 per product).  The
// CG's vector updates and their products stay in FP64 (5 instructions per
// unknown), and the block sums add FP64 partials as integers (fixed-point
// warp sums on the warp's largest exponent), so they use no FP64 instruction
// either.
#pragma once

#include "sea_internal.cuh"

namespace sea {

// -831600 c_k, c_k the order-12 second-difference weights:
// c_0 = -5369/1800, c_1 = 12/7, c_2 = -15/56, c_3 = 10/189, c_4 = -1/112,
// c_5 = 2/1925, c_6 = -1/16632.
#define SEA_FIX_DEN 831600.0
__device__ __forceinline__ constexpr int fix_w(int k) {
  return k == 0 ? 2480478 : k == 1 ? -1425600 : k == 2 ? 222750 : k == 3 ? -44000
       : k == 4 ? 7425 : k == 5 ? -864 : 50;
}

// Limbs of a fixed-point value: X = y 2^28 + x, 0 <= x < 2^28, |y| <= 2^28.
constexpr int FIX_LO = 28;
constexpr int FIX_BITS = 2 * FIX_LO;
constexpr unsigned FIX_MASK = (1u << FIX_LO) - 1u;

__device__ __forceinline__ unsigned long long shr64c(unsigned long long a, unsigned n) {
  unsigned long long r;  // count clamped at 64
  asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(n));
  return r;
}

// p 2^(56 - E) truncated toward zero, |p| < 2^E.
__device__ __forceinline__ int2 fix_quant(double p, int E) {
  const unsigned h = (unsigned)__double2hiint(p), l = (unsigned)__double2loint(p);
  const unsigned e = (h >> 20) & 0x7FFu;
  const unsigned long long m =
      ((unsigned long long)((h & 0xFFFFFu) | 0x100000u) << 32) | (unsigned long long)l;
  long long X = (long long)shr64c(m << 3, (unsigned)(1022 + E) - e);
  if ((int)h < 0) X = -X;
  return make_int2((int)((unsigned)X & FIX_MASK), (int)(X >> FIX_LO));
}

// (hi 2^28 + lo) 2^e0 rounded to nearest, |hi|, |lo| < 2^54.
__device__ __forceinline__ double fix_to_double(long long hi, long long lo, int e0) {
  hi += lo >> FIX_LO;
  unsigned vl = (unsigned)lo & FIX_MASK;
  const unsigned sgn = (unsigned)((unsigned long long)hi >> 32) & 0x80000000u;
  if (sgn) {
    hi = ~hi + (vl == 0u);
    vl = (0u - vl) & FIX_MASK;
  }
  const int sh = min(__clzll(hi), FIX_LO);
  unsigned long long X = ((unsigned long long)hi << sh) | (vl >> (FIX_LO - sh));
  const int lz = __clzll((long long)X);
  X <<= lz;
  const int ex = 63 + 1022 + FIX_LO + e0 - sh - lz;  // biased exponent - 1: mantissa bit 52 adds 1
  const unsigned long long mnt = (X >> 11) + ((X >> 10) & 1ULL);
  const unsigned long long b = mnt + ((unsigned long long)(unsigned)ex << 52);
  if (X == 0ULL || ex < 0) return 0.0;
  return __hiloint2double((int)((unsigned)(b >> 32) | sgn), (int)(unsigned)b);
}

// A warp's or block's sum as X 2^(e - 1080).
struct FixSum {
  long long X;
  int e;
};

__device__ __forceinline__ long long fix_warp_add(long long X) {
  // three limbs of 26 bits (26 + 5 bits per sum) and the signed rest
  const unsigned s0 = __reduce_add_sync(0xffffffffu, (unsigned)X & 0x3FFFFFFu);
  const unsigned s1 = __reduce_add_sync(0xffffffffu, (unsigned)(X >> 26) & 0x3FFFFFFu);
  const int s2 = __reduce_add_sync(0xffffffffu, (int)(X >> 52));
  return ((long long)s2 << 52) + ((long long)s1 << 26) + (long long)s0;
}

// Sum of the warp's FP64 values (finite), each truncated 2^-5 units of the
// last place below the largest: the same in every lane, whatever the order.
__device__ __forceinline__ FixSum fix_warp_sum(double v) {
  const unsigned h = (unsigned)__double2hiint(v), l = (unsigned)__double2loint(v);
  const unsigned e = (h >> 20) & 0x7FFu;
  const unsigned em = __reduce_max_sync(0xffffffffu, e);
  unsigned long long m =
      ((unsigned long long)((h & 0xFFFFFu) | 0x100000u) << 32) | (unsigned long long)l;
  if (e == 0u) m = 0ULL;
  long long X = (long long)shr64c(m << 5, em - e);
  if ((int)h < 0) X = -X;
  return FixSum{fix_warp_add(X), (int)em};
}

// The CTAs that share a box: cluster rank and size.  TEAM: the size, or (3 and
// more) the largest size of a launch.
struct CgTeam {
  int rank, size;
};
template <int TEAM>
__device__ __forceinline__ CgTeam cg_team() {
  if (TEAM == 1) return CgTeam{0, 1};
  unsigned r, n = TEAM;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  if (TEAM > 2) asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
  return CgTeam{(int)r, (int)n};
}
// p's counterpart in the shared memory of the team's CTA `rank`.
template <class T>
__device__ __forceinline__ T* team_ptr(T* p, int rank) {
  unsigned long long a;
  asm("mapa.u64 %0, %1, %2;" : "=l"(a) : "l"((unsigned long long)p), "r"(rank));
  return (T*)a;
}
// Barrier of the team's threads, shared-memory writes to the others included.
__device__ __forceinline__ void team_sync(const CgTeam& T) {
  if (T.size == 1) {
    __syncthreads();
    return;
  }
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// The warp's part of a team's sum and maximum, posted to every CTA of the team.
__device__ __forceinline__ void fix_post(const CgTeam& T, double v, unsigned vmax, int4* slots) {
  const FixSum w = fix_warp_sum(v);
  const unsigned wm = __reduce_max_sync(0xffffffffu, vmax);
  const int lane = threadIdx.x & 31, at = T.rank * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int4 v4 = make_int4((int)(unsigned)w.X, (int)(w.X >> 32), w.e, (int)wm);
  if (T.size == 1) {
    if (lane == 0) slots[at] = v4;
  } else if (lane < T.size) {
    team_ptr(slots, lane)[at] = v4;
  }
}

// The team's sum (and maximum) from the warps' posts, by one whole warp.
__device__ __forceinline__ FixSum fix_combine(const CgTeam& T, const int4* slots, unsigned* bmax) {
  const int lane = threadIdx.x & 31, nw = T.size * (int)(blockDim.x >> 5);
  int4 s = make_int4(0, 0, 0, 0);
  if (lane < nw) s = slots[lane];
  int E = s.z, room = 5;  // bits for 32 warps
  unsigned m = (unsigned)s.w;
  if (T.size > 1)
    for (int k = lane + 32; k < nw; k += 32) {
      E = max(E, slots[k].z);
      m = max(m, (unsigned)slots[k].w);
    }
  E = (int)__reduce_max_sync(0xffffffffu, (unsigned)E);
  *bmax = __reduce_max_sync(0xffffffffu, m);
  if (T.size > 1)
    while ((1 << room) < nw) ++room;
  long long X = (((long long)s.y << 32) | (long long)(unsigned)s.x) >> min(E - s.z + room, 63);
  if (T.size > 1)
    for (int k = lane + 32; k < nw; k += 32) {
      s = slots[k];
      X += (((long long)s.y << 32) | (long long)(unsigned)s.x) >> min(E - s.z + room, 63);
    }
  return FixSum{fix_warp_add(X), E + room};
}

// 1 / b as Y 2^e for a positive sum b (Y = 0 if it is not), good to 2^-59:
// two Newton steps in integer arithmetic from the FP32 reciprocal of b's
// leading 24 bits.
struct FixRecip {
  unsigned long long Y;
  int e;
};
__device__ __forceinline__ FixRecip fix_recip(FixSum b) {
  const int lb = __clzll(b.X);
  const unsigned long long B = (unsigned long long)b.X << lb;
  const float f = __frcp_rn((float)(unsigned)(B >> 40));  // in (2^-24, 2^-23]
  // Y ~ 2^126 / B, kept below 2^63
  unsigned long long Y = ((unsigned long long)(unsigned)(f * 140737488355328.0f) << 39) - 1ULL;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const long long d = (1LL << 62) - (long long)__umul64hi(B, Y);
    Y += (unsigned long long)(__mul64hi((long long)Y, d) << 2);
  }
  return FixRecip{b.X > 0 ? Y : 0ULL, lb - b.e - 126};
}
// a / b from b's reciprocal, for a positive a (else 0), one rounding to FP64.
__device__ __forceinline__ double fix_ratio(FixSum a, FixRecip r) {
  if (a.X <= 0) return 0.0;
  const int la = __clzll(a.X);
  const long long Q = (long long)__umul64hi((unsigned long long)a.X << la, r.Y);
  return scaled_i64(Q, 64 - la + a.e + r.e);
}

// An FP32 value just above the non-negative FP64 value with high word h,
// divided by 2^k (at least 2^-120).
__device__ __forceinline__ float fix_upper(unsigned h, int k) {
  const int ef = (int)(h >> 20) - 1023 - k + 127;
  return __uint_as_float(((unsigned)max(ef, 7) << 23 | (h & 0xFFFFFu) << 3) + 8u);
}

// Scalars of a step that one warp forms for the block.
struct FixScal {
  double as, beta;
  int E, done;
};

// What the lead warp of a CTA keeps between a solve's steps: rr, its
// reciprocal, and the bound M 2^k0 of |p| (M FP32, kept from below by rounding
// up): the next |p| <= |r| + beta |p|.
struct FixLead {
  FixSum rr{0, 0};
  FixRecip irr{0, 0};
  float M = 0.f;
  int k0 = 0;
  // from the posts of (r, r) and the largest |r| at the start: E
  __device__ __forceinline__ void start(const CgTeam& T, const int4* slots, bool post, FixScal& sc) {
    unsigned rmax;
    rr = fix_combine(T, slots, &rmax);
    irr = fix_recip(rr);
    k0 = (int)(rmax >> 20) - 1023;
    M = fix_upper(rmax, k0);
    if (post) sc.E = k0 + (int)(__float_as_uint(M) >> 23) - 126;
  }
  // from the posts of (p, q): alpha s_x
  __device__ __forceinline__ void step(const CgTeam& T, const int4* slots, bool post, FixScal& sc) {
    unsigned none;
    const double as = fix_ratio(rr, fix_recip(fix_combine(T, slots, &none)));
    if (post) sc.as = as;
  }
  // from the posts of the new (r, r): beta, the next E and whether to stop;
  // next() follows, off the critical path
  __device__ __forceinline__ void turn(const CgTeam& T, const int4* slots, double target2, bool post,
                                       FixScal& sc) {
    unsigned rmax;
    rr = fix_combine(T, slots, &rmax);
    const double beta = fix_ratio(rr, irr);
    M = __fmaf_ru(fix_upper((unsigned)__double2hiint(beta), 0), M, fix_upper(rmax, k0));
    if (post) {
      sc.beta = beta;
      sc.E = k0 + (int)(__float_as_uint(M) >> 23) - 126;
      // non-negative FP64 values compare as their bit patterns
      sc.done = __double_as_longlong(scaled_i64(rr.X, rr.e - 1080)) <=
                __double_as_longlong(target2);
    }
  }
  __device__ __forceinline__ void next() { irr = fix_recip(rr); }
};

// What the fixed-point solve needs beside the CG's own arguments.
struct FixArgs {
  double s[3];  // 1 / (831600 h_a^2)
  int mode;     // 0: not used; 1: three axes; 2: equal spacings
};

// sum_a (s_a / s_0) I_a with I_a = axis a's integer stencil sum at padded
// index tp; P: the padded fixed-point direction, unit 2^e0.
template <bool ISO>
__device__ __forceinline__ double fix_stencil(const int2* __restrict__ P, int tp, int x, int ex,
                                              int PXY, double ry, double rz, int e0) {
  const int2 c = P[tp];
  const int2 zero = make_int2(0, 0);
  if (ISO) {
    long long lo = (long long)(3 * fix_w(0)) * c.x, hi = (long long)(3 * fix_w(0)) * c.y;
#pragma unroll
    for (int k = 1; k <= SEA_FDP; ++k) {
      const int2 a = x >= k ? P[tp - k] : zero, b = x + k < ex ? P[tp + k] : zero;
      const int2 d = P[tp - k * ex], e = P[tp + k * ex];
      const int2 f = P[tp - k * PXY], g = P[tp + k * PXY];
      lo += (long long)fix_w(k) * (a.x + b.x + d.x + e.x + f.x + g.x);
      hi += (long long)fix_w(k) * (a.y + b.y + d.y + e.y + f.y + g.y);
    }
    return fix_to_double(hi, lo, e0);
  }
  double q = 0.0;
#pragma unroll
  for (int ax = 2; ax >= 0; --ax) {
    const int st = ax == 0 ? 1 : (ax == 1 ? ex : PXY);
    long long lo = (long long)fix_w(0) * c.x, hi = (long long)fix_w(0) * c.y;
#pragma unroll
    for (int k = 1; k <= SEA_FDP; ++k) {
      const int2 a = (ax > 0 || x >= k) ? P[tp - k * st] : zero;
      const int2 b = (ax > 0 || x + k < ex) ? P[tp + k * st] : zero;
      lo += (long long)fix_w(k) * (a.x + b.x);
      hi += (long long)fix_w(k) * (a.y + b.y);
    }
    const double I = fix_to_double(hi, lo, e0);
    q = ax == 2 ? rz * I : (ax == 1 ? fma(ry, I, q) : I + q);
  }
  return q;
}

}  // namespace sea
