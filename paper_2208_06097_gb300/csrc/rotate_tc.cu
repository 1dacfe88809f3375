// rotate_tc.cu -- the SCDM rotation Phi~ = Phi U (Eq. unitary_scdm) on the
// tensor cores:  out[i][r] = sum_j U[j][i] phi[j][r].
//
// A dense FP64 product of 2 n^2 N operations, 89 times the FP64 unit's rate
// above its bytes at n = 128: bound by the FP64 pipe (11.2 ms for 128 orbitals
// on 72 x 75 x 76 points, its peak).  Here by exact splitting (the Ozaki scheme)
// into balanced base-128 digits held in FP16: phi's values at a point share
// one exponent over the orbitals (|phi_j(r)| < 2^E), U's entries of a column
// one over j (2^F); a value is X 2^(E - 55) with the integer X (|X| < 2^55,
// truncated: the largest values of a point are kept whole), X = sum_k d_k
// 128^(7-k), |d_k| <= 64.  With D_d = sum over k + l = d of the digit planes'
// products,
//   out = 2^(E + F - 61) sum_{d=0}^{7} 128^(7-d) D_d,
// D_d a sum of at most 8 x 512 products below 2^12 (K is taken 512 orbitals at
// a time): an integer of at most 2^24, exact in the FP32 accumulator.  The
// diagonals are combined exactly and rounded once.  Error: the truncations,
// 2^-55 of the point's and the column's largest values, and the dropped
// diagonals d >= 8, about 2^-56 of their product per term: below the
// rounding of an FP64 sum of the products (128 terms, exact rational reference:
// 2.5e-16 of the largest value at worst, the FP64 sum 3.4e-16).
//
// k_rot_udigits, k_rot_digits write the digit images that the tensor core
// reads (K-major core matrices, stage after stage, so that each stage is one
// bulk copy); k_rot_gemm: a CTA per 128 points walks the blocks of 32 outputs,
// one warp loading, one issuing MMAs (M = 128 points, W's planes stacked along
// N as in the contraction with W: 8 MMAs per 16 orbitals), eight converting
// the accumulators.  The points are taken in slabs whose digit images stay in
// L2.  Every wait is bounded; on expiry the kernel sets SEA_FLAG_WAIT, waits
// for work in flight, frees its tensor memory and ends.
#include <algorithm>

#include "cg_fixed.cuh"
#include "sea_internal.cuh"
#include "tcgen05.cuh"

namespace sea {
namespace {

constexpr int RD = 8;     // digits per value
constexpr int RT = 128;   // points per tile (M)
constexpr int RK = 16;    // orbitals per stage
constexpr int RN = 32;    // outputs per block
constexpr int RSEG = 512 / RK;  // stages per exact accumulation
constexpr uint32_t RA_PLANE = RT * RK * 2, RA_STAGE = RD * RA_PLANE, RA_LBO = RT * 16;
constexpr uint32_t RB_STAGE = RD * RN * RK * 2, RB_LBO = RD * RN * 16;
constexpr int R_STAGES = 5;
constexpr int RE_WARPS = 8;                     // epilogue warps
constexpr int R_THREADS = 32 * (RE_WARPS + 2);  // and a loading and an issuing warp
constexpr size_t R_SMEM = R_STAGES * (RA_STAGE + RB_STAGE) + 128;
constexpr uint32_t R_COLS = RD * RN;            // accumulator columns of a block

// Digits of eight consecutive-orbital values (the 16-byte core-matrix row of
// each plane): v's integers against the largest biased exponent em.
__device__ __forceinline__ void digits8_b7(const double (&v)[8], int em, uint4 (&d)[RD]) {
  constexpr unsigned long long BIAS = 0x0081020408102040ULL;  // 64 (128^8 - 1) / 127
  uint32_t w[RD][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    unsigned long long Y[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const unsigned h = (unsigned)__double2hiint(v[2 * i + q]);
      const unsigned l = (unsigned)__double2loint(v[2 * i + q]);
      const unsigned e = (h >> 20) & 0x7FFu;
      const unsigned long long m =
          ((unsigned long long)((h & 0xFFFFFu) | 0x100000u) << 32) | (unsigned long long)l;
      unsigned long long X = e == 0u ? 0ULL : shr64c(m << 2, (unsigned)em - e);
      if ((int)h < 0) X = 0ULL - X;
      Y[q] = X + BIAS;
    }
#pragma unroll
    for (int k = 0; k < RD; ++k) {
      const unsigned mask = k == 0 ? 0xFFu : 0x7Fu;
      const unsigned b0 = (unsigned)(Y[0] >> (49 - 7 * k)) & mask;
      const unsigned b1 = (unsigned)(Y[1] >> (49 - 7 * k)) & mask;
      // FP16 1024 + b from the pattern 0x64bb, less 1088
      asm("add.rn.f16x2 %0, %1, %2;"
          : "=r"(w[k][i])
          : "r"(0x64006400u + b0 + (b1 << 16)), "r"(0xE440E440u));
    }
  }
#pragma unroll
  for (int k = 0; k < RD; ++k) d[k] = make_uint4(w[k][0], w[k][1], w[k][2], w[k][3]);
}

__device__ __forceinline__ int biased_exp(double v) { return (__double2hiint(v) >> 20) & 0x7FF; }

// U's digit image: CTA per block of 32 outputs, ub[block][stage][k group 4096
// B][(plane 32 + i) 16 B], fexp[i] the column's largest biased exponent.
__global__ void __launch_bounds__(256)
    k_rot_udigits(const double* __restrict__ U, int n, int nst, unsigned char* __restrict__ ub,
                  int* __restrict__ fexp) {
  __shared__ int em[RN];
  const int li = threadIdx.x % RN, g = threadIdx.x / RN, i = blockIdx.x * RN + li;
  if (threadIdx.x < RN) em[threadIdx.x] = 0;
  __syncthreads();
  int e = 0;
  if (i < n)
    for (int j = g; j < n; j += 8) e = max(e, biased_exp(U[(size_t)j * n + i]));
  atomicMax(&em[li], e);
  __syncthreads();
  if (threadIdx.x < RN) fexp[blockIdx.x * RN + threadIdx.x] = em[threadIdx.x];
  for (int kg = g; kg < nst * (RK / 8); kg += 8) {
    double v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = (i < n && 8 * kg + q < n) ? U[(size_t)(8 * kg + q) * n + i] : 0.0;
    uint4 d[RD];
    digits8_b7(v, em[li], d);
    unsigned char* dst = ub + ((size_t)blockIdx.x * nst + kg / (RK / 8)) * RB_STAGE + (kg % (RK / 8)) * RB_LBO;
#pragma unroll
    for (int l = 0; l < RD; ++l) *reinterpret_cast<uint4*>(dst + (l * RN + li) * 16) = d[l];
  }
}

// phi's digit image of the slab's tiles (points r0 + 128 blockIdx.x ..), four
// threads a point:
// ab[tile][stage][plane 4 KB][k group 2 KB][point 16 B], eexp[tile][point].
constexpr int RQ = 4;
__global__ void __launch_bounds__(RT* RQ)
    k_rot_digits(const double* __restrict__ phi, int n, size_t N, size_t r0, int nst,
                 unsigned char* __restrict__ ab, int* __restrict__ eexp) {
  __shared__ int em[RQ][RT];
  const int p = threadIdx.x % RT, part = threadIdx.x / RT;
  const size_t r = r0 + (size_t)blockIdx.x * RT + p;
  const double* src = phi + r;
  int e = 0;
  if (r < N)
    for (int j = part; j < n; j += RQ) e = max(e, biased_exp(src[(size_t)j * N]));
  em[part][p] = e;
  __syncthreads();
  for (int q = 0; q < RQ; ++q) e = max(e, em[q][p]);
  if (part == 0) eexp[blockIdx.x * RT + p] = e;
  for (int kg = part; kg < nst * (RK / 8); kg += RQ) {
    double v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = (r < N && 8 * kg + q < n) ? src[(size_t)(8 * kg + q) * N] : 0.0;
    uint4 d[RD];
    digits8_b7(v, e, d);
    unsigned char* dst =
        ab + ((size_t)blockIdx.x * nst + kg / (RK / 8)) * RA_STAGE + (kg % (RK / 8)) * RA_LBO + p * 16;
#pragma unroll
    for (int k = 0; k < RD; ++k) *reinterpret_cast<uint4*>(dst + k * RA_PLANE) = d[k];
  }
}

__global__ void __launch_bounds__(R_THREADS, 1)
    k_rot_gemm(const unsigned char* __restrict__ ab, const unsigned char* __restrict__ ub,
               const int* __restrict__ eexp, const int* __restrict__ fexp, int n, size_t N,
               size_t r0, int nst, double* __restrict__ out, unsigned* __restrict__ status) {
  extern __shared__ unsigned char rt_raw[];
  unsigned char* sA = rt_raw + ((128 - (smem_addr(rt_raw) & 127)) & 127);
  unsigned char* sB = sA + R_STAGES * RA_STAGE;
  __shared__ __align__(8) unsigned long long b_full[R_STAGES], b_free[R_STAGES], b_acc[2], b_read[2],
      b_fin;
  __shared__ uint32_t tmem_base;
  __shared__ volatile int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) tmem_alloc(&tmem_base, 2 * R_COLS);
  if (tid == 0) {
    for (int q = 0; q < R_STAGES; ++q) {
      mbar_init(smem_addr(&b_full[q]), 1);
      mbar_init(smem_addr(&b_free[q]), 1);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(smem_addr(&b_acc[q]), 1);
      mbar_init(smem_addr(&b_read[q]), RE_WARPS);
    }
    mbar_init(smem_addr(&b_fin), 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
    s_fail = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  const int nib = (n + RN - 1) / RN, nseg = (nst + RSEG - 1) / RSEG;

  if (warp == RE_WARPS) {
    // ---- loading thread: the stages in order, A of the tile, B of the block
    if (lane == 0) {
      int s = 0;
      bool ok = true;
      for (int ib = 0; ib < nib && ok; ++ib)
        for (int k = 0; k < nst; ++k, ++s) {
          const int q = s % R_STAGES, use = s / R_STAGES;
          if (use >= 1) ok = mbar_wait(smem_addr(&b_free[q]), (uint32_t)((use - 1) & 1));
          if (!ok || s_fail) {
            ok = false;
            break;
          }
          const uint32_t bar = smem_addr(&b_full[q]);
          mbar_expect_tx(bar, RA_STAGE + RB_STAGE);
          bulk_load(smem_addr(sA + q * RA_STAGE), ab + ((size_t)blockIdx.x * nst + k) * RA_STAGE,
                    RA_STAGE, bar);
          bulk_load(smem_addr(sB + q * RB_STAGE), ub + ((size_t)ib * nst + k) * RB_STAGE, RB_STAGE,
                    bar);
        }
      if (!ok) s_fail = 1;
      // copies in flight land before the shared memory is released
      for (int t = max(0, s - R_STAGES); t < s; ++t)
        mbar_wait(smem_addr(&b_full[t % R_STAGES]), (uint32_t)((t / R_STAGES) & 1));
    }
    __syncwarp();
  } else if (warp == RE_WARPS + 1) {
    // ---- issuing thread
    if (lane == 0) {
      int s = 0, u = 0;  // stages, accumulations
      bool ok = true;
      for (int ib = 0; ib < nib && ok; ++ib)
        for (int seg = 0; seg < nseg && ok; ++seg, ++u) {
          const int buf = u & 1;
          if (u >= 2) ok = mbar_wait(smem_addr(&b_read[buf]), (uint32_t)((u / 2 - 1) & 1));
          const uint32_t dcol = tmem + (uint32_t)buf * R_COLS;
          const int k1 = min(nst, (seg + 1) * RSEG);
          for (int k = seg * RSEG; k < k1 && ok; ++k, ++s) {
            const int q = s % R_STAGES;
            ok = ok && !s_fail && mbar_wait(smem_addr(&b_full[q]), (uint32_t)((s / R_STAGES) & 1));
            if (!ok) break;
            tc_fence_after();
#pragma unroll
            for (int h = 0; h < RK / 16; ++h) {
              const uint64_t b = sdesc(smem_addr(sB + q * RB_STAGE) + h * 2 * RB_LBO, RB_LBO, 128);
#pragma unroll
              for (int d = 0; d < RD; ++d) {
                const uint64_t a =
                    sdesc(smem_addr(sA + q * RA_STAGE) + d * RA_PLANE + h * 2 * RA_LBO, RA_LBO, 128);
                mma_kf16(dcol + (uint32_t)(d * RN), a, b, idesc_kf16((RD - d) * RN, RT, false),
                         (d > 0 || h > 0 || k > seg * RSEG) ? 1u : 0u);
              }
            }
            mma_commit(smem_addr(&b_free[q]));
          }
          if (ok) mma_commit(smem_addr(&b_acc[buf]));
        }
      if (!ok) s_fail = 1;
      // every MMA issued is done before the tensor memory is freed
      mma_commit(smem_addr(&b_fin));
      mbar_wait(smem_addr(&b_fin), 0);
    }
    __syncwarp();
  } else {
    // ---- epilogue: warp w, points 32 (w % 4) .. + 31, outputs 16 (w / 4) .. + 15
    const int p = 32 * (warp & 3) + lane, i0 = 16 * (warp >> 2);
    const size_t r = r0 + (size_t)blockIdx.x * RT + p;
    const int ee = eexp[blockIdx.x * RT + p] - 2 * 1022 - 61;
    const uint32_t la = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)i0;
    int u = 0;
    bool ok = true;
    for (int ib = 0; ib < nib && ok; ++ib)
      for (int seg = 0; seg < nseg; ++seg, ++u) {
        const int buf = u & 1;
        ok = !s_fail && mbar_wait(smem_addr(&b_acc[buf]), (uint32_t)((u / 2) & 1));
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
#pragma unroll 1
        for (int g = 0; g < 2; ++g) {
          uint32_t f[RD][8];
#pragma unroll
          for (int d = 0; d < RD; ++d) tmem_ld8(la + (uint32_t)(buf * R_COLS + d * RN + 8 * g), f[d]);
          tmem_wait_ld();
          if (g == 1) {  // the buffer is read: the next MMAs may overwrite it
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_addr(&b_read[buf]));
          }
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const int i = ib * RN + i0 + 8 * g + c;
            // integers of at most 2^24, exact in FP32
            long long hi = 0, lo = 0;
#pragma unroll
            for (int d = 0; d < 4; ++d) {
              hi += (long long)__float2int_rz(__uint_as_float(f[d][c])) << (7 * (3 - d));
              lo += (long long)__float2int_rz(__uint_as_float(f[d + 4][c])) << (7 * (3 - d));
            }
            if (r < N && i < n) {
              double y = fix_to_double(hi, lo, ee + fexp[i]);
              double* o = out + (size_t)i * N + r;
              if (seg > 0) y += *o;
              *o = y;
            }
          }
        }
      }
    if (!ok && lane == 0) s_fail = 1;
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && s_fail) atomicOr(status, SEA_FLAG_WAIT);
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 2 * R_COLS);
  }
}

}  // namespace

// out[i][r] = sum_j U[j][i] phi[j][r] (n x n U, n x N phi and out) on c's
// stream, the digit images in c->rot.
cudaError_t launch_rotate(sea_ctx* c, const double* phi, int n, size_t N, const double* U,
                          double* out) {
  cudaError_t e =
      cudaFuncSetAttribute(k_rot_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)R_SMEM);
  if (e != cudaSuccess) return e;
  int nsm = 0;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device);
  const int nst = (n + RK - 1) / RK, nib = (n + RN - 1) / RN;
  const size_t tile_bytes = (size_t)nst * RA_STAGE, tiles = (N + RT - 1) / RT;
  // whole waves of CTAs whose digit images fill at most about 3/4 of L2
  const size_t waves = std::max<size_t>(1, (96u << 20) / (tile_bytes * nsm));
  const size_t slab = std::min(tiles, waves * nsm);
  const size_t ubytes = (size_t)nib * nst * RB_STAGE;
  if (!sea_ensure(c, c->rot, slab * tile_bytes + ubytes + (slab * RT + (size_t)nib * RN) * sizeof(int)))
    return cudaErrorMemoryAllocation;
  unsigned char* ab = (unsigned char*)c->rot.p;
  unsigned char* ub = ab + slab * tile_bytes;
  int* eexp = (int*)(ub + ubytes);
  int* fexp = eexp + slab * RT;
  k_rot_udigits<<<nib, 256, 0, c->stream>>>(U, n, nst, ub, fexp);
  c->launches += 1;
  for (size_t t0 = 0; t0 < tiles; t0 += slab) {
    const unsigned g = (unsigned)std::min(slab, tiles - t0);
    k_rot_digits<<<g, RT * RQ, 0, c->stream>>>(phi, n, N, t0 * RT, nst, ab, eexp);
    k_rot_gemm<<<g, R_THREADS, R_SMEM, c->stream>>>(ab, ub, eexp, fexp, n, N, t0 * RT, nst, out,
                                                   (unsigned*)c->status.p);
    c->launches += 2;
  }
  return cudaGetLastError();
}

}  // namespace sea
