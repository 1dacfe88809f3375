// scdm.cu -- SCDM localization of canonical orbitals (Sec. II A).
//
//   Phi^T Pi = Q R               column-pivoted QR of the n x N matrix Phi^T
//                                (Eq. phi_qr); C = the first n pivots
//   B = (Phi^T)_{:,C}            n x n: B[j][k] = phi_j(r_{C_k})
//   X = Phi B,  P_CC = B^T B     (Eq. nonortho_scdm; X^T X dV = B^T B for
//                                orbitals orthonormal with the grid weight)
//   U = B P_CC^{-1/2},  Phi~ = Phi U   (Eqs. ortho_scdm, unitary_scdm)
//
// Only the pivot order of the QR is needed.  Column-pivoted QR picks, at
// step k, the column whose component orthogonal to the span of the k
// columns already chosen is longest; that component's squared norm c_r only
// falls, so a grid point whose density lies below the current largest c can
// not be the next pivot and needs no work yet.  For localized water orbitals
// the last of the n pivots still has c of about 0.4 of the largest density,
// and 0.1 to 0.5% of the grid points ever come into question.  The candidates
// are sorted into classes of a quarter octave of density; k_scdm_step works on
// the open classes only and opens the next one when the largest c falls below
// its lower edge (the points' coefficients on the pivots so far are then made
// up for).  Ties go to the smallest grid index.  Where the classes kept do not
// suffice (a pivot below 1/64 of the largest density, as for nearly dependent
// orbitals, or too many candidates), every grid point is downdated at every
// step against unit vectors orthogonalized twice (k_scdm_pivot,
// k_scdm_downdate).
// U = B P_CC^{-1/2} is the orthogonal polar factor of B: the Newton-Schulz
// iteration X <- X (3 I - X^T X) / 2 from B over the square root of P_CC's
// largest row sum, until X^T X is the identity to rounding.
#include <algorithm>

#include "cg_fixed.cuh"
#include "sea_internal.cuh"

namespace sea {
namespace {

// c[r] = sum_i phi[i][r]^2 (ascending i, fused multiply-add)
__global__ void k_scdm_norms(const double* __restrict__ phi, int n, size_t N,
                             double* __restrict__ c) {
  const size_t r = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= N) return;
  double s = 0.0;
  for (int i = 0; i < n; ++i) {
    const double v = phi[(size_t)i * N + r];
    s = fma(v, v, s);
  }
  c[r] = s;
}

// Per block: the largest c (ties: smallest index); selected points carry -1.
__global__ void __launch_bounds__(256)
    k_argmax1(const double* __restrict__ c, size_t N, double* __restrict__ bv,
              long long* __restrict__ bi) {
  __shared__ double sv[256];
  __shared__ long long si[256];
  double v = -2.0;
  long long idx = -1;
  for (size_t r = (size_t)blockIdx.x * blockDim.x + threadIdx.x; r < N;
       r += (size_t)gridDim.x * blockDim.x)
    if (c[r] > v) {  // strict: keeps the first (smallest) index of this thread's stride
      v = c[r];
      idx = (long long)r;
    }
  sv[threadIdx.x] = v;
  si[threadIdx.x] = idx;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) {
      const double ov = sv[threadIdx.x + h];
      const long long oi = si[threadIdx.x + h];
      if (ov > sv[threadIdx.x] || (ov == sv[threadIdx.x] && oi >= 0 && (si[threadIdx.x] < 0 || oi < si[threadIdx.x]))) {
        sv[threadIdx.x] = ov;
        si[threadIdx.x] = oi;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    bv[blockIdx.x] = sv[0];
    bi[blockIdx.x] = si[0];
  }
}

// Step k, one CTA: the pivot p = argmax over the block results; a = column
// p of Phi^T; two passes of classical Gram-Schmidt against Q[0..k); q_k =
// a / ||a|| into Q[k]; C[k] = p.
__global__ void __launch_bounds__(1024)
    k_scdm_pivot(const double* __restrict__ bv, const long long* __restrict__ bi, int nb,
                 const double* __restrict__ phi, int n, size_t N, int k, double* __restrict__ Q,
                 long long* __restrict__ C, double* __restrict__ work, unsigned* __restrict__ status) {
  __shared__ double sv[1024];
  __shared__ long long si[1024];
  double v = -2.0;
  long long idx = -1;
  for (int b = threadIdx.x; b < nb; b += blockDim.x)
    if (bv[b] > v || (bv[b] == v && bi[b] >= 0 && (idx < 0 || bi[b] < idx))) {
      v = bv[b];
      idx = bi[b];
    }
  sv[threadIdx.x] = v;
  si[threadIdx.x] = idx;
  __syncthreads();
  for (int h = 512; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) {
      const double ov = sv[threadIdx.x + h];
      const long long oi = si[threadIdx.x + h];
      if (ov > sv[threadIdx.x] || (ov == sv[threadIdx.x] && oi >= 0 && (si[threadIdx.x] < 0 || oi < si[threadIdx.x]))) {
        sv[threadIdx.x] = ov;
        si[threadIdx.x] = oi;
      }
    }
    __syncthreads();
  }
  const long long p = si[0];
  if (p < 0) {  // no point left: the orbitals are rank deficient
    if (threadIdx.x == 0) atomicOr(status, SEA_FLAG_NOT_PD);
    return;
  }
  double* a = work;          // [n]
  double* coef = work + n;   // [k]
  for (int i = threadIdx.x; i < n; i += blockDim.x) a[i] = phi[(size_t)i * N + p];
  __syncthreads();
  for (int pass = 0; pass < 2; ++pass) {
    for (int l = threadIdx.x; l < k; l += blockDim.x) {
      double s = 0.0;
      for (int i = 0; i < n; ++i) s = fma(Q[(size_t)l * n + i], a[i], s);
      coef[l] = s;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      double s = a[i];
      for (int l = 0; l < k; ++l) s = fma(-coef[l], Q[(size_t)l * n + i], s);
      a[i] = s;
    }
    __syncthreads();
  }
  double nn = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) nn = fma(a[i], a[i], nn);
  __shared__ double red[1024];
  red[threadIdx.x] = nn;
  __syncthreads();
  for (int h = 512; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  const double inv = red[0] > 0.0 ? 1.0 / sqrt(red[0]) : 0.0;
  if (!(red[0] > 0.0) && threadIdx.x == 0) atomicOr(status, SEA_FLAG_NOT_PD);
  for (int i = threadIdx.x; i < n; i += blockDim.x) Q[(size_t)k * n + i] = a[i] * inv;
  if (threadIdx.x == 0) C[k] = p;
}

// c[r] -= (q_k . a_r)^2 for every grid point; the pivot is marked -1.
__global__ void k_scdm_downdate(const double* __restrict__ phi, int n, size_t N,
                                const double* __restrict__ q, const long long* __restrict__ Ck,
                                double* __restrict__ c) {
  extern __shared__ double sq[];
  for (int i = threadIdx.x; i < n; i += blockDim.x) sq[i] = q[i];
  __syncthreads();
  const size_t r = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= N) return;
  if ((long long)r == *Ck) {
    c[r] = -1.0;
    return;
  }
  if (c[r] < 0.0) return;
  double d = 0.0;
  for (int i = 0; i < n; ++i) d = fma(sq[i], phi[(size_t)i * N + r], d);
  c[r] = fma(-d, d, c[r]);
}

// ---- pivots among the candidates --------------------------------------
constexpr int SC_CLASSES = 24;   // quarter octaves below the largest density
constexpr int SC_THREADS = 512;  // of k_scdm_step
constexpr int SC_ROW = 4;        // its registers for a candidate's row

// The class of density c against the largest cmax: floor(4 log2(cmax / c)),
// decided on cmax 2^(-m/4) (edge m: the lower edge of class m - 1).
__device__ __forceinline__ double sc_edge(double cmax, int m) {
  const double f = (m & 3) == 0 ? 1.0
                   : (m & 3) == 1 ? 0.84089641525371454
                   : (m & 3) == 2 ? 0.70710678118654752 : 0.59460355750136054;
  return cmax * f * (1.0 / (double)(1 << (m >> 2)));
}

// The classes' edges edge[0..SC_CLASSES] from the block maxima of k_argmax1; one
// CTA.  cnt[0..SC_CLASSES] = 0.
__global__ void __launch_bounds__(1024)
    k_scdm_edges(const double* __restrict__ bv, int nb, double* __restrict__ edge,
                 int* __restrict__ cnt) {
  __shared__ double red[32];
  double v = -2.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) v = fmax(v, bv[b]);
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x <= SC_CLASSES) {
    v = red[0];
    for (int w = 1; w < (int)blockDim.x / 32; ++w) v = fmax(v, red[w]);
    edge[threadIdx.x] = sc_edge(v, threadIdx.x);
    cnt[threadIdx.x] = 0;
  }
}

// mode 0: counts the grid points per class; mode 1: writes their indices to
// list at the classes' places (cnt then holds running positions).  The order
// within a class does not matter: a pivot is chosen by value, then index.
__global__ void __launch_bounds__(256)
    k_scdm_classes(const double* __restrict__ c, size_t N, const double* __restrict__ edge_g,
                   int mode, int cap, int* __restrict__ cnt, int* __restrict__ list) {
  __shared__ int n_of[SC_CLASSES], at[SC_CLASSES];
  __shared__ double edge[SC_CLASSES + 1];
  if (threadIdx.x <= SC_CLASSES) edge[threadIdx.x] = edge_g[threadIdx.x];
  const size_t per = (N + gridDim.x - 1) / gridDim.x;
  const size_t b0 = min(N, per * blockIdx.x), b1 = min(N, b0 + per);
  if (threadIdx.x < SC_CLASSES) n_of[threadIdx.x] = 0;
  __syncthreads();
  for (int pass = 0; pass <= mode; ++pass) {
    for (size_t r = b0 + threadIdx.x; r < b1; r += blockDim.x) {
      const double v = c[r];
      if (!(v >= edge[SC_CLASSES])) continue;
      int m = 0;
      while (m < SC_CLASSES - 1 && v < edge[m + 1]) ++m;
      const int k = atomicAdd(pass == 0 ? &n_of[m] : &at[m], 1);
      if (pass == 1 && k < cap) list[k] = (int)r;
    }
    __syncthreads();
    if (pass == 0 && threadIdx.x < SC_CLASSES)
      at[threadIdx.x] = n_of[threadIdx.x] ? atomicAdd(&cnt[threadIdx.x], n_of[threadIdx.x]) : 0;
    __syncthreads();
  }
}

// start[m] = first candidate of class m (start[SC_CLASSES]: their number),
// cnt[m] = the same, for k_scdm_classes mode 1.
__global__ void k_scdm_starts(int* __restrict__ cnt, int* __restrict__ start) {
  int s = 0;
  for (int m = 0; m < SC_CLASSES; ++m) {
    const int n = cnt[m];
    cnt[m] = start[m] = s;
    s += n;
  }
  start[SC_CLASSES] = s;
}

// A[a][i] = phi[i][list[a]], cA[a] = c[list[a]]: a warp per candidate.
__global__ void __launch_bounds__(256)
    k_scdm_collect(const double* __restrict__ phi, int n, size_t N, const int* __restrict__ list,
                   int na, const double* __restrict__ c, double* __restrict__ A,
                   double* __restrict__ cA) {
  const int a = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (a >= na) return;
  const int r = list[a];
  for (int i = lane; i < n; i += 32) A[(size_t)a * n + i] = phi[(size_t)i * N + r];
  if (lane == 0) cA[a] = c[r];
}

// State between steps: pivots found, classes open.  stop: 1 when the
// candidates no longer decide the next pivot.
struct ScState {
  int k, open, stop;
};
struct ScMax {
  double v;
  int r, a;  // grid index, candidate
};
// FP64 values compared as integers (no FP64 instruction), which is their order
// wherever one of them is positive, as every pivot's is.
__device__ __forceinline__ bool sc_better(const ScMax& x, const ScMax& y) {
  const long long a = __double_as_longlong(x.v), b = __double_as_longlong(y.v);
  return a > b || (a == b && x.r < y.r);
}

// One step of the greedy pivot choice (a launch each; the launch boundary is
// the barrier between steps).  From the CTAs' largest c of the step before:
// if the largest lies in the open classes it is the next pivot p and every
// open candidate r gets L[r][k] = q_k . a_r, with
//   (q_k . a_r) = (a_p . a_r - sum_{j<k} L[p][j] L[r][j]) / sqrt(c_p),
// and c_r -= L[r][k]^2; else the next class is opened and its candidates'
// L[r][0..k) formed.  A warp per candidate, the lanes over the orbitals; the
// lanes' sums are added as integers (no FP64 instruction).
// A step is a chain of latencies: the loads that need no result of the step
// before come first, the CTAs of the next step are resident before this one
// ends (programmatic launch: only the wait for the predecessor's results
// remains), and the maxima are compared as integers (as FP64, every warp's
// twenty compares took as long as the dot products).  128 pivots on 72x75x76:
// 14.3 -> 8.3 us a step.
__global__ void __launch_bounds__(SC_THREADS)
    k_scdm_step(const double* __restrict__ A, int n, const int* __restrict__ list,
                const int* __restrict__ start, const int* __restrict__ n_kept,
                const double* __restrict__ edge, double* cA, double* L,
                const ScMax* mx_in, ScMax* mx_out, const ScState* st_in, ScState* st_out,
                int first_open, int* piv_a, long long* __restrict__ C) {
  extern __shared__ double sp[];  // pivot's a_p [n], -L[p] [n], 1 / sqrt(c_p)
  __shared__ ScMax wb[SC_THREADS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gw = blockIdx.x * (SC_THREADS / 32) + warp, nw = gridDim.x * (SC_THREADS / 32);
  const int kept = *n_kept;
  // this warp's first candidate: its row and index do not change between steps
  const bool has = gw < kept;
  double row[SC_ROW];
#pragma unroll
  for (int u = 0; u < SC_ROW; ++u)
    row[u] = has && lane + 32 * u < n ? A[(size_t)gw * n + lane + 32 * u] : 0.0;
  const int r0 = has ? list[gw] : 0;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the step before has ended
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const ScState st0 = *st_in;
  const double c0 = has ? cA[gw] : 0.0;
  ScState st = st0;
  if (st.k >= n || st.stop) {
    if (threadIdx.x == 0 && blockIdx.x == 0) *st_out = st;
    return;
  }
  auto warp_best = [&](ScMax b) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      ScMax y;
      y.v = __shfl_xor_sync(0xffffffffu, b.v, o);
      y.r = __shfl_xor_sync(0xffffffffu, b.r, o);
      y.a = __shfl_xor_sync(0xffffffffu, b.a, o);
      if (sc_better(y, b)) b = y;
    }
    return b;
  };
  // the largest c of the open candidates
  ScMax best{-2.0, 0x7fffffff, -1};
  for (int b = lane; b < (int)gridDim.x; b += 32) {
    const ScMax y = mx_in[b];
    if (sc_better(y, best)) best = y;
  }
  best = warp_best(best);
  // a pivot must not lie below the open classes' lower edge (a closed
  // candidate could be larger) and be positive (with no density at all every
  // edge is 0: the classes then run out and the pass over all points reports it)
  const long long bits = __double_as_longlong(best.v);
  const bool decide = st.open > 0 && bits > 0 && bits >= __double_as_longlong(edge[st.open]);
  ScMax mine{-2.0, 0x7fffffff, -1};
  auto keep = [&](double v, int a) {
    const ScMax y{v, a == gw ? r0 : list[a], a};
    if (sc_better(y, mine)) mine = y;
  };
  auto dot = [&](const double* x, const double* y, int m, double s, double f) {
    for (int i = lane; i < m; i += 32) s = fma(f * x[i], y[i], s);
    return s;
  };
  auto total = [&](double s) {
    const FixSum w = fix_warp_sum(s);
    return scaled_i64(w.X, w.e - 1080);
  };
  if (decide) {
    const double* ap = A + (size_t)best.a * n;
    const double* lp = L + (size_t)best.a * n;
    for (int i = threadIdx.x; i < n; i += SC_THREADS) {
      sp[i] = ap[i];
      sp[n + i] = i < st.k ? -lp[i] : 0.0;
    }
    if (threadIdx.x == 0) sp[2 * n] = 1.0 / sqrt(best.v);
    __syncthreads();
    const double inv = sp[2 * n];
    const int end = min(start[st.open], kept);
    for (int a = gw; a < end; a += nw) {
      double c = a == gw ? c0 : cA[a];
      if (a == best.a) {
        c = -1.0;
      } else if (__double2hiint(c) >= 0) {
        double s = 0.0;
        if (a == gw && n <= 32 * SC_ROW) {
#pragma unroll
          for (int u = 0; u < SC_ROW; ++u)
            if (lane + 32 * u < n) s = fma(row[u], sp[lane + 32 * u], s);
        } else {
          s = dot(A + (size_t)a * n, sp, n, 0.0, 1.0);
        }
        s = dot(L + (size_t)a * n, sp + n, st.k, s, 1.0);
        const double d = total(s) * inv;
        c = fma(-d, d, c);
        if (lane == 0) L[(size_t)a * n + st.k] = d;
      }
      if (lane == 0) cA[a] = c;
      keep(c, a);
    }
    if (threadIdx.x == 0 && blockIdx.x == 0) {
      piv_a[st.k] = best.a;
      C[st.k] = best.r;
      // the pivot's c, for the candidates opened later
      cA[kept + st.k] = best.v;
    }
    ++st.k;
  } else {
    // open the next class (at the start the first first_open ones), if it was
    // kept whole
    const int open = st.open == 0 ? first_open : st.open + 1;
    if (open > SC_CLASSES || start[open] > kept) {
      st.stop = 1;
    } else {
      const int b0 = start[st.open], end = start[open];
      for (int a = gw; a < end; a += nw) {
        if (a < b0) {  // already open: its c stands
          keep(cA[a], a);
          continue;
        }
        double c = cA[a];
        for (int k = 0; k < st.k; ++k) {
          const int pa = piv_a[k];
          double s = dot(A + (size_t)a * n, A + (size_t)pa * n, n, 0.0, 1.0);
          s = dot(L + (size_t)a * n, L + (size_t)pa * n, k, s, -1.0);
          const double d = total(s) / sqrt(cA[kept + k]);
          c = fma(-d, d, c);
          if (lane == 0) L[(size_t)a * n + k] = d;
          __syncwarp();
        }
        if (lane == 0) cA[a] = c;
        keep(c, a);
      }
      st.open = open;
    }
  }
  if (lane == 0) wb[warp] = mine;
  __syncthreads();
  if (warp == 0) {
    mine = warp_best(lane < SC_THREADS / 32 ? wb[lane] : ScMax{-2.0, 0x7fffffff, -1});
    if (lane == 0) {
      mx_out[blockIdx.x] = mine;
      if (blockIdx.x == 0) *st_out = st;
    }
  }
}

// B[j][k] = phi[j][C[k]]
__global__ void k_scdm_gather(const double* __restrict__ phi, int n, size_t N,
                              const long long* __restrict__ C, double* __restrict__ B) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * n) return;
  const int j = t / n, k = t % n;
  B[t] = phi[(size_t)j * N + C[k]];
}

// *s = 1 / sqrt(largest row sum of |P|) (one CTA): at most the inverse of P's
// largest singular value's root.
__global__ void __launch_bounds__(1024)
    k_row_bound(const double* __restrict__ P, int n, double* __restrict__ s) {
  __shared__ double red[32];
  double m = 0.0;
  for (int i = threadIdx.x >> 5; i < n; i += 32) {
    double v = 0.0;
    for (int j = threadIdx.x & 31; j < n; j += 32) v += fabs(P[(size_t)i * n + j]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    m = fmax(m, v);
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 32; ++w) m = fmax(m, red[w]);
    *s = m > 0.0 ? 1.0 / sqrt(m) : 0.0;
  }
}

// X = f B
__global__ void k_scale(const double* __restrict__ B, int n2, const double* __restrict__ f,
                        double* __restrict__ X) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n2) X[t] = B[t] * *f;
}

// One Newton-Schulz product on n x n matrices (row-major).  step 0: T =
// X^T X, and *dev = max |T - I| over the entries (as its bit pattern, by
// atomicMax; zeroed by the caller); step 1: Y = X (3 I - T) / 2.  Tiles of 16
// x 8 outputs by 128 threads, so that n = 128 gives 128 CTAs.
__global__ void __launch_bounds__(128)
    k_ns_product(const double* __restrict__ X, const double* __restrict__ T, int n, int step,
                 double* __restrict__ out, unsigned long long* __restrict__ dev) {
  __shared__ double As[32][17], Bs[32][9];
  const int i0 = blockIdx.y * 16, j0 = blockIdx.x * 8;
  const int ti = threadIdx.x >> 3, tj = threadIdx.x & 7;
  double acc = 0.0;
  for (int k0 = 0; k0 < n; k0 += 32) {
    for (int q = threadIdx.x; q < 32 * 16; q += 128) {
      // step 0 reads X[k][i] (i fastest), step 1 X[i][k] (k fastest)
      const int k = step ? q % 32 : q / 16, i = step ? q / 32 : q % 16;
      const bool in = i0 + i < n && k0 + k < n;
      As[k][i] = in ? (step ? X[(size_t)(i0 + i) * n + k0 + k] : X[(size_t)(k0 + k) * n + i0 + i])
                    : 0.0;
    }
    for (int q = threadIdx.x; q < 32 * 8; q += 128) {
      const int k = q / 8, j = q % 8;
      double v = 0.0;
      if (j0 + j < n && k0 + k < n) {
        if (step)
          v = 0.5 * ((k0 + k == j0 + j ? 3.0 : 0.0) - T[(size_t)(k0 + k) * n + j0 + j]);
        else
          v = X[(size_t)(k0 + k) * n + j0 + j];
      }
      Bs[k][j] = v;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 32; ++k) acc = fma(As[k][ti], Bs[k][tj], acc);
    __syncthreads();
  }
  const int i = i0 + ti, j = j0 + tj;
  double d = 0.0;
  if (i < n && j < n) {
    out[(size_t)i * n + j] = acc;
    d = fabs(acc - (i == j ? 1.0 : 0.0));
  }
  if (step == 0) {
    unsigned long long b = (unsigned long long)__double_as_longlong(d);  // ordered as integers
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long y = __shfl_xor_sync(0xffffffffu, b, o);
      b = y > b ? y : b;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(dev, b);
  }
}

}  // namespace

// The pivots among the candidates; *done = false if they do not decide all
// n of them.  cn: the densities; bv: their block maxima (nb).
static cudaError_t pivots_lazy(sea_ctx* c, const double* cn, const double* bv, int nb,
                               long long* C_dev, bool* done) {
  const int n = c->n_orb;
  const size_t N = c->ng;
  cudaStream_t st = c->stream;
  *done = false;
  int nsm = 0;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device);
  // small state: class edges, counts and starts, step states and maxima
  const size_t small = 256 + 4 * (SC_CLASSES + 1) * 4 + 64 + 2 * (size_t)nsm * sizeof(ScMax) + n * 4;
  if (!sea_ensure(c, c->scdm_s, small)) return cudaErrorMemoryAllocation;
  char* q = (char*)c->scdm_s.p;
  double* edge = (double*)q;
  int* cnt = (int*)(q + 256);
  int* start = cnt + SC_CLASSES + 1;
  int* kept = start + SC_CLASSES + 1;
  ScState* state = (ScState*)(kept + 1);
  ScMax* mx = (ScMax*)(q + ((256 + (2 * (SC_CLASSES + 1) + 1) * 4 + 2 * sizeof(ScState) + 15) & ~(size_t)15));
  int* piv_a = (int*)(mx + 2 * nsm);
  k_scdm_edges<<<1, 1024, 0, st>>>(bv, nb, edge, cnt);
  k_scdm_classes<<<4 * nsm, 256, 0, st>>>(cn, N, edge, 0, 0, cnt, nullptr);
  k_scdm_starts<<<1, 1, 0, st>>>(cnt, start);
  int hs[SC_CLASSES + 1];
  cudaMemcpyAsync(hs, start, sizeof(hs), cudaMemcpyDeviceToHost, st);
  cudaError_t e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return e;
  // whole classes, at most 256 n candidates and 256 MB of rows and L
  const long long cap = std::min<long long>(256LL * n, (256LL << 20) / (16LL * n));
  int m = 0;
  while (m < SC_CLASSES && hs[m + 1] <= cap) ++m;
  const int na = hs[m];
  if (na < n) return cudaSuccess;
  if (!sea_ensure(c, c->scdm_a, (size_t)na * n * 2 * sizeof(double) + (size_t)(na + n) * sizeof(double) +
                                    (size_t)na * sizeof(int)))
    return cudaErrorMemoryAllocation;
  double* A = (double*)c->scdm_a.p;
  double* L = A + (size_t)na * n;
  double* cA = L + (size_t)na * n;
  int* list = (int*)(cA + na + n);
  k_scdm_classes<<<4 * nsm, 256, 0, st>>>(cn, N, edge, 1, na, cnt, list);
  k_scdm_collect<<<(na + 7) / 8, 256, 0, st>>>((const double*)c->vxx_dev.p, n, N, list, na, cn, A, cA);
  const int smem = (2 * n + 1) * (int)sizeof(double);
  if (smem > 48 * 1024) {
    e = sea_allow_smem((const void*)k_scdm_step, smem);
    if (e != cudaSuccess) return e;
  }
  cudaMemcpyAsync(kept, &na, sizeof(int), cudaMemcpyHostToDevice, st);
  cudaMemsetAsync(state, 0, sizeof(ScState), st);
  cudaMemsetAsync(mx, 0xff, (size_t)nsm * sizeof(ScMax), st);  // NaN: no class is open
  // at the start as many classes as two candidates a warp make: their c is
  // kept up to date at every step, which costs less than making up for their
  // coefficients later (0.14 to 0.42 ms a class at n = 128)
  int first = 1;
  while (first < m && hs[first + 1] <= 2 * nsm * (SC_THREADS / 32)) ++first;
  const int launches = n + m - first + 1;  // every pivot, every opening
  for (int l = 0; l < launches; ++l) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nsm);
    cfg.blockDim = dim3(SC_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute early;
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &early;
    cfg.numAttrs = l > 0;  // the first step reads what ordinary launches wrote
    e = cudaLaunchKernelEx(&cfg, k_scdm_step, (const double*)A, n, (const int*)list,
                           (const int*)start, (const int*)kept, (const double*)edge, cA, L,
                           (const ScMax*)(mx + (l & 1) * nsm), mx + ((l + 1) & 1) * nsm,
                           (const ScState*)(state + (l & 1)), state + ((l + 1) & 1), first, piv_a,
                           C_dev);
    if (e != cudaSuccess) return e;
  }
  ScState hst;
  cudaMemcpyAsync(&hst, state + (launches & 1), sizeof(hst), cudaMemcpyDeviceToHost, st);
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return e;
  c->launches += 5 + launches;
  *done = hst.k >= n;
  return cudaGetLastError();
}

// SCDM on the orbitals in c->vxx_dev (n_orb x ng): U (device, n x n) and the
// pivots C (device, n); the localized orbitals go to c->phi.  Synchronizes
// the context stream.
cudaError_t launch_scdm(sea_ctx* c, double* U_dev, long long* C_dev) {
  const int n = c->n_orb;
  const size_t N = c->ng;
  const int nb = 1024;  // blocks of the first argmax stage
  const size_t nn = (size_t)n * n * sizeof(double);
  if (!sea_ensure(c, c->cand_S, std::max<size_t>(N * sizeof(double), 64)) ||
      !sea_ensure(c, c->Mbuf, nn) ||   // Q (rows q_k), then X
      !sea_ensure(c, c->Lbuf, nn) ||   // B
      !sea_ensure(c, c->Linv, nn) ||   // X^T X
      !sea_ensure(c, c->Abuf, (size_t)(2 * n + 4 * nb + 8) * sizeof(double)))
    return cudaErrorMemoryAllocation;
  const double* phi = (const double*)c->vxx_dev.p;
  double* cn = (double*)c->cand_S.p;
  double* Q = (double*)c->Mbuf.p;
  double* B = (double*)c->Lbuf.p;
  double* T = (double*)c->Linv.p;
  double* work = (double*)c->Abuf.p;        // [n] + [n]
  double* bv = work + 2 * n;                 // [nb]
  long long* bi = (long long*)(bv + nb);     // [nb]
  double* sF = bv + 3 * nb;                  // scalar
  unsigned long long* dev = (unsigned long long*)(sF + 1);
  unsigned* status = (unsigned*)c->status.p;
  cudaStream_t st = c->stream;
  const unsigned gN = (unsigned)((N + 255) / 256);
  k_scdm_norms<<<gN, 256, 0, st>>>(phi, n, N, cn);
  k_argmax1<<<nb, 256, 0, st>>>(cn, N, bv, bi);
  c->launches += 2;
  bool done = false;
  cudaError_t e = N < 0x7fffffff ? pivots_lazy(c, cn, bv, nb, C_dev, &done) : cudaSuccess;
  if (e != cudaSuccess) return e;
  if (!done) {
    for (int k = 0; k < n; ++k) {
      if (k) k_argmax1<<<nb, 256, 0, st>>>(cn, N, bv, bi);
      k_scdm_pivot<<<1, 1024, 0, st>>>(bv, bi, nb, phi, n, N, k, Q, C_dev, work, status);
      k_scdm_downdate<<<gN, 256, (size_t)n * sizeof(double), st>>>(phi, n, N, Q + (size_t)k * n,
                                                                    C_dev + k, cn);
    }
    c->launches += 3 * n;
  }
  // B, then its polar factor: X^T X within 1e-8 of the identity before a step
  // (which squares the deviation, to rounding), or no longer approaching it, ends
  // the iteration
  const unsigned gnn = (unsigned)((n * n + 255) / 256);
  const dim3 gp((n + 7) / 8, (n + 15) / 16);
  k_scdm_gather<<<gnn, 256, 0, st>>>(phi, n, N, C_dev, B);
  k_ns_product<<<gp, 128, 0, st>>>(B, nullptr, n, 0, T, dev);
  k_row_bound<<<1, 1024, 0, st>>>(T, n, sF);
  double *X = Q, *Y = U_dev;
  k_scale<<<gnn, 256, 0, st>>>(B, n * n, sF, X);
  c->launches += 4;
  double last = 1e300;
  for (int it = 0; it < 99; ++it) {
    cudaMemsetAsync(dev, 0, sizeof(*dev), st);
    k_ns_product<<<gp, 128, 0, st>>>(X, nullptr, n, 0, T, dev);
    k_ns_product<<<gp, 128, 0, st>>>(X, T, n, 1, Y, nullptr);
    std::swap(X, Y);
    c->launches += 2;
    double d = 0.0;
    if (it % 3 != 2) continue;
    cudaMemcpyAsync(&d, dev, sizeof(d), cudaMemcpyDeviceToHost, st);
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    // the step just taken squares a deviation d below 1/2
    if (!(d > 1e-8) || (d < 1e-3 && !(d < last))) break;
    last = d;
  }
  if (X != U_dev) cudaMemcpyAsync(U_dev, X, nn, cudaMemcpyDeviceToDevice, st);
  return launch_rotate(c, phi, n, N, U_dev, (double*)c->phi.p);
}

}  // namespace sea
