// Per-cluster dense work of one LowRank_Elimination step (Sec. 2.1):
// factor A_ss, form A_ss^{-1}, compress the fill block with column-pivoted
// Householder QR (Eq. lra), build the complement basis V with
// V^T A_ss^{-1} U = 0, the sparsification rows T = [U V]^T A_ss^{-1}
// (Eq. scaling), factor the fine block F = V^T A_ss^{-1} V (Eq. elim) and fold
// its inverse factor into T.  One CTA per cluster of a colour class; all
// clusters of the class run in one launch.  SPD clusters of up to 256 unknowns
// take the blocked kernel of kernels_spd.cu instead; here are the general ones,
// larger SPD ones and the shared helpers.
//
// Matrices are column-major.  `real` is the storage/compute type of the
// factorization (double in float64 mode, float in the mixed modes); the squared
// column norms of the rank-revealing QR are accumulated in it, and its rank
// decision is made in double.  The factor of A_ss and A_ss^{-1} live in shared
// memory when they fit (the host sizes the dynamic shared memory per class);
// everything else is in a per-cluster global workspace that stays in L2.
#include <cfloat>
#include <climits>
#include <cmath>

#include "common.h"

namespace hs {

namespace {

// threads of the per-cluster kernel: 512 in float32 (more warps share each
// barrier-separated step), 256 in float64 (register budget)
template <typename real>
struct PrepThreads {
  static constexpr int value = sizeof(real) == 4 ? 512 : 256;
};
constexpr double kPivotTieRtol = 1e-10;  // LU pivot search
constexpr int kRowsMax = 256;  // triangular inverses with columns or rows in registers
// near-ties of the column-pivoted QR, relative: 1e-10 in float64; float32
// squared norms carry ~1e-7 relative rounding, so ties of exact arithmetic
// are recognised within 1e-5
template <typename real>
__device__ __forceinline__ double qr_tie_rtol() { return sizeof(real) == 8 ? 1e-10 : 1e-5; }

template <typename real>
__device__ __forceinline__ real sqrt_(real x);
template <>
__device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
template <>
__device__ __forceinline__ float sqrt_(float x) { return sqrtf(x); }

// C (M x N, ldc) = op(A) * op(B), whole CTA, RM x RN outputs per thread straight
// from the operands (shared memory, or the workspace through L1); the sum over l
// runs in ascending order in one accumulator.  A thread's rows are strided so
// that a warp reads consecutive ones.  C must not alias A or B.  (Staging 16
// inner indices at a time instead took two barriers per chunk: 43 us for the
// 128 x 128 x 128 product of [U V]^T A_ss^{-1} in shared memory against 17.)
template <typename real, int RM, int RN>
__device__ __forceinline__ void gemm_tiles(int M, int N, int K, const real* A, int ars, int acs,
                                           const real* B, int brs, int bcs, real* C, int ldc) {
  const int nti = (M + RM - 1) / RM, n = nti * ((N + RN - 1) / RN);
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    const int ti = t % nti, jf = t / nti * RN;
    int ao[RM], bo[RN];
#pragma unroll
    for (int r = 0; r < RM; r++) ao[r] = min(ti + r * nti, M - 1) * ars;
#pragma unroll
    for (int c = 0; c < RN; c++) bo[c] = min(jf + c, N - 1) * bcs;
    real acc[RM][RN];
#pragma unroll
    for (int r = 0; r < RM; r++)
#pragma unroll
      for (int c = 0; c < RN; c++) acc[r][c] = 0;
#pragma unroll 4
    for (int l = 0; l < K; l++) {
      real a[RM], b[RN];
#pragma unroll
      for (int r = 0; r < RM; r++) a[r] = A[ao[r] + l * acs];
#pragma unroll
      for (int c = 0; c < RN; c++) b[c] = B[bo[c] + l * brs];
#pragma unroll
      for (int r = 0; r < RM; r++)
#pragma unroll
        for (int c = 0; c < RN; c++) acc[r][c] += a[r] * b[c];
    }
#pragma unroll
    for (int r = 0; r < RM; r++)
#pragma unroll
      for (int c = 0; c < RN; c++)
        if (ti + r * nti < M && jf + c < N) C[ti + r * nti + (int64_t)(jf + c) * ldc] = acc[r][c];
  }
}

// The same for a transposed A in the workspace, float32: the rows a warp
// multiplies are then a leading dimension apart, so 16 inner indices of 128 rows
// at a time go through shared memory (As, kAtElems), read and written without
// bank conflicts, and a warp multiplies four columns whose elements are the same
// for all lanes.  Straight from memory these products were slower from 133
// unknowns on, where [U V] leaves shared memory: [U V]^T A_ss^{-1} of all clusters
// of 128^2 with leaf size 512 86 ms against 13, L^{-T} L^{-1} with the triangular
// inverse before it 126 against 59, the whole step with leaf size 256
// (convection-diffusion) 50 against 35.  (Float64 is bound by its pipe: 163 ms
// straight for the first, 182 staged.)
constexpr int kAtRows = 128, kAtInner = 16, kAtLd = kAtRows + 2, kAtElems = kAtInner * kAtLd;
__device__ __forceinline__ void gemm_staged_at(int M, int N, int K, const float* A, int lda,
                                               const float* B, int brs, int bcs, float* C, int ldc,
                                               float* As) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int i0 = 0; i0 < M; i0 += kAtRows)
    for (int j0 = 0; j0 < N; j0 += 4 * nw) {
      const int jf = j0 + 4 * warp;
      int bo[4];
#pragma unroll
      for (int c = 0; c < 4; c++) bo[c] = min(jf + c, N - 1) * bcs;
      float acc[4][4];
#pragma unroll
      for (int r = 0; r < 4; r++)
#pragma unroll
        for (int c = 0; c < 4; c++) acc[r][c] = 0;
      for (int l0 = 0; l0 < K; l0 += kAtInner) {
        const int lc = min(kAtInner, K - l0);
        for (int e = threadIdx.x; e < kAtRows * kAtInner; e += blockDim.x) {
          const int l = e % kAtInner, i = e / kAtInner;
          As[l * kAtLd + i] = (i0 + i < M && l < lc) ? A[l0 + l + (i0 + i) * lda] : 0.f;
        }
        __syncthreads();
        if (jf < N) {
#pragma unroll 8
          for (int l = 0; l < lc; l++) {
            float a[4], b[4];
#pragma unroll
            for (int r = 0; r < 4; r++) a[r] = As[l * kAtLd + lane + 32 * r];
#pragma unroll
            for (int c = 0; c < 4; c++) b[c] = B[bo[c] + (l0 + l) * brs];
#pragma unroll
            for (int r = 0; r < 4; r++)
#pragma unroll
              for (int c = 0; c < 4; c++) acc[r][c] += a[r] * b[c];
          }
        }
        __syncthreads();
      }
#pragma unroll
      for (int r = 0; r < 4; r++)
#pragma unroll
        for (int c = 0; c < 4; c++)
          if (i0 + lane + 32 * r < M && jf + c < N)
            C[i0 + lane + 32 * r + (int64_t)(jf + c) * ldc] = acc[r][c];
    }
}

template <typename real>
__device__ void cta_gemm(int M, int N, int K, const real* A, int lda, bool ta, const real* B,
                         int ldb, bool tb, real* C, int ldc) {
  const int ars = ta ? lda : 1, acs = ta ? 1 : lda, brs = tb ? ldb : 1, bcs = tb ? 1 : ldb;
  if constexpr (sizeof(real) == 4) {
    if (ta && !__isShared(A)) {  // uniform
      __shared__ float As[kAtElems];
      gemm_staged_at(M, N, K, A, lda, B, brs, bcs, C, ldc, As);
      __syncthreads();
      return;
    }
  }
  if (M * N >= 12 * (int)blockDim.x)
    gemm_tiles<real, 4, 4>(M, N, K, A, ars, acs, B, brs, bcs, C, ldc);
  else
    gemm_tiles<real, 2, 2>(M, N, K, A, ars, acs, B, brs, bcs, C, ldc);
  __syncthreads();
}

// The helpers below map warps to columns and lanes to rows: column-major
// accesses are then contiguous across a warp, and no per-element index
// division is needed.
__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }
__device__ __forceinline__ int warp_id() { return threadIdx.x >> 5; }
__device__ __forceinline__ int num_warps() { return blockDim.x >> 5; }

template <typename real>
__device__ __forceinline__ real warp_sum(real v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename real>
__device__ void cta_copy(int M, int N, const real* A, int64_t lda, real* B, int64_t ldb) {
  for (int j = warp_id(); j < N; j += num_warps())
    for (int i = lane_id(); i < M; i += 32) B[i + j * ldb] = A[i + j * lda];
  __syncthreads();
}

// Zero the strict upper (upper=true) or strict lower part of an n x n matrix.
template <typename real>
__device__ void cta_zero_tri(int n, real* A, int lda, bool upper) {
  for (int j = warp_id(); j < n; j += num_warps()) {
    const int i0 = upper ? 0 : j + 1, i1 = upper ? j : n;
    for (int i = i0 + lane_id(); i < i1; i += 32) A[i + (int64_t)j * lda] = 0;
  }
  __syncthreads();
}

template <typename real>
__device__ void cta_identity(int M, int N, int diag_off, real* A, int lda) {
  for (int j = warp_id(); j < N; j += num_warps())
    for (int i = lane_id(); i < M; i += 32)
      A[i + (int64_t)j * lda] = (i == j + diag_off) ? real(1) : real(0);
  __syncthreads();
}

// In-place lower Cholesky A = L L^T (lower triangle), right-looking, one
// barrier per step: step j subtracts a_ij a_lj / a_jj from the trailing lower
// triangle and, in the same phase, finishes column j-1 (scaling by
// 1/sqrt(d_{j-1})), which step j does not read.  Returns false on every
// thread for a non-positive pivot.
template <typename real>
__device__ bool cta_cholesky(int n, real* A, int lda, int* sflag) {
  (void)sflag;
  const int lane = lane_id(), warp = warp_id(), nw = num_warps();
  real rprev = 0;  // 1 / sqrt(d_{j-1})
  for (int j = 0; j < n; j++) {
    const real d = A[j + (int64_t)j * lda];
    if (!(d > real(0))) return false;  // uniform: every thread read the same d
    const real invd = real(1) / d;
    if (j > 0) {
      real* cp = A + (int64_t)(j - 1) * lda;
      for (int i = j + threadIdx.x; i < n; i += blockDim.x) cp[i] *= rprev;
    }
    const real* cj = A + (int64_t)j * lda;
    for (int l = j + 1 + warp; l < n; l += nw) {
      const real alj = cj[l] * invd;
      real* cl = A + (int64_t)l * lda;
      for (int i = l + lane; i < n; i += 32) cl[i] -= cj[i] * alj;
    }
    __syncthreads();
    // the diagonal of column j-1 was read as d in the previous step only
    if (j > 0 && threadIdx.x == 0) A[(j - 1) + (int64_t)(j - 1) * lda] = real(1) / rprev;
    rprev = real(1) / sqrt_(d);
  }
  if (n > 0 && threadIdx.x == 0) A[(n - 1) + (int64_t)(n - 1) * lda] = real(1) / rprev;
  __syncthreads();
  return true;
}

__device__ double cta_max_d(double v, double* red);
__device__ int cta_min_i(int v, int* red);

// One warp: the pivot row of column c at or below row j -- the largest
// magnitude, near-ties (|a| >= (1 - 1e-10) max, in float32 equal magnitudes) to
// the lowest row; -1 for a zero column.
__device__ __forceinline__ int warp_pivot(int n, int j, const float* c) {
  unsigned mx = 0;
  for (int i = j + lane_id(); i < n; i += 32) {
    const float a = fabsf(c[i]);
    if (a == a) mx = max(mx, __float_as_uint(a));
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  unsigned best = 0xffffffffu;
  for (int i = j + lane_id(); i < n; i += 32)
    if (__float_as_uint(fabsf(c[i])) == mx) best = min(best, (unsigned)i);
  best = __reduce_min_sync(0xffffffffu, best);
  return mx > 0 ? (int)best : -1;
}
__device__ __forceinline__ int warp_pivot(int n, int j, const double* c) {
  double mx = 0;
  for (int i = j + lane_id(); i < n; i += 32) mx = fmax(mx, fabs(c[i]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  unsigned best = 0xffffffffu;
  const double band = (1.0 - kPivotTieRtol) * mx;
  for (int i = j + lane_id(); i < n; i += 32)
    if (fabs(c[i]) >= band) best = min(best, (unsigned)i);
  best = __reduce_min_sync(0xffffffffu, best);
  return mx > 0.0 ? (int)best : -1;
}

// In-place LU with partial pivoting, P A = L U (unit lower L).  piv[j] = row
// swapped with j at step j.  Returns false for an exactly zero pivot column.
// Warp w owns columns w, w + nw, ..: it interchanges and updates them, so a
// step needs one barrier -- the warp owning column j+1 brings that one up to
// date first and searches it for the next pivot while the others still work;
// column j, which everybody reads, is interchanged and scaled in the step
// after.  (Seven barriers and a float64 reduction per step before: 2 us a step
// at any size, 560 us for 128 unknowns.)  Every element sees the same operations
// in the same order as in the plain right-looking form.
template <typename real>
__device__ bool cta_lu(int n, real* A, int lda, int* piv, int* spiv) {
  const int lane = lane_id(), warp = warp_id(), nw = num_warps();
  if (warp == 0) {
    const int p = warp_pivot(n, 0, A);
    if (lane == 0) spiv[0] = p;
  }
  __syncthreads();
  int pp = 0;      // the step before: its pivot row and reciprocal
  real pr = 0;
  for (int j = 0; j < n; j++) {
    const int p = spiv[j & 1];
    if (p < 0) return false;  // uniform
    const real* cj = A + (int64_t)j * lda;
    const real rd = real(1) / cj[p], cjj = cj[j];
    if (threadIdx.x == 0) piv[j] = p;
    for (int l = j + 1 + (warp - (j + 1) % nw + nw) % nw; l < n; l += nw) {
      real* cl = A + (int64_t)l * lda;
      const real u = cl[p], down = cl[j];
      __syncwarp();
      for (int i = j + 1 + lane; i < n; i += 32) {
        const real lij = (i == p ? cjj : cj[i]) * rd;
        cl[i] = (i == p ? down : cl[i]) - lij * u;
      }
      if (lane == 0) cl[j] = u;
      __syncwarp();
      if (l == j + 1) {
        const int q = warp_pivot(n, j + 1, cl);
        if (lane == 0) spiv[(j + 1) & 1] = q;
      }
    }
    // finish column j - 1, then this step's interchange left of column j
    if (j > 0 && warp == (j - 1) % nw) {
      real* c = A + (int64_t)(j - 1) * lda;
      if (lane == 0 && pp != j - 1) {
        const real t = c[j - 1];
        c[j - 1] = c[pp];
        c[pp] = t;
      }
      __syncwarp();
      for (int i = j + lane; i < n; i += 32) c[i] *= pr;
      __syncwarp();
    }
    if (p != j)
      for (int c = warp + nw * lane; c < j; c += nw * 32) {
        real* cc = A + (int64_t)c * lda;
        const real t = cc[j];
        cc[j] = cc[p];
        cc[p] = t;
      }
    pp = p;
    pr = rd;
    __syncthreads();
  }
  return true;
}

// X = L^{-1} for unit lower triangular L (n x n), out of place, zeros above the
// diagonal: every column on its own, x_r -= l_ri x_i for i ascending.  A warp
// keeps four columns in registers (n <= 256), lanes along the rows, and needs no
// barrier; X must not alias L.
template <typename real>
__device__ void cta_trtri_unit(int n, const real* L, int ldl, real* X, int ldx) {
  constexpr int CW = 4, R = 8;
  const int lane = lane_id();
  for (int g0 = warp_id() * CW; g0 < n; g0 += num_warps() * CW) {
    real x[R][CW];
#pragma unroll
    for (int r = 0; r < R; r++)
#pragma unroll
      for (int g = 0; g < CW; g++) x[r][g] = lane + 32 * r == g0 + g ? real(1) : real(0);
#pragma unroll
    for (int rb = 0; rb < R; rb++) {
      if (32 * rb + 31 < g0 || 32 * rb >= n) continue;
      const int hi = min(32, n - 32 * rb);
      for (int ii = max(0, g0 - 32 * rb); ii < hi; ii++) {
        const int i = 32 * rb + ii;
        real xi[CW];
#pragma unroll
        for (int g = 0; g < CW; g++) xi[g] = __shfl_sync(0xffffffffu, x[rb][g], ii);
#pragma unroll
        for (int r = rb; r < R; r++) {
          const int row = lane + 32 * r;
          if (32 * r >= n) break;
          if (row > i && row < n) {
            const real l = L[row + (int64_t)i * ldl];
#pragma unroll
            for (int g = 0; g < CW; g++) x[r][g] -= l * xi[g];
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < R; r++)
#pragma unroll
      for (int g = 0; g < CW; g++)
        if (lane + 32 * r < n && g0 + g < n) X[lane + 32 * r + (int64_t)(g0 + g) * ldx] = x[r][g];
  }
  __syncthreads();
}

// V = U^{-1} for upper triangular U (n x n), out of place, zeros below the
// diagonal: every row on its own, v_il = -(sum over q < l of v_iq u_ql) / u_ll in
// ascending q.  Four rows per warp, lanes along the columns (n <= 256).
template <typename real>
__device__ void cta_trtri_upper_rows(int n, const real* U, int ldu, real* V, int ldv) {
  constexpr int CW = 4, R = 8;
  const int lane = lane_id();
  for (int g0 = warp_id() * CW; g0 < n; g0 += num_warps() * CW) {
    real acc[R][CW], v[R][CW], d[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int c = lane + 32 * r;
      d[r] = c < n ? real(1) / U[c + (int64_t)c * ldu] : real(0);
#pragma unroll
      for (int g = 0; g < CW; g++) acc[r][g] = v[r][g] = 0;
    }
#pragma unroll
    for (int rb = 0; rb < R; rb++) {
      if (32 * rb + 31 < g0 || 32 * rb >= n) continue;
      const int hi = min(32, n - 32 * rb);
      for (int ll = max(0, g0 - 32 * rb); ll < hi; ll++) {
        const int l = 32 * rb + ll;
        real x[CW];
#pragma unroll
        for (int g = 0; g < CW; g++) {
          // this column's entries are final: the lane that holds it
          const real mine = l == g0 + g ? d[rb] : (l > g0 + g ? -acc[rb][g] * d[rb] : real(0));
          if (lane == ll) v[rb][g] = mine;
          x[g] = __shfl_sync(0xffffffffu, mine, ll);
        }
#pragma unroll
        for (int r = rb; r < R; r++) {
          const int c = lane + 32 * r;
          if (32 * r >= n) break;
          if (c > l && c < n) {
            const real u = U[l + (int64_t)c * ldu];
#pragma unroll
            for (int g = 0; g < CW; g++) acc[r][g] += x[g] * u;
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < R; r++)
#pragma unroll
      for (int g = 0; g < CW; g++)
        if (lane + 32 * r < n && g0 + g < n) V[g0 + g + (int64_t)(lane + 32 * r) * ldv] = v[r][g];
  }
  __syncthreads();
}

// X = L^{-1} for lower triangular L (unit diagonal if `unit`), out of place:
// X (n x n, zero above the diagonal) starts as I and every step i subtracts
// l_ri x_ic for rows r > i from all columns c <= i (x_ic = x_ic / l_ii on the
// fly); row i is finished in the next phase.  One barrier per step.
template <typename real>
__device__ void cta_trtri_lower_oop(int n, const real* L, int ldl, bool unit, real* X, int ldx) {
  const int lane = lane_id(), warp = warp_id(), nw = num_warps();
  cta_identity<real>(n, n, 0, X, ldx);
  real dprev = 1;
  for (int i = 0; i < n; i++) {
    const real di = unit ? real(1) : real(1) / L[i + (int64_t)i * ldl];
    if (i > 0 && !unit)
      for (int c = threadIdx.x; c < i; c += blockDim.x) X[(i - 1) + (int64_t)c * ldx] *= dprev;
    const real* li = L + (int64_t)i * ldl;
    for (int c = warp; c <= i; c += nw) {
      real* xc = X + (int64_t)c * ldx;
      const real xic = xc[i] * di;
      for (int r = i + 1 + lane; r < n; r += 32) xc[r] -= li[r] * xic;
    }
    dprev = di;
    __syncthreads();
  }
  if (n > 0 && !unit)
    for (int c = threadIdx.x; c < n; c += blockDim.x) X[(n - 1) + (int64_t)c * ldx] *= dprev;
  __syncthreads();
}

// In-place inverse of an upper triangular matrix, column by column from the
// first.  tmp: n reals.
template <typename real>
__device__ void cta_trtri_upper(int n, real* U, int ld, real* tmp) {
  for (int j = 0; j < n; j++) {
    for (int i = threadIdx.x; i < j; i += blockDim.x) tmp[i] = U[i + (int64_t)j * ld];
    if (threadIdx.x == 0) U[j + (int64_t)j * ld] = real(1) / U[j + (int64_t)j * ld];
    __syncthreads();
    const real d = U[j + (int64_t)j * ld];
    for (int i = threadIdx.x; i < j; i += blockDim.x) {
      real acc = 0;
      for (int l = i; l < j; l++) acc += U[i + (int64_t)l * ld] * tmp[l];
      U[i + (int64_t)j * ld] = -acc * d;
    }
    __syncthreads();
  }
}

// Block reductions: shuffle within each warp, one exchange through shared
// memory (red: at least one slot per warp), two barriers.
__device__ double cta_max_d(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  if (lane_id() == 0) red[warp_id()] = v;
  __syncthreads();
  double r = red[0];
  for (int w = 1; w < num_warps(); w++) r = fmax(r, red[w]);
  __syncthreads();
  return r;
}

__device__ int cta_min_i(int v, int* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
  if (lane_id() == 0) red[warp_id()] = v;
  __syncthreads();
  int r = red[0];
  for (int w = 1; w < num_warps(); w++) r = min(r, red[w]);
  __syncthreads();
  return r;
}

// Householder QR of the m x c matrix G (in place).  Element (i, q) sits at
// G[i * ldg + q] when RowMajor (one thread per column then reads coalesced
// across a warp), else at G[i + q * ldg].  Columns are pivoted by largest
// remaining norm (recomputed every step, near-ties to the lowest original
// index, orig[] tracks original indices), stopping at |r_jj| <= eps |r_11|
// (eps > 0), at |r_jj| <= floor (rounding noise of a block that is zero in
// exact arithmetic), at an all-zero remainder or at kmax steps.  Householder vectors stay in G (v_j in rows j..m of column j);
// tau[j] = 2 / v^T v.  vsh: m reals of shared memory.  Returns the number of
// steps.
template <typename real, bool RowMajor>
__device__ int cta_householder_qr(int m, int c, real* G, int ldg, double* nrm2, double* orig,
                                  real* tau, double eps, int kmax, double floor,
                                  double* red_d, int* red_i, real* vsh, real* rsign = nullptr,
                                  const int* fpiv = nullptr) {
  auto at = [&](int i, int q) -> real& {
    return RowMajor ? G[(int64_t)i * ldg + q] : G[i + (int64_t)q * ldg];
  };
  for (int q = threadIdx.x; q < c; q += blockDim.x) {
    real s = 0;
    for (int i = 0; i < m; i++) {
      const real v = at(i, q);
      s += v * v;
    }
    nrm2[q] = (double)s;
    orig[q] = q;
  }
  __syncthreads();
  double r11 = 0;
  int k = 0;
  const int steps = min(m, c);
  for (int j = 0; j < steps; j++) {
    double mx = 0;
    for (int t = j + threadIdx.x; t < c; t += blockDim.x) mx = fmax(mx, nrm2[t]);
    mx = cta_max_d(mx, red_d);
    if (mx == 0.0) break;
    int best = INT_MAX;
    if (fpiv) {
      // a given pivot order (forced-rank factorization) replaces the search
      best = j < kmax ? fpiv[j] : INT_MAX;
    } else {
      for (int t = j + threadIdx.x; t < c; t += blockDim.x)
        if (nrm2[t] >= (1.0 - qr_tie_rtol<real>()) * mx) best = min(best, (int)orig[t]);
      best = cta_min_i(best, red_i);
    }
    if (threadIdx.x == 0) red_i[blockDim.x] = -1;
    __syncthreads();
    for (int t = j + threadIdx.x; t < c; t += blockDim.x)
      if ((int)orig[t] == best) red_i[blockDim.x] = t;
    __syncthreads();
    const int q = red_i[blockDim.x];
    __syncthreads();
    if (q < 0) break;  // the given pivot names no remaining column
    const double r = sqrt(nrm2[q]);
    if (j == 0) r11 = r;
    if (r <= floor) break;
    if (eps > 0.0 && r <= eps * r11) break;
    if (j >= kmax) break;
    if (q != j) {
      for (int i = threadIdx.x; i < m; i += blockDim.x) {
        real t = at(i, j);
        at(i, j) = at(i, q);
        at(i, q) = t;
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        double t = nrm2[j];
        nrm2[j] = nrm2[q];
        nrm2[q] = t;
        t = orig[j];
        orig[j] = orig[q];
        orig[q] = t;
      }
      __syncthreads();
    }
    // reflector v = x - beta e1, beta = -sign(x0) ||x||, tau = 2 / v^T v
    const double x0 = (double)at(j, j);
    const double beta = (x0 >= 0.0) ? -r : r;
    const double tj = (r > 0.0) ? 1.0 / (r * (r + fabs(x0))) : 0.0;
    __syncthreads();
    for (int i = j + threadIdx.x; i < m; i += blockDim.x) vsh[i] = (i == j) ? (real)(x0 - beta) : at(i, j);
    __syncthreads();
    if (threadIdx.x == 0) {
      at(j, j) = (real)(x0 - beta);
      tau[j] = (real)tj;
      if (rsign) rsign[j] = beta < 0.0 ? real(-1) : real(1);
    }
    const real rt = (real)tj;
    // apply to the remaining columns, CB columns per thread and RB rows per
    // batch of independent loads (memory-level parallelism); recompute the
    // squared norms over rows j+1..m
    constexpr int CB = 4, RB = 4;
    const int nth = blockDim.x;
    for (int t0 = j + 1 + threadIdx.x; t0 < c; t0 += nth * CB) {
      real w[CB];
      bool ok[CB];
#pragma unroll
      for (int g = 0; g < CB; g++) {
        w[g] = 0;
        ok[g] = (t0 + g * nth) < c;
      }
      for (int i = j; i < m; i += RB) {
        real x[RB][CB];
#pragma unroll
        for (int rr = 0; rr < RB; rr++)
#pragma unroll
          for (int g = 0; g < CB; g++)
            x[rr][g] = (ok[g] && i + rr < m) ? at(i + rr, t0 + g * nth) : real(0);
#pragma unroll
        for (int rr = 0; rr < RB; rr++) {
          const real vi = (i + rr < m) ? vsh[i + rr] : real(0);
#pragma unroll
          for (int g = 0; g < CB; g++) w[g] += vi * x[rr][g];
        }
      }
      // squared norms in the working precision: a float64 FMA per element
      // here would bound the float32 path by the float64 rate
      real sq[CB];
#pragma unroll
      for (int g = 0; g < CB; g++) {
        w[g] *= rt;
        sq[g] = 0;
      }
      for (int i = j; i < m; i += RB) {
        real x[RB][CB];
#pragma unroll
        for (int rr = 0; rr < RB; rr++)
#pragma unroll
          for (int g = 0; g < CB; g++)
            x[rr][g] = (ok[g] && i + rr < m) ? at(i + rr, t0 + g * nth) : real(0);
#pragma unroll
        for (int rr = 0; rr < RB; rr++) {
          if (i + rr >= m) break;
          const real vi = vsh[i + rr];
#pragma unroll
          for (int g = 0; g < CB; g++) {
            if (!ok[g]) continue;
            const real v = x[rr][g] - w[g] * vi;
            at(i + rr, t0 + g * nth) = v;
            if (i + rr > j) sq[g] += v * v;
          }
        }
      }
#pragma unroll
      for (int g = 0; g < CB; g++)
        if (ok[g]) nrm2[t0 + g * nth] = (double)sq[g];
    }
    __syncthreads();
    k = j + 1;
  }
  __syncthreads();
  return k;
}

// Q[:, c0:c0+ncols] of Q = H_0 .. H_{k-1} (H_j = I - tau_j v_j v_j^T, v_j in
// rows j..m of column j of V): out (m x ncols) starts as the identity columns
// c0.. and receives the reflectors in reverse order.  One warp per group of
// four columns; lane l owns rows l, l + 32, ... of them (held in registers
// when m <= 256), so the warps never wait for one another and the lanes only
// exchange the four dot products of each reflector (shuffles).
template <typename real, bool RowMajor>
__device__ void cta_form_q(int m, int k, const real* V, int ldv, const real* tau, int c0,
                           int ncols, real* out, int ldo, real* vsh) {
  (void)vsh;
  constexpr int CW = 4, R = 8;
  const int lane = lane_id(), warp = warp_id(), nw = num_warps();
  auto vat = [&](int i, int j) -> real {
    return RowMajor ? V[(int64_t)i * ldv + j] : V[i + (int64_t)j * ldv];
  };
  for (int g0 = warp * CW; g0 < ncols; g0 += nw * CW) {
    const int ng = min(CW, ncols - g0);
    if (m <= 32 * R) {
      real x[R][CW];
#pragma unroll
      for (int r = 0; r < R; r++)
#pragma unroll
        for (int g = 0; g < CW; g++) x[r][g] = (lane + 32 * r == c0 + g0 + g) ? real(1) : real(0);
      for (int j = k - 1; j >= 0; j--) {
        const real tj = tau[j];
        real v[R], d[CW];
#pragma unroll
        for (int g = 0; g < CW; g++) d[g] = 0;
#pragma unroll
        for (int r = 0; r < R; r++) {
          const int i = lane + 32 * r;
          v[r] = (i >= j && i < m) ? vat(i, j) : real(0);
#pragma unroll
          for (int g = 0; g < CW; g++) d[g] += v[r] * x[r][g];
        }
#pragma unroll
        for (int g = 0; g < CW; g++) d[g] = warp_sum(d[g]) * tj;
#pragma unroll
        for (int r = 0; r < R; r++)
#pragma unroll
          for (int g = 0; g < CW; g++) x[r][g] -= d[g] * v[r];
      }
#pragma unroll
      for (int r = 0; r < R; r++) {
        const int i = lane + 32 * r;
        if (i < m)
#pragma unroll
          for (int g = 0; g < CW; g++)
            if (g < ng) out[i + (int64_t)(g0 + g) * ldo] = x[r][g];
      }
    } else {
      for (int g = 0; g < ng; g++)
        for (int i = lane; i < m; i += 32)
          out[i + (int64_t)(g0 + g) * ldo] = (i == c0 + g0 + g) ? real(1) : real(0);
      for (int j = k - 1; j >= 0; j--) {
        const real tj = tau[j];
        real d[CW];
#pragma unroll
        for (int g = 0; g < CW; g++) d[g] = 0;
        for (int i = lane; i < m; i += 32) {
          if (i < j) continue;
          const real v = vat(i, j);
#pragma unroll
          for (int g = 0; g < CW; g++)
            if (g < ng) d[g] += v * out[i + (int64_t)(g0 + g) * ldo];
        }
#pragma unroll
        for (int g = 0; g < CW; g++) d[g] = warp_sum(d[g]) * tj;
        for (int i = lane; i < m; i += 32) {
          if (i < j) continue;
          const real v = vat(i, j);
#pragma unroll
          for (int g = 0; g < CW; g++)
            if (g < ng) out[i + (int64_t)(g0 + g) * ldo] -= d[g] * v;
        }
      }
    }
  }
  __syncthreads();
}

// Householder QR without pivoting of the m x k matrix X (column-major, in
// place): v_j in rows j..m of column j (its head x_jj - beta, beta =
// -sign(x_jj) ||x_j||), tau[j] = 1 / (r (r + |x_jj|)).  Warp w owns columns
// w, w + nw, ..; in step j the owner of column j+1 brings it up to date first and
// forms the next reflector, so a step takes one barrier.
template <typename real>
__device__ void cta_qr_np(int m, int k, real* X, int ldx, real* tau) {
  const int lane = lane_id(), warp = warp_id(), nw = num_warps();
  const auto form = [&](int j) {  // the owning warp
    real* xj = X + (int64_t)j * ldx;
    real sq = 0;
    for (int i = j + lane; i < m; i += 32) sq += xj[i] * xj[i];
    sq = warp_sum(sq);
    const real x0 = xj[j];
    real head, t;
    householder_scalars(sq, x0, &head, &t);
    __syncwarp();
    if (lane == 0) {
      xj[j] = head;
      tau[j] = t;
    }
  };
  if (k > 0 && warp == 0) form(0);
  __syncthreads();
  for (int j = 0; j < k; j++) {
    const real* vj = X + (int64_t)j * ldx;
    const real tj = tau[j];
    for (int t = j + 1 + (warp - (j + 1) % nw + nw) % nw; t < k; t += nw) {
      real* xt = X + (int64_t)t * ldx;
      real d = 0;
      for (int i = j + lane; i < m; i += 32) d += vj[i] * xt[i];
      d = warp_sum(d) * tj;
      for (int i = j + lane; i < m; i += 32) xt[i] -= d * vj[i];
      __syncwarp();
      if (t == j + 1) form(t);
    }
    __syncthreads();
  }
}

// pos[c] = row of P A holding original row c after the swaps piv[0..n-1] in
// order (inverse = false), or the original row that row c of P A holds.
__device__ void cta_permutation(int n, const int* piv, int* pos, bool inverse) {
  for (int c = threadIdx.x; c < n; c += blockDim.x) {
    int q = c;
    if (!inverse) {
      for (int j = 0; j < n; j++) {
        const int p = piv[j];
        q = p == q ? j : (j == q ? p : q);
      }
    } else {
      for (int j = n - 1; j >= 0; j--) {
        const int p = piv[j];
        q = p == q ? j : (j == q ? p : q);
      }
    }
    pos[c] = q;
  }
  __syncthreads();
}

// Y = X P: column c of Y is column pos[c] of X.
template <typename real>
__device__ void cta_permute_cols(int n, const int* pos, const real* X, int ldx, real* Y, int ldy) {
  for (int c = warp_id(); c < n; c += num_warps())
    for (int i = lane_id(); i < n; i += 32)
      Y[i + (int64_t)c * ldy] = X[i + (int64_t)pos[c] * ldx];
  __syncthreads();
}

template <typename real>
__device__ void report(DevError* err, int code, int s, int level, int* rank, int m) {
  if (threadIdx.x == 0) {
    if (atomicCAS(&err->code, 0, code) == 0) {
      err->cluster = s;
      err->level = level;
    }
    rank[s] = m;  // leave the cluster untouched downstream
  }
}

template <typename real>
__global__ void __launch_bounds__(PrepThreads<real>::value)
prep_kernel(const PrepTask* __restrict__ tasks, real* __restrict__ arena, real* __restrict__ fac,
            real* __restrict__ ws_all, double* __restrict__ wsd_all,
            const Seg* __restrict__ segs, int* rank, int* __restrict__ piv_all,
            const int* __restrict__ fpiv, double eps, double noise_rtol, int sym, int max_rank,
            int smem_mats, int smem_m,
            DevError* err, int level, long long* dbg) {
  __shared__ double red_d[PrepThreads<real>::value];
  __shared__ int red_i[PrepThreads<real>::value + 1];
  __shared__ int sflag;
  __shared__ int s_ncol;
  __shared__ double s_amax;
  extern __shared__ unsigned char dsm[];
  const PrepTask tk = tasks[blockIdx.x];
  const int m = tk.m;
  // optional per-phase clock stamps (profiling): dbg[task * 8 + checkpoint]
  long long* stamp = dbg ? dbg + (int64_t)blockIdx.x * 8 : nullptr;
  auto mark = [&](int i) {
    if (stamp && threadIdx.x == 0) stamp[i] = clock64();
  };
  mark(0);
  if (threadIdx.x == 0) sflag = 0;
  __syncthreads();
  const int64_t mm = (int64_t)m * m;
  real* ws = ws_all + tk.ws;
  real* smat = reinterpret_cast<real*>(dsm);
  real* vsh = smat + (int64_t)smem_mats * (smem_m | 1) * smem_m;  // m reals
  real* tsh = vsh + smem_m;                                  // m reals
  // shared-memory matrices get an odd leading dimension: loops that give one
  // column to each thread then touch 32 different banks
  const int64_t reg = (int64_t)(smem_m | 1) * smem_m;  // one shared region
  int ldA = smem_mats >= 1 ? (m | 1) : m;
  int ldB = smem_mats >= 2 ? (m | 1) : m;
  const int ldU = smem_mats >= 3 ? (m | 1) : m;
  real* W_A = smem_mats >= 1 ? smat : ws;                  // A_ss -> factor -> inverse factor
  real* W_B = smem_mats >= 2 ? smat + reg : ws + mm;       // A_ss^{-1}
  // [U V_L] as one m x m matrix: U in columns 0..k, V_L in columns k..m
  real* W_U = smem_mats >= 3 ? smat + 2 * reg : ws + 2 * mm;
  real* W_X = ws + 3 * mm;   // X = B U, then its reflectors
  real* W_V = W_U + (int64_t)0;  // V_L = columns k..m of W_U (set below)
  real* W_T = ws + 4 * mm;   // [U V_L]^T B
  real* W_F = W_T + mm;      // F, then its factor / inverse factor (general)
  real* W_L = W_F + mm;      // general: L^{-1} P, (U_F^{-1})
  real* W_C = W_L + mm;      // C = U^T B U
  real* W_R = W_C + mm;      // general: V_R
  real* W_S = W_R + mm;      // general: scratch
  real* W_G = W_S + mm;      // G (m x ncolG)
  double* nrm2 = wsd_all + tk.wsd;
  double* orig = nrm2 + tk.ncolG;
  real* tau = reinterpret_cast<real*>(orig + tk.ncolG);
  real* tau2 = tau + m;
  real* rsign = tau2 + m;  // sign of R's diagonal in the pivoted QR
  int* piv = reinterpret_cast<int*>(rsign + m);
  int* pos = reinterpret_cast<int*>(vsh);  // m ints (vsh: the in-kernel QR's, spent by then)
  real* T = fac + tk.T;

  // ---- A_ss, its largest magnitude (scale of the noise floor), its factor
  cta_copy<real>(m, m, arena + tk.a_ss, tk.ld, W_A, ldA);
  {
    real mx = 0;  // (the float64 pipe issues two lanes per clock)
    for (int j = warp_id(); j < m; j += num_warps())
      for (int i = lane_id(); i < m; i += 32) mx = fmax(mx, fabs(W_A[i + (int64_t)j * ldA]));
    const double all = cta_max_d((double)mx, red_d);
    if (threadIdx.x == 0) s_amax = all;
    __syncthreads();
  }
  const bool ok = sym ? cta_cholesky<real>(m, W_A, ldA, &sflag)
                      : cta_lu<real>(m, W_A, ldA, piv, red_i);
  if (!ok) {
    report<real>(err, sym ? (int)HSOLVE_ERR_NOT_SPD : (int)HSOLVE_ERR_SINGULAR, tk.s, level, rank, m);
    return;
  }

  mark(1);
  const bool sketched = tk.l > 0;
  const bool qr_done = tk.qr == 2;  // done by the thread-block-cluster kernel
  // ---- gather the nonzero fill columns into G (Eq. lra input), row-major
  // (not needed when the pivoted QR runs on the sketch Y = G Omega or was
  // done by the cluster kernel)
  if (!sketched && !qr_done) {
    const int nc = tk.ncolG;
    // flag nonzero columns: one thread per column, batched independent loads
    for (int q = threadIdx.x; q < nc; q += blockDim.x) {
      int64_t p;
      int st;
      seg_col(segs + tk.gcol, tk.ngcol, q, &p, &st);
      bool nz = false;
      for (int i = 0; i < m; i += 8) {
        real x[8];
#pragma unroll
        for (int rr = 0; rr < 8; rr++) x[rr] = (i + rr < m) ? arena[p + (int64_t)(i + rr) * st] : real(0);
#pragma unroll
        for (int rr = 0; rr < 8; rr++) nz |= (x[rr] != real(0));
      }
      orig[q] = nz ? 1.0 : 0.0;
    }
    __syncthreads();
    // exclusive scan of the flags: contiguous chunk per thread
    const int per = (nc + blockDim.x - 1) / blockDim.x;
    const int c0 = min(nc, (int)threadIdx.x * per), c1 = min(nc, c0 + per);
    int cnt = 0;
    for (int q = c0; q < c1; q++) cnt += (orig[q] != 0.0);
    red_i[threadIdx.x] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
      int acc = 0;
      for (int t = 0; t < (int)blockDim.x; t++) {
        int v = red_i[t];
        red_i[t] = acc;
        acc += v;
      }
      s_ncol = acc;
    }
    __syncthreads();
    int dst = red_i[threadIdx.x];
    for (int q = c0; q < c1; q++) orig[q] = (orig[q] != 0.0) ? (double)(dst++) : -1.0;
    __syncthreads();
    const int ncomp = s_ncol;
    // copy: one thread per column; consecutive threads write consecutive
    // entries of a row of the row-major G
    for (int q = threadIdx.x; q < nc; q += blockDim.x) {
      const int d = (int)orig[q];
      if (d < 0) continue;
      int64_t p;
      int st;
      seg_col(segs + tk.gcol, tk.ngcol, q, &p, &st);
      for (int i = 0; i < m; i += 8) {
        real x[8];
#pragma unroll
        for (int rr = 0; rr < 8; rr++) x[rr] = (i + rr < m) ? arena[p + (int64_t)(i + rr) * st] : real(0);
#pragma unroll
        for (int rr = 0; rr < 8; rr++)
          if (i + rr < m) W_G[(int64_t)(i + rr) * ncomp + d] = x[rr];
      }
    }
    __syncthreads();
  }
  mark(2);
  const int ncol = sketched ? tk.l : s_ncol;
  int k = 0;
  int kmax = m;
  if (max_rank > 0) kmax = min(kmax, max_rank);
  if (max_rank < 0) {  // forced rank (set by the host in rank[s]): no eps, no floor
    kmax = min(kmax, rank[tk.s]);
    eps = 0.0;
    noise_rtol = 0.0;
  }
  if (qr_done) {
    k = rank[tk.s];
  } else if (sketched) {
    // pivoted QR of the sketch (column-major m x l), in the shared memory of
    // the not yet used A_ss^{-1} and [U V] buffers when it fits; the kept
    // reflectors then move to W_G (column-major, ld m) for U
    real* Ysrc = ws_all + tk.Y;
    const bool ysm = smem_mats >= 3 && (int64_t)(m | 1) * tk.l <= 2 * reg;
    real* Yq = ysm ? W_B : Ysrc;
    const int ldY = ysm ? (m | 1) : m;
    if (ysm) cta_copy<real>(m, tk.l, Ysrc, m, Yq, ldY);
    k = cta_householder_qr<real, false>(m, tk.l, Yq, ldY, nrm2, orig, tau, eps, kmax,
                                        noise_rtol * s_amax, red_d, red_i, vsh, rsign,
                                        fpiv ? fpiv + tk.pv : nullptr);
    cta_copy<real>(m, k, Yq, ldY, W_G, m);
  } else if (ncol > 0) {
    k = cta_householder_qr<real, true>(m, ncol, W_G, ncol, nrm2, orig, tau, eps, kmax,
                                       noise_rtol * s_amax, red_d, red_i, vsh, rsign,
                                       fpiv ? fpiv + tk.pv : nullptr);
  }
  __syncthreads();
  if (threadIdx.x == 0) rank[tk.s] = k;
  // pivot order (the cluster kernel recorded its own): orig[j] is the
  // compacted (or sketch) column chosen at step j
  if (!qr_done)
    for (int j = threadIdx.x; j < k; j += blockDim.x) piv_all[tk.pv + j] = (int)orig[j];
  mark(3);
  if (k == m) return;  // untouched: all unknowns coarse, E_s = I
  const int f = m - k;

  if (sym) {
    // L^{-1} into the home of A_ss^{-1}, then B = L^{-T} L^{-1} into the
    // home of the (spent) factor; the two buffers then trade names
    cta_trtri_lower_oop<real>(m, W_A, ldA, false, W_B, ldB);
    if (k == 0) {  // E_s = I: T' = L^{-1}
      cta_copy<real>(m, m, W_B, ldB, T, m);
      return;
    }
    cta_gemm<real>(m, m, m, W_B, ldB, true, W_B, ldB, false, W_A, ldA);
    real* tp = W_A;
    W_A = W_B;
    W_B = tp;
    const int tl = ldA;
    ldA = ldB;
    ldB = tl;
  } else {
    // L^{-1} (unit lower) into W_L, U^{-1} into W_S
    if (m <= kRowsMax) {
      cta_trtri_unit<real>(m, W_A, ldA, W_L, m);
      cta_trtri_upper_rows<real>(m, W_A, ldA, W_S, m);
    } else {
      cta_trtri_lower_oop<real>(m, W_A, ldA, true, W_L, m);
      cta_copy<real>(m, m, W_A, ldA, W_S, m);
      cta_trtri_upper<real>(m, W_S, m, tsh);
      cta_zero_tri<real>(m, W_S, m, false);
    }
    cta_permutation(m, piv, pos, false);
    if (k == 0) {
      // E_s = I: T' = L^{-1} P, T'_R^T = (U^{-1})^T
      cta_permute_cols<real>(m, pos, W_L, m, T, m);
      real* TRt = fac + tk.TR;
      for (int idx = threadIdx.x; idx < m * m; idx += blockDim.x) {
        int i = idx % m, j = idx / m;
        TRt[i + (int64_t)j * m] = W_S[j + (int64_t)i * m];
      }
      __syncthreads();
      return;
    }
    // B = U^{-1} L^{-1} P
    cta_gemm<real>(m, m, m, W_S, m, false, W_L, m, false, W_F, m);
    cta_permute_cols<real>(m, pos, W_F, m, W_B, ldB);
  }

  mark(4);
  // ---- U = first k columns of Q of the pivoted QR
  if (sketched || qr_done)
    cta_form_q<real, false>(m, k, W_G, m, tau, 0, k, W_U, ldU, vsh);
  else
    cta_form_q<real, true>(m, k, W_G, ncol, tau, 0, k, W_U, ldU, vsh);
  // orient U so that R has a positive diagonal (Gram-Schmidt directions)
  for (int idx = threadIdx.x; idx < m * k; idx += blockDim.x) {
    int i = idx % m, j = idx / m;
    W_U[i + (int64_t)j * ldU] *= rsign[j];
  }
  __syncthreads();

  // ---- V_L: complement of X = B U (full QR of X, V = Q[:, k:]); X takes the
  // (spent) home of the factor of A_ss
  W_X = W_A;
  const int ldX = ldA;
  cta_gemm<real>(m, k, m, W_B, ldB, false, W_U, ldU, false, W_X, ldX);
  cta_qr_np<real>(m, k, W_X, ldX, tau2);
  W_V = W_U + (int64_t)k * ldU;
  cta_form_q<real, false>(m, k, W_X, ldX, tau2, k, f, W_V, ldU, vsh);

  mark(5);
  // ---- T = [U V_L]^T B (one product); C = U^T B U -> coarse (s,s) block
  cta_gemm<real>(m, m, m, W_U, ldU, true, W_B, ldB, false, W_T, m);
  cta_gemm<real>(k, k, m, W_T, m, false, W_U, ldU, false, W_C, m);

  if (sym) {
    // F = V^T B V; L_F^{-1}; T' rows k.. = L_F^{-1} V^T B.  F lives where the
    // factor of A_ss was (shared memory when it fits): that factor is spent.
    W_F = W_A;
    const int ldF = ldA;
    mark(6);
    cta_gemm<real>(f, f, m, W_T + k, m, false, W_V, ldU, false, W_F, ldF);
    if (!cta_cholesky<real>(f, W_F, ldF, &sflag)) {
      report<real>(err, (int)HSOLVE_ERR_NOT_SPD, tk.s, level, rank, m);
      return;
    }
    cta_trtri_lower_oop<real>(f, W_F, ldF, false, W_L, m);
    cta_copy<real>(k, m, W_T, m, T, m);
    cta_gemm<real>(f, m, f, W_L, m, false, W_T + k, m, false, T + k, m);
    // D = C U^T (k x m) for the coarse-to-far update C (U^T A_sw)
    cta_gemm<real>(k, m, k, W_C, m, false, W_U, ldU, true, ws_all + tk.D, m);
  } else {
    // V_R: complement of B^T U
    cta_gemm<real>(m, k, m, W_B, ldB, true, W_U, ldU, false, W_X, ldX);
    cta_qr_np<real>(m, k, W_X, ldX, tau2);
    cta_form_q<real, false>(m, k, W_X, ldX, tau2, k, f, W_R, m, vsh);
    // F = V_L^T B V_R (f x f) and its LU, in the home of X
    W_F = W_A;
    const int ldF = ldA;
    cta_gemm<real>(f, f, m, W_T + k, m, false, W_R, m, false, W_F, ldF);
    if (!cta_lu<real>(f, W_F, ldF, piv, red_i)) {
      report<real>(err, (int)HSOLVE_ERR_SINGULAR, tk.s, level, rank, m);
      return;
    }
    // T' rows k.. = L_F^{-1} P_F V_L^T B; P_F V_L^T B beside the workspace's
    // spent inverse, L_F^{-1} over the spent V_L
    cta_permutation(f, piv, pos, true);
    real* W_P = ws + 5 * mm;
    for (int c = warp_id(); c < m; c += num_warps())
      for (int i = lane_id(); i < f; i += 32)
        W_P[i + (int64_t)c * m] = W_T[k + pos[i] + (int64_t)c * m];
    if (f <= kRowsMax) cta_trtri_unit<real>(f, W_F, ldF, W_L, m);
    else cta_trtri_lower_oop<real>(f, W_F, ldF, true, W_L, m);
    cta_copy<real>(k, m, W_T, m, T, m);
    cta_gemm<real>(f, m, f, W_L, m, false, W_P, m, false, T + k, m);
    // T'_R = B [U, V_R U_F^{-1}]; store its transpose
    const real* W_Ui = W_F;
    int ldi = ldF;
    if (f <= kRowsMax) {
      cta_trtri_upper_rows<real>(f, W_F, ldF, W_L, m);
      W_Ui = W_L;
      ldi = m;
    } else {
      cta_trtri_upper<real>(f, W_F, ldF, tsh);
      cta_zero_tri<real>(f, W_F, ldF, false);
    }
    cta_gemm<real>(m, f, f, W_R, m, false, W_Ui, ldi, false, W_S, m);
    real* TRt = fac + tk.TR;
    cta_gemm<real>(k, m, m, W_U, ldU, true, W_B, ldB, true, TRt, m);
    cta_gemm<real>(f, m, m, W_S, m, true, W_B, ldB, true, TRt + k, m);
    cta_gemm<real>(k, m, k, W_C, m, false, W_U, ldU, true, ws_all + tk.D, m);
    cta_gemm<real>(k, m, k, W_C, m, true, W_U, ldU, true, ws_all + tk.D2, m);
  }
  // write C into the (s,s) block (coarse part); done last: A_ss was copied
  real* blk_ss = arena + tk.a_ss;
  for (int idx = threadIdx.x; idx < k * k; idx += blockDim.x) {
    int i = idx % k, j = idx / k;
    blk_ss[i + (int64_t)j * tk.ld] = W_C[i + (int64_t)j * m];
  }
  mark(7);
}

}  // namespace

template <typename real>
void Launch<real>::prep(const PrepTask* tasks_dev, int ntask, real* arena, real* fac, real* ws,
                        double* wsd, const Seg* segs, int* rank, int* piv, const int* fpiv,
                        double eps,
                        int sym, int max_rank, int maxm, DevError* err, int level,
                        long long* dbg, cudaStream_t st) {
  if (ntask <= 0) return;
  // rounding-noise floor of the rank decision, relative to max |A_ss|: the
  // oracle's 1e-14 in float64; float32 blocks carry ~1e-7 relative noise
  const double noise_rtol = sizeof(real) == 8 ? 1e-14 : 1e-6;
  // the factor of A_ss and A_ss^{-1} in shared memory when they fit
  const size_t budget = 208 * 1024;
  const size_t one = sizeof(real) * (size_t)(maxm | 1) * maxm;
  const size_t vec = sizeof(real) * 2 * (size_t)maxm;
  int mats = 0;
  if (3 * one + vec <= budget) mats = 3;
  else if (2 * one + vec <= budget) mats = 2;
  else if (one + vec <= budget) mats = 1;
  const size_t smem = mats * one + vec;
  // the limit is raised once to the budget and never lowered: host threads
  // factoring different matrices launch this kernel concurrently
  static const bool limit_set = [budget] {
    cudaFuncSetAttribute(prep_kernel<real>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)budget);
    return true;
  }();
  (void)limit_set;
  count_launch();
  prep_kernel<real><<<ntask, PrepThreads<real>::value, smem, st>>>(tasks_dev, arena, fac, ws, wsd, segs,
                                                        rank, piv, fpiv, eps, noise_rtol, sym, max_rank, mats,
                                                        maxm, err, level, dbg);
}

template struct Launch<double>;
template struct Launch<float>;

}  // namespace hs
