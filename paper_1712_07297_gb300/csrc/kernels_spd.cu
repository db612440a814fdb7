// Per-cluster dense work of one LowRank_Elimination step (Sec. 2.1) on the SPD
// path, behind the pivoted QR of the fill blocks: one CTA per cluster of a
// colour class.
//
//   A_ss = L L^T, Li = L^{-1}                       (k = 0: T' = Li, done)
//   U = first k columns of Q of the pivoted QR
//   P = Li U,  C = P^T P = U^T A_ss^{-1} U,  D = C U^T,  X = Li^T P = A_ss^{-1} U
//   V = complement of X (its Householder Q, columns k..)      (V^T X = 0)
//   Z = Li V,  F = Z^T Z = V^T A_ss^{-1} V = L_F L_F^T        (Eq. elim)
//   T' = [X^T; (Z L_F^{-T})^T Li] = [U^T; L_F^{-1} V^T] A_ss^{-1}  (Eq. scaling)
//
// What bounds it.  In float32 the chain of CTA-wide phases: the factorizations
// and the two orthogonal bases used to take one to three barriers per column
// (573 us per class at level 1 of 64^3, where the products need about 20).
// Here every step works on blocks of 32 columns: one warp factors and inverts
// a diagonal block in registers, the rest are products; the bases are formed
// from the compact WY form of their reflectors (Schreiber and Van Loan 1989),
// and the one QR of this kernel keeps its columns in registers with one barrier
// per step.  In float64 the products' count (1.9 per clock and SM): A_ss^{-1}
// is never formed, which leaves 5.9 of 9.8 million products at m = 128, k = 35.
// Per factorization, the general kernel -> this one: 64^3 51 -> 27 ms in float32,
// 341 -> 195 in float64; 96^3 120 -> 71; 29 x 37 x 23 (eps 1e-4, float64)
// 272 -> 122; 64^2 2.5 -> 1.5.
//
// Matrices are column-major.  Three m x m regions: R1 holds A_ss, L, Li; R2 and
// R3 the rest; in shared memory (odd leading dimension) as far as they fit, the
// others in the cluster's workspace.
#include <cfloat>
#include <cmath>

#include "common.h"

namespace hs {

namespace {

constexpr int NT = 512;      // threads
constexpr int NB = 32;       // block of the factorizations: one warp's lanes
constexpr int kMaxM = 256;   // largest cluster (larger ones take the general kernel)

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }
__device__ __forceinline__ int warp_id() { return threadIdx.x >> 5; }
__device__ __forceinline__ float sqrt_(float x) { return sqrtf(x); }
__device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }

template <typename real>
__device__ __forceinline__ real warp_sum(real v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Ranges of the inner index of a product, from the structure of its operands
enum Lo { kFrom0, kFromRow, kFromCol };  // l >= 0, l >= i, l >= j
enum Hi { kToEnd, kToRow, kToCol };      // l < K, l <= i, l <= j

// emit(i, j, sum_l A(i, l) B(l, j)) for i < M, j < N (lower: only tiles with an
// element i >= j), A(i, l) = A[i * ars + l * acs], B(l, j) = B[l * brs + j * bcs].
// RM x RN outputs per thread, tiles dealt out from thread `first` on.  float32:
// a thread's rows are strided so that a warp reads consecutive ones (no bank
// conflicts); float64: contiguous, so that triangular structure shortens the
// inner ranges (the float64 pipe is the bound, not shared memory).  No barrier.
template <typename real, int RM, int RN, Lo LO, Hi HI, typename Emit>
__device__ __forceinline__ void product_tiles(int M, int N, int K, const real* A, int ars, int acs,
                                              const real* B, int brs, int bcs, bool lower,
                                              int first, Emit&& emit) {
  constexpr bool kStride = sizeof(real) == 4;
  const int nti = (M + RM - 1) / RM, ntj = (N + RN - 1) / RN, n = nti * ntj;
  for (int t = (threadIdx.x + NT - first % NT) % NT; t < n; t += NT) {
    const int ti = t % nti, tj = t / nti;
    const auto row = [&](int r) { return kStride ? ti + r * nti : ti * RM + r; };
    const int jf = tj * RN, jl = min(N, jf + RN) - 1;
    const int fi = row(0), li = min(M - 1, row(RM - 1));
    if (lower && li < jf) continue;
    const int lo = LO == kFromRow ? fi : LO == kFromCol ? jf : 0;
    const int hi = HI == kToRow ? min(K, li + 1) : HI == kToCol ? min(K, jl + 1) : K;
    int ao[RM], bo[RN];
#pragma unroll
    for (int r = 0; r < RM; r++) ao[r] = min(row(r), M - 1) * ars;
#pragma unroll
    for (int c = 0; c < RN; c++) bo[c] = min(jf + c, N - 1) * bcs;
    real acc[RM][RN];
#pragma unroll
    for (int r = 0; r < RM; r++)
#pragma unroll
      for (int c = 0; c < RN; c++) acc[r][c] = 0;
#pragma unroll 4
    for (int l = lo; l < hi; l++) {
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
        if (row(r) < M && jf + c < N) emit(row(r), jf + c, acc[r][c]);
  }
}

// Tiles of 4 x 4 where that still occupies the threads, else 2 x 2.
template <typename real, Lo LO, Hi HI, typename Emit>
__device__ __forceinline__ void product(int M, int N, int K, const real* A, int ars, int acs,
                                        const real* B, int brs, int bcs, bool lower, int first,
                                        Emit&& emit) {
  if (M * N >= 6144)
    product_tiles<real, 4, 4, LO, HI>(M, N, K, A, ars, acs, B, brs, bcs, lower, first, emit);
  else
    product_tiles<real, 2, 2, LO, HI>(M, N, K, A, ars, acs, B, brs, bcs, lower, first, emit);
}

// 1 / sqrt(d), to the last bit or two
__device__ __forceinline__ float inv_sqrt(float d) {
  const float y = rsqrtf(d);
  return fmaf(y * 0.5f, fmaf(-d * y, y, 1.f), y);
}
__device__ __forceinline__ double inv_sqrt(double d) { return rsqrt(d); }

// One warp: L = chol of the lower n x n block at A (n <= 32), then L^{-1} in its
// place (zeros above the diagonal); factor = false: the block is lower
// triangular already.  False for a pivot that is not positive.  A lane keeps a
// row (of L), then a column (of the inverse) in registers that move down by one
// per step, so that the step's column is always register 0: fully unrolled
// steps instead took 15 us, and as much again to fetch their instructions in
// every CTA.
template <typename real>
__device__ __noinline__ bool warp_chol_inv(int n, real* A, int ld, bool factor) {
  const int lane = lane_id();
  real a[NB], dinv = 1;
  if (factor) {
#pragma unroll
    for (int j = 0; j < NB; j++) a[j] = (j <= lane && lane < n) ? A[lane + j * ld] : real(0);
#pragma unroll 1
    for (int j = 0; j < n; j++) {
      const real d = __shfl_sync(0xffffffffu, a[0], j);
      if (!(d > real(0))) return false;
      const real rs = inv_sqrt(d);
      const real c = a[0] * rs;
      if (lane == j) dinv = rs;
      if (lane >= j && lane < n) A[lane + j * ld] = c;
#pragma unroll
      for (int t0 = 1; t0 < NB; t0 += 8) {
        if (j + t0 >= n) break;
#pragma unroll
        for (int t = t0; t < t0 + 8; t++)
          if (t < NB) a[t - 1] = a[t] - c * __shfl_sync(0xffffffffu, c, j + t);
      }
    }
    __syncwarp();
  } else if (lane < n) {
    dinv = real(1) / A[lane + lane * ld];
  }
  // column `lane` of the inverse: row i is final at step i, the rows below it
  // lose l_ri times it
#pragma unroll
  for (int r = 0; r < NB; r++) a[r] = r == lane ? real(1) : real(0);
#pragma unroll 1
  for (int i = 0; i < n; i++) {
    const real x = a[0] * __shfl_sync(0xffffffffu, dinv, i);
    const real* Li = A + i * ld;
#pragma unroll
    for (int t0 = 1; t0 < NB; t0 += 8) {
      if (i + t0 >= n) break;
#pragma unroll
      for (int t = t0; t < t0 + 8; t++)
        if (t < NB) a[t - 1] = a[t] - Li[min(i + t, n - 1)] * x;
    }
    __syncwarp();
    // (column i of L is not read again; row i of the inverse needs row i only)
    if (lane <= i) A[i + lane * ld] = x;
    __syncwarp();
  }
  for (int j = 1 + lane; j < n; j += 32)
    for (int i = 0; i < j; i++) A[i + j * ld] = 0;
  __syncwarp();
  return true;
}

// In place: the lower triangle of A (n x n) whose diagonal blocks of 32 hold
// their inverses already becomes the inverse of the whole, pairs of blocks at
// a time: X21 = -X22 (L21 X11).  tmp: at most n^2 / 4 elements (the pairs' n2 x w,
// n2 + w <= 2 w and summing to at most n).
template <typename real>
__device__ void tri_inv_levels(int n, real* A, int ld, real* tmp) {
  for (int w = NB; w < n; w *= 2) {
    // the pairs' products W = L21 X11 (n2 x w), side by side in tmp
    int first = 0, off = 0;
    for (int b = 0; b + w < n; b += 2 * w) {
      const int n2 = min(w, n - b - w);
      real* W = tmp + off;
      product<real, kFromCol, kToEnd>(n2, w, w, A + (b + w) + b * ld, 1, ld, A + b + b * ld, 1, ld,
                                      false, first, [&](int i, int j, real v) { W[i + j * n2] = v; });
      first += 256;
      off += n2 * w;
    }
    __syncthreads();
    first = off = 0;
    for (int b = 0; b + w < n; b += 2 * w) {
      const int n2 = min(w, n - b - w);
      const real* W = tmp + off;
      real* X21 = A + (b + w) + b * ld;
      product<real, kFrom0, kToRow>(n2, w, n2, A + (b + w) + (b + w) * ld, 1, ld, W, 1, n2, false,
                                    first, [&](int i, int j, real v) { X21[i + j * ld] = -v; });
      first += 256;
      off += n2 * w;
    }
    __syncthreads();
  }
}

__host__ __device__ inline int round32(int n) { return (n + 31) / 32 * 32; }
// Elements of the blocked routines' scratch for matrices of up to n columns:
// a panel of 32 columns, or the products of tri_inv_levels (at most n / 2
// pairs' worth of w x w)
__host__ __device__ inline int scratch_elems(int n) {
  const int a = n * NB, r = round32(n), b = r * r / 4 + NB * NB;
  return a > b ? a : b;
}

// A (n x n, lower triangle) becomes L^{-1} of its Cholesky factor L, zeros
// above the diagonal; false (for every thread) when a pivot is not positive.
// factored() is called between the factorization and the rest of the inverse.
template <typename real, typename Mark>
__device__ bool chol_inverse(int n, real* A, int ld, real* tmp, int* flag, Mark&& factored) {
  for (int p = 0; p < n; p += NB) {
    const int nb = min(NB, n - p), rest = n - p - nb;
    real* D = A + p + p * ld;
    if (warp_id() == 0) {
      const bool ok = warp_chol_inv<real>(nb, D, ld, true);
      if (lane_id() == 0) *flag = ok ? 1 : 0;
    }
    __syncthreads();
    if (!*flag) return false;
    if (rest > 0) {
      // L21 = A21 X11^T, through tmp into its place
      real* A21 = D + nb;
      product<real, kFrom0, kToCol>(rest, nb, nb, A21, 1, ld, D, ld, 1, false, 0,
                                    [&](int i, int j, real v) { tmp[i + j * rest] = v; });
      __syncthreads();
      for (int j = warp_id(); j < nb; j += NT / 32)
        for (int i = lane_id(); i < rest; i += 32) A21[i + j * ld] = tmp[i + j * rest];
      real* A22 = A21 + nb * ld;
      product<real, kFrom0, kToEnd>(rest, rest, nb, tmp, 1, rest, tmp, rest, 1, true, 0,
                                    [&](int i, int j, real v) {
                                      if (i >= j) A22[i + j * ld] -= v;
                                    });
    }
    __syncthreads();
  }
  for (int j = warp_id(); j < n; j += NT / 32)
    for (int i = lane_id(); i < j; i += 32) A[i + j * ld] = 0;
  __syncthreads();
  factored();
  tri_inv_levels<real>(n, A, ld, tmp);
  return true;
}

// W (m x k): reflectors, zeros above their heads; tau.  S (k x k, ld lds)
// becomes the lower triangular inverse of (triu(W^T W, 1) + diag(1 / tau))^T,
// so that H_0 .. H_{k-1} = I - W S^T W^T (compact WY form).
template <typename real>
__device__ void wy_factor(int m, int k, const real* W, int ldw, const real* tau, real* S, int lds,
                          real* tmp) {
  product<real, kFromRow, kToEnd>(k, k, m, W, ldw, 1, W, 1, ldw, true, 0,
                                  [&](int i, int j, real v) {
                                    S[i + j * lds] =
                                        i > j ? v : (i == j ? real(1) / tau[i] : real(0));
                                  });
  __syncthreads();
  // (tiles wholly above the diagonal were left out)
  for (int j = warp_id(); j < k; j += NT / 32)
    for (int i = lane_id(); i < j; i += 32) S[i + j * lds] = 0;
  __syncthreads();
  for (int b = warp_id() * NB; b < k; b += NT)
    warp_chol_inv<real>(min(NB, k - b), S + b + b * lds, lds, false);
  __syncthreads();
  tri_inv_levels<real>(k, S, lds, tmp);
}

// Householder QR without pivoting of X (m x k), columns in registers: warp w
// of the CTA keeps columns w, w + 16, ..; lane l rows l, l + 32, ..  Step j: the
// warp owning column j forms the reflector and publishes it (two buffers, one
// barrier per step), every warp applies it to its columns.  X receives the
// reflectors with zeros above their heads.  m <= 128, k <= 128.
template <typename real>
__device__ void qr_registers(int m, int k, real* X, int ldx, real* tau, real* vbuf, real* tbuf) {
  constexpr int W = NT / 32, CPW = 8, RPL = 4;
  const int lane = lane_id(), warp = warp_id();
  real x[CPW][RPL];
#pragma unroll
  for (int s = 0; s < CPW; s++)
#pragma unroll
    for (int r = 0; r < RPL; r++) {
      const int c = s * W + warp, i = lane + 32 * r;
      x[s][r] = (c < k && i < m) ? X[i + c * ldx] : real(0);
    }
#pragma unroll
  for (int s = 0; s < CPW; s++) {
    for (int w = 0; w < W; w++) {
      const int j = s * W + w;
      if (j >= k) break;
      real* v = vbuf + (j & 1) * 128;
      if (warp == w) {
        real sq = 0;
#pragma unroll
        for (int r = 0; r < RPL; r++)
          if (lane + 32 * r >= j) sq += x[s][r] * x[s][r];
        sq = warp_sum(sq);
        real h = 0;
#pragma unroll
        for (int r = 0; r < RPL; r++)
          if (r == j / 32) h = x[s][r];
        const real x0 = __shfl_sync(0xffffffffu, h, j % 32);
        real head, t;
        householder_scalars(sq, x0, &head, &t);
#pragma unroll
        for (int r = 0; r < RPL; r++) {
          const int i = lane + 32 * r;
          const real y = i < j ? real(0) : (i == j ? head : x[s][r]);
          v[i] = y;
          if (i < m) X[i + j * ldx] = y;
        }
        if (lane == 0) {
          tbuf[j & 1] = t;
          tau[j] = t;
        }
      }
      __syncthreads();
      const real t = tbuf[j & 1];
      real y[RPL];
#pragma unroll
      for (int r = 0; r < RPL; r++) y[r] = v[lane + 32 * r];
#pragma unroll
      for (int q = 0; q < CPW; q++) {
        const int c = q * W + warp;
        if (q < s || c <= j || c >= k) continue;
        real d = 0;
#pragma unroll
        for (int r = 0; r < RPL; r++) d += y[r] * x[q][r];
        d = warp_sum(d) * t;
#pragma unroll
        for (int r = 0; r < RPL; r++) x[q][r] -= d * y[r];
      }
    }
  }
  __syncthreads();
}

// The same on X in memory (larger m), two barriers per step.
template <typename real>
__device__ void qr_memory(int m, int k, real* X, int ldx, real* tau) {
  constexpr int W = NT / 32;
  const int lane = lane_id(), warp = warp_id();
  for (int j = 0; j < k; j++) {
    real* xj = X + j * ldx;
    if (warp == j % W) {
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
    }
    __syncthreads();
    const real t = tau[j];
    for (int c = j + 1 + warp; c < k; c += W) {
      real* xc = X + c * ldx;
      real d = 0;
      for (int i = j + lane; i < m; i += 32) d += xj[i] * xc[i];
      d = warp_sum(d) * t;
      for (int i = j + lane; i < m; i += 32) xc[i] -= d * xj[i];
    }
    __syncthreads();
  }
  for (int j = warp; j < k; j += W)
    for (int i = lane; i < j; i += 32) X[i + j * ldx] = 0;
  __syncthreads();
}

template <typename real>
__device__ void fail(DevError* err, int s, int level, int* rank, int m) {
  if (threadIdx.x == 0) {
    if (atomicCAS(&err->code, 0, (int)HSOLVE_ERR_NOT_SPD) == 0) {
      err->cluster = s;
      err->level = level;
    }
    rank[s] = m;  // leave the cluster untouched downstream
  }
}

template <typename real>
__global__ void __launch_bounds__(NT)
prep_spd_kernel(const PrepTask* __restrict__ tasks, real* __restrict__ arena,
                real* __restrict__ fac, real* __restrict__ ws_all, double* __restrict__ wsd_all,
                int* rank, int smem_mats, int smem_m, DevError* err, int level, long long* dbg) {
  extern __shared__ __align__(16) unsigned char spd_smem[];
  __shared__ real vbuf[2 * 128];
  __shared__ real tbuf[2];
  __shared__ int flag;
  const PrepTask tk = tasks[blockIdx.x];
  // optional per-phase clock stamps (profiling), the general kernel's
  // checkpoints: 0 -> 1 factor, 3 -> 4 inverse, -> 5 bases, -> 6 Z, -> 7 F and T'
  long long* stamp = dbg ? dbg + (int64_t)blockIdx.x * 8 : nullptr;
  const auto mark = [&](int i) {
    if (stamp && threadIdx.x == 0) stamp[i] = clock64();
  };
  mark(0);
  const int m = tk.m;
  const int64_t mm = (int64_t)m * m, reg = (int64_t)(smem_m | 1) * smem_m;
  real* sm = reinterpret_cast<real*>(spd_smem);
  real* ws = ws_all + tk.ws;
  const int ld1 = smem_mats >= 1 ? (m | 1) : m;
  const int ld2 = smem_mats >= 2 ? (m | 1) : m;
  const int ld3 = smem_mats >= 3 ? (m | 1) : m;
  real* R1 = smem_mats >= 1 ? sm : ws;
  real* R2 = smem_mats >= 2 ? sm + reg : ws + mm;
  real* R3 = smem_mats >= 3 ? sm + 2 * reg : ws + 2 * mm;
  real* tmp = sm + smem_mats * reg;      // scratch_elems(smem_m)
  real* tau2 = tmp + scratch_elems(smem_m);  // smem_m
  real* W_C = ws + 3 * mm;
  const real* W_G = ws + 10 * mm;        // reflectors of the pivoted QR
  const real* tau = reinterpret_cast<const real*>(wsd_all + tk.wsd + 2 * (int64_t)tk.ncolG);
  const real* rsign = tau + 2 * m;
  real* T = fac + tk.T;
  // (a cluster without fill columns has no QR; its rank is 0 also where forced)
  const int k = tk.ncolG > 0 ? rank[tk.s] : 0, f = m - k;
  if (tk.ncolG == 0 && threadIdx.x == 0) rank[tk.s] = 0;
  const int lane = lane_id(), warp = warp_id();
  constexpr int W = NT / 32;
  for (int j = warp; j < m; j += W)
    for (int i = lane; i < m; i += 32) R1[i + j * ld1] = arena[tk.a_ss + i + (int64_t)j * tk.ld];
  __syncthreads();
  if (!chol_inverse<real>(m, R1, ld1, tmp, &flag, [&] {
        mark(1);
        mark(3);
      })) {
    fail<real>(err, tk.s, level, rank, m);
    return;
  }
  mark(4);
  if (k == m) return;  // untouched: all unknowns coarse, E_s = I
  if (k == 0) {  // E_s = I: T' = L^{-1}
    for (int j = warp; j < m; j += W)
      for (int i = lane; i < m; i += 32) T[i + (int64_t)j * m] = R1[i + j * ld1];
    return;
  }
  // ---- U = first k columns of Q, oriented so that R has a positive diagonal
  // (Gram-Schmidt directions): U = (E_k - W M) sign, M = S^T W_1^T upper
  // triangular, W_1 the first k rows of W
  for (int j = warp; j < k; j += W)
    for (int i = lane; i < m; i += 32) R3[i + j * ld3] = i >= j ? W_G[i + (int64_t)j * m] : real(0);
  __syncthreads();
  real* M = 2 * (int64_t)k * k <= (int64_t)m * m ? R2 + k * k : W_C;  // k x k, ld k
  wy_factor<real>(m, k, R3, ld3, tau, R2, k, tmp);
  product<real, kFromRow, kToCol>(k, k, k, R2, k, 1, R3, ld3, 1, false, 0,
                                  [&](int i, int j, real v) { M[i + j * k] = v; });
  __syncthreads();
  // column blocks from the last to the first: block j needs W's columns <= j
  for (int j0 = (k - 1) / NB * NB; j0 >= 0; j0 -= NB) {
    const int nb = min(NB, k - j0);
    product<real, kFrom0, kToEnd>(m, nb, j0 + nb, R3, 1, ld3, M + j0 * k, 1, k, false, 0,
                                  [&](int i, int j, real v) {
                                    tmp[i + j * m] = ((i == j0 + j ? real(1) : real(0)) - v) *
                                                     rsign[j0 + j];
                                  });
    __syncthreads();
    for (int j = warp; j < nb; j += W)
      for (int i = lane; i < m; i += 32) R3[i + (j0 + j) * ld3] = tmp[i + j * m];
    __syncthreads();
  }
  // ---- P = Li U (R2), C = P^T P, D = C U^T, X = Li^T P (R3)
  product<real, kFrom0, kToRow>(m, k, m, R1, 1, ld1, R3, 1, ld3, false, 0,
                                [&](int i, int j, real v) { R2[i + j * ld2] = v; });
  __syncthreads();
  product<real, kFrom0, kToEnd>(k, k, m, R2, ld2, 1, R2, 1, ld2, true, 0,
                                [&](int i, int j, real v) {
                                  if (i < j) return;
                                  W_C[i + j * m] = v;
                                  W_C[j + i * m] = v;
                                });
  __syncthreads();
  {
    real* D = ws_all + tk.D;
    product<real, kFrom0, kToEnd>(k, m, k, W_C, 1, m, R3, ld3, 1, false, 0,
                                  [&](int i, int j, real v) { D[i + (int64_t)j * m] = v; });
  }
  __syncthreads();
  product<real, kFromRow, kToEnd>(m, k, m, R1, ld1, 1, R2, 1, ld2, false, 0,
                                  [&](int i, int j, real v) {
                                    R3[i + j * ld3] = v;
                                    T[j + (int64_t)i * m] = v;  // coarse rows: X^T
                                  });
  __syncthreads();
  // ---- V (R3, columns k..): E_f - W M, M = S^T W_2^T (k x f), W_2 the rows k..
  if (m <= 128 && k <= 128) qr_registers<real>(m, k, R3, ld3, tau2, vbuf, tbuf);
  else qr_memory<real>(m, k, R3, ld3, tau2);
  wy_factor<real>(m, k, R3, ld3, tau2, R2, k, tmp);
  {
    real* M2 = R2 + k * k;
    product<real, kFromRow, kToEnd>(k, f, k, R2, k, 1, R3 + k, ld3, 1, false, 0,
                                    [&](int i, int j, real v) { M2[i + j * k] = v; });
    __syncthreads();
    product<real, kFrom0, kToEnd>(m, f, k, R3, 1, ld3, M2, 1, k, false, 0,
                                  [&](int i, int j, real v) {
                                    R3[i + (k + j) * ld3] = (i == k + j ? real(1) : real(0)) - v;
                                  });
  }
  __syncthreads();
  mark(5);
  // ---- Z = Li V (R2), F = Z^T Z (R3) and the inverse of its factor
  product<real, kFrom0, kToRow>(m, f, m, R1, 1, ld1, R3 + k * ld3, 1, ld3, false, 0,
                                [&](int i, int j, real v) { R2[i + j * ld2] = v; });
  __syncthreads();
  mark(6);
  product<real, kFrom0, kToEnd>(f, f, m, R2, ld2, 1, R2, 1, ld2, true, 0,
                                [&](int i, int j, real v) { R3[i + j * ld3] = v; });
  __syncthreads();
  if (!chol_inverse<real>(f, R3, ld3, tmp, &flag, [] {})) {
    fail<real>(err, tk.s, level, rank, m);
    return;
  }
  // ---- T' fine rows = (Z L_F^{-T})^T Li: Z L_F^{-T} in place, column blocks
  // from the last to the first
  for (int j0 = (f - 1) / NB * NB; j0 >= 0; j0 -= NB) {
    const int nb = min(NB, f - j0);
    product<real, kFrom0, kToEnd>(m, nb, j0 + nb, R2, 1, ld2, R3 + j0, ld3, 1, false, 0,
                                  [&](int i, int j, real v) { tmp[i + j * m] = v; });
    __syncthreads();
    for (int j = warp; j < nb; j += W)
      for (int i = lane; i < m; i += 32) R2[i + (j0 + j) * ld2] = tmp[i + j * m];
    __syncthreads();
  }
  product<real, kFromCol, kToEnd>(f, m, m, R2, ld2, 1, R1, 1, ld1, false, 0,
                                  [&](int i, int j, real v) { T[k + i + (int64_t)j * m] = v; });
  mark(7);
  // C into the (s,s) block (coarse part); last: A_ss was copied
  real* ss = arena + tk.a_ss;
  for (int j = warp; j < k; j += W)
    for (int i = lane; i < k; i += 32) ss[i + (int64_t)j * tk.ld] = W_C[i + j * m];
}

// X = L^{-1} of the Cholesky factor of the lower n x n block at A, on one CTA,
// by the same blocks of 32 (128 unknowns: about 100 us; one column at a time by the
// whole CTA took 198).
template <typename real>
__global__ void __launch_bounds__(NT)
chol_inv_leaf_kernel(const real* __restrict__ A, int64_t lda, real* __restrict__ X, int64_t ldx,
                     int n, DevError* err, int level) {
  extern __shared__ __align__(16) unsigned char spd_smem[];
  __shared__ int flag;
  real* R = reinterpret_cast<real*>(spd_smem);
  const int ld = n | 1;
  real* tmp = R + n * ld;
  for (int j = warp_id(); j < n; j += NT / 32)
    for (int i = lane_id(); i < n; i += 32) R[i + j * ld] = A[i + (int64_t)j * lda];
  __syncthreads();
  if (!chol_inverse<real>(n, R, ld, tmp, &flag, [] {})) {
    if (threadIdx.x == 0 && atomicCAS(&err->code, 0, (int)HSOLVE_ERR_NOT_SPD) == 0) {
      err->cluster = 0;
      err->level = level;
    }
    return;
  }
  for (int j = warp_id(); j < n; j += NT / 32)
    for (int i = lane_id(); i < n; i += 32) X[i + (int64_t)j * ldx] = R[i + j * ld];
}

}  // namespace

void chol_inv_leaf(float* A, int64_t lda, float* X, int64_t ldx, int n, DevError* err, int level,
                   cudaStream_t st) {
  const auto bytes = [](int v) { return sizeof(float) * ((size_t)(v | 1) * v + scratch_elems(v)); };
  static const bool limit_set = [&] {
    cudaFuncSetAttribute(chol_inv_leaf_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)bytes(128));
    return true;
  }();
  (void)limit_set;
  count_launch();
  chol_inv_leaf_kernel<float><<<1, NT, bytes(n), st>>>(A, lda, X, ldx, n, err, level);
}

template <typename real>
bool Launch<real>::prep_spd(const PrepTask* tasks, int ntask, real* arena, real* fac, real* ws,
                            double* wsd, int* rank, int maxm, DevError* err, int level,
                            long long* dbg, cudaStream_t st) {
  if (maxm > kMaxM) return false;
  if (ntask <= 0) return true;
  const size_t budget = 224 * 1024;
  const size_t one = sizeof(real) * (size_t)(maxm | 1) * maxm;
  const size_t fix = sizeof(real) * (size_t)(scratch_elems(maxm) + maxm);
  int mats = 0;
  while (mats < 3 && (mats + 1) * one + fix <= budget) mats++;
  static const bool limit_set = [budget] {
    cudaFuncSetAttribute(prep_spd_kernel<real>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)budget);
    return true;
  }();
  (void)limit_set;
  count_launch();
  prep_spd_kernel<real><<<ntask, NT, mats * one + fix, st>>>(tasks, arena, fac, ws, wsd, rank, mats,
                                                            maxm, err, level, dbg);
  return true;
}

template bool Launch<float>::prep_spd(const PrepTask*, int, float*, float*, float*, double*, int*,
                                      int, DevError*, int, long long*, cudaStream_t);
template bool Launch<double>::prep_spd(const PrepTask*, int, double*, double*, double*, double*,
                                       int*, int, DevError*, int, long long*, cudaStream_t);

}  // namespace hs
