// Substitution sweeps of Alg. 2, one launch per colour class and direction.
//
// Forward (y <- W_s y for the clusters of a class): z_s = T' y_s with T' =
// diag(I, L_F^{-1} [P_F]) [U V_L]^T A_ss^{-1}, y_N -= B_L z_f, y_s = z_s.
// Backward (x <- W_s^T x): z_s = [x_c; x_f - B_R x_N], x_s = T_R'^T z_s.
// Clusters of one class touch disjoint slots (their neighbour sets are
// disjoint, Sec. 3.2), so no atomics are needed.
//
// A sweep is a chain of hundreds of dependent classes whose operators are
// small: its time is the time of one link, not the operator bytes.  So a
// class is one launch (fwd_sweep_kernel, bwd_sweep_kernel): a cluster's rows
// and neighbour columns are split over the CTAs of a thread-block cluster,
// which exchange z_s (or the partial sums of B_R x_N) through distributed
// shared memory instead of through a second launch; and the launches are
// programmatic dependents of one another: a class's CTAs start while the
// class before still runs, copy their operator slices (which no sweep
// writes) into shared memory, and only then wait for the vectors.
// The figures are at sweep_shape.
//
// The dense top (one cluster, nothing but a triangular T' of thousands of
// unknowns) has kernels of its own that stream the triangle once from HBM.
// Clusters too large for the shared-memory vectors of the fused kernels, and
// large ones with many right-hand sides (kManyRhs), take the unfused ones:
// fwd_t, fwd_nbr, bwd_part, bwd_z, bwd_t.
#include <algorithm>
#include <cooperative_groups.h>
#include <type_traits>
#include <utility>

#include "common.h"

namespace cg = cooperative_groups;

namespace hs {

namespace {

constexpr int kRows = 64;   // output rows per CTA in the T' products
constexpr int kCols = 64;   // neighbour columns per CTA
// right-hand sides per CTA (grid z runs over the groups): 8 when there are
// several, 1 for a single one (a wider group's predicated-off products would
// still be issued, which the float64 pipe cannot afford)
constexpr int kRbWide = 8;

// The right-hand-side group of this CTA: columns r0 .. r0 + nr, groups of
// rb <= RB columns (rb is smaller when RB slot vectors would not fit in
// shared memory).
struct RhsGroup {
  int r0, nr;
  __device__ RhsGroup(int nrhs, int rb)
      : r0(blockIdx.z * rb), nr(min(rb, nrhs - (int)blockIdx.z * rb)) {}
};

// Sums of RB values over a warp.  RB = 8: a reduce-scatter butterfly (9
// shuffles instead of 8 x 5): each exchange halves the set of values a lane
// carries, lane l ending with the total of value rs_index(l); lanes 0..7
// hold the 8 totals once each.  RB = 1: the plain butterfly in every lane.
__device__ __forceinline__ int rs_index(int lane) {
  return ((lane & 1) << 2) | (lane & 2) | ((lane & 4) >> 2);
}

template <typename real>
__device__ __forceinline__ real warp_sum8(const real (&v)[8]) {
  const int lane = threadIdx.x & 31;
  real a[4], b[2];
  const bool h1 = lane & 1, h2 = lane & 2, h4 = lane & 4;
#pragma unroll
  for (int j = 0; j < 4; j++)
    a[j] = (h1 ? v[4 + j] : v[j]) + __shfl_xor_sync(0xffffffffu, h1 ? v[j] : v[4 + j], 1);
#pragma unroll
  for (int j = 0; j < 2; j++)
    b[j] = (h2 ? a[2 + j] : a[j]) + __shfl_xor_sync(0xffffffffu, h2 ? a[j] : a[2 + j], 2);
  real c = (h4 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, h4 ? b[0] : b[1], 4);
  c += __shfl_xor_sync(0xffffffffu, c, 8);
  c += __shfl_xor_sync(0xffffffffu, c, 16);
  return c;
}

// Reduce acc[0..RB) over the warp; returns the total that this lane reports
// and sets *r to its right-hand side (-1: this lane reports nothing).
template <typename real, int RB>
__device__ __forceinline__ real warp_sums(real (&acc)[RB], int* r) {
  const int lane = threadIdx.x & 31;
  if constexpr (RB == 8) {
    const real t = warp_sum8<real>(acc);
    *r = lane < 8 ? rs_index(lane) : -1;
    return t;
  } else {
    real t = acc[0];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    *r = lane == 0 ? 0 : -1;
    return t;
  }
}

template <typename real, int RB>
__global__ void __launch_bounds__(256)
fwd_t_kernel(const ApplyRec* __restrict__ recs, const int* __restrict__ ids,
             const real* __restrict__ fac, const real* __restrict__ y, real* __restrict__ z,
             int64_t ldy, int nrhs, int rb) {
  extern __shared__ unsigned char smem_raw[];
  real* ys = reinterpret_cast<real*>(smem_raw);  // RB x m
  __shared__ real red[RB][256];
  const ApplyRec rc = recs[ids[blockIdx.y]];
  const int m = rc.m;
  if (rc.k == m) return;
  const int i0 = blockIdx.x * kRows;
  if (i0 >= m) return;
  const RhsGroup g(nrhs, rb);
  const real* T = fac + rc.T;
  const int ii = threadIdx.x % kRows, part = threadIdx.x / kRows;  // 4 parts over l
  const int i = i0 + ii;
  for (int r = 0; r < g.nr; r++)
    for (int l = threadIdx.x; l < m; l += blockDim.x)
      ys[r * m + l] = y[rc.voff + l + (int64_t)(g.r0 + r) * ldy];
  __syncthreads();
  real acc[RB];
#pragma unroll
  for (int r = 0; r < RB; r++) acc[r] = 0;
  if (i < m) {
    // four independent loads in flight per step
    int l = part;
    for (; l + 12 < m; l += 16) {
      const real t0 = __ldg(T + i + (int64_t)l * m);
      const real t1 = __ldg(T + i + (int64_t)(l + 4) * m);
      const real t2 = __ldg(T + i + (int64_t)(l + 8) * m);
      const real t3 = __ldg(T + i + (int64_t)(l + 12) * m);
#pragma unroll
      for (int r = 0; r < RB; r++)
        if (r < g.nr)
          acc[r] += t0 * ys[r * m + l] + t1 * ys[r * m + l + 4] + t2 * ys[r * m + l + 8] +
                    t3 * ys[r * m + l + 12];
    }
    for (; l < m; l += 4) {
      const real t = __ldg(T + i + (int64_t)l * m);
#pragma unroll
      for (int r = 0; r < RB; r++)
        if (r < g.nr) acc[r] += t * ys[r * m + l];
    }
  }
#pragma unroll
  for (int r = 0; r < RB; r++) red[r][threadIdx.x] = acc[r];
  __syncthreads();
  if (part == 0 && i < m)
    for (int r = 0; r < g.nr; r++)
      z[rc.voff + i + (int64_t)(g.r0 + r) * ldy] =
          red[r][ii] + red[r][ii + 64] + red[r][ii + 128] + red[r][ii + 192];
}

template <typename real, int RB>
__global__ void __launch_bounds__(256)
fwd_nbr_kernel(const ApplyRec* __restrict__ recs, const int* __restrict__ ids,
               const real* __restrict__ fac, const int64_t* __restrict__ vmap,
               real* __restrict__ y, const real* __restrict__ z, int64_t ldy, int nrhs, int rb) {
  extern __shared__ unsigned char smem_raw[];
  real* zsh = reinterpret_cast<real*>(smem_raw);  // RB x f: z_f, read once per CTA
  __shared__ real dsh[RB][kCols];                 // the column sums of this CTA
  const ApplyRec rc = recs[ids[blockIdx.y]];
  const int m = rc.m, k = rc.k, f = m - k;
  if (k == m) return;
  const RhsGroup g(nrhs, rb);
  if (blockIdx.x == 0)
    for (int r = 0; r < g.nr; r++)
      for (int i = threadIdx.x; i < m; i += blockDim.x)
        y[rc.voff + i + (int64_t)(g.r0 + r) * ldy] = z[rc.voff + i + (int64_t)(g.r0 + r) * ldy];
  const int c0 = blockIdx.x * kCols;
  if (c0 >= rc.nw) return;
  const int c1 = min(rc.nw, c0 + kCols);
  for (int r = 0; r < g.nr; r++)
    for (int i = threadIdx.x; i < f; i += blockDim.x)
      zsh[r * f + i] = z[rc.voff + k + i + (int64_t)(g.r0 + r) * ldy];
  __syncthreads();
  const real* BL = fac + (rc.sym ? rc.Y : rc.XT) + k;  // column c: B_L[c, :]
  const int64_t* vm = vmap + rc.map;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  for (int c = c0 + warp; c < c1; c += nwarp) {
    const real* col = BL + (int64_t)c * m;
    real acc[RB];
#pragma unroll
    for (int r = 0; r < RB; r++) acc[r] = 0;
    for (int i = lane; i < f; i += 32) {
      const real b = col[i];
#pragma unroll
      for (int r = 0; r < RB; r++)
        if (r < g.nr) acc[r] += b * zsh[r * f + i];
    }
    int rr;
    const real t = warp_sums<real, RB>(acc, &rr);
    if (rr >= 0) dsh[rr][c - c0] = t;
  }
  __syncthreads();
  // y_N -= B_L z_f: every thread one (column, right-hand side) of the CTA;
  // the neighbour slots of a column range are contiguous runs
  const int nc = c1 - c0;
  for (int e = threadIdx.x; e < nc * g.nr; e += blockDim.x) {
    const int c = e % nc, r = e / nc;
    y[vm[c0 + c] + (int64_t)(g.r0 + r) * ldy] -= dsh[r][c];
  }
}

template <typename real, int RB>
__global__ void __launch_bounds__(256)
bwd_part_kernel(const ApplyRec* __restrict__ recs, const int* __restrict__ ids,
                const real* __restrict__ fac, const int64_t* __restrict__ vmap,
                const real* __restrict__ y, real* __restrict__ part, int64_t ldy, int nrhs, int rb) {
  __shared__ real xn[RB][kCols];
  const ApplyRec rc = recs[ids[blockIdx.y]];
  const int m = rc.m, k = rc.k, f = m - k;
  if (k == m) return;
  const int c0 = blockIdx.x * kCols;
  if (c0 >= rc.nw) return;
  const RhsGroup g(nrhs, rb);
  const int nc = min(rc.nw, c0 + kCols) - c0;
  const int nchunk = (rc.nw + kCols - 1) / kCols;
  const real* BR = fac + rc.Y + k;
  const int64_t* vm = vmap + rc.map;
  real* pr = part + rc.part * nrhs;
  for (int r = 0; r < g.nr; r++)
    for (int c = threadIdx.x; c < nc; c += blockDim.x)
      xn[r][c] = y[vm[c0 + c] + (int64_t)(g.r0 + r) * ldy];
  __syncthreads();
  for (int i = threadIdx.x; i < f; i += blockDim.x) {
    real acc[RB];
#pragma unroll
    for (int r = 0; r < RB; r++) acc[r] = 0;
    const real* Bi = BR + i + (int64_t)c0 * m;
    int c = 0;
    // four independent loads in flight per step
    for (; c + 3 < nc; c += 4) {
      const real b0 = __ldg(Bi + (int64_t)c * m), b1 = __ldg(Bi + (int64_t)(c + 1) * m);
      const real b2 = __ldg(Bi + (int64_t)(c + 2) * m), b3 = __ldg(Bi + (int64_t)(c + 3) * m);
#pragma unroll
      for (int r = 0; r < RB; r++)
        acc[r] += b0 * xn[r][c] + b1 * xn[r][c + 1] + b2 * xn[r][c + 2] + b3 * xn[r][c + 3];
    }
    for (; c < nc; c++) {
      const real b = __ldg(Bi + (int64_t)c * m);
#pragma unroll
      for (int r = 0; r < RB; r++) acc[r] += b * xn[r][c];
    }
#pragma unroll
    for (int r = 0; r < RB; r++)
      if (r < g.nr) pr[((int64_t)(g.r0 + r) * nchunk + blockIdx.x) * f + i] = acc[r];
  }
}

template <typename real, int RB>
__global__ void __launch_bounds__(256)
bwd_z_kernel(const ApplyRec* __restrict__ recs, const int* __restrict__ ids,
             const real* __restrict__ y, real* __restrict__ z, const real* __restrict__ part,
             int64_t ldy, int nrhs, int rb) {
  const ApplyRec rc = recs[ids[blockIdx.x]];
  const int m = rc.m, k = rc.k, f = m - k;
  if (k == m) return;
  const RhsGroup g(nrhs, rb);
  const int nchunk = (rc.nw + kCols - 1) / kCols;
  const real* pr = part + rc.part * nrhs;
  for (int r = g.r0; r < g.r0 + g.nr; r++) {
    const real* ys = y + rc.voff + (int64_t)r * ldy;
    real* zs = z + rc.voff + (int64_t)r * ldy;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
      real v = ys[i];
      if (i >= k)
        for (int q = 0; q < nchunk; q++) v -= pr[((int64_t)r * nchunk + q) * f + (i - k)];
      zs[i] = v;
    }
  }
}

template <typename real, int RB>
__global__ void __launch_bounds__(256)
bwd_t_kernel(const ApplyRec* __restrict__ recs, const int* __restrict__ ids,
             const real* __restrict__ fac, real* __restrict__ y, const real* __restrict__ z,
             int64_t ldy, int nrhs, int rb) {
  extern __shared__ unsigned char smem_raw[];
  real* zsm = reinterpret_cast<real*>(smem_raw);  // RB x m
  const ApplyRec rc = recs[ids[blockIdx.y]];
  const int m = rc.m;
  if (rc.k == m) return;
  const int i0 = blockIdx.x * kRows;
  if (i0 >= m) return;
  const RhsGroup g(nrhs, rb);
  const int i1 = min(m, i0 + kRows);
  const real* TRt = fac + (rc.sym ? rc.T : rc.TR);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  for (int r = 0; r < g.nr; r++)
    for (int l = threadIdx.x; l < m; l += blockDim.x)
      zsm[r * m + l] = z[rc.voff + l + (int64_t)(g.r0 + r) * ldy];
  __syncthreads();
  for (int i = i0 + warp; i < i1; i += nwarp) {
    const real* col = TRt + (int64_t)i * m;
    real acc[RB];
#pragma unroll
    for (int r = 0; r < RB; r++) acc[r] = 0;
    for (int l = lane; l < m; l += 32) {
      const real t = col[l];
#pragma unroll
      for (int r = 0; r < RB; r++)
        if (r < g.nr) acc[r] += t * zsm[r * m + l];
    }
    int rr;
    const real tot = warp_sums<real, RB>(acc, &rr);
    if (rr >= 0 && rr < g.nr) y[rc.voff + i + (int64_t)(g.r0 + rr) * ldy] = tot;
  }
}

// ---------------------------------------------------------------------------
// Fused sweeps: one launch per class and direction
// ---------------------------------------------------------------------------
constexpr int kSweepThreads = 256;
constexpr int kSweepMaxCl = 8;  // CTAs per cluster, the portable limit

// Programmatic dependent launch: the kernel after this one may start; this
// kernel waits until the one before it has completed and its writes are
// visible.  Every CTA executes the wait, also those without work: a launch
// whose CTAs all left early would otherwise count as completed while the one
// before it still ran.
__device__ __forceinline__ void pdl_launch() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ void cp_async(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Leading dimension of the transposed T' tile: 7 or 9 modulo 16, so that the
// 4 rows x 8 columns a warp reads at once overlap in at most one bank and the
// transposing copies (a warp writes one column) meet no conflict.
__host__ __device__ constexpr int sweep_ld(int n) {
  int v = n;
  while ((v & 15) != 7 && (v & 15) != 9) v++;
  return v;
}

// Leading dimension of staged columns of m elements.  When the columns are
// whole 16-byte units they are spread to 8 or 24 modulo 32 elements (4 columns
// x 8 rows meet no bank conflict; an unspread 128 would meet four); else the
// columns are copied as they stand in memory.
template <typename real>
__host__ __device__ constexpr int column_ld(int m) {
  constexpr int unit = 16 / (int)sizeof(real);
  int v = m;
  if (m % unit == 0)
    while ((v & 31) != 8 && (v & 31) != 24) v += unit;
  return v;
}

// Stride of a vector block in shared memory, [index][right-hand side]: RB
// padded to an odd number of 16-byte units, so that eight consecutive indices
// read with 16-byte loads fall into different banks.
template <typename real, int RB>
struct VecStride {
  static constexpr int unit = 16 / (int)sizeof(real);
  static constexpr int value = (RB % unit == 0 && (RB / unit) % 2 == 0) ? RB + unit : RB;
};

// dst[r * ldd + c] = src[r + c * lds], asynchronously (r < nrow runs along
// global memory): the rows of T' a CTA multiplies.
template <typename real>
__device__ __forceinline__ void stage_rows(real* dst, int ldd, const real* __restrict__ src,
                                           int lds, int nrow, int ncol) {
  // lanes along the rows, several columns per warp when they are few
  int p2 = 32;
  while (p2 > 4 && p2 / 2 >= nrow) p2 >>= 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = 32 / p2;
  for (int c = warp * per + lane / p2; c < ncol; c += (kSweepThreads / 32) * per)
    for (int r = lane & (p2 - 1); r < nrow; r += p2)
      cp_async(dst + r * ldd + c, src + r + (int64_t)c * lds);
}

// ncol whole columns of m elements (contiguous in memory from `src`) into
// `dst` with leading dimension column_ld(m), asynchronously in 16-byte units:
// four times fewer copy instructions than element by element, which crowded
// out the CTAs already computing on the same SM.  Returns where column 0
// starts: columns that are not whole units are copied as one stretch from the
// 16-byte boundary before `src` (the arena starts on one and ends on one).
template <typename real>
__device__ __forceinline__ const real* stage_columns(real* dst, const real* __restrict__ src,
                                                     int m, int ncol) {
  constexpr int unit = 16 / (int)sizeof(real);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (m % unit == 0) {
    const int ld = column_ld<real>(m), n = m / unit;
    int p2 = 32;
    while (p2 > 4 && p2 / 2 >= n) p2 >>= 1;
    const int per = 32 / p2;
    for (int c = warp * per + lane / p2; c < ncol; c += (kSweepThreads / 32) * per)
      for (int u = lane & (p2 - 1); u < n; u += p2)
        cp_async16(dst + c * ld + u * unit, src + (int64_t)c * m + u * unit);
    return dst;
  }
  const int shift = (int)((reinterpret_cast<uintptr_t>(src) & 15) / sizeof(real));
  const int n = ncol > 0 ? (shift + ncol * m + unit - 1) / unit : 0;
  const real* s = src - shift;
  for (int u = threadIdx.x; u < n; u += kSweepThreads) cp_async16(dst + u * unit, s + u * unit);
  return dst + shift;
}

template <typename real, int RB>
__device__ __forceinline__ void load_vec(const real* v, real (&x)[RB]) {
  if constexpr (RB * sizeof(real) % 16 == 0) {
    constexpr int U = 16 / (int)sizeof(real);
#pragma unroll
    for (int u = 0; u < RB / U; u++) {
      const int4 q = *reinterpret_cast<const int4*>(v + u * U);
      const real* e = reinterpret_cast<const real*>(&q);
#pragma unroll
      for (int w = 0; w < U; w++) x[u * U + w] = e[w];
    }
  } else {
#pragma unroll
    for (int r = 0; r < RB; r++) x[r] = v[r];
  }
}

// dst[l][r] = y[slot(l)] of right-hand side r0 + r for l < n, zeros for the
// group's missing right-hand sides.  A warp takes one right-hand side at a
// time (several warps share one when there are fewer than eight) and keeps
// eight loads in flight: right after the wait for the class before, this
// latency is on the chain.
template <typename real, int RB, typename Slot>
__device__ __forceinline__ void load_block(real* dst, const real* y, int64_t ldy, int r0, int nr,
                                           int n, Slot&& slot) {
  constexpr int VS = VecStride<real, RB>::value;
  constexpr int W = RB < 8 ? RB : 8, SUB = 8 / W, RW = RB / W, U = 8 / RW;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int b = (warp / W) * 32 + lane; b < n; b += SUB * 32 * U) {
    real v[U][RW];
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int l = b + u * SUB * 32;
      const int64_t at = l < n ? slot(l) : 0;
#pragma unroll
      for (int w = 0; w < RW; w++) {
        const int r = warp % W + w * W;
        v[u][w] = (l < n && r < nr) ? __ldcg(y + at + (int64_t)(r0 + r) * ldy) : real(0);
      }
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int l = b + u * SUB * 32;
      if (l < n)
#pragma unroll
        for (int w = 0; w < RW; w++) dst[l * VS + warp % W + w * W] = v[u][w];
    }
  }
}

// y[slot(l)] of right-hand side r0 + r = src[l][r] for l < n, r < nr.
template <typename real, int RB, typename Slot>
__device__ __forceinline__ void store_block(real* y, const real* src, int64_t ldy, int r0, int nr,
                                            int n, Slot&& slot) {
  constexpr int VS = VecStride<real, RB>::value;
  constexpr int W = RB < 8 ? RB : 8, SUB = 8 / W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int l = (warp / W) * 32 + lane; l < n; l += SUB * 32) {
    real* yl = y + slot(l) + (int64_t)r0 * ldy;
    for (int r = warp % W; r < nr; r += W) yl[r * ldy] = src[l * VS + r];
  }
}

// The 16-byte units (single elements for one right-hand side) of a vector
// block that are exchanged through distributed shared memory.
template <typename real, int RB>
struct Unit {
  static constexpr bool wide = RB * sizeof(real) % 16 == 0;
  static constexpr int n = wide ? 16 / (int)sizeof(real) : 1;  // elements
  static constexpr int per = RB / n;                           // units per index
  alignas(16) real v[n];
  __device__ __forceinline__ void load(const real* p) {
    if constexpr (wide) *reinterpret_cast<int4*>(v) = *reinterpret_cast<const int4*>(p);
    else v[0] = p[0];
  }
  __device__ __forceinline__ void store(real* p) const {
    if constexpr (wide) *reinterpret_cast<int4*>(p) = *reinterpret_cast<const int4*>(v);
    else p[0] = v[0];
  }
};

// Sum N values over the 8 lanes of a group (xor masks MASK, 2 MASK, ..): every
// exchange halves the set a lane carries while more than one is left.
template <typename real, int N, int MASK>
__device__ __forceinline__ void group_reduce(real* a, int lane, int* base) {
  if constexpr (MASK < 8) {
    if constexpr (N > 1) {
      const bool up = lane & MASK;
#pragma unroll
      for (int j = 0; j < N / 2; j++) {
        const real keep = up ? a[N / 2 + j] : a[j];
        const real send = up ? a[j] : a[N / 2 + j];
        a[j] = keep + __shfl_xor_sync(0xffffffffu, send, MASK);
      }
      if (up) *base += N / 2;
      group_reduce<real, N / 2, MASK * 2>(a, lane, base);
    } else {
      a[0] += __shfl_xor_sync(0xffffffffu, a[0], MASK);
      group_reduce<real, 1, MASK * 2>(a, lane, base);
    }
  }
}

// out(o, r) = sum_l A[o * lda + l] v[l][r] for o < nout: eight lanes share NO
// outputs, 32 NO outputs per pass of the CTA.  emit(o, r, value) is called once
// per output and right-hand side.
template <typename real, int RB, int NO, typename Emit>
__device__ __forceinline__ void sweep_dots_by(const real* A, int lda, int nout, int inner,
                                              const real* v, Emit& emit) {
  constexpr int VS = VecStride<real, RB>::value;
  constexpr int kLeft = RB >= 8 ? RB / 8 : 1;  // values a lane ends with
  constexpr int kGroups = kSweepThreads / 8;
  const int lane = threadIdx.x & 31, p = threadIdx.x & 7, g = threadIdx.x >> 3;
  for (int base0 = 0; base0 < nout; base0 += kGroups * NO) {
    // (a warp whose outputs are all missing from the last pass leaves the pipes
    // to the others)
    if (base0 + (g & ~3) >= nout) break;
    const real* row[NO];
#pragma unroll
    for (int w = 0; w < NO; w++) row[w] = A + min(base0 + g + w * kGroups, nout - 1) * lda;
    real acc[NO][RB];
#pragma unroll
    for (int w = 0; w < NO; w++)
#pragma unroll
      for (int r = 0; r < RB; r++) acc[w][r] = 0;
    constexpr int kUnroll = NO * RB >= 32 ? 1 : (NO * RB >= 8 ? 2 : 4);
    int l = p;
    for (; l + 8 * (kUnroll - 1) < inner; l += 8 * kUnroll) {
      real a[kUnroll][NO];
#pragma unroll
      for (int u = 0; u < kUnroll; u++)
#pragma unroll
        for (int w = 0; w < NO; w++) a[u][w] = row[w][l + 8 * u];
#pragma unroll
      for (int u = 0; u < kUnroll; u++) {
        real x[RB];
        load_vec<real, RB>(v + (l + 8 * u) * VS, x);
#pragma unroll
        for (int w = 0; w < NO; w++)
#pragma unroll
          for (int r = 0; r < RB; r++) acc[w][r] += a[u][w] * x[r];
      }
    }
    for (; l < inner; l += 8) {
      real x[RB];
      load_vec<real, RB>(v + l * VS, x);
#pragma unroll
      for (int w = 0; w < NO; w++) {
        const real a = row[w][l];
#pragma unroll
        for (int r = 0; r < RB; r++) acc[w][r] += a * x[r];
      }
    }
    // fewer right-hand sides than lanes: the first lane holding a total
    const bool mine = RB >= 8 || p < (RB == 4 ? 4 : 1);
#pragma unroll
    for (int w = 0; w < NO; w++) {
      int base = 0;
      group_reduce<real, RB, 1>(acc[w], lane, &base);
      const int o = base0 + g + w * kGroups;
      if (mine && o < nout)
#pragma unroll
        for (int j = 0; j < kLeft; j++) emit(o, base + j, acc[w][j]);
    }
  }
}

// Several outputs per group where there are enough: they share the vector's
// loads and overlap one another's latency (a forward link of 96^3's level 3, 490
// columns per CTA and 8 right-hand sides, spent 5.2 of its 12.5 us in passes of
// one output).  One application, one output -> several: 64^3 2.08 -> 1.96 ms, 96^3
// with variable coefficients 6.44 -> 5.88, 96^3 with 8 right-hand sides 15.2 ->
// 14.2.  Float64 takes one: its pipe is the bound, and the last pass's missing
// outputs are multiplied all the same (64^3 4.62 -> 5.36).
template <typename real, int RB, typename Emit>
__device__ __forceinline__ void sweep_dots(const real* A, int lda, int nout, int inner,
                                           const real* v, Emit&& emit) {
  constexpr int NO = sizeof(real) == 8 ? 1 : (RB >= 32 ? 2 : 4);
  if (NO > 1 && nout > kSweepThreads / 8) sweep_dots_by<real, RB, NO>(A, lda, nout, inner, v, emit);
  else sweep_dots_by<real, RB, 1>(A, lda, nout, inner, v, emit);
}

// out[i][r] (+)= sum_c A[c * lda + i] x[c][r] for i < nrow, c < ncol.  Lanes run
// along the rows (no bank conflicts for any lda), the warps split the row
// blocks and the columns; the column parts are added through `red`
// (max(256, nrow) rows).  Ends with a barrier.
template <typename real, int RB>
__device__ __forceinline__ void sweep_columns(const real* A, int lda, int nrow, int ncol,
                                              const real* x, real* red, real* out, bool add) {
  constexpr int VS = VecStride<real, RB>::value;
  constexpr int W = kSweepThreads / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int nb = 1;  // row blocks side by side: a power of two up to the warps
  while (nb < W && nb * 32 < nrow) nb *= 2;
  const int P = W / nb, part = warp / nb;
  for (int i0 = 0; i0 < nrow; i0 += 32 * nb) {
    const int i = i0 + (warp % nb) * 32 + lane;
    real acc[RB];
#pragma unroll
    for (int r = 0; r < RB; r++) acc[r] = 0;
    if (i < nrow) {
      const real* Ai = A + i;
      constexpr int kUnroll = RB >= 32 ? 2 : 4;
      int c = part;
      for (; c + P * (kUnroll - 1) < ncol; c += P * kUnroll) {
        real a[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; u++) a[u] = Ai[(c + u * P) * lda];
#pragma unroll
        for (int u = 0; u < kUnroll; u++) {
          real v[RB];
          load_vec<real, RB>(x + (c + u * P) * VS, v);
#pragma unroll
          for (int r = 0; r < RB; r++) acc[r] += a[u] * v[r];
        }
      }
      for (; c < ncol; c += P) {
        const real a = Ai[c * lda];
        real v[RB];
        load_vec<real, RB>(x + c * VS, v);
#pragma unroll
        for (int r = 0; r < RB; r++) acc[r] += a * v[r];
      }
    }
    real* mine = red + (part * nb * 32 + (warp % nb) * 32 + lane) * VS;
#pragma unroll
    for (int r = 0; r < RB; r++) mine[r] = acc[r];
    __syncthreads();
    const int nr = min(32 * nb, nrow - i0);
    for (int e = threadIdx.x; e < nr * RB; e += kSweepThreads) {
      const int q = e / RB, r = e % RB;
      real s = add ? out[(i0 + q) * VS + r] : real(0);
      for (int p = 0; p < P; p++) s += red[(p * nb * 32 + q) * VS + r];
      out[(i0 + q) * VS + r] = s;
    }
    __syncthreads();
  }
}

// Tile extents of a class's launch: TS rows (of T') and CS neighbour columns
// staged at a time.
struct SweepTiles {
  int maxm, TS, CS;
};

// Shared memory of one CTA, in elements of `real` (then CS ints).
template <typename real, int RB>
struct SweepSmem {
  int v0, v1, out, red, T, B, total;
  __host__ __device__ SweepSmem(const SweepTiles& t, bool fwd) {
    constexpr int VS = VecStride<real, RB>::value;
    const auto al = [](int n) { return (n + 3) / 4 * 4; };
    // columns of a smaller cluster may be spread wider than the largest's
    const int ldc = t.maxm + 31, unit = 16 / (int)sizeof(real);
    v0 = 0;
    v1 = v0 + al(t.maxm * VS);
    out = v1 + al(t.maxm * VS);
    red = out + al((t.CS > t.TS ? t.CS : t.TS) * VS);
    T = red + (fwd ? 0 : al((t.maxm > 256 ? (t.maxm + 31) / 32 * 32 : 256) * VS));
    B = T + al(fwd ? t.TS * sweep_ld(t.maxm) : t.TS * ldc + 2 * unit);
    total = B + al(t.CS * ldc + 2 * unit);
  }
  __host__ __device__ size_t bytes(const SweepTiles& t) const {
    return sizeof(real) * (size_t)total + sizeof(int) * (size_t)t.CS;
  }
};

// The forward step of a class.  A link of the chain is the wait for the class
// before, the vector loads, the T' product, the exchange and the B_L product:
// 3.8 us for classes of a few clusters (float32, one right-hand side), where
// two dependent launches took about 20; large classes are bound by staging
// their operators (22 us for 202 clusters of 128 unknowns, 66 MB).
template <typename real, int RB>
__global__ void __launch_bounds__(kSweepThreads)
fwd_sweep_kernel(const ApplyRec* __restrict__ recs, const int* __restrict__ ids,
                 const real* __restrict__ fac, const int64_t* __restrict__ vmap, real* y,
                 int64_t ldy, int nrhs, SweepTiles t) {
  constexpr int VS = VecStride<real, RB>::value;
  extern __shared__ __align__(16) unsigned char sweep_smem[];
  pdl_launch();
  cg::cluster_group cl = cg::this_cluster();
  const int CL = (int)cl.num_blocks(), cr = (int)cl.block_rank();
  const ApplyRec rc = recs[ids[blockIdx.y]];
  const int m = rc.m, k = rc.k, f = m - k, nw = rc.nw;
  if (k == m) {  // untouched cluster (all CTAs of it leave)
    pdl_wait();
    return;
  }
  const SweepSmem<real, RB> L(t, true);
  real* sm = reinterpret_cast<real*>(sweep_smem);
  real* ys = sm + L.v0;
  real* zs = sm + L.v1;
  real* yn = sm + L.out;
  real* sT = sm + L.T;
  real* sB = sm + L.B;
  int* vmi = reinterpret_cast<int*>(sm + L.total);
  const int mr = (m + CL - 1) / CL, i0 = min(m, cr * mr), i1 = min(m, i0 + mr);
  const int cw = (nw + CL - 1) / CL, c0 = min(nw, cr * cw), c1 = min(nw, c0 + cw);
  const int ldT = sweep_ld(m), ldB = column_ld<real>(m);
  const real* T = fac + rc.T;
  const real* BL = fac + (rc.sym ? rc.Y : rc.XT);  // column c, rows k..: B_L[c, :]
  const int64_t* vm = vmap + rc.map;
  const int r0 = blockIdx.z * RB, nr = min(RB, nrhs - r0);
  // operators of the first tiles and the neighbour slots: no sweep writes them
  int it = i0, tn = min(t.TS, i1 - i0);
  stage_rows<real>(sT, ldT, T + it, m, tn, m);
  cp_async_commit();
  int ct = c0, cn = min(t.CS, c1 - c0);
  const real* cB = stage_columns<real>(sB, BL + (int64_t)ct * m, m, cn);
  cp_async_commit();
  for (int c = threadIdx.x; c < cn; c += kSweepThreads) vmi[c] = (int)vm[ct + c];
  cl.sync();  // every CTA of the cluster runs before its memory is written
  pdl_wait();
  auto load_yn = [&] {
    load_block<real, RB>(yn, y, ldy, r0, nr, cn, [&](int c) { return (int64_t)vmi[c]; });
  };
  load_block<real, RB>(ys, y, ldy, r0, nr, m, [&](int l) { return rc.voff + l; });
  load_yn();
  cp_async_wait<1>();
  __syncthreads();
  while (true) {
    sweep_dots<real, RB>(sT, ldT, tn, m, ys,
                         [&](int o, int r, real v) { zs[(it + o) * VS + r] = v; });
    it += tn;
    if (it >= i1) break;
    __syncthreads();
    tn = min(t.TS, i1 - it);
    stage_rows<real>(sT, ldT, T + it, m, tn, m);
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
  }
  cp_async_wait<0>();
  __syncthreads();
  if (CL > 1) {
    // this CTA's z rows into every other CTA's z
    using U = Unit<real, RB>;
    const int n = (i1 - i0) * U::per;
    for (int e = threadIdx.x; e < n * CL; e += kSweepThreads) {
      const int q = e / n, u = e - q * n;
      const int at = (i0 + u / U::per) * VS + (u % U::per) * U::n;
      if (q == cr) continue;
      U x;
      x.load(zs + at);
      x.store(cl.map_shared_rank(zs, q) + at);
    }
    cl.sync();
  }
  // y_s = z_s: every CTA of the cluster has read y_s by now
  store_block<real, RB>(y, zs + i0 * VS, ldy, r0, nr, i1 - i0,
                        [&](int l) { return rc.voff + i0 + l; });
  // y_N -= B_L z_f over this CTA's columns
  while (ct < c1) {
    sweep_dots<real, RB>(cB + k, ldB, cn, f, zs + k * VS,
                         [&](int o, int r, real v) { yn[o * VS + r] -= v; });
    __syncthreads();
    store_block<real, RB>(y, yn, ldy, r0, nr, cn, [&](int c) { return (int64_t)vmi[c]; });
    ct += cn;
    if (ct >= c1) break;
    __syncthreads();
    cn = min(t.CS, c1 - ct);
    cB = stage_columns<real>(sB, BL + (int64_t)ct * m, m, cn);
    cp_async_commit();
    for (int c = threadIdx.x; c < cn; c += kSweepThreads) vmi[c] = (int)vm[ct + c];
    __syncthreads();
    load_yn();
    cp_async_wait<0>();
    __syncthreads();
  }
}

// The backward step of a class: each CTA multiplies its columns of B_R, the
// partial sums are added through distributed shared memory, each CTA then
// writes a share of the rows (5-6 us per link for small classes).
template <typename real, int RB>
__global__ void __launch_bounds__(kSweepThreads)
bwd_sweep_kernel(const ApplyRec* __restrict__ recs, const int* __restrict__ ids,
                 const real* __restrict__ fac, const int64_t* __restrict__ vmap, real* y,
                 int64_t ldy, int nrhs, SweepTiles t) {
  constexpr int VS = VecStride<real, RB>::value;
  extern __shared__ __align__(16) unsigned char sweep_smem[];
  pdl_launch();
  cg::cluster_group cl = cg::this_cluster();
  const int CL = (int)cl.num_blocks(), cr = (int)cl.block_rank();
  const ApplyRec rc = recs[ids[blockIdx.y]];
  const int m = rc.m, k = rc.k, f = m - k, nw = rc.nw;
  if (k == m) {
    pdl_wait();
    return;
  }
  const SweepSmem<real, RB> L(t, false);
  real* sm = reinterpret_cast<real*>(sweep_smem);
  real* xs = sm + L.v0;   // x_s, then z_s
  real* ps = sm + L.v1;   // this CTA's partial sums of B_R x_N (f rows)
  real* xn = sm + L.out;  // x_N of the staged columns, then the output rows
  real* sT = sm + L.T;
  real* sB = sm + L.B;
  int* vmi = reinterpret_cast<int*>(sm + L.total);
  const int mr = (m + CL - 1) / CL, i0 = min(m, cr * mr), i1 = min(m, i0 + mr);
  const int cw = (nw + CL - 1) / CL, c0 = min(nw, cr * cw), c1 = min(nw, c0 + cw);
  const int ldc = column_ld<real>(m);
  const real* TRt = fac + (rc.sym ? rc.T : rc.TR);
  const real* BR = fac + rc.Y;  // rows k..
  const int64_t* vm = vmap + rc.map;
  const int r0 = blockIdx.z * RB, nr = min(RB, nrhs - r0);
  int ct = c0, cn = min(t.CS, c1 - c0);
  const real* cB = stage_columns<real>(sB, BR + (int64_t)ct * m, m, cn);
  cp_async_commit();
  int it = i0, tn = min(t.TS, i1 - i0);
  const real* cT = stage_columns<real>(sT, TRt + (int64_t)it * m, m, tn);
  cp_async_commit();
  for (int c = threadIdx.x; c < cn; c += kSweepThreads) vmi[c] = (int)vm[ct + c];
  __syncthreads();
  pdl_wait();
  auto load_xn = [&] {
    load_block<real, RB>(xn, y, ldy, r0, nr, cn, [&](int c) { return (int64_t)vmi[c]; });
  };
  load_xn();
  load_block<real, RB>(xs, y, ldy, r0, nr, m, [&](int l) { return rc.voff + l; });
  if (cn == 0)  // no columns here
    for (int e = threadIdx.x; e < f * VS; e += kSweepThreads) ps[e] = 0;
  cp_async_wait<1>();
  __syncthreads();
  while (ct < c1) {
    sweep_columns<real, RB>(cB + k, ldc, f, cn, xn, sm + L.red, ps, ct > c0);
    ct += cn;
    if (ct >= c1) break;
    cn = min(t.CS, c1 - ct);
    cB = stage_columns<real>(sB, BR + (int64_t)ct * m, m, cn);
    cp_async_commit();
    for (int c = threadIdx.x; c < cn; c += kSweepThreads) vmi[c] = (int)vm[ct + c];
    __syncthreads();
    load_xn();
    cp_async_wait<0>();
    __syncthreads();
  }
  cp_async_wait<0>();
  cl.sync();
  // z_f = x_f - the CTAs' partial sums in rank order: each CTA adds up a
  // share of the rows and hands them to the others
  {
    using U = Unit<real, RB>;
    const int fr = (f + CL - 1) / CL, f0 = min(f, cr * fr), n = (min(f, f0 + fr) - f0) * U::per;
    for (int e = threadIdx.x; e < n; e += kSweepThreads) {
      const int at = (f0 + e / U::per) * VS + (e % U::per) * U::n;
      U p[kSweepMaxCl];
#pragma unroll
      for (int q = 0; q < kSweepMaxCl; q++)
        if (q < CL) p[q].load(cl.map_shared_rank(ps, q) + at);
      U z;
      z.load(xs + k * VS + at);
#pragma unroll
      for (int w = 0; w < U::n; w++) {
        real s = p[0].v[w];
#pragma unroll
        for (int q = 1; q < kSweepMaxCl; q++)
          if (q < CL) s += p[q].v[w];
        z.v[w] -= s;
      }
#pragma unroll
      for (int q = 0; q < kSweepMaxCl; q++)
        if (q < CL) z.store(cl.map_shared_rank(xs, q) + k * VS + at);
    }
  }
  cl.sync();
  while (it < i1) {
    sweep_dots<real, RB>(cT, ldc, tn, m, xs, [&](int o, int r, real v) { xn[o * VS + r] = v; });
    __syncthreads();
    store_block<real, RB>(y, xn, ldy, r0, nr, tn, [&](int l) { return rc.voff + it + l; });
    it += tn;
    if (it >= i1) break;
    __syncthreads();
    tn = min(t.TS, i1 - it);
    cT = stage_columns<real>(sT, TRt + (int64_t)it * m, m, tn);
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// The dense top: z = T' y and y = T_R'^T z with T' and T_R'^T n x n, read
// once from HBM (lower triangular but for the permuted columns of a general
// T': tri).  A thread-block cluster of CL CTAs shares 64 rows (forward)
// or 32 columns (backward), each CTA a stretch of the other index, and adds
// the CTAs' sums through distributed shared memory: 93 x 8 and 185 x 8 CTAs
// for 5,909 unknowns keep enough loads in flight for the HBM rate, which one
// CTA per 64 rows (93 CTAs, four loads each) did not.
// ---------------------------------------------------------------------------
constexpr int kTopRows = 64, kTopCols = 32, kTopChunk = 256;

template <typename real, int RB, int CL>
__global__ void __launch_bounds__(kSweepThreads)
fwd_top_kernel(const ApplyRec* __restrict__ recs, const int* __restrict__ ids,
               const real* __restrict__ fac, const real* y, real* z, int64_t ldy, int nrhs,
               int tri) {
  __shared__ __align__(16) real ys[kTopChunk * RB];
  __shared__ real red[kTopRows * RB];
  pdl_launch();
  cg::cluster_group cl = cg::this_cluster();
  const int cr = (int)cl.block_rank();
  const ApplyRec rc = recs[ids[0]];
  const int n = rc.m;
  // the longest rows first
  const int i0 = ((int)gridDim.y - 1 - (int)blockIdx.y) * kTopRows;
  const int r0 = blockIdx.z * RB, nr = min(RB, nrhs - r0);
  const int cols = tri ? min(n, i0 + kTopRows) : n;
  const int per = (cols + CL - 1) / CL;
  const int l0 = min(cols, cr * per), l1 = min(cols, l0 + per);
  const int ii = threadIdx.x % kTopRows, part = threadIdx.x / kTopRows;
  const int i = min(i0 + ii, n - 1);
  const real* T = fac + rc.T + i;
  pdl_wait();
  real acc[RB];
#pragma unroll
  for (int r = 0; r < RB; r++) acc[r] = 0;
  for (int lc = l0; lc < l1; lc += kTopChunk) {
    const int nl = min(kTopChunk, l1 - lc);
    __syncthreads();
    for (int r = 0; r < RB; r++)
      for (int l = threadIdx.x; l < nl; l += kSweepThreads)
        ys[l * RB + r] = r < nr ? y[rc.voff + lc + l + (int64_t)(r0 + r) * ldy] : real(0);
    __syncthreads();
    int l = part;
    for (; l + 28 < nl; l += 32) {  // eight loads in flight per thread
      real a[8];
#pragma unroll
      for (int u = 0; u < 8; u++) a[u] = __ldg(T + (int64_t)(lc + l + 4 * u) * n);
#pragma unroll
      for (int u = 0; u < 8; u++)
#pragma unroll
        for (int r = 0; r < RB; r++) acc[r] += a[u] * ys[(l + 4 * u) * RB + r];
    }
    for (; l < nl; l += 4) {
      const real a = __ldg(T + (int64_t)(lc + l) * n);
#pragma unroll
      for (int r = 0; r < RB; r++) acc[r] += a * ys[l * RB + r];
    }
  }
  // the four parts of this CTA in turn, then the CTAs in rank order
  for (int q = 0; q < 4; q++) {
    if (part == q)
#pragma unroll
      for (int r = 0; r < RB; r++) red[r * kTopRows + ii] = q == 0 ? acc[r] : red[r * kTopRows + ii] + acc[r];
    __syncthreads();
  }
  cl.sync();
  for (int e = cr * kSweepThreads + threadIdx.x; e < kTopRows * nr; e += CL * kSweepThreads) {
    const int a = e % kTopRows;
    real s = 0;
#pragma unroll
    for (int q = 0; q < CL; q++) s += cl.map_shared_rank(red, q)[e];
    if (i0 + a < n) z[rc.voff + i0 + a + (int64_t)(r0 + e / kTopRows) * ldy] = s;
  }
  cl.sync();
}

template <typename real, int RB, int CL>
__global__ void __launch_bounds__(kSweepThreads)
bwd_top_kernel(const ApplyRec* __restrict__ recs, const int* __restrict__ ids,
               const real* __restrict__ fac, real* y, const real* z, int64_t ldy, int nrhs) {
  constexpr int kPer = kTopCols / (kSweepThreads / 32);  // columns per warp
  __shared__ real zs[RB * kTopChunk];
  __shared__ real red[kTopCols * RB];
  pdl_launch();
  cg::cluster_group cl = cg::this_cluster();
  const int cr = (int)cl.block_rank();
  const ApplyRec rc = recs[ids[0]];
  const int n = rc.m;
  const int i0 = blockIdx.y * kTopCols;
  const int r0 = blockIdx.z * RB, nr = min(RB, nrhs - r0);
  // rows i0.. only: T_R'^T is lower triangular
  const int rows = n - i0, per = (rows + CL - 1) / CL;
  const int l0 = min(n, i0 + cr * per), l1 = min(n, l0 + per);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const real* T = fac + (rc.sym ? rc.T : rc.TR);
  const real* col[kPer];
#pragma unroll
  for (int w = 0; w < kPer; w++) col[w] = T + (int64_t)min(i0 + warp * kPer + w, n - 1) * n;
  pdl_wait();
  real acc[kPer][RB];
#pragma unroll
  for (int w = 0; w < kPer; w++)
#pragma unroll
    for (int r = 0; r < RB; r++) acc[w][r] = 0;
  for (int lc = l0; lc < l1; lc += kTopChunk) {
    const int nl = min(kTopChunk, l1 - lc);
    __syncthreads();
    for (int r = 0; r < RB; r++)
      for (int l = threadIdx.x; l < kTopChunk; l += kSweepThreads)
        zs[r * kTopChunk + l] =
            (r < nr && l < nl) ? z[rc.voff + lc + l + (int64_t)(r0 + r) * ldy] : real(0);
    __syncthreads();
    for (int l = lane; l < nl; l += 64) {
      const bool two = l + 32 < nl;
      real a[2][kPer];
#pragma unroll
      for (int w = 0; w < kPer; w++) {
        a[0][w] = __ldg(col[w] + lc + l);
        a[1][w] = two ? __ldg(col[w] + lc + l + 32) : real(0);
      }
#pragma unroll
      for (int h = 0; h < 2; h++)
#pragma unroll
        for (int r = 0; r < RB; r++) {
          // (a second index past the chunk's end multiplies a zero operator)
          const real x = zs[r * kTopChunk + min(l + 32 * h, kTopChunk - 1)];
#pragma unroll
          for (int w = 0; w < kPer; w++) acc[w][r] += a[h][w] * x;
        }
    }
  }
#pragma unroll
  for (int w = 0; w < kPer; w++)
#pragma unroll
    for (int r = 0; r < RB; r++) {
      real v = acc[w][r];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) red[r * kTopCols + warp * kPer + w] = v;
    }
  cl.sync();
  for (int e = cr * kSweepThreads + threadIdx.x; e < kTopCols * nr; e += CL * kSweepThreads) {
    const int a = e % kTopCols;
    real s = 0;
#pragma unroll
    for (int q = 0; q < CL; q++) s += cl.map_shared_rank(red, q)[e];
    if (i0 + a < n) y[rc.voff + i0 + a + (int64_t)(r0 + e / kTopCols) * ldy] = s;
  }
  cl.sync();
}

// Right-hand sides per CTA: rbmax, fewer when rbmax slot vectors of maxm
// entries would exceed 160 KB of shared memory (the dense top's long
// vectors).
template <typename real>
int group_size(int maxm, int rbmax) {
  const size_t per = sizeof(real) * (size_t)std::max(maxm, 1);
  return (int)std::max<size_t>(1, std::min<size_t>(rbmax, (160u * 1024u) / per));
}

// The dynamic shared-memory limit of a kernel is raised once, to a ceiling
// above every request (at most 160 KB of slot vectors) plus its static arrays,
// and never lowered: a CUDA graph captured earlier may hold a launch of the
// same kernel with a larger request than the current one.
constexpr int kSmemCeiling = 192 * 1024;
template <auto Kernel>
void set_smem() {
  static const bool once = [] {
    cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCeiling);
    return true;
  }();
  (void)once;
}

template <typename real, int RB>
void launch_fwd(const ApplyRec* recs, const int* ids, int nids, int maxm, int maxnw,
                const real* fac, const int64_t* vmap, real* y, real* z, int64_t ldy, int nrhs,
                cudaStream_t st) {
  const int rb = group_size<real>(maxm, RB);
  const int nz = (nrhs + rb - 1) / rb;
  const size_t sm = sizeof(real) * (size_t)rb * std::max(maxm, 1);
  set_smem<fwd_t_kernel<real, RB>>();
  dim3 g1((maxm + kRows - 1) / kRows, nids, nz);
  count_launch();
  fwd_t_kernel<real, RB><<<g1, 256, sm, st>>>(recs, ids, fac, y, z, ldy, nrhs, rb);
  dim3 g2(std::max(1, (maxnw + kCols - 1) / kCols), nids, nz);
  set_smem<fwd_nbr_kernel<real, RB>>();
  count_launch();
  fwd_nbr_kernel<real, RB><<<g2, 256, sm, st>>>(recs, ids, fac, vmap, y, z, ldy, nrhs, rb);
}

template <typename real, int RB>
void launch_bwd(const ApplyRec* recs, const int* ids, int nids, int maxm, int maxnw,
                const real* fac, const int64_t* vmap, real* y, real* z, real* part, int64_t ldy,
                int nrhs, cudaStream_t st) {
  const int rb = group_size<real>(maxm, RB);
  const int nz = (nrhs + rb - 1) / rb;
  if (maxnw > 0) {
    dim3 g1((maxnw + kCols - 1) / kCols, nids, nz);
    count_launch();
    bwd_part_kernel<real, RB><<<g1, 256, 0, st>>>(recs, ids, fac, vmap, y, part, ldy, nrhs, rb);
  }
  count_launch();
  bwd_z_kernel<real, RB><<<dim3(nids, 1, nz), 256, 0, st>>>(recs, ids, y, z, part, ldy, nrhs,
                                                             rb);
  const size_t sm = sizeof(real) * (size_t)rb * std::max(maxm, 1);
  set_smem<bwd_t_kernel<real, RB>>();
  dim3 g3((maxm + kRows - 1) / kRows, nids, nz);
  count_launch();
  bwd_t_kernel<real, RB><<<g3, 256, sm, st>>>(recs, ids, fac, y, z, ldy, nrhs, rb);
}

// A launch over thread-block clusters of CL CTAs that may start before the
// kernel ahead of it has completed.
template <typename... KArgs, typename... Args>
void launch_pdl(void (*kernel)(KArgs...), dim3 grid, int CL, size_t smem, cudaStream_t st,
                Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kSweepThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = CL;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  count_launch();
  cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

struct SweepShape {
  int CL = 0;  // CTAs per cluster; 0: the fused kernels cannot take the class
  size_t smem = 0;
  SweepTiles t{};
};

// Split of a class over the chip.  More CTAs per cluster shorten a link (each
// stages and multiplies a smaller slice) until the class fills the chip about
// twice over, and let a slice be staged in one piece of at most kShare (two
// CTAs per SM).  One application, CTAs wanted / share: 2 / 104 KB takes 2.08
// ms at 64^3 (float32, 1 right-hand side), 15.2 ms at 96^3 (8) and 7.2 ms at
// 512^2 (124); 4 / 56 KB took 2.03, 16.0 and 11.8 ms, 4 / 150 KB 2.35, 16.0
// and 7.7 ms, all with one output per lane group in the products (several: 1.95,
// 14.2 and 6.95 ms).  The four-launch form took 6.4, 34.2 and 18.8 ms.
constexpr size_t kShare = 104 * 1024;
template <typename real, int RB>
SweepShape sweep_shape(bool fwd, int nids, int maxm, int maxnw, int nrhs) {
  SweepShape s;
  const int64_t cl0 = (int64_t)nids * ((nrhs + RB - 1) / RB);
  SweepTiles t{};
  const auto bytes = [&] { return SweepSmem<real, RB>(t, fwd).bytes(t); };
  const auto tiles = [&](int CL) {
    t.maxm = maxm;
    t.TS = std::max(1, (maxm + CL - 1) / CL);
    t.CS = std::max(1, (maxnw + CL - 1) / CL);
  };
  int CL = 1;
  tiles(1);
  while (CL < kSweepMaxCl && std::max(maxnw, maxm) >= CL * 2 * 8 &&
         (cl0 * CL * 2 <= 152 * 2 || bytes() > kShare)) {
    CL *= 2;
    tiles(CL);
  }
  // shared memory: all of an SM's for a class that leaves SMs idle, else a
  // share that keeps several CTAs resident
  const int64_t ctas = cl0 * CL;
  const size_t cap = ctas <= 152 ? 190 * 1024 : kShare;
  const auto halve = [](int v) { return std::max(1, (v + 1) / 2); };
  while (bytes() > cap && (t.TS > 32 || t.CS > 32)) {
    if (t.CS > 32 && (t.CS >= t.TS || t.TS <= 32)) t.CS = std::max(32, halve(t.CS));
    else t.TS = std::max(32, halve(t.TS));
  }
  if (bytes() > kSmemCeiling) return s;
  s.CL = CL;
  s.smem = bytes();
  s.t = t;
  return s;
}

// The right-hand sides a CTA takes: groups of 1, 4, 8 or (float32) 32.  Each
// operator element read from shared memory serves the whole group; a wider
// group than there are right-hand sides multiplies zeros, which the float64
// pipe cannot afford.  A class of few clusters takes the smallest group whose
// CTAs still run at once (kAtOnce): its SMs would be idle otherwise, and a
// narrower group is a shorter link (29 x 37 x 23, float64, 3 right-hand sides:
// 3.2 ms per application against 5.8 with the group chosen by the count alone;
// 64^3 with 32: 6.2 against 7.1; twice as many CTAs: 96^3 with 8 gains
// nothing, 64^3 with 32 loses 0.4 ms).
constexpr int kAtOnce = 2 * 152;
template <typename real, int RB>
bool try_sweep(bool fwd, const ApplyRec* recs, const int* ids, int nids, int maxm, int maxnw,
               const real* fac, const int64_t* vmap, real* y, int64_t ldy, int nrhs,
               cudaStream_t st) {
  const SweepShape s = sweep_shape<real, RB>(fwd, nids, maxm, maxnw, nrhs);
  if (s.CL == 0) return false;
  const dim3 grid(s.CL, nids, (nrhs + RB - 1) / RB);
  if (fwd) {
    set_smem<fwd_sweep_kernel<real, RB>>();
    launch_pdl(fwd_sweep_kernel<real, RB>, grid, s.CL, s.smem, st, recs, ids, fac, vmap, y, ldy,
               nrhs, s.t);
  } else {
    set_smem<bwd_sweep_kernel<real, RB>>();
    launch_pdl(bwd_sweep_kernel<real, RB>, grid, s.CL, s.smem, st, recs, ids, fac, vmap, y, ldy,
               nrhs, s.t);
  }
  return true;
}

// Large clusters with many right-hand sides take the unfused kernels: a link's
// latency no longer counts, and each group of right-hand sides stages the class's
// operators anew and multiplies by slices of T' that leave lanes idle.  One
// application with 128 right-hand sides, fused -> these clusters unfused:
// float64, clusters of 183 (36^3) 40.3 -> 35.9 ms, 160 equal, 144 22.2 -> 22.9; float32
// (whose fused groups of 32 end at 256 unknowns) 350 (150 x 148) 3.76 -> 2.44, 264
// (33 x 32^2) 6.23 -> 4.93, 256 equal, 184 5.54 -> 5.86.  With 64: 183 21.9 -> 20.7, 256
// (float64) 4.67 -> 4.86, 264 3.62 -> 3.64; with 32 the fused ones win throughout.
constexpr int kManyRhs = 64, kWideF64 = 160, kWideF32 = 256;

template <typename real>
bool sweep_class(bool fwd, const ApplyRec* recs, const int* ids, int nids, int maxm, int maxnw,
                 const real* fac, const int64_t* vmap, real* y, int64_t ldy, int nrhs,
                 cudaStream_t st) {
  if (nids > 65535 || nrhs > 65535) return false;
  if (nrhs > kManyRhs && maxm > (sizeof(real) == 8 ? kWideF64 : kWideF32)) return false;
  const auto fits = [&](int rb) {
    return (int64_t)nids * kSweepMaxCl * ((nrhs + rb - 1) / rb) <= kAtOnce;
  };
  const auto go = [&](auto rb) {
    return try_sweep<real, decltype(rb)::value>(fwd, recs, ids, nids, maxm, maxnw, fac, vmap, y,
                                                ldy, nrhs, st);
  };
  if (nrhs == 1 || fits(1)) return go(std::integral_constant<int, 1>{});
  if (nrhs <= 4 || fits(4)) return go(std::integral_constant<int, 4>{});
  if constexpr (sizeof(real) == 4)
    if (nrhs > 16 && maxm <= 256 && !fits(8) && go(std::integral_constant<int, 32>{})) return true;
  return go(std::integral_constant<int, 8>{});
}

// CTAs per cluster of a top of n unknowns whose launch has `tiles` clusters: 8,
// fewer when the chip stays full without them and a CTA's stretch would be
// shorter than a staged chunk, as in a small top with many right-hand sides: its
// start and the exchange then cost more than its products (float64, one
// application with 256 right-hand sides, 8 CTAs -> the rule: 400 unknowns 0.52 ->
// 0.29 ms, 1,000 1.42 -> 0.83).
int top_ctas(int n, int64_t tiles) {
  int CL = kSweepMaxCl;
  while (CL > 2 && n < CL * kTopChunk && tiles * CL / 2 >= kAtOnce) CL /= 2;
  return CL;
}

template <typename real, int RB>
void launch_top(bool fwd, const ApplyRec* recs, const int* ids, int n, bool sym, const real* fac,
                real* y, real* z, int64_t ldy, int nrhs, cudaStream_t st) {
  const int nz = (nrhs + RB - 1) / RB, per = fwd ? kTopRows : kTopCols, nt = (n + per - 1) / per;
  const auto go = [&](auto cl) {
    constexpr int CL = decltype(cl)::value;
    const dim3 grid(CL, nt, nz);
    if (fwd)
      launch_pdl(fwd_top_kernel<real, RB, CL>, grid, CL, 0, st, recs, ids, fac, y, z, ldy, nrhs,
                 sym ? 1 : 0);
    else
      launch_pdl(bwd_top_kernel<real, RB, CL>, grid, CL, 0, st, recs, ids, fac, y, z, ldy, nrhs);
  };
  if constexpr (RB >= 8) {  // (fewer right-hand sides leave too few tiles)
    const int CL = top_ctas(n, (int64_t)nt * nz);
    if (CL == 2) return go(std::integral_constant<int, 2>{});
    if (CL == 4) return go(std::integral_constant<int, 4>{});
  }
  go(std::integral_constant<int, kSweepMaxCl>{});
}

}  // namespace

template <typename real>
int Launch<real>::apply_max_m() {
  return (int)(kSmemCeiling / sizeof(real));
}

template <typename real>
void Launch<real>::apply_fwd(const ApplyRec* recs, const int* ids, int nids, int maxm, int maxnw,
                             const real* fac, const int64_t* vmap, real* y, real* z, int64_t ldy,
                             int nrhs, cudaStream_t st) {
  if (nids <= 0) return;
  if (sweep_class<real>(true, recs, ids, nids, maxm, maxnw, fac, vmap, y, ldy, nrhs, st)) return;
  if (nrhs == 1)
    launch_fwd<real, 1>(recs, ids, nids, maxm, maxnw, fac, vmap, y, z, ldy, nrhs, st);
  else
    launch_fwd<real, kRbWide>(recs, ids, nids, maxm, maxnw, fac, vmap, y, z, ldy, nrhs, st);
}

template <typename real>
void Launch<real>::apply_bwd(const ApplyRec* recs, const int* ids, int nids, int maxm, int maxnw,
                             const real* fac, const int64_t* vmap, real* y, real* z, real* part,
                             int64_t ldy, int nrhs, cudaStream_t st) {
  if (nids <= 0) return;
  if (sweep_class<real>(false, recs, ids, nids, maxm, maxnw, fac, vmap, y, ldy, nrhs, st)) return;
  if (nrhs == 1)
    launch_bwd<real, 1>(recs, ids, nids, maxm, maxnw, fac, vmap, y, z, part, ldy, nrhs, st);
  else
    launch_bwd<real, kRbWide>(recs, ids, nids, maxm, maxnw, fac, vmap, y, z, part, ldy, nrhs,
                              st);
}

template <typename real>
void Launch<real>::apply_top(const ApplyRec* recs, const int* ids, int n, bool sym,
                             const real* fac, real* y, real* z, int64_t ldy, int nrhs,
                             cudaStream_t st) {
  for (int pass = 0; pass < 2; pass++) {
    if (nrhs == 1)
      launch_top<real, 1>(pass == 0, recs, ids, n, sym, fac, y, z, ldy, nrhs, st);
    else if (nrhs <= 4)
      launch_top<real, 4>(pass == 0, recs, ids, n, sym, fac, y, z, ldy, nrhs, st);
    else
      launch_top<real, 8>(pass == 0, recs, ids, n, sym, fac, y, z, ldy, nrhs, st);
  }
}

template struct Launch<double>;
template struct Launch<float>;

}  // namespace hs
