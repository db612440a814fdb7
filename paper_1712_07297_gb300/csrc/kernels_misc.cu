// Batched products, scatters and the substitution sweeps.
//
// gemm_gather  C = A * Bg for every cluster of a colour class, where the
//              columns of Bg are gathered from the cluster's blocks (the
//              neighbour coupling A_sN for Eq. scaling's coarse rows and the
//              fine-elimination factor; the fill blocks A_sw for the
//              coarse-to-far coupling C Z).
// schur        A_nn -= B_L B_R (Eq. elim): the product of a cluster's two
//              factor panels, written straight into the neighbour blocks
//              through a row/column map (clusters of a colour touch disjoint
//              blocks, so no atomics).
// scatter      coarse rows/columns of a processed cluster into its blocks.
// float64 Krylov helpers: CSR SpMV, deterministic dot products, axpy forms.
#include <algorithm>
#include <atomic>
#include <cmath>

#include "common.h"

namespace hs {

static std::atomic<int64_t> g_launches{0};
int64_t launches_total() { return g_launches.load(); }
std::mutex& device_mutex() {
  static std::mutex m;
  return m;
}
void count_launch(int n) { g_launches += n; }

namespace {

constexpr int TM = 64, TN = 64, TK = 16;
constexpr int kMaxGridYZ = 65535;  // grid y/z limit: larger task lists are split

template <typename real>
struct alignas(4 * sizeof(real) > 16 ? 16 : 4 * sizeof(real)) Quad {
  real v[4];
};
template <typename real>
struct alignas(2 * sizeof(real)) Pair {
  real v[2];
};

// One tile of gemm_gather: 16 S rows from i0, TN columns from j0.  The thread
// (tx, ty) has rows tx + 16 p and columns 4 ty + q.
template <typename real, int S, int KC>
__device__ __forceinline__ void gather_tile(const GemmTask& tk, const real* __restrict__ A,
                                            const real* __restrict__ Bbase, real* C, int M, int i0,
                                            int j0, const int64_t* cp, const int* cst, real* As,
                                            real* Bs) {
  constexpr int PB = TN + 4;
  const int N = tk.N, K = tk.K;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  real acc[S][4];
#pragma unroll
  for (int a = 0; a < S; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) acc[a][b] = 0;
  for (int l0 = 0; l0 < K; l0 += KC) {
    const int lc = min(KC, K - l0);
    // consecutive threads along rows of A, and along the gathered columns
#pragma unroll
    for (int h = 0; h < KC; h += 16) {
      if (h >= lc) break;
#pragma unroll
      for (int u = 0; u < S; u++) {
        const int i = tx + 16 * u, l = h + ty;
        As[l * TM + i] =
            (i0 + i < M && l < lc) ? A[i0 + i + (int64_t)(l0 + l) * tk.lda] : real(0);
      }
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const int j = ty + 16 * u, l = h + tx;
        Bs[l * PB + j] =
            (l < lc && j0 + j < N) ? Bbase[cp[j] + (int64_t)(l0 + l) * cst[j]] : real(0);
      }
    }
    __syncthreads();
#pragma unroll 8
    for (int l = 0; l < lc; l++) {
      real a[S];
#pragma unroll
      for (int p = 0; p < S; p++) a[p] = As[l * TM + tx + 16 * p];
      const Quad<real> b = *reinterpret_cast<const Quad<real>*>(Bs + l * PB + 4 * ty);
#pragma unroll
      for (int p = 0; p < S; p++)
#pragma unroll
        for (int q = 0; q < 4; q++) acc[p][q] += a[p] * b.v[q];
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < 4; q++)
#pragma unroll
    for (int p = 0; p < S; p++) {
      const int gi = i0 + tx + 16 * p, gj = j0 + 4 * ty + q;
      if (gi < M && gj < N) C[gi + (int64_t)gj * tk.ldc] = acc[p][q];
    }
}

// rows of A (M), inner K and skip rule from the rank of the cluster:
//   mode 0: M = task.M, K = task.K; skip when rank == m (untouched)
//   mode 1: M = rank; skip when rank == 0 or rank == m
//
// Bound: the FP64 pipe in float64, latency of short tiles in float32.  The rows
// go in equal tiles of a whole number of 16-row strips (S = 1 to 4), so a
// cluster of 130 unknowns computes 144 rows and not 192, and a rank of 20
// computes 32 and not 64; S is a template argument since a strip skipped inside
// the product loop costs more than it saves (fill products 73 ms against 65).
// Chunks of 32 and a vector read of the gathered operand as in the Schur
// update.  Both products per factorization, before -> now: float64 64^3 115 ->
// 77 ms, 96^3 40 -> 29, convection-diffusion 64^3 31 -> 23.
template <typename real>
__global__ void __launch_bounds__(256, sizeof(real) == 8 ? 2 : 5)
gemm_gather_kernel(const GemmTask* __restrict__ tasks, const real* __restrict__ Abase,
                   real* __restrict__ Cbase, const real* __restrict__ Bbase,
                   const Seg* __restrict__ segs, const int* __restrict__ rank) {
  const GemmTask tk = tasks[blockIdx.z];
  const int r = rank[tk.s];
  int M = tk.M;
  if (tk.mode == 0) {
    if (r == tk.K) return;
  } else {
    if (r == 0 || r == tk.K) return;
    M = r;
  }
  const int nt = (M + TM - 1) / TM, j0 = blockIdx.x * TN;
  if ((int)blockIdx.y >= nt || j0 >= tk.N) return;
  const int S = (M + 16 * nt - 1) / (16 * nt), i0 = blockIdx.y * 16 * S;
  if (i0 >= M) return;
  constexpr int KC = 32;
  __shared__ __align__(16) real As[KC * TM];
  __shared__ __align__(16) real Bs[KC * (TN + 4)];
  __shared__ int64_t cp[TN];
  __shared__ int cst[TN];
  // this tile's gathered columns: offset and stride, resolved once
  if (threadIdx.x < TN && j0 + threadIdx.x < tk.N)
    seg_col(segs + tk.bcol, tk.nseg, j0 + threadIdx.x, &cp[threadIdx.x], &cst[threadIdx.x]);
  __syncthreads();
  const real* A = Abase + tk.A;
  real* C = Cbase + tk.C;
  if (S == 4)
    gather_tile<real, 4, KC>(tk, A, Bbase, C, M, i0, j0, cp, cst, As, Bs);
  else if (S == 3)
    gather_tile<real, 3, KC>(tk, A, Bbase, C, M, i0, j0, cp, cst, As, Bs);
  else if (S == 2)
    gather_tile<real, 2, KC>(tk, A, Bbase, C, M, i0, j0, cp, cst, As, Bs);
  else
    gather_tile<real, 1, KC>(tk, A, Bbase, C, M, i0, j0, cp, cst, As, Bs);
}

// SplitMix64 output function (Steele, Lea, Flood 2014; Vigna's public
// domain reference implementation).
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Y (m x l) = G Omega: G's columns gathered through descriptors, Omega
// generated on the fly (Rademacher, +-1/sqrt(l)); the randomized variant of
// the compression of Eq. lra.  64 x 64 output tiles, inner chunks of 16
// gathered columns.
template <typename real>
__global__ void __launch_bounds__(256)
sketch_kernel(const SketchTask* __restrict__ tasks, const real* __restrict__ arena,
              real* __restrict__ ws, const Seg* __restrict__ segs) {
  const SketchTask tk = tasks[blockIdx.z];
  const int i0 = blockIdx.y * TM, j0 = blockIdx.x * TN;
  if (i0 >= tk.m || j0 >= tk.l) return;
  __shared__ real As[TK][TM + 1];
  __shared__ real Bs[TK][TN + 1];
  const real scale = real(1) / sqrt((real)tk.l);
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  real acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) acc[a][b] = 0;
  __shared__ int64_t cp[TK];
  __shared__ int cst[TK];
  for (int q0 = 0; q0 < tk.ncol; q0 += TK) {
    if (threadIdx.x < TK && q0 + threadIdx.x < tk.ncol)
      seg_col(segs + tk.gcol, tk.nseg, q0 + threadIdx.x, &cp[threadIdx.x], &cst[threadIdx.x]);
    __syncthreads();
    for (int e = threadIdx.x; e < TM * TK; e += 256) {
      int i = e % TM, l = e / TM;
      int gi = i0 + i, q = q0 + l;
      real v = 0;
      if (gi < tk.m && q < tk.ncol) v = arena[cp[l] + (int64_t)gi * cst[l]];
      As[l][i] = v;
    }
    for (int e = threadIdx.x; e < TK * TN; e += 256) {
      int l = e % TK, j = e / TK;
      int q = q0 + l, gj = j0 + j;
      real v = 0;
      if (q < tk.ncol && gj < tk.l) {
        uint64_t z = splitmix64(((uint64_t)q << 32) | (uint64_t)gj);
        v = (z >> 63) ? -scale : scale;
      }
      Bs[l][j] = v;
    }
    __syncthreads();
#pragma unroll
    for (int l = 0; l < TK; l++) {
      real a[4], b[4];
#pragma unroll
      for (int q = 0; q < 4; q++) {
        a[q] = As[l][ty + 16 * q];
        b[q] = Bs[l][tx + 16 * q];
      }
#pragma unroll
      for (int p = 0; p < 4; p++)
#pragma unroll
        for (int q = 0; q < 4; q++) acc[p][q] += a[p] * b[q];
    }
    __syncthreads();
  }
  real* Y = ws + tk.Y;
#pragma unroll
  for (int p = 0; p < 4; p++)
#pragma unroll
    for (int q = 0; q < 4; q++) {
      int gi = i0 + ty + 16 * p, gj = j0 + tx + 16 * q;
      if (gi < tk.m && gj < tk.l) Y[gi + (int64_t)gj * tk.m] = acc[p][q];
    }
}

// C_mapped[r, c] -= sum_i P[k+i, r] Q[k+i, c], i < f = m - rank.  For an
// SPD factorization (P = Q) the update is symmetric: only the tiles on or
// below the diagonal compute, and each writes its elements to both (r, c)
// and (c, r) -- bitwise the values the full product would give, since
// P[., r] Q[., c] and P[., c] Q[., r] are the same products summed in the
// same order.
//
// Bound: L1 and DRAM latency of short tiles (K = f is 20 to 130; at level 3 of
// 96^3 a CTA multiplies for 3,000 cycles and then updates 8,192 elements).  So
// the operands come in chunks of 32 (one or two round trips to L2 instead of
// four), the products read shared memory in vectors (three loads per 16 FMA
// instead of eight), and the update has eight loads in flight instead of a
// load and a store in turn; that costs registers (64, four CTAs per SM) and
// pays all the same: with one load in flight the kernel ran at 1.7 TB/s with
// six CTAs per SM.  Updates per factorization, before -> now: 96^3 138 -> 83
// ms, convection-diffusion 64^3 28 -> 18, float64 64^3 127 -> 111.  Fewer loads
// in flight: four 92, two 103; six CTAs per SM with eight: 96 (spills).
template <typename real>
__global__ void __launch_bounds__(256)
schur_kernel(const SchurTask* __restrict__ tasks, const real* __restrict__ fac,
             real* __restrict__ arena, const Seg* __restrict__ segs,
             const int64_t* __restrict__ base, const SchurNbr* __restrict__ nbr,
             const int* __restrict__ rank) {
  const SchurTask tk = tasks[blockIdx.z];
  const int k = rank[tk.s];
  const int f = tk.m - k;
  if (f <= 0) return;
  const int N = tk.nw;
  const int i0 = blockIdx.y * TM, j0 = blockIdx.x * TN;
  if (i0 >= N || j0 >= N) return;
  const bool sym = tk.P == tk.Q;
  if (sym && j0 > i0) return;
  // the operand tiles, then (after the products) the output tile Cs[j][i]
  constexpr int KC = 32, PA = TM + 4, PB = TN + 2;
  __shared__ __align__(16) real tile[KC * (PA + PB)];
  static_assert(TN * (TM + 1) <= KC * (PA + PB), "the output tile takes the operands' place");
  real* As = tile;
  real* Bs = tile + KC * PA;
  real(*Cs)[TM + 1] = reinterpret_cast<real(*)[TM + 1]>(tile);
  const real* P = fac + tk.P + k;
  const real* Q = fac + tk.Q + k;
  const int ld = tk.m;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  real acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) acc[a][b] = 0;
  for (int l0 = 0; l0 < f; l0 += KC) {
    const int lc = min(KC, f - l0);
#pragma unroll
    for (int h = 0; h < KC; h += 16) {
      if (h >= lc) break;
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const int l = h + tx, i = ty + 16 * u, gi = i0 + i, gj = j0 + i;
        const bool in = l < lc;
        As[l * PA + i] = (in && gi < N) ? P[l0 + l + (int64_t)gi * ld] : real(0);
        Bs[l * PB + i] = (in && gj < N) ? Q[l0 + l + (int64_t)gj * ld] : real(0);
      }
    }
    __syncthreads();
#pragma unroll 8
    for (int l = 0; l < lc; l++) {
      real a[4], b[4];
      const Quad<real> qa = *reinterpret_cast<const Quad<real>*>(As + l * PA + 4 * ty);
#pragma unroll
      for (int q = 0; q < 4; q++) a[q] = qa.v[q];
#pragma unroll
      for (int q = 0; q < 2; q++) {
        const Pair<real> pb = *reinterpret_cast<const Pair<real>*>(Bs + l * PB + 32 * q + 2 * tx);
        b[2 * q] = pb.v[0];
        b[2 * q + 1] = pb.v[1];
      }
#pragma unroll
      for (int p = 0; p < 4; p++)
#pragma unroll
        for (int q = 0; q < 4; q++) acc[p][q] += a[p] * b[q];
    }
    __syncthreads();
  }
  // neighbour (run) and local index of every row/column of the tile: the
  // runs of a cluster's neighbour columns, one per neighbour
  __shared__ int rblk[TM], rloc[TM], cblk[TN], cloc[TN];
  const Seg* sg = segs + tk.map;
  for (int e = threadIdx.x; e < TM + TN; e += blockDim.x) {
    const int r = (e < TM) ? i0 + e : j0 + (e - TM);
    int a = 0, lr = 0;
    if (r < N) {
      int lo = 0, hi = tk.nb - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (sg[mid].colstart <= r) lo = mid;
        else hi = mid - 1;
      }
      a = lo;
      lr = r - sg[lo].colstart;
    }
    if (e < TM) {
      rblk[e] = a;
      rloc[e] = lr;
    } else {
      cblk[e - TM] = a;
      cloc[e - TM] = lr;
    }
  }
#pragma unroll
  for (int p = 0; p < 4; p++)
#pragma unroll
    for (int q = 0; q < 4; q++)
      Cs[32 * (q / 2) + 2 * tx + q % 2][4 * ty + p] = acc[p][q];
  __syncthreads();
  // read-modify-write of the target blocks from the staged tile, consecutive
  // threads on consecutive rows of a block (column-major: contiguous), RB loads
  // in flight before the first store
  constexpr int RB = 8;
  static_assert(TM == 64 && TN == 64, "four columns (rows) of the tile per pass of 256 threads");
  const int64_t* bs = base + tk.base;
  const SchurNbr* nb = nbr + tk.nbr;
  const int e0 = threadIdx.x % 64, e1 = threadIdx.x / 64;
  if (i0 + e0 < N) {
    const int gi = i0 + e0, a = rblk[e0], jend = min(TN, (sym ? gi + 1 : N) - j0);
    const int64_t* row = bs + a * tk.nb;
    real* col = arena + rloc[e0];
    const int lda = nb[a].ld;
    for (int j = e1; j < jend; j += 4 * RB) {
      real* t[RB];
      real v[RB];
#pragma unroll
      for (int u = 0; u < RB; u++) {
        const int jj = min(j + 4 * u, TN - 1);
        t[u] = col + row[cblk[jj]] + (int64_t)cloc[jj] * lda;
      }
#pragma unroll
      for (int u = 0; u < RB; u++)
        if (j + 4 * u < jend) v[u] = *t[u];
#pragma unroll
      for (int u = 0; u < RB; u++)
        if (j + 4 * u < jend) *t[u] = v[u] - Cs[j + 4 * u][e0];
    }
  }
  if (!sym) return;
  // the mirror elements (c, r) of the strictly lower part: row gj of block
  // (cblk, rblk), column gi; consecutive threads on consecutive rows gj
  if (j0 + e0 < N) {
    const int gj = j0 + e0, b = cblk[e0], iend = min(TM, N - i0);
    const int64_t* row = bs + b * tk.nb;
    real* col = arena + cloc[e0];
    const int lda = nb[b].ld;
    for (int i = e1; i < iend; i += 4 * RB) {
      real* t[RB];
      real v[RB];
#pragma unroll
      for (int u = 0; u < RB; u++) {
        const int ii = min(i + 4 * u, TM - 1);
        t[u] = col + row[rblk[ii]] + (int64_t)rloc[ii] * lda;
      }
#pragma unroll
      for (int u = 0; u < RB; u++)
        if (i + 4 * u < iend && i0 + i + 4 * u > gj) v[u] = *t[u];
#pragma unroll
      for (int u = 0; u < RB; u++)
        if (i + 4 * u < iend && i0 + i + 4 * u > gj) *t[u] = v[u] - Cs[e0][i + 4 * u];
    }
  }
}

// base[a * nb + b] = arena offset of block (neighbour a, neighbour b) of every
// task, one thread per pair, by bisection of the pattern row.  (The host built
// and uploaded this table: 124 of 170 ms of its work per factorization of 96^3
// went into it; here it takes about 4 us per class.  Looking the blocks up in
// the Schur update itself put the searches in front of every tile: 140 to 160
// ms of updates at 96^3 against 132.)
__global__ void schur_targets_kernel(const SchurTask* __restrict__ tasks,
                                     const SchurNbr* __restrict__ nbr, DevPattern P,
                                     int64_t* __restrict__ base, DevError* err) {
  const SchurTask tk = tasks[blockIdx.y];
  const SchurNbr* nb = nbr + tk.nbr;
  const int n = tk.nb * tk.nb;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const int i = nb[e / tk.nb].id, j = nb[e % tk.nb].id;
    int lo = P.ptr[i], hi = P.ptr[i + 1];
    const int end = hi;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (P.col[mid] < j) lo = mid + 1;
      else hi = mid;
    }
    const bool have = lo < end && P.col[lo] == j;
    // two neighbours of a cluster are within distance two: the block exists
    if (!have && atomicCAS(&err->code, 0, (int)HSOLVE_ERR_CUDA) == 0) err->cluster = tk.s;
    base[tk.base + e] = have ? P.off[lo] : 0;
  }
}

// One segment per (cluster, other-cluster) coupling: rows 0..k of the
// source columns go to rows 0..k of block (s, o); their transpose (or the
// second source, general case) to columns 0..k of block (o, s).
// Two passes, so that both stores run along contiguous elements (the source is
// in L1 for the second); the grid has about 1,024 elements of a segment per CTA
// (a CTA per 64 x 4 elements of the widest instead meant 16,000 nearly empty
// CTAs per class at level 3 of 96^3).  96^3: 29.5 -> 11.7 ms per factorization.
template <typename real>
__global__ void __launch_bounds__(128)
scatter_kernel(const ScatterSeg* __restrict__ segs, const real* __restrict__ src, real* arena,
               const int* __restrict__ rank) {
  const ScatterSeg sg = segs[blockIdx.y];
  const int k = rank[sg.s];
  if (k == 0 || k == sg.m) return;
  const int total = k * sg.width, first = blockIdx.x * blockDim.x + threadIdx.x;
  const int step = gridDim.x * blockDim.x;
  for (int e = first; e < total; e += step) {
    const int i = e % k, c = e / k;
    arena[sg.dst_row + i + (int64_t)c * sg.ld_s] = src[sg.src + i + (int64_t)c * sg.ld_src];
  }
  const real* t = src + (sg.src2 >= 0 ? sg.src2 : sg.src);
  for (int e = first; e < total; e += step) {
    const int c = e % sg.width, i = e / sg.width;
    arena[sg.dst_col + c + (int64_t)i * sg.ld_o] = t[i + (int64_t)c * sg.ld_src];
  }
}

template <typename real>
__global__ void copy_blocks_kernel(const CopyTask* __restrict__ tasks, const real* __restrict__ src,
                                   real* __restrict__ dst) {
  const CopyTask t = tasks[blockIdx.y];
  const int total = t.rows * t.cols;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    int i = e % t.rows, j = e / t.rows;
    dst[t.dst + i + (int64_t)j * t.ld_dst] = src[t.src + i + (int64_t)j * t.ld_src];
  }
}

template <typename real>
__global__ void scatter_csr_kernel(const int64_t* __restrict__ dst, const double* __restrict__ val,
                                   int64_t nnz, real* __restrict__ arena) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz;
       e += (int64_t)gridDim.x * blockDim.x)
    arena[dst[e]] += (real)val[e];
}

// The level-to-level copies sit between two sweeps that are programmatic
// dependents of one another (kernels_apply.cu) and take part in the chain.
// The kernel ahead still writes `src` when they start, so they make no promise
// that it is read-only (no __restrict__: such loads may go through the
// non-coherent cache) and read it from L2.
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... KArgs, typename... Args>
void launch_pdl(void (*kernel)(KArgs...), int grid, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  count_launch();
  cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

template <typename real>
__global__ void gather_vec_kernel(const int64_t* __restrict__ idx, int64_t n, const real* src,
                                  int64_t lds, real* dst, int64_t ldd, int nrhs) {
  pdl_begin();
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * nrhs;
       e += (int64_t)gridDim.x * blockDim.x) {
    int64_t p = e % n;
    int r = (int)(e / n);
    dst[p + r * ldd] = __ldcg(src + idx[p] + r * lds);
  }
}

template <typename real>
__global__ void scatter_vec_kernel(const int64_t* __restrict__ idx, int64_t n, const real* src,
                                   int64_t lds, real* dst, int64_t ldd, int nrhs) {
  pdl_begin();
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * nrhs;
       e += (int64_t)gridDim.x * blockDim.x) {
    int64_t p = e % n;
    int r = (int)(e / n);
    dst[idx[p] + r * ldd] = __ldcg(src + p + r * lds);
  }
}

template <typename real>
__global__ void perm_in_kernel(const int64_t* __restrict__ perm, const double* __restrict__ S,
                               int64_t n, const double* __restrict__ src, int64_t lds,
                               real* __restrict__ dst, int64_t ldd, int nrhs) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * nrhs;
       e += (int64_t)gridDim.x * blockDim.x) {
    int64_t p = e % n;
    int r = (int)(e / n);
    const int64_t g = perm[p];
    const double v = src[g + r * lds];
    dst[p + r * ldd] = (real)(S ? S[g] * v : v);
  }
}

template <typename real>
__global__ void perm_out_kernel(const int64_t* __restrict__ perm, const double* __restrict__ S,
                                int64_t n, const real* __restrict__ src, int64_t lds,
                                double* __restrict__ dst, int64_t ldd, int nrhs) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * nrhs;
       e += (int64_t)gridDim.x * blockDim.x) {
    int64_t p = e % n;
    int r = (int)(e / n);
    const int64_t g = perm[p];
    const double v = (double)src[p + r * lds];
    dst[g + r * ldd] = S ? S[g] * v : v;
  }
}

inline int grid_for(int64_t work, int threads) {
  int64_t g = (work + threads - 1) / threads;
  if (g < 1) g = 1;
  if (g > 152 * 32) g = 152 * 32;
  return (int)g;
}

// ---- float64 Krylov helpers ----------------------------------------------

__global__ void spmv_kernel(int64_t n, const int64_t* __restrict__ rp, const int* __restrict__ ci,
                            const double* __restrict__ v, const double* __restrict__ x, int64_t ldx,
                            double* __restrict__ y, int64_t ldy, int nrhs) {
  for (int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; row < n;
       row += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = rp[row], e = rp[row + 1];
    for (int r = blockIdx.y; r < nrhs; r += gridDim.y) {
      double acc = 0;
      const double* xr = x + r * ldx;
      for (int64_t p = b; p < e; p++) acc += v[p] * xr[ci[p]];
      y[row + r * ldy] = acc;
    }
  }
}

constexpr int kDotBlocks = 256;

// partial[c * kDotBlocks + b] = sum over this block's rows of
// a[:,c] * b[:, c mod bmod], one column c per grid row: a block that took the
// columns in turn held the device to 256 blocks and eight barriers per column
// (a PCG solve of 512^2 with 124 columns 120.6 -> 112.9 ms).  The order of every
// sum is unchanged.
__global__ void dots_partial(int64_t n, const double* __restrict__ a, int64_t lda,
                             const double* __restrict__ b, int64_t ldb, int ncol, int bmod,
                             double* __restrict__ part) {
  __shared__ double red[256];
  for (int c = blockIdx.y; c < ncol; c += gridDim.y) {
    const double* ac = a + c * lda;
    const double* bc = b + (int64_t)(c % bmod) * ldb;
    double s = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
      s += ac[i] * bc[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int st = blockDim.x / 2; st > 0; st >>= 1) {
      if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
      __syncthreads();
    }
    if (threadIdx.x == 0) part[c * kDotBlocks + blockIdx.x] = red[0];
    __syncthreads();
  }
}

__global__ void dots_final(const double* __restrict__ part, int ncol, double* __restrict__ out) {
  int c = blockIdx.x;
  __shared__ double red[kDotBlocks];
  red[threadIdx.x] = part[c * kDotBlocks + threadIdx.x];
  __syncthreads();
  for (int st = kDotBlocks / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[c] = red[0];
}

// w[:, c] += sign * sum_i coef[i * nrhs + c] V_i[:, c] for the nv blocks
// V_i (n x nrhs, ld n, block stride n * nrhs)
__global__ void block_multi_axpy_kernel(int64_t n, int nv, int nrhs, const double* __restrict__ V,
                                        const double* __restrict__ coef, double sign,
                                        double* __restrict__ w, int64_t ldw) {
  const int64_t bs = n * nrhs;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < bs;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e % n;
    const int c = (int)(e / n);
    double acc = 0;
    for (int j = 0; j < nv; j++) acc += V[j * bs + e] * coef[j * nrhs + c];
    w[i + c * ldw] += sign * acc;
  }
}

__global__ void axpby_kernel(int64_t n, int nrhs, const double* __restrict__ alpha,
                             const double* __restrict__ x, int64_t ldx,
                             const double* __restrict__ beta, double* __restrict__ y, int64_t ldy) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * nrhs;
       e += (int64_t)gridDim.x * blockDim.x) {
    int64_t i = e % n;
    int r = (int)(e / n);
    y[i + r * ldy] = alpha[r] * x[i + r * ldx] + beta[r] * y[i + r * ldy];
  }
}

}  // namespace

template <typename real>
void Launch<real>::gemm_gather(const GemmTask* tasks_dev, int ntask, int maxM, int maxN,
                               const real* Abase, real* Cbase, const real* Bbase,
                               const Seg* segs, const int* rank,
                               cudaStream_t st) {
  if (ntask <= 0 || maxM <= 0 || maxN <= 0) return;
  for (int t0 = 0; t0 < ntask; t0 += kMaxGridYZ) {
    dim3 grid((maxN + TN - 1) / TN, (maxM + TM - 1) / TM, std::min(kMaxGridYZ, ntask - t0));
    count_launch();
    gemm_gather_kernel<real><<<grid, 256, 0, st>>>(tasks_dev + t0, Abase, Cbase, Bbase, segs,
                                                    rank);
  }
}

template <typename real>
void Launch<real>::sketch(const SketchTask* tasks_dev, int ntask, int maxm, int maxl,
                          const real* arena, real* ws, const Seg* segs, cudaStream_t st) {
  if (ntask <= 0 || maxm <= 0 || maxl <= 0) return;
  for (int t0 = 0; t0 < ntask; t0 += kMaxGridYZ) {
    dim3 grid((maxl + TN - 1) / TN, (maxm + TM - 1) / TM, std::min(kMaxGridYZ, ntask - t0));
    count_launch();
    sketch_kernel<real><<<grid, 256, 0, st>>>(tasks_dev + t0, arena, ws, segs);
  }
}

template <typename real>
void Launch<real>::schur(const SchurTask* tasks_dev, int ntask, int maxnw, const real* fac,
                         real* arena, const Seg* segs, const int64_t* base, const SchurNbr* nbr,
                         const int* rank, cudaStream_t st) {
  if (ntask <= 0 || maxnw <= 0) return;
  for (int t0 = 0; t0 < ntask; t0 += kMaxGridYZ) {
    dim3 grid((maxnw + TN - 1) / TN, (maxnw + TM - 1) / TM, std::min(kMaxGridYZ, ntask - t0));
    count_launch();
    schur_kernel<real><<<grid, 256, 0, st>>>(tasks_dev + t0, fac, arena, segs, base, nbr, rank);
  }
}

void schur_targets(const SchurTask* tasks, int ntask, int maxnb, const SchurNbr* nbr,
                   const DevPattern& P, int64_t* base, DevError* err, cudaStream_t st) {
  if (ntask <= 0 || maxnb <= 0) return;
  for (int t0 = 0; t0 < ntask; t0 += kMaxGridYZ) {
    const int64_t pairs = (int64_t)maxnb * maxnb;
    dim3 grid((int)std::min<int64_t>(128, (pairs + 255) / 256), std::min(kMaxGridYZ, ntask - t0));
    count_launch();
    schur_targets_kernel<<<grid, 256, 0, st>>>(tasks + t0, nbr, P, base, err);
  }
}

template <typename real>
void Launch<real>::scatter(const ScatterSeg* segs_dev, int nseg, int maxw, int maxm,
                           const real* src, real* arena, const int* rank, cudaStream_t st) {
  if (nseg <= 0) return;
  for (int t0 = 0; t0 < nseg; t0 += kMaxGridYZ) {
    // (ranks are about a quarter of the unknowns)
    dim3 grid(std::max(1, std::min(64, maxw * maxm / 4096)), std::min(kMaxGridYZ, nseg - t0));
    count_launch();
    scatter_kernel<real><<<grid, 128, 0, st>>>(segs_dev + t0, src, arena, rank);
  }
}

template <typename real>
void Launch<real>::copy_blocks(const CopyTask* tasks_dev, int ntask, const real* src, real* dst,
                               cudaStream_t st) {
  if (ntask <= 0) return;
  for (int t0 = 0; t0 < ntask; t0 += kMaxGridYZ) {
    dim3 grid(8, std::min(kMaxGridYZ, ntask - t0));
    count_launch();
    copy_blocks_kernel<real><<<grid, 256, 0, st>>>(tasks_dev + t0, src, dst);
  }
}

template <typename real>
void Launch<real>::scatter_csr(const int64_t* dst, const double* val, int64_t nnz, real* arena,
                               cudaStream_t st) {
  if (nnz <= 0) return;
  count_launch();
  scatter_csr_kernel<real><<<grid_for(nnz, 256), 256, 0, st>>>(dst, val, nnz, arena);
}

template <typename real>
void Launch<real>::gather_vec(const int64_t* idx, int64_t n, const real* src, int64_t lds,
                              real* dst, int64_t ldd, int nrhs, cudaStream_t st) {
  if (n <= 0) return;
  launch_pdl(gather_vec_kernel<real>, grid_for(n * nrhs, 256), st, idx, n, src, lds, dst, ldd,
             nrhs);
}

template <typename real>
void Launch<real>::scatter_vec(const int64_t* idx, int64_t n, const real* src, int64_t lds,
                               real* dst, int64_t ldd, int nrhs, cudaStream_t st) {
  if (n <= 0) return;
  launch_pdl(scatter_vec_kernel<real>, grid_for(n * nrhs, 256), st, idx, n, src, lds, dst, ldd,
             nrhs);
}

template <typename real>
void Launch<real>::perm_in(const int64_t* perm, const double* S, int64_t n, const double* src,
                           int64_t lds, real* dst, int64_t ldd, int nrhs, cudaStream_t st) {
  if (n <= 0) return;
  count_launch();
  perm_in_kernel<real><<<grid_for(n * nrhs, 256), 256, 0, st>>>(perm, S, n, src, lds, dst, ldd,
                                                                  nrhs);
}

template <typename real>
void Launch<real>::perm_out(const int64_t* perm, const double* S, int64_t n, const real* src,
                            int64_t lds, double* dst, int64_t ldd, int nrhs, cudaStream_t st) {
  if (n <= 0) return;
  count_launch();
  perm_out_kernel<real><<<grid_for(n * nrhs, 256), 256, 0, st>>>(perm, S, n, src, lds, dst, ldd,
                                                                   nrhs);
}


template struct Launch<double>;
template struct Launch<float>;

namespace {
__global__ void expand_runs_kernel(const VRun* __restrict__ runs, int64_t nrun,
                                   int64_t* __restrict__ out) {
  for (int64_t r = blockIdx.x; r < nrun; r += gridDim.x) {
    const VRun v = runs[r];
    for (int q = threadIdx.x; q < v.w; q += blockDim.x) out[v.dst + q] = v.src + q;
  }
}
}  // namespace

void expand_runs(const VRun* runs, int64_t nrun, int64_t* out, cudaStream_t st) {
  if (nrun <= 0) return;
  count_launch();
  expand_runs_kernel<<<(int)std::min<int64_t>(nrun, 152 * 32), 128, 0, st>>>(runs, nrun, out);
}

void spmv_csr(int64_t n, const int64_t* rp, const int* ci, const double* v, const double* x,
              int64_t ldx, double* y, int64_t ldy, int nrhs, cudaStream_t st) {
  count_launch();
  // (a matrix of few rows spreads its right-hand sides over the grid)
  const int gx = grid_for(n, 256), gy = std::max(1, std::min(nrhs, 152 * 16 / gx));
  spmv_kernel<<<dim3(gx, gy), 256, 0, st>>>(n, rp, ci, v, x, ldx, y, ldy, nrhs);
}

// out[c] = a[:,c] . b[:,c]; partial sums in a fixed order (deterministic).
// `out` must have room for nrhs * (kDotBlocks + 1) doubles: the first
// nrhs * kDotBlocks hold partials, results go to out[nrhs*kDotBlocks + c].
void dots(int64_t n, const double* a, int64_t lda, const double* b, int64_t ldb, int nrhs,
          double* out, cudaStream_t st) {
  count_launch();
  dots_partial<<<dim3(kDotBlocks, std::min(nrhs, kMaxGridYZ)), 256, 0, st>>>(n, a, lda, b, ldb,
                                                                            nrhs, nrhs, out);
  count_launch();
  dots_final<<<nrhs, kDotBlocks, 0, st>>>(out, nrhs, out + (int64_t)nrhs * kDotBlocks);
}

void block_multi_dot(int64_t n, int nv, int nrhs, const double* V, const double* w,
                     double* out, cudaStream_t st) {
  // column q = i * nrhs + c of the nv blocks is V_i[:, c] (stride n); it
  // meets w[:, c] = w[:, q mod nrhs]
  const int ncol = nv * nrhs;
  count_launch();
  dots_partial<<<dim3(kDotBlocks, std::min(ncol, kMaxGridYZ)), 256, 0, st>>>(n, V, n, w, n, ncol,
                                                                            nrhs, out);
  count_launch();
  dots_final<<<ncol, kDotBlocks, 0, st>>>(out, ncol, out + (int64_t)ncol * kDotBlocks);
}

void block_multi_axpy(int64_t n, int nv, int nrhs, const double* V, const double* coef,
                      double sign, double* w, int64_t ldw, cudaStream_t st) {
  count_launch();
  block_multi_axpy_kernel<<<grid_for(n * nrhs, 256), 256, 0, st>>>(n, nv, nrhs, V, coef, sign,
                                                                    w, ldw);
}

void axpby_cols(int64_t n, int nrhs, const double* alpha, const double* x, int64_t ldx,
                const double* beta, double* y, int64_t ldy, cudaStream_t st) {
  count_launch();
  axpby_kernel<<<grid_for(n * nrhs, 256), 256, 0, st>>>(n, nrhs, alpha, x, ldx, beta, y, ldy);
}

}  // namespace hs
