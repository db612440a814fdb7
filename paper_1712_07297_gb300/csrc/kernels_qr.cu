// Truncated column-pivoted Householder QR of a cluster's fill block (Eq. lra)
// spread over a thread-block cluster.
//
// The fill block G (m x c, c often in the thousands) is split by columns over
// the CL CTAs of a thread-block cluster.  qr_reg_kernel keeps the columns in
// registers for the whole factorization (float32 Cholesky path, clusters of up to
// 256 unknowns, fill blocks that 16 CTAs hold); qr_cluster_kernel keeps them in
// shared memory (the others).  Per step the CTAs agree on the pivot through distributed
// shared memory: the largest remaining column norm over the cluster, then the
// lowest original column index among the columns within the tie tolerance of
// it (the tie rule of the single-CTA path); the reflector is formed from the
// pivot column and every CTA updates its columns.  Two cluster barriers per
// step; every CTA takes the same branches (its decisions use the same
// exchanged values), so the barriers always match.
//
// A count pass first flags and counts the nonzero gathered columns, so that
// each CTA holds an equal share of the nonzero ones and the cluster size and
// shared memory are chosen for the compacted block.
//
// Outputs, in the layout the per-cluster kernel expects: the rank k in
// rank[s], the reflectors v_j as column j of W_G (column-major, ld m, rows
// j..m), tau_j and the sign of R's diagonal in the per-cluster double
// workspace.
#include <climits>
#include <cooperative_groups.h>

#include "common.h"

namespace cg = cooperative_groups;

namespace hs {

namespace {

constexpr size_t kQrSmemCap = 200 * 1024;  // dynamic shared memory per CTA, at most
constexpr int kQrThreads = 256;  // threads per CTA of the cluster QR (more only add barrier cost)
constexpr int kMaxGrid = 1 << 20;

// Dynamic shared memory of one CTA: every array starts on a 16-byte boundary
// (the same computation sizes the launch and carves the buffer).
struct QrSmem {
  size_t G, nrm, oidx, vloc, total;
  __host__ __device__ static size_t al(size_t b) { return (b + 15) / 16 * 16; }
  __host__ __device__ QrSmem(int ldsm, int cc, int sz) {
    G = 0;
    nrm = G + al((size_t)ldsm * cc * sz);
    oidx = nrm + al((size_t)cc * sizeof(double));  // (float32 norms use half of it)
    vloc = oidx + al((size_t)cc * sizeof(int));
    total = vloc + al((size_t)ldsm * sz);
  }
};

// Squared norms as keys: maxima of non-negative floating point numbers are
// integer maxima of their bit patterns, one instruction per warp, and float32
// stays off the float64 pipe (two lanes per clock on this chip).
template <typename real>
struct NormKey;
template <>
struct NormKey<float> {  // non-negative floats order as their bit patterns
  using type = unsigned;
  static __device__ __forceinline__ type of(float v) { return __float_as_uint(v); }
  static __device__ __forceinline__ float value(type k) { return __uint_as_float(k); }
  static __device__ __forceinline__ type warp_max(type k) {
    return __reduce_max_sync(0xffffffffu, k);
  }
  static __device__ __forceinline__ float band(float M) { return tie_band(M); }
  // the largest float x with x <= v
  static __device__ __forceinline__ float floor_of(double v) { return __double2float_rd(v); }
};
template <>
struct NormKey<double> {
  using type = unsigned long long;
  static __device__ __forceinline__ type of(double v) { return __double_as_longlong(v); }
  static __device__ __forceinline__ double value(type k) { return __longlong_as_double(k); }
  static __device__ __forceinline__ type warp_max(type k) {
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32));
    const unsigned lo =
        __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32) == hi ? (unsigned)k : 0u);
    return ((type)hi << 32) | lo;
  }
  static __device__ __forceinline__ double band(double M) { return (1.0 - 1e-10) * M; }
  static __device__ __forceinline__ double floor_of(double v) { return v; }
};

template <typename real>
struct Exchange {
  real val;        // largest local squared norm
  real candnrm;    // squared norm of the local candidate
  int cand;        // lowest original index among the local candidates
  int loc;         // local column of the candidate
};

__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v) {
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long x = __shfl_xor_sync(0xffffffffu, v, o);
    v = x < v ? x : v;
  }
  return v;
}

template <typename real>
__global__ void __launch_bounds__(kQrThreads)
qr_cluster_kernel(const PrepTask* __restrict__ tasks, const int* __restrict__ order,
                  const real* __restrict__ arena,
                  real* __restrict__ ws_all, double* __restrict__ wsd_all,
                  const Seg* __restrict__ segs, int* rank, int* __restrict__ piv,
                  const int* __restrict__ fpiv, const int* __restrict__ cnt, double eps,
                  double noise_rtol, int max_rank, int ldsm, int ccmax) {
  cg::cluster_group cl = cg::this_cluster();
  const int CL = (int)cl.num_blocks();
  const int cr = (int)cl.block_rank();
  const int task = order[blockIdx.x / CL];
  const PrepTask tk = tasks[task];
  const int m = tk.m, c = tk.ncolG;
  using Key = NormKey<real>;
  __shared__ real red_n[kQrThreads / 32];
  __shared__ int scan[kQrThreads / 32];
  __shared__ Exchange<real> xch;
  extern __shared__ __align__(16) unsigned char dsm[];
  const QrSmem lay(ldsm, ccmax, (int)sizeof(real));
  real* Gs = reinterpret_cast<real*>(dsm + lay.G);  // ldsm x ccmax, column-major
  real* nrm = reinterpret_cast<real*>(dsm + lay.nrm);
  int* oidx = reinterpret_cast<int*>(dsm + lay.oidx);
  real* vloc = reinterpret_cast<real*>(dsm + lay.vloc);  // the step's reflector

  // per-cluster outputs (same layout as the per-cluster kernel)
  double* nrm2_g = wsd_all + tk.wsd;
  real* tau_g = reinterpret_cast<real*>(nrm2_g + 2 * (int64_t)tk.ncolG);
  real* rsign_g = tau_g + 2 * m;
  real* W_G = ws_all + tk.ws + 10 * (int64_t)m * m;

  // scale of the rounding-noise floor: max |A_ss|
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  real amx = 0;
  for (int j = warp; j < m; j += nwarp)
    for (int i = lane; i < m; i += 32) amx = fmax(amx, fabs(arena[tk.a_ss + i + (int64_t)j * tk.ld]));
  amx = Key::value(Key::warp_max(Key::of(amx)));
  if (lane == 0) red_n[warp] = amx;
  __syncthreads();
  for (int w = 0; w < nwarp; w++) amx = fmax(amx, red_n[w]);
  // forced ranks keep every direction up to the forced count (no floor)
  const double floor = max_rank < 0 ? 0.0 : noise_rtol * (double)amx;

  // The count pass flagged the nonzero gathered columns (flags[q] != 0) and
  // counted them (nz); CTA cr keeps nonzero columns cr*cz .. (cr+1)*cz - 1
  // in gathered order, so every CTA holds at most cz columns.
  const int* flags = reinterpret_cast<const int*>(nrm2_g + tk.ncolG);
  const int nz = cnt[task];
  const int cz = (nz + CL - 1) / CL;
  const int z0 = cr * cz, z1 = min(nz, z0 + cz);
  {
    const int per = (c + blockDim.x - 1) / blockDim.x;
    const int a0 = min(c, (int)threadIdx.x * per), a1 = min(c, a0 + per);
    int n = 0;
    for (int q = a0; q < a1; q++) n += flags[q];
    int inc = n;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) scan[warp] = inc;
    __syncthreads();
    int zq = inc - n;
    for (int w = 0; w < warp; w++) zq += scan[w];
    // the gathered column of each of this CTA's slots
    for (int q = a0; q < a1; q++) {
      if (flags[q] == 0) continue;
      if (zq >= z0 && zq < z1) oidx[zq - z0] = q;
      zq++;
    }
    __syncthreads();
  }
  const int nloc = max(0, z1 - z0);
  for (int d = warp; d < nloc; d += nwarp) {
    int64_t p;
    int st;
    seg_col(segs + tk.gcol, tk.ngcol, oidx[d], &p, &st);
    for (int i = lane; i < m; i += 32) Gs[i + (int64_t)d * ldsm] = arena[p + (int64_t)i * st];
  }
  __syncthreads();
  // squared norms in the working precision (float64 arithmetic per element
  // would bound the float32 path by the float64 rate), compared in it with
  // thresholds that keep the float64 decisions (NormKey)
  for (int t = threadIdx.x; t < nloc; t += blockDim.x) {
    real s = 0;
    for (int i = 0; i < m; i++) {
      const real x = Gs[i + (int64_t)t * ldsm];
      s += x * x;
    }
    nrm[t] = s;
  }
  __syncthreads();

  // max_rank < 0: the rank of every cluster is forced to rank[s] (set by the
  // host before the launch, read before any CTA of the cluster can write it)
  const int kmax = max_rank > 0 ? min(m, max_rank) : (max_rank < 0 ? min(m, rank[tk.s]) : m);
  if (max_rank < 0) eps = 0.0;
  const int steps = min(m, c);
  real stop = 0;  // a squared norm at or below this ends the factorization
  int k = 0;
  __shared__ unsigned long long red_u[kQrThreads / 32];
  __shared__ real s_M, s_r2;
  __shared__ int s_owner;
  for (int j = 0; j < steps; j++) {
    // 1. largest remaining norm over the cluster
    real lmx = 0;
    for (int t = threadIdx.x; t < nloc; t += blockDim.x) lmx = fmax(lmx, nrm[t]);
    lmx = Key::value(Key::warp_max(Key::of(lmx)));
    if (lane == 0) red_n[warp] = lmx;
    __syncthreads();
    if (threadIdx.x == 0) {
      real v = red_n[0];
      for (int w = 1; w < nwarp; w++) v = fmax(v, red_n[w]);
      xch.val = v;
    }
    cl.sync();
    if (warp == 0) {
      const real v = (lane < CL) ? cl.map_shared_rank(&xch, lane)->val : real(0);
      const real x = Key::value(Key::warp_max(Key::of(v)));
      if (lane == 0) s_M = x;
    }
    __syncthreads();
    const real M = s_M;
    if (!(M > real(0))) break;
    const real band = Key::band(M);
    // 2. lowest original index among the near-maximal columns: one key
    //    (original index, local slot) per candidate, the smallest wins; a
    //    given pivot order (fpiv) makes its column the only candidate
    unsigned long long key = ~0ull;
    const int fq = fpiv ? fpiv[tk.pv + j] : -1;
    for (int t = threadIdx.x; t < nloc; t += blockDim.x)
      if (fpiv ? (z0 + t == fq && nrm[t] >= real(0)) : (nrm[t] >= band)) {
        const unsigned long long kk = ((unsigned long long)oidx[t] << 32) | (unsigned)t;
        key = kk < key ? kk : key;
      }
    key = warp_min_u64(key);
    if (lane == 0) red_u[warp] = key;
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned long long v = red_u[0];
      for (int w = 1; w < nwarp; w++) v = red_u[w] < v ? red_u[w] : v;
      const bool any = v != ~0ull;
      xch.cand = any ? (int)(v >> 32) : INT_MAX;
      xch.loc = any ? (int)(v & 0xffffffffu) : -1;
      xch.candnrm = any ? nrm[(int)(v & 0xffffffffu)] : real(-1);
    }
    cl.sync();
    if (warp == 0) {
      unsigned long long v = ~0ull;
      if (lane < CL)
        v = ((unsigned long long)(unsigned)cl.map_shared_rank(&xch, lane)->cand << 8) | lane;
      v = warp_min_u64(v);
      if (lane == 0) {
        s_owner = (int)(v & 0xff);
        s_r2 = cl.map_shared_rank(&xch, (int)(v & 0xff))->candnrm;
      }
    }
    __syncthreads();
    const int owner = s_owner;
    const real r2 = s_r2;
    if (!(r2 >= real(0))) break;  // a given pivot that names no remaining column
    if (j == 0) {
      // |r_jj| <= floor or |r_jj| <= eps |r_11|, on the squares
      double s2 = floor * floor;
      if (eps > 0.0) s2 = fmax(s2, eps * eps * (double)r2);
      stop = Key::floor_of(s2);
    }
    if (r2 <= stop || j >= kmax) break;
    // 3. every CTA forms the reflector v = x - beta e1, beta = -sign(x0) ||x||
    //    from the pivot column in the owner's shared memory (read through
    //    distributed shared memory; that column is never written again, so
    //    no further cluster barrier is needed); the owner also stores it
    const int oloc = cl.map_shared_rank(&xch, owner)->loc;
    const real* ocol = cl.map_shared_rank(Gs, owner) + (int64_t)oloc * ldsm;
    const real x0 = ocol[j];
    real head, tj;
    householder_scalars(r2, x0, &head, &tj);
    for (int i = j + threadIdx.x; i < m; i += blockDim.x) {
      const real v = (i == j) ? head : ocol[i];
      vloc[i] = v;
      if (cr == owner) W_G[i + (int64_t)j * m] = v;
    }
    if (cr == owner && threadIdx.x == 0) {
      tau_g[j] = tj;
      rsign_g[j] = x0 >= real(0) ? real(-1) : real(1);
      nrm[oloc] = real(-1);  // used: out of every later step
      // the pivot as an index among the nonzero gathered columns: slot t of
      // CTA cr holds nonzero column z0 + t
      piv[tk.pv + j] = z0 + oloc;
    }
    __syncthreads();
    // 4. every CTA applies the reflector to its remaining columns and
    //    recomputes their squared norms over rows j+1..m
    for (int t = threadIdx.x; t < nloc; t += blockDim.x) {
      if (nrm[t] < real(0)) continue;
      real* col = Gs + (int64_t)t * ldsm;
      // four independent partial sums (combined in a fixed order) keep four
      // products in flight instead of one dependent chain
      real w0 = 0, w1 = 0, w2 = 0, w3 = 0;
      int i = j;
      for (; i + 3 < m; i += 4) {
        w0 += vloc[i] * col[i];
        w1 += vloc[i + 1] * col[i + 1];
        w2 += vloc[i + 2] * col[i + 2];
        w3 += vloc[i + 3] * col[i + 3];
      }
      for (; i < m; i++) w0 += vloc[i] * col[i];
      const real w = ((w0 + w1) + (w2 + w3)) * tj;
      col[j] -= w * vloc[j];
      real s0 = 0, s1 = 0, s2 = 0, s3 = 0;
      i = j + 1;
      for (; i + 3 < m; i += 4) {
        const real a0 = col[i] - w * vloc[i], a1 = col[i + 1] - w * vloc[i + 1];
        const real a2 = col[i + 2] - w * vloc[i + 2], a3 = col[i + 3] - w * vloc[i + 3];
        col[i] = a0;
        col[i + 1] = a1;
        col[i + 2] = a2;
        col[i + 3] = a3;
        s0 += a0 * a0;
        s1 += a1 * a1;
        s2 += a2 * a2;
        s3 += a3 * a3;
      }
      for (; i < m; i++) {
        const real a = col[i] - w * vloc[i];
        col[i] = a;
        s0 += a * a;
      }
      nrm[t] = (s0 + s1) + (s2 + s3);
    }
    __syncthreads();
    k = j + 1;
  }
  if (cr == 0 && threadIdx.x == 0) rank[tk.s] = k;
  // no CTA leaves while another may still read its shared memory
  cl.sync();
}

// ---------------------------------------------------------------------------
// Register-resident pivoted QR
// ---------------------------------------------------------------------------
// TPC threads share a column, thread h of them rows h, h + TPC, .. (RPT of
// them, zero beyond m), so a step reads only the reflector from shared memory
// (16-byte broadcasts) where the shared-memory form reads each element twice,
// writes it once and reads two scalars of the reflector beside it.  What else a
// step pays for is latency, so: columns lie on the warps in gathered order,
// and the winner -- the lowest index within the tie band of the largest norm
// -- is in the first warp whose own maximum reaches the band, found without a
// second reduction (two CTA barriers per step; with several CTAs one and two
// cluster barriers); and float32 stays off the float64 pipe (two lanes per
// clock on this chip): norms compare as integers, thresholds are rounded to
// float32 once, the reflector's scalars are formed in float32 pairs.  (The
// float64 path is bound by that pipe, 56,000 products per step and SM at 128 x
// 280, and keeps the shared-memory form, whose rows end exactly at m; so does
// the float32 general path.)  Per step: search 1.0 us, publish 1.2-1.6, apply
// 1.1-1.3 (two cluster barriers among them; the shared-memory form took 6 to
// 8).  All fill blocks of a factorization, shared memory -> registers: 64^3
// 47.5 -> 20 ms, 96^3 184 -> 99 ms.
// CTAs of a thread-block cluster: 16 (beyond the portable 8) hold the coarse
// levels' widest fill blocks
constexpr int kRegMaxCl = 16;

template <typename real, int RPT, int TPC, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
qr_reg_kernel(const PrepTask* __restrict__ tasks, const int* __restrict__ order,
              const real* __restrict__ arena,
              real* __restrict__ ws_all, double* __restrict__ wsd_all,
              const Seg* __restrict__ segs, int* rank, int* __restrict__ piv,
              const int* __restrict__ fpiv, const int* __restrict__ cnt, double eps,
              double noise_rtol, int max_rank) {
  using Key = NormKey<real>;
  using key_t = typename Key::type;
  constexpr int kBlk = 8, kBlocks = RPT / kBlk;
  constexpr int kPad = 16 / (int)sizeof(real);  // threads of a column on other banks
  constexpr int kLdv = RPT + kPad;
  // the launches of a class run beside one another: each lets the next one
  // start at once and ends only after the one before it has
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  cg::cluster_group cl = cg::this_cluster();
  const int CL = (int)cl.num_blocks(), cr = (int)cl.block_rank();
  const int task = order[blockIdx.x / CL];
  const PrepTask tk = tasks[task];
  const int m = tk.m, c = tk.ncolG;
  // the step's reflector, by thread of a column, then its squared norm, its
  // tau and the pivot's index
  constexpr int kInfo = TPC * kLdv, kVs = kInfo + kPad;
  __shared__ __align__(16) real vs[2][kVs];
  __shared__ key_t wmax[2][32];                     // largest norm of every warp
  __shared__ key_t xmax[2][kRegMaxCl];              // and of every CTA
  __shared__ int scan[33];
  __shared__ int slot_col[NT / TPC];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const int t = threadIdx.x / TPC, h = threadIdx.x % TPC;

  double* nrm2_g = wsd_all + tk.wsd;
  real* tau_g = reinterpret_cast<real*>(nrm2_g + 2 * (int64_t)tk.ncolG);
  real* rsign_g = tau_g + 2 * m;
  real* W_G = ws_all + tk.ws + 10 * (int64_t)m * m;

  // this CTA's columns: nonzero columns cr * cz .. (cr + 1) * cz - 1 in
  // gathered order, one per slot
  const int* flags = reinterpret_cast<const int*>(nrm2_g + tk.ncolG);
  const int nz = cnt[task];
  const int cz = (nz + CL - 1) / CL;
  const int z0 = min(nz, cr * cz), z1 = min(nz, z0 + cz), nloc = z1 - z0;
  {
    const int per = (c + blockDim.x - 1) / blockDim.x;
    const int a0 = min(c, (int)threadIdx.x * per), a1 = min(c, a0 + per);
    int n = 0;
    for (int q = a0; q < a1; q++) n += flags[q];
    int inc = n;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) scan[warp] = inc;
    __syncthreads();
    int before = inc - n;
    for (int w = 0; w < warp; w++) before += scan[w];
    for (int q = a0; q < a1; q++) {
      if (flags[q] == 0) continue;
      if (before >= z0 && before < z1) slot_col[before - z0] = q;
      before++;
    }
    __syncthreads();
  }
  real col[RPT];
#pragma unroll
  for (int r = 0; r < RPT; r++) col[r] = 0;
  if (t < nloc) {
    int64_t p;
    int st;
    seg_col(segs + tk.gcol, tk.ngcol, slot_col[t], &p, &st);
#pragma unroll
    for (int r = 0; r < RPT; r++) {
      const int i = r * TPC + h;
      if (i < m) col[r] = arena[p + (int64_t)i * st];
    }
  }
  // scale of the rounding-noise floor: max |A_ss|
  real amx = 0;
  for (int j = warp; j < m; j += 4 * nwarp)
    for (int i = lane; i < m; i += 32) {
      real x[4];
#pragma unroll
      for (int q = 0; q < 4; q++)
        x[q] = j + q * nwarp < m ? arena[tk.a_ss + i + (int64_t)(j + q * nwarp) * tk.ld] : real(0);
#pragma unroll
      for (int q = 0; q < 4; q++) amx = fmax(amx, fabs(x[q]));
    }
  const auto column_sum = [](real s) {
#pragma unroll
    for (int o = 1; o < TPC; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  };
  real nrm;
  {
    real s[4] = {0, 0, 0, 0};
#pragma unroll
    for (int r = 0; r < RPT; r++) s[r & 3] += col[r] * col[r];
    nrm = column_sum((s[0] + s[1]) + (s[2] + s[3]));
  }
  {
    const key_t a = Key::warp_max(Key::of(amx));
    if (lane == 0) wmax[1][warp] = a;
  }
  __syncthreads();
  amx = Key::value(Key::warp_max(lane < nwarp ? wmax[1][lane] : key_t(0)));
  // forced ranks keep every direction up to the forced count (no floor)
  const double floor = max_rank < 0 ? 0.0 : noise_rtol * (double)amx;
  const int kmax = max_rank > 0 ? min(m, max_rank) : (max_rank < 0 ? min(m, rank[tk.s]) : m);
  if (max_rank < 0) eps = 0.0;
  const int steps = min(m, c);
  const int nblk = (m + kBlk * TPC - 1) / (kBlk * TPC);  // row blocks that hold rows
  real stop = 0;  // a squared norm at or below this ends the factorization
  bool used = false;
  int k = 0;
  cl.sync();  // rank[s] is read, and every CTA runs before its memory is written
  for (int j = 0; j < steps; j++) {
    const int par = j & 1;
    // 1. largest remaining norm, and which warp's columns hold the pivot
    const key_t mine = used ? key_t(0) : Key::of(nrm);
    const key_t wm = Key::warp_max(mine);
    if (lane == 0) wmax[par][warp] = wm;
    __syncthreads();
    const key_t wl = lane < nwarp ? wmax[par][lane] : key_t(0);
    key_t M = Key::warp_max(wl);
    int owner = 0;
    const int fq = fpiv ? fpiv[tk.pv + j] : -1;
    if (CL > 1) {
      if (warp == 0 && lane < CL) *cl.map_shared_rank(&xmax[par][cr], lane) = M;
      cl.sync();
      const key_t xl = lane < CL ? xmax[par][lane] : key_t(0);
      M = Key::warp_max(xl);
      owner = __ffs(__ballot_sync(0xffffffffu, lane < CL && Key::value(xl) >=
                                                              Key::band(Key::value(M)))) - 1;
    }
    if (!(Key::value(M) > real(0))) break;
    const real band = Key::band(Key::value(M));
    int ww;
    if (fpiv) {  // a given pivot order names its column
      if (fq < 0 || fq >= nz) break;
      owner = fq / cz;
      ww = (fq - owner * cz) * TPC / 32;
    } else {
      ww = __ffs(__ballot_sync(0xffffffffu, lane < nwarp && Key::value(wl) >= band)) - 1;
    }
    // 2. the winner's warp publishes the reflector
    if (cr == owner && warp == ww) {
      const bool cand = fpiv ? (z0 + t == fq) : (!used && nrm >= band);
      const int src = (__ffs(__ballot_sync(0xffffffffu, cand)) - 1) / TPC * TPC;
      const bool win = lane / TPC * TPC == src;
      if (win) {
#pragma unroll
        for (int r = 0; r < RPT; r++)
          vs[par][h * kLdv + r] = r * TPC + h >= j ? col[r] : real(0);
      }
      __syncwarp();
      const real x0 = vs[par][(j % TPC) * kLdv + j / TPC];
      const real r2 = __shfl_sync(0xffffffffu, used ? real(-1) : nrm, src);
      __syncwarp();
      real head, tau;
      householder_scalars(r2, x0, &head, &tau);
      if (lane == 0) {
        vs[par][(j % TPC) * kLdv + j / TPC] = head;
        vs[par][kInfo] = r2;
        vs[par][kInfo + 1] = tau;
      }
      if (lane == src) vs[par][kInfo + 2] = __int_as_float(z0 + t);
      __syncwarp();
      if (CL > 1) {
        // into the other CTAs' shared memory, 16 bytes at a time
        constexpr int kUnits = kVs / kPad;
        for (int e = lane; e < kUnits * CL; e += 32) {
          const int q = e / kUnits, u = e % kUnits * kPad;
          if (q != cr)
            *reinterpret_cast<int4*>(cl.map_shared_rank(&vs[par][0], q) + u) =
                *reinterpret_cast<const int4*>(&vs[par][u]);
        }
      }
      used = used || win;
    }
    if (CL > 1) cl.sync();
    else __syncthreads();
    const real r2 = vs[par][kInfo];
    if (!(r2 >= real(0))) break;  // a given pivot that is used already
    if (j == 0) {
      // |r_jj| <= floor or |r_jj| <= eps |r_11|, on the squares
      double s2 = floor * floor;
      if (eps > 0.0) s2 = fmax(s2, eps * eps * (double)r2);
      stop = Key::floor_of(s2);
    }
    if (r2 <= stop || j >= kmax) break;
    // the reflector leaves for the per-cluster kernel behind the barrier, from
    // the CTAs in turn: a barrier waits for the stores before it
    if (cr == j % CL) {
      for (int i = j + threadIdx.x; i < m; i += blockDim.x)
        W_G[i + (int64_t)j * m] = vs[par][(i % TPC) * kLdv + i / TPC];
      if (threadIdx.x == 0) {
        tau_g[j] = vs[par][kInfo + 1];
        rsign_g[j] = vs[par][(j % TPC) * kLdv + j / TPC] >= real(0) ? real(-1) : real(1);
        piv[tk.pv + j] = __float_as_int(vs[par][kInfo + 2]);
      }
    }
    // 3. apply it to the remaining columns; squared norms of rows j+1..m (row
    //    j of a column is not needed again and set to zero)
    const real tau = vs[par][kInfo + 1];
    const real* v = &vs[par][h * kLdv];
    const int jb = j / (kBlk * TPC);
    real w[4] = {0, 0, 0, 0};
#pragma unroll
    for (int b = 0; b < kBlocks; b++) {
      if (b < jb || b >= nblk) continue;
      real x[kBlk];
#pragma unroll
      for (int q = 0; q < kBlk; q += kPad)
        *reinterpret_cast<int4*>(x + q) = *reinterpret_cast<const int4*>(v + b * kBlk + q);
#pragma unroll
      for (int q = 0; q < kBlk; q++) w[q & 3] += x[q] * col[b * kBlk + q];
    }
    const real wt = column_sum((w[0] + w[1]) + (w[2] + w[3])) * tau;
    real s[4] = {0, 0, 0, 0};
#pragma unroll
    for (int b = 0; b < kBlocks; b++) {
      if (b < jb || b >= nblk) continue;
      real x[kBlk];
#pragma unroll
      for (int q = 0; q < kBlk; q += kPad)
        *reinterpret_cast<int4*>(x + q) = *reinterpret_cast<const int4*>(v + b * kBlk + q);
      if (b == jb) {
#pragma unroll
        for (int q = 0; q < kBlk; q++) {
          const real a = (b * kBlk + q) * TPC + h > j ? col[b * kBlk + q] - wt * x[q] : real(0);
          col[b * kBlk + q] = a;
          s[q & 3] += a * a;
        }
      } else {
#pragma unroll
        for (int q = 0; q < kBlk; q++) {
          const real a = col[b * kBlk + q] - wt * x[q];
          col[b * kBlk + q] = a;
          s[q & 3] += a * a;
        }
      }
    }
    nrm = column_sum((s[0] + s[1]) + (s[2] + s[3]));
    k = j + 1;
  }
  if (cr == 0 && threadIdx.x == 0) rank[tk.s] = k;
  // no CTA leaves while another may still write its shared memory
  cl.sync();
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Count pass: flag the nonzero gathered columns of every task (flags in the
// task's double workspace after the norms) and count them.  Grid (task,
// chunk of 256 columns), one thread per column with eight loads in flight;
// the counts are accumulated atomically into cnt (zeroed by the caller).
template <typename real>
__global__ void __launch_bounds__(256)
count_nz_kernel(const PrepTask* __restrict__ tasks, const real* __restrict__ arena,
                double* __restrict__ wsd_all, const Seg* __restrict__ segs, int* cnt) {
  const PrepTask tk = tasks[blockIdx.x];
  int* flags = reinterpret_cast<int*>(wsd_all + tk.wsd + tk.ncolG);
  __shared__ int red[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  int n = 0;
  for (int q = blockIdx.y * blockDim.x + threadIdx.x; q < tk.ncolG;
       q += gridDim.y * blockDim.x) {
    int64_t p;
    int st;
    seg_col(segs + tk.gcol, tk.ngcol, q, &p, &st);
    bool nz = false;
    for (int i = 0; i < tk.m; i += 8) {
      real x[8];
#pragma unroll
      for (int r = 0; r < 8; r++) x[r] = (i + r < tk.m) ? arena[p + (int64_t)(i + r) * st] : real(0);
#pragma unroll
      for (int r = 0; r < 8; r++) nz |= (x[r] != real(0));
    }
    flags[q] = nz ? 1 : 0;
    n += nz;
  }
  for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  if (lane == 0) red[warp] = n;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < nwarp; w++) t += red[w];
    if (t) atomicAdd(cnt + blockIdx.x, t);
  }
}

}  // namespace

template <typename real>
void Launch<real>::count_nz(const PrepTask* tasks_dev, int ntask, int maxc, const real* arena,
                            double* wsd, const Seg* segs, int* cnt, cudaStream_t st) {
  if (ntask <= 0) return;
  cudaMemsetAsync(cnt, 0, sizeof(int) * ntask, st);
  const int chunks = std::max(1, std::min((maxc + 255) / 256, 64));
  for (int t0 = 0; t0 < ntask; t0 += kMaxGrid) {
    const int nt = std::min(kMaxGrid, ntask - t0);
    count_launch();
    count_nz_kernel<real><<<dim3(nt, chunks), 256, 0, st>>>(tasks_dev + t0, arena, wsd, segs,
                                                            cnt + t0);
  }
}

template <typename real>
int Launch<real>::qr_cluster_size(int maxm, int maxc) {
  for (int CL = 1; CL <= 16; CL *= 2) {
    if (qr_cluster_smem(maxm, maxc, CL) <= kQrSmemCap) return CL;
  }
  return 0;
}

template <typename real>
size_t Launch<real>::qr_cluster_smem(int maxm, int maxc, int CL) {
  const int cc = (maxc + CL - 1) / CL;
  return QrSmem((maxm + 1) | 1, cc, (int)sizeof(real)).total;
}

template <typename real>
void Launch<real>::qr_cluster(const PrepTask* tasks_dev, const int* order, int ntask, int maxm,
                              int maxc, int CL, const real* arena, real* ws, double* wsd, const Seg* segs,
                              int* rank, int* piv, const int* fpiv, const int* cnt, double eps,
                              int max_rank, cudaStream_t st) {
  if (ntask <= 0) return;
  const double noise_rtol = sizeof(real) == 8 ? 1e-14 : 1e-6;
  const size_t smem = qr_cluster_smem(maxm, maxc, CL);
  const int cc = (maxc + CL - 1) / CL;
  // the limit is raised once to the sizing cap (qr_cluster_size keeps every
  // launch at or below it) and never lowered: host threads factoring
  // different matrices launch this kernel concurrently
  static const bool limit_set = [] {
    cudaFuncSetAttribute(qr_cluster_kernel<real>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)kQrSmemCap);
    // clusters of 16 CTAs (the largest qr_cluster_size picks) are non-portable
    cudaFuncSetAttribute(qr_cluster_kernel<real>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return true;
  }();
  (void)limit_set;
  for (int t0 = 0; t0 < ntask; t0 += 4096) {
    const int nt = std::min(4096, ntask - t0);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nt * CL);
    cfg.blockDim = dim3(kQrThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    count_launch();
    cudaLaunchKernelEx(&cfg, qr_cluster_kernel<real>, tasks_dev, order + t0, arena, ws, wsd, segs, rank,
                       piv, fpiv, cnt, eps, noise_rtol, max_rank, (maxm + 1) | 1, cc);
  }
}

namespace {
// The forms of the register kernel (float32): rows per thread, threads per
// column, most threads and CTAs per SM the registers are cut for.  The first
// form with room for the class is taken: fewer rows per thread make a shorter
// step, more threads per column leave fewer columns per CTA.
struct QrForm {
  int maxm, tpc, threads;
  int cols() const { return threads / tpc; }
};
constexpr QrForm kQrForms[] = {{32, 4, 1024},  {32, 2, 1024}, {64, 4, 1024}, {64, 2, 1024},
                               {128, 4, 576}, {128, 2, 576}, {256, 4, 512}};

// The form for clusters of up to m unknowns and c columns, and its cluster
// size (a portable one of any form before a larger one); -1 when none has
// room.
int reg_form(int m, int c, int* CL) {
  for (int most = 8; most <= kRegMaxCl; most *= 2)
    for (int i = 0; i < (int)(sizeof(kQrForms) / sizeof(kQrForms[0])); i++)
      for (*CL = 1; m <= kQrForms[i].maxm && *CL <= most; *CL *= 2)
        if ((c + *CL - 1) / *CL <= kQrForms[i].cols()) return i;
  return -1;
}

template <typename real, int RPT, int TPC, int NT, int MINB>
void launch_qr_reg(int CL, int cols, bool beside, const PrepTask* tasks, const int* order,
                   int ntask, const real* arena, real* ws, double* wsd, const Seg* segs, int* rank,
                   int* piv, const int* fpiv, const int* cnt, double eps, double noise,
                   int max_rank, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  static const bool limit_set = [] {
    cudaFuncSetAttribute(qr_reg_kernel<real, RPT, TPC, NT, MINB>,
                         cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return true;
  }();
  (void)limit_set;
  cfg.blockDim = dim3(std::max(64, (cols * TPC + 31) / 32 * 32));
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CL;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  for (int t0 = 0; t0 < ntask; t0 += 4096) {
    attr[1].val.programmaticStreamSerializationAllowed = beside || t0 > 0;
    cfg.gridDim = dim3(std::min(4096, ntask - t0) * CL);
    count_launch();
    cudaLaunchKernelEx(&cfg, qr_reg_kernel<real, RPT, TPC, NT, MINB>, tasks, order + t0, arena, ws,
                       wsd, segs, rank, piv, fpiv, cnt, eps, noise, max_rank);
  }
}
}  // namespace

template <typename real>
int Launch<real>::qr_reg_form(int m, int c, int* CL) {
  return sizeof(real) == 4 ? reg_form(m, c, CL) : -1;
}

template <typename real>
void Launch<real>::qr_reg(int form, int CL, int maxc, bool beside, const PrepTask* tasks,
                          const int* order, int ntask, const real* arena, real* ws, double* wsd,
                          const Seg* segs, int* rank, int* piv, const int* fpiv, const int* cnt,
                          double eps, int max_rank, cudaStream_t st) {
  if (ntask <= 0) return;
  const int cols = std::max(1, (maxc + CL - 1) / CL);
  const auto go = [&](auto launch) {
    launch(CL, cols, beside, tasks, order, ntask, arena, ws, wsd, segs, rank, piv, fpiv, cnt, eps,
           1e-6, max_rank, st);
  };
  if constexpr (sizeof(real) == 4) {
    switch (form) {
      case 0: go(launch_qr_reg<real, 8, 4, 1024, 1>); break;
      case 1: go(launch_qr_reg<real, 16, 2, 1024, 1>); break;
      case 2: go(launch_qr_reg<real, 16, 4, 1024, 1>); break;
      case 3: go(launch_qr_reg<real, 32, 2, 1024, 1>); break;
      case 4: go(launch_qr_reg<real, 32, 4, 576, 2>); break;
      case 5: go(launch_qr_reg<real, 64, 2, 576, 1>); break;
      case 6: go(launch_qr_reg<real, 64, 4, 512, 1>); break;
      default: break;
    }
  }
}

template struct Launch<double>;
template struct Launch<float>;

}  // namespace hs
