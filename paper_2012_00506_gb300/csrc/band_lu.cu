// band_lu.cu -- shifted band LU with partial pivoting inside the band and the
// multi-right-hand-side solves of eq. (10) of arXiv 2012.00506:
//     (z_j I - B) Q^(j) = X~,   j = 1..n_e.
//
// The band of semi-bandwidth b is handled as a block band of T x T tiles
// (T = 32, block semi-bandwidth bt = ceil(b/T)).  Partial pivoting over the
// rows k..k+b of column k is the same as pivoting over the (bt+1)T rows of
// the block panel, because the rows past k+b are structurally zero there, so
// the pivots equal those of LAPACK's gbtrf (first maximum of |Re|+|Im|).
// The U factor fills to 2b superdiagonals (2bt tiles).
//
// factor_kernel: a thread-block cluster per shifted system (the L2 level of the
//   paper's parallelism is the batch dimension; the cluster is the L3 level,
//   inside one factorization).  Per block column K: the panel ((bt+1)T x T) is
//   factored by one CTA; the panel permutation is gathered into each trailing
//   block column on load; the top tile is multiplied by the inverted unit-lower
//   diagonal block and the tiles below get the T-deep Schur update.
// diag_inverse_kernel: the inverses of the diagonal blocks, so that every solve
//   step is a tile product.
// solve kernels: one thread block per (system, block of 8 to 64 right-hand
//   sides, solve_width); forward L sweep then backward U sweep (trans = 0), or U^H then
//   L^H and the inverse permutation (trans = 1, the conjugate node conj(z)
//   of a Hermitian band).  Factor tiles stream from L2/HBM through shared
//   memory; each is reused by the right-hand sides of the block.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "band_lu.cuh"
#include "quotient.cuh"

namespace cg = cooperative_groups;

namespace pdeshep {

constexpr int kThreads = 256;
constexpr int kLdt = kTile + 1;

// ---------------------------------------------------------------------------
// init: tiles of z I - B (identity padding past n, zero fill slots)
// ---------------------------------------------------------------------------
template <typename C>
__global__ void __launch_bounds__(kThreads) init_factor_kernel(FactorGeom g, int cplx,
                                                              const double* __restrict__ band,
                                                              int64_t ldab, const SysDesc* sys,
                                                              char* arena) {
  using R = typename real_of<C>::type;
  const int s = blockIdx.y;
  const SysDesc d = sys[s];
  FactorPtr<C> f = factor_ptr<C>(g, arena + d.factor_off);
  const int T = kTile;
  for (int64_t t = blockIdx.x; t < g.tiles; t += gridDim.x) {
    const int I = (int)(t / g.nslot);
    const int J = I + (int)(t % g.nslot) - g.bt;
    C* tile = f.tiles + t * g.tile_elems;
    for (int e = threadIdx.x; e < T * T; e += blockDim.x) {
      const int r = e % T, c = e / T;
      const int64_t i = (int64_t)I * T + r, j = (int64_t)J * T + c;
      R vr = 0, vi = 0;
      if (J >= 0 && J < g.Nb) {
        if (i >= g.n || j >= g.n) {
          vr = (i == j) ? R(1) : R(0);
        } else {
          const int64_t dd = i - j;
          if (dd >= -g.b && dd <= g.b) {
            double br, bi;
            if (dd >= 0) {
              if (cplx) {
                br = band[2 * (dd + j * ldab)];
                bi = band[2 * (dd + j * ldab) + 1];
              } else {
                br = band[dd + j * ldab];
                bi = 0.0;
              }
            } else {
              if (cplx) {
                br = band[2 * (-dd + i * ldab)];
                bi = -band[2 * (-dd + i * ldab) + 1];
              } else {
                br = band[-dd + i * ldab];
                bi = 0.0;
              }
            }
            if (i == j) {
              vr = (R)(d.zre - br);
              vi = (R)d.zim;
            } else {
              vr = (R)(-br);
              vi = (R)(-bi);
            }
          }
        }
      }
      tile[e] = cmk<C>(vr, vi);
    }
  }
}

// ---------------------------------------------------------------------------
// factorization.  The chain of a block column is its panel: 32 columns of pivot
// search, row interchange and elimination, in which the next column waits for the
// last.  One CTA per system spent 88 us (b = 64) to 150 us (b = 128) per block
// column on it and on what followed it (serial inverses of the diagonal blocks,
// updates through shared memory), with all but a few SMs idle when a call has few
// systems.  Here
//  * a cluster of G CTAs shares a system: CTA 0 updates the next block column and
//    factors it while the others apply the current panel to the block columns
//    right of it (look-ahead of one); one cluster barrier per block column.  In
//    FP64, where the updates of a block column take longer than a barrier, its
//    columns are spread over the cluster as well (`spread`, a second barrier);
//  * rows of the panel do not move: each carries its logical index.  complex64: a thread per row, the row in
//    registers, every warp searching the column's entries itself (panel_lu_rows); complex128, where the
//    FP64 pipes of all four quadrants are needed, a row in four threads and a warp that searches
//    ahead (panel_lu_parts);
//  * a warp updates NC columns on its own (gathered through the permutation,
//    rows in registers), without barriers;
//  * the inverses of the diagonal blocks that only the solves need are left to
//    diag_inverse_kernel, parallel over blocks and systems.
// Every entry sees the operations of the one-CTA form in the same order
// (complex64 factors keep their bits; in FP64 the top block comes from forward
// substitution instead of the product with the inverse).
// Measured, us per block column against one CTA with a panel in shared memory: complex64 b = 64, 8
// systems 24.5 against 88, 64 systems 25 against 89, 256 systems 54 (two waves of 89 before); b = 128, 16
// systems 30 against 151; complex128 b = 32, 8 systems 81 against 454, b = 128, 2 systems 182 against
// 1558.  What remains (b = 64) is the panel: 32 columns of about 1200 clocks, each a search (300), a
// reciprocal (two dependent divisions, 170), two barriers and the row's updates (440).
// ---------------------------------------------------------------------------
// a b with each rounding spelled out, so that the factors' bits do not depend on how the compiler
// contracts the expression: (a.x b.x - [a.y b.y], a.x b.y + [a.y b.x]), products in brackets rounded.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
template <typename C>
__device__ __forceinline__ C cmul_rn(C a, C b) {
  return cmk<C>(fma(a.x, b.x, -mul_rn(a.y, b.y)), fma(a.x, b.y, mul_rn(a.y, b.x)));
}

// order-preserving integer key of v >= 0 (0 for NaN, which is never a pivot; > 1 if v > 0)
__device__ __forceinline__ unsigned long long pivot_key(float v) {
  return v == v ? (unsigned long long)__float_as_uint(v) + 1 : 0ull;
}
__device__ __forceinline__ unsigned long long pivot_key(double v) {  // (an FP64 comparison takes 64 clocks)
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  return (u << 1) <= 0xFFE0000000000000ull ? u + 1 : 0ull;
}
template <typename R>
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long k) {
  if constexpr (sizeof(R) == 4) return __reduce_max_sync(0xffffffffu, (unsigned)k);
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32));
  const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32) == hi ? (unsigned)k : 0u);
  return ((unsigned long long)hi << 32) | lo;
}
__device__ __forceinline__ float2 shfl_c(float2 v, int src) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
__device__ __forceinline__ double2 shfl_c(double2 v, int src) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

constexpr int kRowsMax = 256;  // panel rows that panel_lu_rows takes

// One column's pivot, from the warp that searches to those that eliminate.
template <typename C>
struct Pivot {
  C inv;
  int row, log, ok;  // its row and logical row; whether there is one
};

// shared memory of one CTA
template <typename C>
struct FactorSmem {
  C* Pan;   // [T][ldp] panel: packed L\U of the top block and L below, logical row r at perm[r]
            // (panel_lu_rows: multipliers only) or at r (panel_lu_parts)
  C* Li;    // [T][T+1] rows of the inverse of the unit lower top block (complex64)
  C* top;   // [warps][2][NC][T] top rows of a warp's columns
  int* perm;            // [Pmax]
  unsigned long long* keys;  // panel_lu_parts: [2][Pmax] keys of the rows' entries of the current column
  int* logs;            // ... [2][Pmax] and their logical rows
  Pivot<C>* pivot;      // ... [2]
  C* U;                 // panel_lu_rows: [T][T+2] pivot rows, each from its column on
  C* col;               // ... [2][kRowsMax] the rows' entries of the current column
  unsigned* key;        // ... [2][kRowsMax] and their keys
  int* log;             // ... [kRowsMax] logical rows
  int* win;             // ... [T] pivot row of each column
};

template <typename C, bool ROWS>
__host__ __device__ inline size_t factor_cluster_smem(int Pmax, int nw, int nc) {
  const size_t base = sizeof(C) * ((size_t)kTile * (Pmax + 1) + (size_t)kTile * (kTile + 1) + (size_t)nw * 2 * nc * kTile) +
                      sizeof(int) * Pmax + 64;
  return base + (ROWS ? sizeof(C) * (kTile * (kTile + 2) + 2 * kRowsMax) + sizeof(int) * (3 * kRowsMax + kTile)
                      : (sizeof(unsigned long long) + sizeof(int)) * 2 * Pmax + 2 * sizeof(Pivot<C>));
}

// complex64: LU with partial pivoting of the panel of block column K (rows K .. K+nbb), thread r holding
// panel row r.  The row's registers move down one place per column (w[0] is the current column), which
// the elimination does for free by its choice of destination and which keeps the loop rolled: four
// stages of 8 columns, their widths 32, 24, 16 and 8 (unrolled over 32 columns the code would not stay
// in the instruction cache).  Per column, every row's entry of that column is in shared memory; each warp
// searches all of them and takes the reciprocal itself, while the pivot row's thread writes its row
// out: one round of warp reductions and two short barriers (a search per warp and then one among the
// warps took as long at b = 64 and 3% longer at b = 128).  Multipliers go to sm.Pan at the row's own place, pivot rows to
// sm.U.  The pivot of a column is the largest |re| + |im|, the lowest logical row on ties.
// A warp of its own (unit_lower_rows) follows with the inverse of the unit lower top block, whose row c
// needs no more than the pivot row of column c.
// The steps after which that warp may go on; each has a named barrier of its own (2 ..), on which the
// panel's warps only arrive, so that it may lag behind them.
constexpr unsigned kHelperSteps = 1u << 7 | 1u << 15 | 1u << 19 | 1u << 23 | 1u << 25 | 1u << 27 | 1u << 29 | 1u << 30 |
                                  1u << 31;
__device__ __forceinline__ int helper_barrier(int c) { return 2 + __popc(kHelperSteps & ((1u << c) - 1)); }
__device__ __forceinline__ void helper_arrive(int c, int nthreads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(helper_barrier(c)), "r"(nthreads) : "memory");
}
__device__ __forceinline__ void panel_barrier(int nthreads) {
  asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
}
// order-preserving key of a candidate pivot (0: a row that is done, or NaN; > 1: a positive pivot)
__device__ __forceinline__ unsigned candidate_key(float2 a, bool active) {
  const float v = cabs1(a);
  return active && v == v ? __float_as_uint(v) + 1 : 0u;
}
constexpr int kURow = kTile + 2;  // a pivot row in sm.U, from its column on: 16-byte words
// NQ: rows / 32, at most
template <int W, int NQ>
__device__ __forceinline__ void panel_stage(float2 (&w)[kTile], int& mylog, int nwp, int ldp,
                                            const FactorSmem<float2>& sm, int64_t k0, int64_t n, int* sh_status,
                                            int32_t* ipiv) {
  constexpr int T = kTile;
  const int tid = threadIdx.x, lane = tid & 31;
#pragma unroll 1
  for (int c = T - W; c < T - W + 8; ++c) {
    const unsigned* keys = sm.key + (c & 1) * kRowsMax;
    panel_barrier(nwp * 32);
    unsigned k[NQ], key = 0;
#pragma unroll
    for (int q = 0; q < NQ; ++q) k[q] = keys[q * 32 + lane];  // (0 past the last row)
#pragma unroll
    for (int q = 0; q < NQ; ++q) key = max(key, k[q]);
    const unsigned best = __reduce_max_sync(0xffffffffu, key);
    unsigned hits = 0;
#pragma unroll
    for (int q = 0; q < NQ; ++q) hits |= (k[q] == best ? 1u : 0u) << q;
    int r = 32 * (__ffs(hits) - 1) + lane;
    unsigned who = __ballot_sync(0xffffffffu, hits != 0);
    if (__ballot_sync(0xffffffffu, (hits & (hits - 1)) != 0) | (who & (who - 1))) {  // equal keys: the lowest logical row
      int lg = 0x7fffffff;
#pragma unroll 1
      for (int q = 0; q < nwp; ++q) {
        const int l = sm.log[q * 32 + lane];
        if (keys[q * 32 + lane] == best && l >= c && l < lg) {
          lg = l;
          r = q * 32 + lane;
        }
      }
      who = __ballot_sync(0xffffffffu, lg == __reduce_min_sync(0xffffffffu, lg));
    }
    r = __shfl_sync(0xffffffffu, r, __ffs(who) - 1);  // the pivot row (nothing but NaN: row c, no interchange)
    if (tid == r) {
#pragma unroll
      for (int q = 0; q < W; q += 2)
        *(float4*)&sm.U[c * kURow + q] = make_float4(w[q].x, w[q].y, w[q + 1].x, w[q + 1].y);
      sm.win[c] = r;
    }
    const float2 a = sm.col[(c & 1) * kRowsMax + r];
    const int p = sm.log[r];
    const bool ok = best > 1;  // a positive pivot
    // 1 / a with Smith's scaling (crecip), the parts' divisions in lanes 0 and 1
    const bool big = fabsf(a.x) >= fabsf(a.y);
    const float rr = (big ? a.y : a.x) / (big ? a.x : a.y);
    const float den = big ? fmaf(a.y, rr, a.x) : fmaf(a.x, rr, a.y);
    const float q2 = (lane == 0 ? (big ? 1.f : rr) : (big ? -rr : -1.f)) / den;
    const float2 inv = make_float2(__shfl_sync(0xffffffffu, q2, 0), __shfl_sync(0xffffffffu, q2, 1));
    const int nlog = mylog == p ? c : (mylog == c ? p : mylog);
    const int nx = ((c + 1) & 1) * kRowsMax + tid;
    panel_barrier(nwp * 32);
    const float2* u = sm.U + c * kURow;
    if (ok) {
      const float2 l = cmul_rn(w[0], inv);
      w[0] = w[1];
      cfms(w[0], l, u[1]);
      sm.key[nx] = candidate_key(w[0], nlog > c);
      sm.col[nx] = w[0];
      sm.Pan[tid + c * ldp] = l;
#pragma unroll
      for (int q = 2; q < W; q += 2) {
        const float4 v = *(const float4*)&u[q];
        w[q - 1] = w[q];
        cfms(w[q - 1], l, make_float2(v.x, v.y));
        w[q] = w[q + 1 < W ? q + 1 : q];
        cfms(w[q], l, make_float2(v.z, v.w));
      }
    } else {
      sm.Pan[tid + c * ldp] = w[0];
#pragma unroll
      for (int q = 0; q < W - 1; ++q) w[q] = w[q + 1];
      sm.key[nx] = candidate_key(w[0], nlog > c);
      sm.col[nx] = w[0];
      if (tid == 0 && *sh_status == 0) *sh_status = (int)(k0 + c + 1);
    }
    if (nlog != mylog) sm.log[tid] = nlog;
    mylog = nlog;
    if ((kHelperSteps >> c) & 1u) helper_arrive(c, nwp * 32 + 32);
    if (ipiv && tid == 0 && k0 + c < n) ipiv[k0 + c] = (int32_t)(k0 + p);
  }
}

// Rows of the inverse X of the unit lower top block, those up to column c once the panel's warps have
// passed step c of kHelperSteps: lane = column, X(c, j) = -sum_{k=j}^{c-1} L(c, k) X(k, j), terms in
// ascending k.
__device__ __forceinline__ void unit_lower_rows(int nwp, int ldp, const FactorSmem<float2>& sm) {
  constexpr int T = kTile;
  const int j = threadIdx.x & 31;
  int c = 0;
  for (int e = 0; e < T; ++e) {
    if (!((kHelperSteps >> e) & 1u)) continue;
    asm volatile("bar.sync %0, %1;" ::"r"(helper_barrier(e)), "r"(nwp * 32 + 32) : "memory");
    for (; c <= e; ++c) {
      const float2* L = sm.Pan + sm.win[c];
      float2 s = make_float2(0.f, 0.f);
#pragma unroll 8
      for (int k = 0; k < c; ++k) {
        const float2 a = L[k * ldp], x = sm.Li[k * (T + 1) + j];
        if (k >= j) cfma(s, a, x);
      }
      sm.Li[c * (T + 1) + j] = j == c ? make_float2(1.f, 0.f) : j < c ? make_float2(-s.x, -s.y) : make_float2(0.f, 0.f);
      __syncwarp();
    }
  }
}

template <int NQ>
__device__ void panel_lu_rows(const FactorGeom& g, const FactorPtr<float2>& f, int K, const FactorSmem<float2>& sm,
                              int* sh_status, int32_t* ipiv) {
  constexpr int T = kTile;
  const int tid = threadIdx.x;
  const int nbb = min(g.bt, g.Nb - 1 - K);
  const int P = (nbb + 1) * T, Pmax = (g.bt + 1) * T, ldp = Pmax + 1, nwp = P / 32;
  if (tid < P) {
    float2 w[T];
    const float2* src = f.tiles + g.tile_index(K + tid / T, K) * g.tile_elems + (tid & (T - 1));
#pragma unroll
    for (int i = 0; i < T; ++i) w[i] = src[i * T];
    int mylog = tid;
    sm.log[tid] = tid;
    sm.col[tid] = w[0];
    sm.key[tid] = candidate_key(w[0], true);
    for (int q = nwp; q < NQ; ++q)  // no rows here
      if (tid < 32) sm.key[q * 32 + tid] = sm.key[kRowsMax + q * 32 + tid] = 0;
    const int64_t k0 = (int64_t)K * T;
    panel_stage<32, NQ>(w, mylog, nwp, ldp, sm, k0, g.n, sh_status, ipiv);
    panel_stage<24, NQ>(w, mylog, nwp, ldp, sm, k0, g.n, sh_status, ipiv);
    panel_stage<16, NQ>(w, mylog, nwp, ldp, sm, k0, g.n, sh_status, ipiv);
    panel_stage<8, NQ>(w, mylog, nwp, ldp, sm, k0, g.n, sh_status, ipiv);
    sm.perm[mylog] = tid;
  } else if (tid < P + 32) {
    unit_lower_rows(nwp, ldp, sm);
  }
  __syncthreads();
}
// ... and its results to global memory (L\U of the top block, L below, in logical row order; the inverse of
// the unit lower block; the permutation), with every thread of the CTA
__device__ void store_panel_rows(const FactorGeom& g, const FactorPtr<float2>& f, int K,
                                 const FactorSmem<float2>& sm) {
  constexpr int T = kTile;
  const int nbb = min(g.bt, g.Nb - 1 - K);
  const int P = (nbb + 1) * T, Pmax = (g.bt + 1) * T, ldp = Pmax + 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  float2* li = f.inv + (int64_t)(2 * K) * g.tile_elems + lane;
  for (int c = warp; c < T; c += nw) li[c * T] = sm.Li[lane * (T + 1) + c];
  for (int q = 0; q <= nbb; ++q) {
    const float2* L = sm.Pan + sm.perm[q * T + lane];
    float2* dst = f.tiles + g.tile_index(K + q, K) * g.tile_elems + lane;
#pragma unroll 4
    for (int c = warp; c < T; c += nw)
      dst[c * T] = q == 0 && lane <= c ? sm.U[lane * kURow + c - lane] : L[c * ldp];
  }
  int16_t* pg = f.perm + (int64_t)K * Pmax;
  for (int e = threadIdx.x; e < Pmax; e += blockDim.x) pg[e] = (int16_t)(e < P ? sm.perm[e] : e);
}

// Reciprocal of a pivot by one warp, its parts' divisions in two lanes at once (lane 0: re, lane 1: im).
// complex64 (Smith's form, whose bits the factors keep): two divisions in a row.
__device__ __forceinline__ float pivot_reciprocal(float2 a, int lane) {
  const bool big = fabsf(a.x) >= fabsf(a.y);
  const float lo = big ? a.y : a.x, hi = big ? a.x : a.y;
  const float r0 = lo / hi;
  return (lane == 0 ? (big ? 1.0f : r0) : (big ? -r0 : -1.0f)) / fmaf(lo, r0, hi);
}
// complex128: the same with the divisions in integers (conj(a) / |a|^2 with one division takes as long, the searcher
// being ahead, and has more error: at most 3.1 units of 2^-53 |1/a| against 1.6, 0.78 against 0.62 on average)
__device__ __forceinline__ double pivot_reciprocal(double2 a, int lane) {
  const bool big = ((unsigned long long)__double_as_longlong(a.x) << 1) >=
                   ((unsigned long long)__double_as_longlong(a.y) << 1);
  const double lo = big ? a.y : a.x, hi = big ? a.x : a.y;
  const double r0 = divide(lo, hi);
  return divide(lane == 0 ? (big ? 1.0 : r0) : (big ? -r0 : -1.0), fma(lo, r0, hi));
}

// The same with a row in PARTS threads: complex128, and complex64 panels of more than kRowsMax rows.
// FP64 issue bounds the complex128 panel (64 clocks a warp instruction and quadrant, so the row's entries can
// stay in shared memory for nothing); the search and the reciprocal of a column are integer work (quotient.cuh), as
// long again.  So the CTA's last warp searches the next column and takes its reciprocal while the others still
// apply the current one: a warp has 32 rows (lane = row, where it was) and every PARTS-th column after
// the current one, the first of them before the rest, with the keys of its entries.  Two named barriers carry
// this: kKeys (the next column's keys are there; arrivals only) and kPivot (so is its pivot).  The loops stay rolled.
// (With the rows in registers, eight unrolled bodies, a search per warp followed by one among the warps and
// FP64 divisions, a block column of b = 32 took 145 us, b = 128 282 us; now 81 and 182.
// The FP64 instructions of a column, 22 a warp on average and two warps a quadrant at b = 32, are 3.3k of its 4.8k clocks.)
// Results in sm.Pan (logical row order) / sm.perm and in global memory.
template <typename C, int PARTS>
__device__ void panel_lu_parts(const FactorGeom& g, const FactorPtr<C>& f, int K, const FactorSmem<C>& sm, int* sh_status,
                         int32_t* ipiv) {
  using R = typename real_of<C>::type;
  constexpr int T = kTile, kPivot = 1, kKeys = 2;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nbb = min(g.bt, g.Nb - 1 - K);
  const int P = (nbb + 1) * T, Pmax = (g.bt + 1) * T, ldp = Pmax + 1;
  const int part = warp / (nbb + 1), rg = warp - part * (nbb + 1), r = rg * T + lane;
  const bool searcher = warp == (int)(blockDim.x >> 5) - 1;
  const bool has = part < PARTS && !searcher;  // a short last panel leaves warps without rows
  C* W = sm.Pan + r;  // this row; column q at q ldp
  if (has) {
    const C* src = f.tiles + g.tile_index(K + rg, K) * g.tile_elems + lane;
#pragma unroll 4
    for (int q = part; q < T; q += PARTS) W[q * ldp] = src[q * T];
    if (part == 0) {
      sm.keys[r] = pivot_key(cabs1(W[0]));
      sm.logs[r] = r;
    }
  }
  int mylog = r;
  __syncthreads();
  if (searcher) {
#pragma unroll 1
    for (int c = 0; c < T; ++c) {
      if (c > 0) asm volatile("bar.sync %0, %1;" ::"n"(kKeys), "r"(P + 32) : "memory");
      // the largest key, the lowest logical row on ties
      const unsigned long long* kc = sm.keys + (c & 1) * Pmax;
      const int* lc = sm.logs + (c & 1) * Pmax;
      unsigned long long best = 0;
      int blog = 0x7fffffff, brow = 0;
      for (int x = lane; x < P; x += 32) {
        const unsigned long long k = kc[x];
        const int lg = lc[x];
        if (k > best || (k == best && k > 0 && lg < blog)) {
          best = k;
          blog = lg;
          brow = x;
        }
      }
      const unsigned long long m = warp_max_key<R>(best);
      unsigned who = __ballot_sync(0xffffffffu, best == m);
      if (who & (who - 1)) {
        const int p = __reduce_min_sync(0xffffffffu, best == m ? blog : 0x7fffffff);
        who = __ballot_sync(0xffffffffu, best == m && blog == p);
      }
      const int at = __ffs(who) - 1;
      const int rs = __shfl_sync(0xffffffffu, brow, at);
      const bool ok = m > 1;                                              // a positive pivot
      const int p = m == 0 ? c : __shfl_sync(0xffffffffu, blog, at);  // nothing but NaN: no interchange
      Pivot<C>* out = sm.pivot + (c & 1);
      if (ok) {
        const R q = pivot_reciprocal(sm.Pan[rs + c * ldp], lane);
        if (lane < 2) ((R*)&out->inv)[lane] = q;
      }
      if (lane == 0) {
        out->row = rs;
        out->log = p;
        out->ok = ok;
        const int64_t k = (int64_t)K * T + c;
        if (ipiv && k < g.n) ipiv[k] = (int32_t)((int64_t)K * T + p);
        if (!ok && *sh_status == 0) *sh_status = (int)(k + 1);
      }
      asm volatile("bar.arrive %0, %1;" ::"n"(kPivot), "r"(P * PARTS + 32) : "memory");
    }
  } else if (has) {
    C l = cmk<C>(0, 0);
    bool done = false;  // l is the row's multiplier of the previous column, still to be stored
#pragma unroll 1
    for (int c = 0; c < T; ++c) {
      asm volatile("bar.sync %0, %1;" ::"n"(kPivot), "r"(P * PARTS + 32) : "memory");
      const Pivot<C> pv = sm.pivot[c & 1];
      if (part == 0 && done) W[(c - 1) * ldp] = l;  // (column c - 1 is read no more)
      const bool act = mylog >= c && mylog != pv.log;
      done = pv.ok && act;
      mylog = mylog == pv.log ? c : (mylog == c ? pv.log : mylog);
      const C* U = sm.Pan + pv.row;
      l = cmul_rn(W[c * ldp], pv.inv);
      int q = c + 1 + part;
      if (part == 0 && q < T) {  // the next column first, with its keys
        C x = W[q * ldp];
        if (done) {
          cfms(x, l, U[q * ldp]);
          W[q * ldp] = x;
        }
        sm.keys[((c + 1) & 1) * Pmax + r] = mylog > c ? pivot_key(cabs1(x)) : 0ull;
        sm.logs[((c + 1) & 1) * Pmax + r] = mylog;
        asm volatile("bar.arrive %0, %1;" ::"n"(kKeys), "r"(P + 32) : "memory");
        q += PARTS;
      }
      if (done) {
#pragma unroll 2
        for (; q < T; q += PARTS) {
          C x = W[q * ldp];
          cfms(x, l, U[q * ldp]);
          W[q * ldp] = x;
        }
      }
    }
    if (part == 0 && done) W[(T - 1) * ldp] = l;
  }
  // rows to their logical places
  C w[T / PARTS];
  __syncthreads();
  if (has) {
#pragma unroll
    for (int i = 0; i < T / PARTS; ++i) w[i] = W[(i * PARTS + part) * ldp];
  }
  __syncthreads();
  if (has) {
#pragma unroll
    for (int i = 0; i < T / PARTS; ++i) sm.Pan[mylog + (i * PARTS + part) * ldp] = w[i];
    if (part == 0) sm.perm[mylog] = r;
  }
  __syncthreads();
  for (int e = tid; e < P * T; e += blockDim.x) {
    const int q = e / (T * T), x = e % (T * T);
    f.tiles[g.tile_index(K + q, K) * g.tile_elems + x] = sm.Pan[q * T + x % T + (x / T) * ldp];
  }
  int16_t* pg = f.perm + (int64_t)K * Pmax;
  for (int e = tid; e < Pmax; e += blockDim.x) pg[e] = (int16_t)(e < P ? sm.perm[e] : e);
}

// Inverse of the panel's unit lower top block into sm.Li and global memory: lane = row, a warp takes
// 4 columns at a time; X(i, j) = -sum_{k=j}^{i-1} L(i, k) X(k, j), terms in ascending k, each X(k, j)
// passed on by a shuffle once it is final.
template <typename C>
__device__ void unit_lower_inverse(const FactorGeom& g, const FactorPtr<C>& f, int K, const FactorSmem<C>& sm) {
  using R = typename real_of<C>::type;
  constexpr int T = kTile;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int ldp = (g.bt + 1) * T + 1;
  const C* L = sm.Pan + lane;
  C* out = f.inv + (int64_t)(2 * K) * g.tile_elems;
  for (int j0 = 4 * warp; j0 < T; j0 += 4 * nw) {
    C s[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] = cmk<C>(0, 0);
#pragma unroll 4
    for (int k = 0; k < T - 1; ++k) {
      const C a = L[k * ldp];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        C x = shfl_c(s[q], k);
        x = k == j0 + q ? cmk<C>(R(1), R(0)) : cmk<C>(-x.x, -x.y);
        if (lane > k && k >= j0 + q) cfma(s[q], a, x);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = j0 + q;
      const C x = lane == j ? cmk<C>(R(1), R(0)) : (lane > j ? cmk<C>(-s[q].x, -s[q].y) : cmk<C>(0, 0));
      sm.Li[lane * (T + 1) + j] = x;
      out[lane + j * T] = x;
    }
  }
}

// Panel K applied to columns c0 .. c0+NC-1 of block column Jc by one warp: rows gathered through the
// panel's permutation, U(K, Jc) = L^{-1} (top rows), then rows below -= L U.
template <typename C, int NC, bool ROWS>
__device__ __forceinline__ void update_columns(const FactorGeom& g, const FactorPtr<C>& f, int K, int Jc, int c0,
                                               const FactorSmem<C>& sm) {
  constexpr int T = kTile;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nbb = min(g.bt, g.Nb - 1 - K);
  const int ldp = (g.bt + 1) * T + 1;
  C* top = sm.top + (size_t)warp * 2 * NC * T;  // the top block in use
  C* raw = top + NC * T;                        // the top rows before the permutation
  auto at = [&](int row, int c) -> C* {  // window row `row` of the block column
    return f.tiles + g.tile_index(K + (row >> 5), Jc) * g.tile_elems + (row & 31) + c * T;
  };
  // A row below the top block is either where it was or an old top row (interchanges bring rows up
  // only as pivots), so only old top rows are read after their place is written: from `raw`.
  auto request = [&](int q, int sr, C (&v)[NC]) {
    if (sr >= T) {
#pragma unroll
      for (int j = 0; j < NC; ++j) v[j] = *at(sr, c0 + j);
    }
  };
  auto complete = [&](int sr, C (&v)[NC]) {
    if (sr < T) {
#pragma unroll
      for (int j = 0; j < NC; ++j) v[j] = raw[j * T + sr];
    }
  };
  C x[NC], nx[NC];
  const int s0 = sm.perm[lane];
  int s1 = nbb > 0 ? sm.perm[T + lane] : 0;
  {
    C y[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) y[j] = *at(lane, c0 + j);
    request(0, s0, x);
    request(1, s1, nx);
#pragma unroll
    for (int j = 0; j < NC; ++j) raw[j * T + lane] = y[j];
  }
  __syncwarp();
  complete(s0, x);
  if constexpr (sizeof(C) == sizeof(float2)) {
#pragma unroll
    for (int j = 0; j < NC; ++j) top[j * T + lane] = x[j];
    __syncwarp();
#pragma unroll
    for (int j = 0; j < NC; ++j) x[j] = cmk<C>(0, 0);
#pragma unroll 4
    for (int k = 0; k < T; k += 2) {
      const C a0 = sm.Li[lane * (T + 1) + k], a1 = sm.Li[lane * (T + 1) + k + 1];
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        const float4 u = *(const float4*)&top[j * T + k];
        cfma(x[j], a0, cmk<C>(u.x, u.y));
        cfma(x[j], a1, cmk<C>(u.z, u.w));
      }
    }
    __syncwarp();
  } else {
    const C* L = sm.Pan + (ROWS ? s0 : lane);
    for (int k = 0; k < T - 1; ++k) {
      const C a = L[k * ldp];
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        const C u = shfl_c(x[j], k);
        C y = x[j];
        cfms(y, a, u);
        if (lane > k) x[j] = y;
      }
    }
  }
#pragma unroll
  for (int j = 0; j < NC; ++j) top[j * T + lane] = x[j];
  __syncwarp();
#pragma unroll
  for (int j = 0; j < NC; ++j) *at(lane, c0 + j) = x[j];
  for (int q = 1; q <= nbb; ++q) {
    const C* L = sm.Pan + (ROWS ? s1 : q * T + lane);
    complete(s1, nx);
    C acc[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) acc[j] = nx[j];
    if (q < nbb) {
      s1 = sm.perm[(q + 1) * T + lane];
      request(q + 1, s1, nx);
    }
    if constexpr (sizeof(C) == sizeof(float2)) {
#pragma unroll 4
      for (int k = 0; k < T; k += 2) {
        const C a0 = L[k * ldp], a1 = L[(k + 1) * ldp];
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          const float4 u = *(const float4*)&top[j * T + k];
          cfms(acc[j], a0, cmk<C>(u.x, u.y));
          cfms(acc[j], a1, cmk<C>(u.z, u.w));
        }
      }
    } else {
#pragma unroll 8
      for (int k = 0; k < T; ++k) {
        const C a = L[k * ldp];
#pragma unroll
        for (int j = 0; j < NC; ++j) cfms(acc[j], a, top[j * T + k]);
      }
    }
#pragma unroll
    for (int j = 0; j < NC; ++j) *at(q * T + lane, c0 + j) = acc[j];
  }
  __syncwarp();
}

// Columns [0, ncol) of the block columns from Jc0 on, in groups of NC, over the warps of `nc` CTAs.
template <typename C, int NC, bool ROWS>
__device__ __forceinline__ void update_range(const FactorGeom& g, const FactorPtr<C>& f, int K, int Jc0, int ncol,
                                             int cta, int nc, const FactorSmem<C>& sm) {
  const int nw = blockDim.x >> 5;
  for (int u = cta + nc * (int)(threadIdx.x >> 5); u * NC < ncol; u += nc * nw)
    update_columns<C, NC, ROWS>(g, f, K, Jc0 + u * NC / kTile, (u * NC) % kTile, sm);
}

// PARTS: 0 for panel_lu_rows (-1: of more than 160 rows), else the threads of a row; NCF: columns a warp takes at once in the next
// block column, NC: in the others; MAXT: the largest CTA; MINB: CTAs that share an SM.
template <typename C, int PARTS, int NCF, int NC, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
    factor_kernel(FactorGeom g, const SysDesc* sys, char* arena, int* status, int32_t* ipiv, int spread) {
  extern __shared__ __align__(16) char smem[];
  __shared__ int sh_status;
  constexpr int T = kTile, NCM = NCF > NC ? NCF : NC;
  constexpr bool ROWS = PARTS <= 0;
  cg::cluster_group cl = cg::this_cluster();
  const int G = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int sidx = blockIdx.x / G;
  const SysDesc d = sys[sidx];
  const FactorPtr<C> f = factor_ptr<C>(g, arena + d.factor_off);
  const int Pmax = (g.bt + 1) * T, ldp = Pmax + 1, nw = blockDim.x >> 5;
  auto align16 = [](void* p) { return (void*)(((uintptr_t)p + 15) & ~(uintptr_t)15); };
  FactorSmem<C> sm;
  sm.top = (C*)smem;  // first: read as 16-byte words
  sm.Li = sm.top + (size_t)nw * 2 * NCM * T;
  sm.Pan = sm.Li + T * (T + 1);
  if constexpr (ROWS) {
    sm.U = (C*)align16(sm.Pan + (size_t)T * ldp);
    sm.col = sm.U + T * (T + 2);
    sm.key = (unsigned*)(sm.col + 2 * kRowsMax);
    sm.log = (int*)(sm.key + 2 * kRowsMax);
    sm.win = sm.log + kRowsMax;
    sm.perm = sm.win + T;
  } else {
    sm.pivot = (Pivot<C>*)align16(sm.Pan + (size_t)T * ldp);
    sm.keys = (unsigned long long*)(sm.pivot + 2);
    sm.logs = (int*)(sm.keys + 2 * Pmax);
    sm.perm = sm.logs + 2 * Pmax;
  }
  int32_t* piv = ipiv ? ipiv + (int64_t)sidx * g.n : nullptr;
  if (threadIdx.x == 0) sh_status = 0;
  __syncthreads();
  auto panel = [&](int K) {
    if constexpr (ROWS) {
      panel_lu_rows<(PARTS < 0 ? 8 : 5)>(g, f, K, sm, &sh_status, piv);
      store_panel_rows(g, f, K, sm);
    } else {
      panel_lu_parts<C, PARTS>(g, f, K, sm, &sh_status, piv);
      if (sizeof(C) == sizeof(float2)) unit_lower_inverse<C>(g, f, K, sm);
    }
  };
  auto csync = [&]() {
    if (G > 1)
      cl.sync();
    else
      __syncthreads();
  };
  if (rank == 0) panel(0);
  csync();
  for (int K = 0; K < g.Nb - 1; ++K) {
    const int nbb = min(g.bt, g.Nb - 1 - K), nbr = min(2 * g.bt, g.Nb - 1 - K);
    const int P = (nbb + 1) * T;
    if (rank != 0) {  // CTA 0 holds the panel already
      const int16_t* pg = f.perm + (int64_t)K * Pmax;
      for (int e = threadIdx.x; e < P; e += blockDim.x) sm.perm[e] = pg[e];
      const int lane = threadIdx.x & 31;
      for (int q = 0; q <= nbb; ++q) {
        const C* src = f.tiles + g.tile_index(K + q, K) * g.tile_elems + lane;
        C* dst = sm.Pan + (ROWS ? (int)pg[q * T + lane] : q * T + lane);
        for (int c = threadIdx.x >> 5; c < T; c += nw) dst[c * ldp] = src[c * T];
      }
      if (sizeof(C) == sizeof(float2)) {
        const C* li = f.inv + (int64_t)(2 * K) * g.tile_elems;
        for (int c = threadIdx.x >> 5; c < T; c += nw) sm.Li[lane * (T + 1) + c] = li[lane + c * T];
      }
      __syncthreads();
    }
    if (spread) {
      update_range<C, NCF, ROWS>(g, f, K, K + 1, T, rank, G, sm);
      csync();
    } else if (rank == 0) {
      update_range<C, NCF, ROWS>(g, f, K, K + 1, T, 0, 1, sm);
      __syncthreads();
    }
    if (G == 1 || rank != 0)
      update_range<C, NC, ROWS>(g, f, K, K + 2, (nbr - 1) * T, G == 1 ? 0 : rank - 1, G == 1 ? 1 : G - 1, sm);
    if (G == 1) __syncthreads();
    if (rank == 0) panel(K + 1);
    csync();
  }
  if (rank == 0 && threadIdx.x == 0) status[sidx] = sh_status;
}

// Inverses of the diagonal blocks, one warp per block and system, lane = column: Uinv of the upper
// triangle and, in FP64, Linv of the unit lower one.
template <typename C>
__global__ void __launch_bounds__(64) diag_inverse_kernel(FactorGeom g, const SysDesc* sys, char* arena) {
  using R = typename real_of<C>::type;
  constexpr int T = kTile;
  __shared__ C D[T * T];   // the packed diagonal block, element (r, c) at r + c T
  __shared__ C X[2][T * T];
  const int K = blockIdx.x, lane = threadIdx.x & 31, which = threadIdx.x >> 5;
  const FactorPtr<C> f = factor_ptr<C>(g, arena + sys[blockIdx.y].factor_off);
  const C* src = f.tiles + g.tile_index(K, K) * g.tile_elems;
  for (int e = threadIdx.x; e < T * T; e += blockDim.x) D[e] = src[e];
  __syncthreads();
  const int j = lane;
  if (which == 0) {
    C* U = X[0];
    U[(T - 1) * T + j] = j == T - 1 ? crecip(D[j + j * T]) : cmk<C>(0, 0);
    for (int i = T - 2; i >= 0; --i) {
      C s = cmk<C>(0, 0);
#pragma unroll 4
      for (int k = i + 1; k < T; ++k)
        if (k <= j) cfma(s, D[i + k * T], U[k * T + j]);
      const C ri = crecip(D[i + i * T]);
      const C u = cmul_rn(cmk<C>(s.x, s.y), ri);  // real part of s ri; the imaginary part below
      U[i * T + j] = i == j ? ri : i > j ? cmk<C>(0, 0) : cmk<C>(-u.x, -fma(s.y, ri.x, mul_rn(s.x, ri.y)));
    }
  } else if (sizeof(C) == sizeof(double2)) {
    C* L = X[1];
    for (int i = 0; i < T; ++i) {
      C s = cmk<C>(0, 0);
#pragma unroll 4
      for (int k = 0; k < i; ++k)
        if (k >= j) cfma(s, D[i + k * T], L[k * T + j]);
      L[i * T + j] = i == j ? cmk<C>(R(1), R(0)) : i < j ? cmk<C>(0, 0) : cmk<C>(-s.x, -s.y);
    }
  }
  __syncthreads();
  C* ui = f.inv + (int64_t)(2 * K + 1) * g.tile_elems;
  C* li = f.inv + (int64_t)(2 * K) * g.tile_elems;
  for (int e = threadIdx.x; e < T * T; e += blockDim.x) {
    ui[e] = X[0][(e % T) * T + e / T];
    if (sizeof(C) == sizeof(double2)) li[e] = X[1][(e % T) * T + e / T];
  }
}

// ---------------------------------------------------------------------------
// solve helpers.  A solve block covers CW right-hand sides with 8 warps: lane
// = row of a tile, warp w owns columns w + 8 jj, jj < NJ = CW / 8.
// ---------------------------------------------------------------------------
// Load one T x T tile into Tb (ld kLdt); conjugate-transposed if CT.
template <typename C, bool CT>
__device__ __forceinline__ void load_tile(C* Tb, const C* __restrict__ src) {
  for (int e = threadIdx.x; e < kTile * kTile; e += blockDim.x) {
    const int r = e % kTile, c = e / kTile;
    const C v = src[e];
    if (CT)
      Tb[c + r * kLdt] = cconj(v);
    else
      Tb[r + c * kLdt] = v;
  }
}

// acc[jj] += / -= Tb(lane, :) * Bm(:, col_jj), Bm with leading dimension ldb.
template <typename C, int NJ, bool SUB>
__device__ __forceinline__ void tile_mul(C acc[NJ], const C* Tb, const C* Bm, int ldb) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll 8
  for (int k = 0; k < kTile; ++k) {
    const C a = Tb[lane + k * kLdt];
#pragma unroll
    for (int jj = 0; jj < NJ; ++jj) {
      const C bv = Bm[k + (warp + 8 * jj) * ldb];
      if (SUB)
        cfms(acc[jj], a, bv);
      else
        cfma(acc[jj], a, bv);
    }
  }
}

template <typename C, int NJ>
__device__ __forceinline__ void load_rhs_block(C* dst, int ldd, const C* __restrict__ Y, int64_t n,
                                               int64_t row0, int col0, int ncols) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int jj = 0; jj < NJ; ++jj) {
    const int c = warp + 8 * jj;
    const int64_t i = row0 + lane;
    C v = cmk<C>(0, 0);
    if (i < n && col0 + c < ncols) v = Y[i + (int64_t)(col0 + c) * n];
    dst[lane + c * ldd] = v;
  }
}

template <typename C, int NJ>
__device__ __forceinline__ void store_rows(C* __restrict__ X, int64_t n, int64_t row0, int col0,
                                           int ncols, const C acc[NJ]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int jj = 0; jj < NJ; ++jj) {
    const int c = warp + 8 * jj;
    const int64_t i = row0 + lane;
    if (i < n && col0 + c < ncols) X[i + (int64_t)(col0 + c) * n] = acc[jj];
  }
}

template <typename C, int NJ>
__device__ __forceinline__ void load_acc(C acc[NJ], const C* __restrict__ X, int64_t n, int64_t row0,
                                         int col0, int ncols) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int jj = 0; jj < NJ; ++jj) {
    const int c = warp + 8 * jj;
    const int64_t i = row0 + lane;
    acc[jj] = (i < n && col0 + c < ncols) ? X[i + (int64_t)(col0 + c) * n] : cmk<C>(0, 0);
  }
}

template <typename C, int NJ>
__device__ __forceinline__ void put_acc(C* dst, int ldd, const C acc[NJ]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int jj = 0; jj < NJ; ++jj) dst[lane + (warp + 8 * jj) * ldd] = acc[jj];
}

template <typename C, int NJ>
__device__ __forceinline__ void get_acc(C acc[NJ], const C* src, int lds) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int jj = 0; jj < NJ; ++jj) acc[jj] = src[lane + (warp + 8 * jj) * lds];
}

template <typename C, int NJ>
__device__ __forceinline__ void zero_acc(C acc[NJ]) {
#pragma unroll
  for (int jj = 0; jj < NJ; ++jj) acc[jj] = cmk<C>(0, 0);
}

// ---------------------------------------------------------------------------
// Factor tiles reach shared memory through a two-slot cp.async pipeline: the
// tile of the next step is requested before the current one is used, so its
// L2/HBM latency overlaps the current tile product.  Tiles keep their stored
// layout (element (r, c) at r + c kLdt); conjugate-transposed use reads them
// transposed (tile_mul_ct).
// ---------------------------------------------------------------------------
template <typename C>
__device__ __forceinline__ void cp_async_tile(C* dst, const C* __restrict__ src) {
  for (int e = threadIdx.x; e < kTile * kTile; e += blockDim.x) {
    const int r = e % kTile, c = e / kTile;
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst + r + c * kLdt);
    if constexpr (sizeof(C) == 8)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src + e));
    else
      asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src + e));
  }
  asm volatile("cp.async.commit_group;\n" ::);
}

// acc[jj] += / -= Tc(:, lane)^H-row times Bm: a = conj(Traw(k, lane))
template <typename C, int NJ, bool SUB>
__device__ __forceinline__ void tile_mul_ct(C acc[NJ], const C* Traw, const C* Bm, int ldb) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll 8
  for (int k = 0; k < kTile; ++k) {
    const C a = cconj(Traw[k + lane * kLdt]);
#pragma unroll
    for (int jj = 0; jj < NJ; ++jj) {
      const C bv = Bm[k + (warp + 8 * jj) * ldb];
      if (SUB)
        cfms(acc[jj], a, bv);
      else
        cfma(acc[jj], a, bv);
    }
  }
}

// Ordered tile requests of one sweep.  next() returns the source of the
// following request (nullptr after the last); acquire() starts the request
// after the current one, waits for the current one and returns its slot.
template <typename C>
struct TilePipe {
  C* slot[2];
  int cur = 0;
  const C* pending = nullptr;  // source of the request issued into slot[cur ^ 1]
  __device__ void start(const C* first, const C* second) {
    cur = 0;
    cp_async_tile(slot[0], first);
    pending = second;
    if (second) cp_async_tile(slot[1], second);
  }
  // current tile is ready on return; `after_next` is the request after the pending one
  __device__ C* acquire() {
    if (pending)
      asm volatile("cp.async.wait_group 1;\n" ::);
    else
      asm volatile("cp.async.wait_group 0;\n" ::);
    __syncthreads();
    return slot[cur];
  }
  // the current slot is free again (every thread is past its use): refill it
  __device__ void release(const C* after_next) {
    __syncthreads();
    cur ^= 1;
    const C* next = after_next;
    if (pending && next) cp_async_tile(slot[cur ^ 1], next);
    pending = pending ? next : nullptr;
  }
};

// Iterators over the tile requests of each sweep (same order as the sweeps).
struct SweepIt {
  int K, q;
};

// ---------------------------------------------------------------------------
// trans = 0: forward (P, L) then backward (U), for columns col0 .. col0+CW-1
// ---------------------------------------------------------------------------
template <typename C, int CW>
__device__ void solve_n_body(const FactorGeom& g, const SysDesc& d, int col0, const char* arena, const C* rhs,
                             C* out, char* smem) {
  constexpr int NJ = CW / 8;
  const int T = kTile, bt = g.bt;
  const int Pmax = (bt + 1) * T;
  const int ldw = Pmax;
  const FactorPtr<C> f = factor_ptr<C>(g, (char*)arena + d.factor_off);
  const C* Y = rhs + d.rhs_off;
  C* X = out + d.out_off;
  const int64_t n = g.n;
  const int ncols = d.ncols;
  const int tid = threadIdx.x;
  const int Nb = g.Nb;

  TilePipe<C> pipe;
  pipe.slot[0] = (C*)smem;                     // T x kLdt
  pipe.slot[1] = pipe.slot[0] + T * kLdt;      // T x kLdt
  C* tS = pipe.slot[1] + T * kLdt;             // T x CW
  C* U0 = tS + T * CW;                         // union area
  C* Wn = U0;                                  // Pmax x CW
  C* G = U0 + (size_t)Pmax * CW;               // Pmax x CW
  C* xwin = U0;                                // 2bt slots of T x CW

  // forward requests: per K, Linv(K) then L(K+q, K), q = 1..min(bt, Nb-1-K)
  auto fsrc = [&](SweepIt it) -> const C* {
    if (it.K >= Nb) return nullptr;
    return it.q == 0 ? f.inv + (int64_t)(2 * it.K) * g.tile_elems
                     : f.tiles + g.tile_index(it.K + it.q, it.K) * g.tile_elems;
  };
  auto fnext = [&](SweepIt it) -> SweepIt {
    if (it.q < min(bt, Nb - 1 - it.K)) return SweepIt{it.K, it.q + 1};
    return SweepIt{it.K + 1, 0};
  };
  // ---------------- forward ----------------
  {
    SweepIt it0{0, 0};
    SweepIt it1 = fnext(it0);
    SweepIt it2 = fnext(it1);
    pipe.start(fsrc(it0), fsrc(it1));
    const int nbb0 = min(bt, Nb - 1);
    for (int q = 0; q <= nbb0; ++q) load_rhs_block<C, NJ>(Wn + q * T, ldw, Y, n, (int64_t)q * T, col0, ncols);
    __syncthreads();
    for (int K = 0; K < Nb; ++K) {
      const int nbb = min(bt, Nb - 1 - K);
      const int P = (nbb + 1) * T;
      const int16_t* pm = f.perm + (int64_t)K * Pmax;
      for (int e = tid; e < P * CW; e += blockDim.x) {
        const int r = e % P, c = e / P;
        G[r + c * ldw] = Wn[pm[r] + c * ldw];
      }
      C* Tb = pipe.acquire();
      C acc[NJ];
      zero_acc<C, NJ>(acc);
      tile_mul<C, NJ, false>(acc, Tb, G, ldw);
      pipe.release(fsrc(it2));
      it2 = fnext(it2);
      put_acc<C, NJ>(G, ldw, acc);
      store_rows<C, NJ>(X, n, (int64_t)K * T, col0, ncols, acc);
      __syncthreads();
      for (int q = 1; q <= nbb; ++q) {
        Tb = pipe.acquire();
        get_acc<C, NJ>(acc, G + q * T, ldw);
        tile_mul<C, NJ, true>(acc, Tb, G, ldw);
        put_acc<C, NJ>(G + q * T, ldw, acc);
        pipe.release(fsrc(it2));
        it2 = fnext(it2);
      }
      if (K + 1 < Nb) {
        for (int e = tid; e < nbb * T * CW; e += blockDim.x) {
          const int r = e % (nbb * T), c = e / (nbb * T);
          Wn[r + c * ldw] = G[T + r + c * ldw];
        }
        const int nbn = min(bt, Nb - 2 - K);
        if (nbn == nbb)
          load_rhs_block<C, NJ>(Wn + nbb * T, ldw, Y, n, (int64_t)(K + bt + 1) * T, col0, ncols);
        __syncthreads();
      }
    }
  }
  // backward requests: per K (descending), U(K, K+q), q = 1..min(2bt, Nb-1-K), then Uinv(K)
  auto bsrc = [&](SweepIt it) -> const C* {
    if (it.K < 0) return nullptr;
    return it.q > 0 ? f.tiles + g.tile_index(it.K, it.K + it.q) * g.tile_elems
                    : f.inv + (int64_t)(2 * it.K + 1) * g.tile_elems;
  };
  auto bfirst = [&](int K) -> SweepIt { return SweepIt{K, min(2 * bt, Nb - 1 - K) > 0 ? 1 : 0}; };
  auto bnext = [&](SweepIt it) -> SweepIt {
    if (it.q > 0 && it.q < min(2 * bt, Nb - 1 - it.K)) return SweepIt{it.K, it.q + 1};
    if (it.q > 0) return SweepIt{it.K, 0};
    return it.K - 1 >= 0 ? bfirst(it.K - 1) : SweepIt{-1, 0};
  };
  // ---------------- backward ----------------
  {
    const int ns = 2 * bt;
    SweepIt it0 = bfirst(Nb - 1);
    SweepIt it1 = bnext(it0);
    SweepIt it2 = bnext(it1);
    pipe.start(bsrc(it0), bsrc(it1));
    for (int K = Nb - 1; K >= 0; --K) {
      const int nbr = min(2 * bt, Nb - 1 - K);
      C acc[NJ];
      load_acc<C, NJ>(acc, X, n, (int64_t)K * T, col0, ncols);
      for (int q = 1; q <= nbr; ++q) {
        C* Tb = pipe.acquire();
        tile_mul<C, NJ, true>(acc, Tb, xwin + ((K + q) % ns) * T * CW, T);
        pipe.release(bsrc(it2));
        it2 = bnext(it2);
      }
      put_acc<C, NJ>(tS, T, acc);
      C* Tb = pipe.acquire();
      zero_acc<C, NJ>(acc);
      tile_mul<C, NJ, false>(acc, Tb, tS, T);
      put_acc<C, NJ>(xwin + (K % ns) * T * CW, T, acc);
      store_rows<C, NJ>(X, n, (int64_t)K * T, col0, ncols, acc);
      pipe.release(bsrc(it2));
      it2 = bnext(it2);
    }
  }
}

// ---------------------------------------------------------------------------
// trans = 1: forward U^H, backward L^H then P^T
// ---------------------------------------------------------------------------
template <typename C, int CW>
__device__ void solve_c_body(const FactorGeom& g, const SysDesc& d, int col0, const char* arena, const C* rhs,
                             C* out, char* smem) {
  constexpr int NJ = CW / 8;
  const int T = kTile, bt = g.bt;
  const int Pmax = (bt + 1) * T;
  const int ldw = Pmax;
  const FactorPtr<C> f = factor_ptr<C>(g, (char*)arena + d.factor_off);
  const C* Y = rhs + d.rhs_off;
  C* X = out + d.out2_off;
  const int64_t n = g.n;
  const int ncols = d.ncols;
  const int tid = threadIdx.x;
  const int Nb = g.Nb;

  TilePipe<C> pipe;
  pipe.slot[0] = (C*)smem;
  pipe.slot[1] = pipe.slot[0] + T * kLdt;
  C* tS = pipe.slot[1] + T * kLdt;
  C* U0 = tS + T * CW;
  C* wwin = U0;                        // 2bt slots of T x CW
  C* V = U0;                           // Pmax x CW
  C* Vn = U0 + (size_t)Pmax * CW;      // Pmax x CW

  // forward requests: per K, U(K-q, K), q = 1..min(2bt, K), then Uinv(K)
  auto fsrc = [&](SweepIt it) -> const C* {
    if (it.K >= Nb) return nullptr;
    return it.q > 0 ? f.tiles + g.tile_index(it.K - it.q, it.K) * g.tile_elems
                    : f.inv + (int64_t)(2 * it.K + 1) * g.tile_elems;
  };
  auto ffirst = [&](int K) -> SweepIt { return SweepIt{K, min(2 * bt, K) > 0 ? 1 : 0}; };
  auto fnext = [&](SweepIt it) -> SweepIt {
    if (it.q > 0 && it.q < min(2 * bt, it.K)) return SweepIt{it.K, it.q + 1};
    if (it.q > 0) return SweepIt{it.K, 0};
    return ffirst(it.K + 1);
  };
  // ---------------- forward: U^H w = y ----------------
  {
    const int ns = 2 * bt;
    SweepIt it0 = ffirst(0);
    SweepIt it1 = fnext(it0);
    SweepIt it2 = fnext(it1);
    pipe.start(fsrc(it0), fsrc(it1));
    for (int K = 0; K < Nb; ++K) {
      C acc[NJ];
      load_acc<C, NJ>(acc, Y, n, (int64_t)K * T, col0, ncols);
      const int nq = min(2 * bt, K);
      for (int q = 1; q <= nq; ++q) {
        C* Tb = pipe.acquire();
        tile_mul_ct<C, NJ, true>(acc, Tb, wwin + ((K - q) % ns) * T * CW, T);
        pipe.release(fsrc(it2));
        it2 = fnext(it2);
      }
      put_acc<C, NJ>(tS, T, acc);
      C* Tb = pipe.acquire();
      zero_acc<C, NJ>(acc);
      tile_mul_ct<C, NJ, false>(acc, Tb, tS, T);
      put_acc<C, NJ>(wwin + (K % ns) * T * CW, T, acc);
      store_rows<C, NJ>(X, n, (int64_t)K * T, col0, ncols, acc);
      pipe.release(fsrc(it2));
      it2 = fnext(it2);
    }
  }
  // backward requests: per K (descending), L(K+q, K), q = 1..min(bt, Nb-1-K), then Linv(K)
  auto bsrc = [&](SweepIt it) -> const C* {
    if (it.K < 0) return nullptr;
    return it.q > 0 ? f.tiles + g.tile_index(it.K + it.q, it.K) * g.tile_elems
                    : f.inv + (int64_t)(2 * it.K) * g.tile_elems;
  };
  auto bfirst = [&](int K) -> SweepIt { return SweepIt{K, min(bt, Nb - 1 - K) > 0 ? 1 : 0}; };
  auto bnext = [&](SweepIt it) -> SweepIt {
    if (it.q > 0 && it.q < min(bt, Nb - 1 - it.K)) return SweepIt{it.K, it.q + 1};
    if (it.q > 0) return SweepIt{it.K, 0};
    return it.K - 1 >= 0 ? bfirst(it.K - 1) : SweepIt{-1, 0};
  };
  // ---------------- backward: x = P_0^T E_0^H ... P_{Nb-1}^T E_{Nb-1}^H w ----------------
  {
    SweepIt it0 = bfirst(Nb - 1);
    SweepIt it1 = bnext(it0);
    SweepIt it2 = bnext(it1);
    pipe.start(bsrc(it0), bsrc(it1));
    for (int K = Nb - 1; K >= 0; --K) {
      const int nbb = min(bt, Nb - 1 - K);
      const int P = (nbb + 1) * T;
      C acc[NJ];
      load_acc<C, NJ>(acc, X, n, (int64_t)K * T, col0, ncols);
      for (int q = 1; q <= nbb; ++q) {
        C* Tb = pipe.acquire();
        tile_mul_ct<C, NJ, true>(acc, Tb, V + q * T, ldw);
        pipe.release(bsrc(it2));
        it2 = bnext(it2);
      }
      put_acc<C, NJ>(tS, T, acc);
      C* Tb = pipe.acquire();
      zero_acc<C, NJ>(acc);
      tile_mul_ct<C, NJ, false>(acc, Tb, tS, T);
      pipe.release(bsrc(it2));
      it2 = bnext(it2);
      put_acc<C, NJ>(V, ldw, acc);
      __syncthreads();
      const int16_t* pm = f.perm + (int64_t)K * Pmax;
      for (int e = tid; e < P * CW; e += blockDim.x) {
        const int r = e % P, c = e / P;
        Vn[pm[r] + c * ldw] = V[r + c * ldw];
      }
      __syncthreads();
      if (nbb == bt) {
        // block K+bt is final
#pragma unroll
        for (int jj = 0; jj < NJ; ++jj) acc[jj] = Vn[bt * T + (tid & 31) + ((tid >> 5) + 8 * jj) * ldw];
        store_rows<C, NJ>(X, n, (int64_t)(K + bt) * T, col0, ncols, acc);
      }
      const int nbn = min(bt, Nb - K);  // window blocks kept for step K-1 (beyond its top block)
      for (int e = tid; e < nbn * T * CW; e += blockDim.x) {
        const int r = e % (nbn * T), c = e / (nbn * T);
        V[T + r + c * ldw] = Vn[r + c * ldw];
      }
      __syncthreads();
    }
    // remaining window blocks 0 .. min(bt, Nb)-1 sit in V[T : ...]
    const int nrem = min(bt, Nb);
    for (int q = 0; q < nrem; ++q) {
      C acc[NJ];
#pragma unroll
      for (int jj = 0; jj < NJ; ++jj) acc[jj] = V[T + q * T + (tid & 31) + ((tid >> 5) + 8 * jj) * ldw];
      store_rows<C, NJ>(X, n, (int64_t)q * T, col0, ncols, acc);
    }
  }
}

// Persistent solve: the grid holds as many blocks as fit on the GPU at once;
// each block takes (system, column block) items from a shared counter until
// the list is exhausted, so systems of uneven m0 keep every SM busy.  A column
// block of 8 (complex128) takes the items of 16 columns in halves.
template <typename C, int CW, int TRANS>
__global__ void __launch_bounds__(kThreads) solve_kernel(FactorGeom g, const SysDesc* sys, const char* arena,
                                                        const C* rhs, C* out, const int2* items, int nitems,
                                                        int* counter) {
  extern __shared__ __align__(16) char smem[];
  __shared__ int sh_item;
  for (;;) {
    if (threadIdx.x == 0) sh_item = atomicAdd(counter, 1);
    __syncthreads();
    const int item = sh_item;
    __syncthreads();  // every thread has its item before thread 0 fetches the next one
    if (item >= nitems) return;
    int2 w = items[CW == 8 ? item >> 1 : item];
    if (CW == 8) w.y += 8 * (item & 1);
    const SysDesc d = sys[w.x];
    if (w.y >= d.ncols) continue;  // (the same for every thread)
    if (TRANS == 0)
      solve_n_body<C, CW>(g, d, w.y, arena, rhs, out, smem);
    else
      solve_c_body<C, CW>(g, d, w.y, arena, rhs, out, smem);
    __syncthreads();
  }
}

size_t solve_smem_bytes(const FactorGeom& g, int chunk, size_t es, int trans) {
  (void)trans;
  const int T = kTile;
  const size_t Pmax = (size_t)(g.bt + 1) * T;
  size_t uni = 2 * Pmax * (size_t)chunk;
  size_t win = (size_t)2 * g.bt * T * chunk;
  if (win > uni) uni = win;
  return es * ((size_t)2 * T * kLdt + (size_t)T * chunk + uni);  // two tile slots
}

// The widest band the factorization takes (the shared memory of two panels, their
// permutations and the diagonal inverses; what the callers' workspaces were planned for).
static bool factor_band_ok(const FactorGeom& g, size_t es) {
  const size_t Pmax = (size_t)(g.bt + 1) * kTile;
  return es * (2 * (Pmax + 1) * kTile + 2 * (size_t)kTile * kTile) + sizeof(int) * 3 * Pmax <= 227 * 1024;
}

template <typename C, int PARTS, int NCF, int NC, int MAXT, int MINB>
static int launch_factor_cluster(const FactorGeom& g, int G, int spread, int nsys, const SysDesc* d_sys,
                                 char* factor_arena, int* d_status, int32_t* d_ipiv, cudaStream_t st) {
  const int Pmax = (g.bt + 1) * kTile, threads = PARTS > 0 ? Pmax * PARTS + 32 : MAXT;
  const size_t smem = factor_cluster_smem<C, (PARTS <= 0)>(Pmax, threads / 32, NCF > NC ? NCF : NC);
  auto kern = factor_kernel<C, PARTS, NCF, NC, MAXT, MINB>;
  PD_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  if (G > 8) PD_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)nsys * (unsigned)G);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = G;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  PD_CK(cudaLaunchKernelEx(&cfg, kern, g, d_sys, factor_arena, d_status, d_ipiv, spread));
  count_launch();
  return 0;
}

template <typename C>
int launch_factor(const FactorGeom& g, int cplx, const void* band, int64_t ldab, int nsys,
                  const SysDesc* d_sys, char* factor_arena, int* d_status, int32_t* d_ipiv,
                  cudaStream_t st) {
  if (nsys <= 0) return 0;
  dim3 gi((unsigned)(g.tiles < 4096 ? g.tiles : 4096), (unsigned)nsys);
  init_factor_kernel<C><<<gi, kThreads, 0, st>>>(g, cplx, (const double*)band, ldab, d_sys, factor_arena);
  PD_CK_LAUNCH();
  if (!factor_band_ok(g, sizeof(C))) {
    set_last_error_msg("band too wide for the factor kernel's shared memory");
    return PDESHEP_CUDA_ERROR;
  }
  // The cluster: as many CTAs as still shorten a block column, while all clusters run at once (76, 36
  // and 15 clusters of 2, 4 and 8 fit at one CTA per SM).  complex64: a second CTA takes the updates off
  // the panel's chain (b = 64: 34 -> 24.5 us per block column), at b > 64 four (68, 44, 30 us for 1, 2, 4);
  // more change nothing.  complex128: every CTA shortens the updates (b = 32: 203, 106, 87, 81 us for 1 to 8;
  // b = 128: 1316, 1117, 399, 183).
  const int most = sizeof(C) == sizeof(double2) ? 8 : g.bt > 2 ? 4 : 2;
  const int G = most >= 8 && nsys <= 15 ? 8 : most >= 4 && nsys <= 36 ? 4 : nsys <= 76 ? 2 : 1;
  if constexpr (sizeof(C) == sizeof(float2)) {
    if ((g.bt + 1) * kTile > kRowsMax)
      PD_TRY((launch_factor_cluster<C, 2, 2, 2, 832, 1>(g, G, 0, nsys, d_sys, factor_arena, d_status, d_ipiv, st)));
    else if ((g.bt + 1) * kTile > 160)
      PD_TRY((launch_factor_cluster<C, -1, 4, 4, 288, 1>(g, G, 0, nsys, d_sys, factor_arena, d_status, d_ipiv, st)));
    else if (nsys <= 152)
      PD_TRY((launch_factor_cluster<C, 0, 4, 4, 256, 1>(g, G, 0, nsys, d_sys, factor_arena, d_status, d_ipiv, st)));
    else  // more systems than SMs: two per SM, with some registers spilled (256 systems, b = 64: 54 against 70 us)
      PD_TRY((launch_factor_cluster<C, 0, 4, 4, 256, 2>(g, G, 0, nsys, d_sys, factor_arena, d_status, d_ipiv, st)));
  } else {
    PD_TRY((launch_factor_cluster<C, 4, 1, 1, 672, 1>(g, G, G > 1, nsys, d_sys, factor_arena, d_status, d_ipiv, st)));
  }
  diag_inverse_kernel<C><<<dim3((unsigned)g.Nb, (unsigned)nsys), 64, 0, st>>>(g, d_sys, factor_arena);
  PD_CK_LAUNCH();
  return 0;
}

// Scratch of the solve work queue for nsys systems of at most max_cols
// right-hand sides (enough for the narrowest column block, 16).
size_t solve_queue_bytes(int nsys, int max_cols) {
  Arena a;
  a.take<int>(1);
  a.take<int2>((size_t)nsys * ceil_div(max_cols, 16));
  return a.used();
}

// Work list of (system, first column) items of `chunk` right-hand sides into
// the queue scratch (counter first, then the items).  Returns the item count.
int upload_solve_items(int nsys, const SysDesc* h_sys, int chunk, void* queue, cudaStream_t st, int* nitems) {
  if (chunk == kTcChunk) chunk = kTmChunk;  // the tensor-core solve also takes 128 right-hand sides per item
  if (chunk == 8) chunk = 16;               // halves of 16-column items
  std::vector<int2> it;
  for (int s = 0; s < nsys; ++s)
    for (int c = 0; c < h_sys[s].ncols; c += chunk) it.push_back(make_int2(s, c));
  *nitems = (int)it.size();
  if (it.empty()) return 0;
  Arena qa(queue, ~size_t(0));
  qa.take<int>(1);
  int2* d_items = qa.take<int2>(it.size());
  PD_CK(cudaMemcpyAsync(d_items, it.data(), sizeof(int2) * it.size(), cudaMemcpyHostToDevice, st));
  return 0;
}

template <typename C, int CW, int TRANS>
static int launch_solve_cw(const FactorGeom& g, int nitems, const SysDesc* d_sys, const char* factor_arena,
                           const C* rhs_arena, C* out_arena, void* queue, cudaStream_t st) {
  const size_t smem = solve_smem_bytes(g, CW, sizeof(C), TRANS);
  if (smem > 227 * 1024) {
    set_last_error_msg("band too wide for the solve kernel's shared memory at this column block");
    return PDESHEP_CUDA_ERROR;
  }
  if (!nitems) return 0;
  Arena qa(queue, ~size_t(0));
  int* counter = qa.take<int>(1);
  const int2* d_items = qa.take<int2>((size_t)nitems);
  if (CW == 8) nitems *= 2;
  auto kern = solve_kernel<C, CW, TRANS>;
  PD_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = 0, dev = 0, sms = 0;
  PD_CK(cudaGetDevice(&dev));
  PD_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  PD_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, smem));
  // complex128: no more blocks on an SM than every SM has items for.  One fills the FP64 pipes, and with a block
  // per item some SMs took two at once while others had none (152 items among 160 halves, b = 32, n = 2000:
  // 5.05 ms, now 2.7).  complex64 blocks hide one another's latency.
  if (std::is_same<C, double2>::value) per_sm = std::min(per_sm, std::max(1, nitems / sms));
  const int grid = std::max(1, std::min(nitems, sms * std::max(1, per_sm)));
  PD_CK(cudaMemsetAsync(counter, 0, sizeof(int), st));
  kern<<<grid, kThreads, smem, st>>>(g, d_sys, factor_arena, rhs_arena, out_arena, d_items, nitems, counter);
  PD_CK_LAUNCH();
  return 0;
}

template <typename C>
int launch_solve_queued(const FactorGeom& g, int trans, int nitems, const SysDesc* d_sys, const char* factor_arena,
                        const C* rhs_arena, C* out_arena, int chunk, void* queue, cudaStream_t st) {
  if (chunk == kTmChunk || chunk == kTcChunk) {
    if constexpr (std::is_same<C, float2>::value) {
      if (chunk == kTcChunk)
        return launch_solve_tc(g, trans, nitems, d_sys, factor_arena, rhs_arena, out_arena, queue, st);
      return launch_solve_tm(g, trans, nitems, d_sys, factor_arena, rhs_arena, out_arena, queue, st);
    }
    set_last_error_msg("the tensor-memory and tensor-core solves are complex64 only");
    return PDESHEP_CUDA_ERROR;
  }
  if constexpr (std::is_same<C, double2>::value) {
    if (chunk == 8)
      return trans ? launch_solve_cw<C, 8, 1>(g, nitems, d_sys, factor_arena, rhs_arena, out_arena, queue, st)
                   : launch_solve_cw<C, 8, 0>(g, nitems, d_sys, factor_arena, rhs_arena, out_arena, queue, st);
  }
  switch (chunk * 2 + (trans ? 1 : 0)) {
    case 32: return launch_solve_cw<C, 16, 0>(g, nitems, d_sys, factor_arena, rhs_arena, out_arena, queue, st);
    case 33: return launch_solve_cw<C, 16, 1>(g, nitems, d_sys, factor_arena, rhs_arena, out_arena, queue, st);
    case 64: return launch_solve_cw<C, 32, 0>(g, nitems, d_sys, factor_arena, rhs_arena, out_arena, queue, st);
    case 65: return launch_solve_cw<C, 32, 1>(g, nitems, d_sys, factor_arena, rhs_arena, out_arena, queue, st);
    case 128: return launch_solve_cw<C, 64, 0>(g, nitems, d_sys, factor_arena, rhs_arena, out_arena, queue, st);
    case 129: return launch_solve_cw<C, 64, 1>(g, nitems, d_sys, factor_arena, rhs_arena, out_arena, queue, st);
    default:
      set_last_error_msg("right-hand-side block width must be 8 (FP64), 16, 32 or 64");
      return PDESHEP_CUDA_ERROR;
  }
}

// The column block of the solve for these systems, by an item's time and the items of 152 SMs.
// complex128 is bound by its SM's FP64 pipe, an item's time by its columns (b = 32: 1.34, 2.58, 5.04, 10.0 us
// per row for 8, 16, 32, 64 columns, in the same ratios from b = 8 to 128; 152 items of 8 run 3.8 times as fast as
// 40 of 32).
// complex64, us per row: items of 16 and 32 columns are bound by the chain of a step while they are alone on an SM and
// by the SM's throughput when several share it, with a loss in the last, unfilled round; an item of 128 columns of the
// tensor-memory kernel has an SM for itself.  Fitted to 144 calls (b = 16, 64, 128, 8 to 152 systems of 60 to
// 384 columns): the choice costs 0.2% over the best width on average, 13% at most.  Few systems are fastest with 16
// columns (b = 64, 8 of 200: 0.33 against 0.45 and 1.09), full rounds of 128 columns with 128 (b = 64, 64 of
// 250: 1.52, 1.34, 1.12; b = 128, 128 of 250: 5.06, 4.47, 3.51).  64 columns never won.
int solve_width(const FactorGeom& g, size_t es, int nsys, const SysDesc* h_sys) {
  const bool dbl = es == sizeof(double2);
  int best = 16;
  double best_t = 1e300;
  auto rounds = [&](int cw) {  // items per SM
    int64_t items = 0;
    for (int s = 0; s < nsys; ++s) items += ceil_div(h_sys[s].ncols, cw);
    return (double)items / 152.0;
  };
  auto consider = [&](int cw, double t) {
    if (t >= best_t) return;
    best_t = t;
    best = cw;
  };
  for (int cw = dbl ? 8 : 16; cw <= (dbl ? 64 : 32); cw *= 2) {
    if (cw > 16 && solve_smem_bytes(g, cw, es, 0) > 227 * 1024) break;
    const double r = rounds(cw);
    if (dbl)
      consider(cw, ceil(r) * (0.1 + 0.155 * cw));
    else if (cw == 16)
      consider(16, std::max(0.107 + 0.11 * g.bt, 0.11 + (0.0285 + 0.0816 * g.bt) * (0.65 * r + 0.35 * ceil(r))));
    else
      consider(32, std::max(0.13 + 0.155 * g.bt, 0.17 + (0.0343 + 0.1423 * g.bt) * (0.6 * r + 0.4 * ceil(r))));
  }
  if (!dbl && solve_tm_supported(g)) consider(kTmChunk, ceil(rounds(kTmChunk)) * (0.49 + 0.3125 * g.bt));
  return best;
}

template <typename C>
int launch_solve(const FactorGeom& g, int trans, int nsys, const SysDesc* h_sys, const SysDesc* d_sys,
                 const char* factor_arena, const C* rhs_arena, C* out_arena, int chunk, void* queue,
                 cudaStream_t st) {
  if (nsys <= 0) return 0;
  if (chunk <= 0) chunk = solve_width(g, sizeof(C), nsys, h_sys);
  if (chunk != 8 && chunk != 16 && chunk != 32 && chunk != 64 && chunk != kTmChunk && chunk != kTcChunk) {
    set_last_error_msg("right-hand-side block width must be 8 (FP64), 16, 32, 64, 128 or 256");
    return PDESHEP_CUDA_ERROR;
  }
  int nitems = 0;
  PD_TRY(upload_solve_items(nsys, h_sys, chunk, queue, st, &nitems));
  return launch_solve_queued<C>(g, trans, nitems, d_sys, factor_arena, rhs_arena, out_arena, chunk, queue, st);
}

template int launch_factor<float2>(const FactorGeom&, int, const void*, int64_t, int, const SysDesc*,
                                   char*, int*, int32_t*, cudaStream_t);
template int launch_factor<double2>(const FactorGeom&, int, const void*, int64_t, int, const SysDesc*,
                                    char*, int*, int32_t*, cudaStream_t);
template int launch_solve_queued<float2>(const FactorGeom&, int, int, const SysDesc*, const char*, const float2*,
                                         float2*, int, void*, cudaStream_t);
template int launch_solve_queued<double2>(const FactorGeom&, int, int, const SysDesc*, const char*, const double2*,
                                          double2*, int, void*, cudaStream_t);
template int launch_solve<float2>(const FactorGeom&, int, int, const SysDesc*, const SysDesc*, const char*,
                                  const float2*, float2*, int, void*, cudaStream_t);
template int launch_solve<double2>(const FactorGeom&, int, int, const SysDesc*, const SysDesc*, const char*,
                                   const double2*, double2*, int, void*, cudaStream_t);

}  // namespace pdeshep
