// inertia.cu -- Sylvester inertia of B - sigma I by a pivot-free LDL^T (real)
// or LDL^H (complex) factorization in FP64, many shifts sigma at once.
//
// The paper counts the eigenvalues of each slice from the inertia of
// D - b_i I at both ends of the slice (Section 3.2, "Validation and Other
// Details"), using a band LDL^H that keeps no L.  Here the count is computed
// for many shifts at once: a thread-block cluster of 1 to 16 CTAs per shift
// eliminates panels of 8 columns with the active window in (distributed) shared
// memory (inertia_panel_kernel); calls with enough shifts to fill the GPU, and
// bands too wide for a cluster (window in a per-shift slice of the workspace, L2
// resident), take one CTA per shift and one column at a time (inertia_kernel).
//
// Every floating-point operation is explicitly rounded (__dmul_rn, __dsub_rn, no
// contraction; quotients to nearest, quotient.cuh), in the same order as the CPU
// reference, so the counts and pivots are bit-reproducible:
//   d_k = W(k,k) (zero -> -pivmin);  l_i = W(i,k) / d_k;
//   W(i,j) -= l_i * conj(W(j,k))  for k < j <= i <= k+b,
// with t = l*conj(a) formed as (l.re*a.re + l.im*a.im, l.im*a.re - l.re*a.im)
// and only the real part applied on the diagonal.
#include <cooperative_groups.h>
#include <float.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "common.cuh"
#include "quotient.cuh"

namespace cg = cooperative_groups;

namespace pdeshep {

// ---------------------------------------------------------------------------
// max over stored entries of max(|Re|,|Im|) (as ordered uint64 bits of a
// non-negative double) and a non-finite flag.
// ---------------------------------------------------------------------------
__global__ void band_amax_kernel(int64_t n, int b, int cplx, const double* __restrict__ band,
                                 int64_t ldab, unsigned long long* amax_bits, int* nonfinite) {
  const int64_t per = cplx ? 2 : 1;
  const int64_t total = n * (int64_t)(b + 1);
  double m = 0.0;
  int bad = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    int64_t j = e / (b + 1);
    int d = (int)(e - j * (b + 1));
    if (j + d >= n) continue;
    const double* p = band + (d + j * ldab) * per;
    for (int c = 0; c < per; ++c) {
      double v = p[c];
      if (!isfinite(v)) bad = 1;
      double a = fabs(v);
      if (a > m) m = a;
    }
  }
  // warp reduce
  for (int o = 16; o > 0; o >>= 1) {
    double t = __shfl_down_sync(0xffffffffu, m, o);
    m = t > m ? t : m;
    bad |= __shfl_down_sync(0xffffffffu, bad, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(amax_bits, (unsigned long long)__double_as_longlong(m));
    if (bad) atomicOr(nonfinite, 1);
  }
}

template <bool CPLX>
struct InertiaElem;
template <>
struct InertiaElem<false> {
  using T = double;
};
template <>
struct InertiaElem<true> {
  using T = double2;
};

// The active window (rows and columns k..k+b at step k) is stored by
// diagonals: diagonal d (d = i - j, 0..b) is a ring of R_d = b + 1 - d
// entries, entry (i, j) at ring_base(d) + (j mod R_d).  At step k column j
// = k + s of the window holds rows j..k+b, so diagonal d holds the columns
// k..k+b-d: exactly R_d entries, (b+1)(b+2)/2 in all (half of a square
// window).  After step k the entries of column k are dead; the row k+b+1 that
// enters next lands in exactly those slots (its entry on diagonal d is column
// k+b+1-d = k + R_d).
__host__ __device__ __forceinline__ int ring_base(int d, int b) { return d * (b + 1) - d * (d - 1) / 2; }

// Row r of B - sigma I (entries (r, j), j = max(0, r-b)..r) into the rings; h[d] = k mod R_d for the
// step k that first uses the row (only the column index modulo R_d is needed: j mod R_d).
template <bool CPLX>
__device__ __forceinline__ void load_row(typename InertiaElem<CPLX>::T* W, int b, int64_t r, int64_t k,
                                         const int* h, const double* band, int64_t ldab, double sigma) {
  for (int d = threadIdx.x; d <= b; d += blockDim.x) {
    const int64_t j = r - d;
    if (j < 0 || j < k) continue;
    // j - k = b - d' for the row r = k + b (window bottom row), so j mod R_d = h[d] + (j - k) wrapped
    const int R = b + 1 - d;
    int pos = h[d] + (int)(j - k);
    if (pos >= R) pos -= R;
    const int e = ring_base(d, b) + pos;
    if constexpr (CPLX) {
      const double* p = band + 2 * (d + j * ldab);
      double2 v = make_double2(p[0], p[1]);
      if (d == 0) v = make_double2(__dsub_rn(v.x, sigma), 0.0);
      W[e] = v;
    } else {
      double v = band[d + j * ldab];
      if (d == 0) v = __dsub_rn(v, sigma);
      W[e] = v;
    }
  }
}

// One CTA per shift, one column per step.  Shared memory: pair table (s,u)
// packed as int32, the multipliers L[0..b], the ring heads h[0..b] and (if
// `gwin` is null) the window rings W[(b+1)(b+2)/2].  It serves calls with enough
// shifts to fill the GPU: its half-square window lets four CTAs of b = 64 complex
// share an SM and hide each other's barriers, and it spends fewer FP64
// instructions per column than the panel kernel below (504 shifts, n = 2048,
// b = 64 complex: 22.6 us per column against 26.6).  Bands that no cluster's
// shared memory holds also come here (window in the workspace).
template <bool CPLX>
__global__ void __launch_bounds__(256) inertia_kernel(int64_t n, int b, const double* __restrict__ band,
                                                      int64_t ldab, const double* __restrict__ sigmas,
                                                      const unsigned long long* amax_bits,
                                                      int64_t* __restrict__ neg_out,
                                                      double* __restrict__ piv_out, char* gwin,
                                                      size_t gwin_stride) {
  using T = typename InertiaElem<CPLX>::T;
  extern __shared__ __align__(16) char smem[];
  const int B1 = b + 1;
  const int npairs = b * (b + 1) / 2;
  int* pairs = (int*)smem;
  T* L = (T*)(smem + (((size_t)npairs * 4 + 15) & ~size_t(15)));
  int* h = (int*)(L + B1);
  T* W = gwin ? (T*)(gwin + gwin_stride * blockIdx.x)
              : (T*)((char*)h + (((size_t)B1 * sizeof(int) + 15) & ~size_t(15)));

  const int sid = blockIdx.x;
  const double sigma = sigmas[sid];
  const double amax = __longlong_as_double((long long)*amax_bits);
  const double a2 = __dmul_rn(amax, amax);
  const double pivmin = DBL_MIN * (a2 > 1.0 ? a2 : 1.0);

  // pair table: s in 1..b (column offset), u in 0..b-s (row offset from the column)
  for (int p = threadIdx.x; p < npairs; p += blockDim.x) {
    // invert p = sum_{s'<s} (b - s' + 1) + u  -- small loop, done once
    int s = 1, rem = p;
    while (rem >= b - s + 1) {
      rem -= b - s + 1;
      ++s;
    }
    pairs[p] = (s << 16) | rem;
  }
  for (int d = threadIdx.x; d < B1; d += blockDim.x) h[d] = 0;  // k = 0: 0 mod R_d
  __syncthreads();
  // rows 0..b of the first window: entry (r, j) of diagonal d = r - j at ring position j (j < R_d)
  for (int64_t r = 0; r < B1 && r < n; ++r) {
    for (int d = threadIdx.x; d <= b; d += blockDim.x) {
      const int64_t j = r - d;
      if (j < 0) continue;
      const int e = ring_base(d, b) + (int)j;
      if constexpr (CPLX) {
        const double* pp = band + 2 * (d + j * ldab);
        double2 v = make_double2(pp[0], pp[1]);
        if (d == 0) v = make_double2(__dsub_rn(v.x, sigma), 0.0);
        W[e] = v;
      } else {
        double v = band[d + j * ldab];
        if (d == 0) v = __dsub_rn(v, sigma);
        W[e] = v;
      }
    }
  }
  __syncthreads();

  int64_t neg = 0;
  for (int64_t k = 0; k < n; ++k) {
    const int kmax = (int)((n - 1 - k) < b ? (n - 1 - k) : b);  // rows below k inside the matrix
    // column k sits at ring position h[d] of every diagonal d
    double dk;
    if constexpr (CPLX)
      dk = W[h[0]].x;
    else
      dk = W[h[0]];
    if (dk == 0.0) dk = -pivmin;
    if (threadIdx.x == 0) {
      if (dk < 0.0) ++neg;
      if (piv_out) piv_out[(int64_t)sid * n + k] = dk;
    }
    if (threadIdx.x < kmax) {
      const Divisor by = divisor(dk);
      for (int d = 1 + threadIdx.x; d <= kmax; d += blockDim.x) {
        T a = W[ring_base(d, b) + h[d]];
        if constexpr (CPLX)
          L[d] = make_double2(quotient(a.x, by), quotient(a.y, by));
        else
          L[d] = quotient(a, by);
      }
    }
    __syncthreads();
    for (int p = threadIdx.x; p < npairs; p += blockDim.x) {
      const int pr = pairs[p];
      const int s = pr >> 16, u = pr & 0xffff;
      if (s + u > kmax) continue;
      // W(k+s+u, k+s): diagonal u, column k+s -> position h[u] + s (mod R_u; s <= b - u < R_u)
      int pos = h[u] + s;
      const int R = B1 - u;
      if (pos >= R) pos -= R;
      T a = W[ring_base(s, b) + h[s]];  // W(k+s, k)
      T l = L[s + u];
      T* e = &W[ring_base(u, b) + pos];
      if constexpr (CPLX) {
        double p1 = __dmul_rn(l.x, a.x);
        double p2 = __dmul_rn(l.y, a.y);
        double tre = __dadd_rn(p1, p2);
        if (u == 0) {
          e->x = __dsub_rn(e->x, tre);
        } else {
          double p3 = __dmul_rn(l.y, a.x);
          double p4 = __dmul_rn(l.x, a.y);
          double tim = __dsub_rn(p3, p4);
          double2 v = *e;
          v.x = __dsub_rn(v.x, tre);
          v.y = __dsub_rn(v.y, tim);
          *e = v;
        }
      } else {
        *e = __dsub_rn(*e, __dmul_rn(l, a));
      }
    }
    __syncthreads();
    // column k is finished: advance the ring heads to k + 1 and bring in row k + 1 + b
    for (int d = threadIdx.x; d < B1; d += blockDim.x) {
      const int R = B1 - d;
      h[d] = h[d] + 1 == R ? 0 : h[d] + 1;
    }
    __syncthreads();
    if (k + B1 < n) load_row<CPLX>(W, b, k + B1, k + 1, h, band, ldab, sigma);
    __syncthreads();
  }
  if (threadIdx.x == 0) neg_out[sid] = neg;
}

// The pivot in use (zero -> -pivmin), counted in neg if negative; on the bits, since an FP64
// comparison costs 64 clocks of the step's chain.
__device__ __forceinline__ double pivot(double dk, double pivmin, int64_t& neg) {
  long long bits = __double_as_longlong(dk);
  if ((bits << 1) == 0) {
    dk = -pivmin;
    bits = __double_as_longlong(dk);
  }
  neg += bits < 0 && (unsigned long long)(bits << 1) <= 0xffe0000000000000ull;  // negative, not NaN
  return dk;
}

// ---------------------------------------------------------------------------
// Panel elimination on a thread-block cluster.  FP64 is the scarce resource
// (about 1.7 lanes per clock and SM; a warp instruction holds its quadrant's
// pipe for 64 clocks however few lanes are active, a division takes about 600),
// so one CTA per shift left 143 of 152 SMs idle at 9 shifts, and one column at a
// time paid four barriers and the latency of a band row per column.  Here
//  * a cluster of G CTAs shares one shift: row i of the window belongs to CTA
//    i mod G (cyclic: every CTA keeps an even share of the shrinking triangle),
//    which holds its b + 1 entries (i, i-d) at offset d of a row slot;
//  * kPan = 8 columns are eliminated per round, with two cluster barriers: every
//    CTA factors the panel's 8 x 8 triangle redundantly together with its own
//    rows' 8 entries, sends those rows' entries (the a of W -= l conj(a)) to the
//    other CTAs through distributed shared memory, then applies the 8 updates to
//    its rows in registers, one read and one write of the window per 8 columns;
//  * real and imaginary parts are separate lanes (4 FP64 operations each per
//    update) and the triangle's rows are paired shortest with longest, so that
//    the lanes of a warp are all in use;
//  * band rows arrive by cp.async one round ahead.
// Each entry sees the same rounded operations in the same (ascending column)
// order as with one column at a time, so counts and pivots keep their bits.
// Measured against one CTA per shift and one column per step (us per column, all
// shifts of the call): b = 64 complex, 1 shift 1.4 against 6.6, 9 shifts 1.7
// against 6.6, 63 shifts 4.3 against 6.6; b = 128 complex, 17 shifts 5.0 against
// 22.2; b = 32 real, 64 shifts 0.93 against 1.48.  (With the FP64 division, 9 shifts
// took 2.0 and 64 real ones 1.25.)  What remains at few shifts (b = 64 complex, 8 CTAs
// a shift) is the chain of a column, a division and four dependent operations, 1.3k of
// 3.6k clocks, the share of the updates (1.6k) and two cluster barriers per 8.
// ---------------------------------------------------------------------------
constexpr int kPan = 8;
constexpr int kPanThreads = 256;
static_assert(kPan * 32 == kPanThreads, "one warp per panel column");

struct PanelShape {
  int nslot;   // row slots of one CTA
  int rown;    // own rows below a panel, at most
  int chunks;  // warps that hold one panel column (a lane per entry and part)
  size_t smem;
};
static PanelShape panel_shape(int b, int cplx, int G) {
  PanelShape s;
  s.nslot = (int)ceil_div(b + 2 * kPan, G);  // rows k .. k+b+2 kPan-1 are live during panel k
  s.rown = (int)ceil_div(b, G);
  const size_t np = cplx ? 2 : 1;
  s.chunks = (int)ceil_div((kPan + s.rown) * (int64_t)np, 32);
  s.smem = sizeof(double) * np *
           ((size_t)s.nslot * (b + 1) + (size_t)kPan * kPan + (size_t)2 * (kPan + s.rown) * kPan +
            (G > 1 ? (size_t)b * kPan : 0));
  return s;
}

__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}

// v - t with t = l a (real) or the `part` (0: real, 1: imaginary) of l conj(a):
// re: l.re a.re + l.im a.im, im: l.im a.re - l.re a.im, every operation rounded
__device__ __forceinline__ double sub_prod(double v, double l, double a) { return __dsub_rn(v, __dmul_rn(l, a)); }
__device__ __forceinline__ double sub_prod(double v, double2 l, double2 a, int part) {
  const double l1 = part ? l.y : l.x, l2 = part ? -l.x : l.y;
  return __dsub_rn(v, __dadd_rn(__dmul_rn(l1, a.x), __dmul_rn(l2, a.y)));
}

template <bool CPLX, int NC>
__global__ void __launch_bounds__(kPanThreads)
    inertia_panel_kernel(int64_t n, int b, const double* __restrict__ band, int64_t ldab,
                         const double* __restrict__ sigmas, const unsigned long long* amax_bits,
                         int64_t* __restrict__ neg_out, double* __restrict__ piv_out, int nslot, int rown,
                         int chunks) {
  using T = typename InertiaElem<CPLX>::T;
  constexpr int NP = CPLX ? 2 : 1;
  extern __shared__ __align__(16) char smem[];
  cg::cluster_group cl = cg::this_cluster();
  const int G = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int sid = blockIdx.x / G;
  const int tid = threadIdx.x;
  const int rl = (b + 1) * NP;                      // doubles of a row slot
  double* W = (double*)smem;                        // [nslot][b + 1][NP]
  double* Tri = W + (size_t)nslot * rl;             // [kPan][kPan][NP]: panel rows (r, c), r >= c
  const int lda = kPan + rown;
  T* L = (T*)(Tri + kPan * kPan * NP);              // [kPan][lda]: column c's l of the panel rows, then own rows
  T* A = L + (size_t)lda * kPan;                    // the same for the a of column c
  T* Ap = G > 1 ? A + (size_t)lda * kPan : A + kPan;  // column c, row k + kPan + j, of all CTAs at c * ldp + j
  const int ldp = G > 1 ? b : lda;
  __shared__ double sh_d;                              // the pivot of the next column
  const int warp = tid >> 5, lane = tid & 31;
  const double sigma = sigmas[sid];
  const double amax = __longlong_as_double((long long)*amax_bits);
  const double a2 = __dmul_rn(amax, amax);
  const double pivmin = DBL_MIN * (a2 > 1.0 ? a2 : 1.0);

  const int lg = 31 - __clz(G);  // G is a power of two
  auto first_own = [&](int64_t i) -> int64_t {  // the first row >= i of this CTA
    return i + ((rank - (int)i) & (G - 1));
  };
  auto slot_of = [&](int64_t i) -> int { return (int)((unsigned)(i >> lg) % (unsigned)nslot); };
  // own rows r0 <= r < r0 + cnt requested (8-byte copies: the band is only known to be 8-byte aligned), row
  // number x by warp 1 + x mod 7: in the loop below warp 0 has the panel's first division meanwhile
  auto request_rows = [&](int64_t r0, int cnt) {
    const int64_t r1 = r0 + cnt < n ? r0 + cnt : n, r = first_own(r0);
    if (warp == 0 || r >= r1) return;
    const int q0 = slot_of(r);
    for (int x = warp - 1; r + (int64_t)x * G < r1; x += kPan - 1) {
      const int64_t i = r + (int64_t)x * G;
      const int q = q0 + x;  // (at most nslot rows are requested at once)
      double* s = W + (size_t)(q >= nslot ? q - nslot : q) * rl;
      const int last = i < b ? (int)i : b;
      const double* p = band + NP * (lane + (i - lane) * ldab);
      for (int d = lane; d <= last; d += 32, p += NP * 32 * (1 - ldab)) {
        cp_async8(s + NP * d, p);
        if (CPLX) cp_async8(s + NP * d + 1, p + 1);
      }
    }
  };
  // ... and finished: the thread that copied a diagonal entry shifts it (own copies are visible to it)
  auto finish_rows = [&](int64_t r0, int cnt) {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    const int64_t r1 = r0 + cnt < n ? r0 + cnt : n, r = first_own(r0);
    if (warp == 0 || lane > 0 || r >= r1) return;
    const int q0 = slot_of(r);
    for (int x = warp - 1; r + (int64_t)x * G < r1; x += kPan - 1) {
      const int q = q0 + x;
      double* s = W + (size_t)(q >= nslot ? q - nslot : q) * rl;
      s[0] = __dsub_rn(s[0], sigma);
      if (CPLX) s[1] = 0.0;
    }
  };
  auto csync = [&]() {
    if (G > 1)
      cl.sync();
    else
      __syncthreads();
  };
  // rows k .. k+kPan-1, columns k .. of them, to every CTA's triangle; q: the slot of the first own one
  auto send_triangle = [&](int64_t k, int q) {
    const int i0 = (rank - (int)k) & (G - 1);
    const int nown = i0 < kPan ? ((kPan - 1 - i0) >> lg) + 1 : 0;
    for (int e = tid; e < nown * (kPan * NP << lg); e += kPanThreads) {
      const int part = e % NP, c = (e / NP) % kPan, g = (e / (NP * kPan)) & (G - 1), x = (e / (NP * kPan)) >> lg;
      const int i = i0 + (x << lg);
      if (c > i || k + i >= n) continue;
      const double* s = W + (size_t)(q + x >= nslot ? q + x - nslot : q + x) * rl;
      const double v = i - c <= b ? s[NP * (i - c) + part] : 0.0;
      double* t = G > 1 ? cl.map_shared_rank(Tri, g) : Tri;
      t[(i * kPan + c) * NP + part] = v;
    }
  };
  request_rows(0, b + kPan);
  finish_rows(0, b + kPan);
  csync();
  send_triangle(0, 0);
  csync();

  int64_t neg = 0;
  for (int64_t k = 0; k < n; k += kPan) {
    const int pk = (int)(n - k < kPan ? n - k : kPan);
    const int nrows = (int)(n - k - pk < b ? n - k - pk : b);  // rows k+kPan .. of the panel
    const int64_t i0 = first_own(k + kPan);
    const int off0 = (int)(i0 - (k + kPan));
    const int s0 = slot_of(i0);
    auto own = [&](int t) -> double* {  // slot of own row i0 + t G
      const int q = s0 + t;
      return W + (size_t)(q >= nslot ? q - nslot : q) * rl;
    };
    const int T0 = off0 < nrows ? ((nrows - 1 - off0) >> lg) + 1 : 0;  // own rows among them: i0 + t G
    const int64_t new0 = k + kPan + b;
    if (NC > 1) request_rows(new0, kPan);
    // ---- the panel.  Its entries live in registers: chunk u of column j (32 lanes of rows: the
    // triangle's, then the own ones) belongs to warp (j + u) mod 8, so the divisions of a column and
    // the updates of the others spread over the SM's four FP64 pipes.
    double v[NC];
    int rho[NC];  // row - k of this lane's entry in chunk u; past every reach if there is none
    const int part = lane % NP;
#pragma unroll
    for (int u = 0; u < NC; ++u) {
      const int r = (32 * u + lane) / NP, j = (warp - u) & (kPan - 1), t = r - kPan;
      const double* src = Tri;
      rho[u] = 1 << 30;
      if (r < kPan) {
        if (r < pk) rho[u] = r;
        src = Tri + (r * kPan + j) * NP;
      } else if (t < T0) {
        rho[u] = kPan + off0 + t * G;
        if (rho[u] - j <= b) src = own(t) + NP * (rho[u] - j);
      }
      v[u] = src[part];
      if (NC > 1 && u == 0 && warp == 0 && lane == 0) sh_d = v[u];
    }
    if (NC > 1) __syncthreads();
#pragma unroll 1
    for (int c = 0; c < pk; ++c) {
      // With one chunk per column the warp of column c has the pivot among its lanes and goes on to the
      // division at once; the other warps' updates by column c - 1 run beside it.
      if (NC == 1 && c == 0) request_rows(new0, kPan);
      if (NC > 1 || warp == c) {
        const double dk = pivot(NC > 1 ? sh_d : __shfl_sync(0xffffffffu, v[0], c * NP), pivmin, neg);
        const Divisor by = divisor(dk);
        const bool first = NC > 1 ? tid == 0 : lane == 0;
        if (piv_out && first && rank == 0) piv_out[(int64_t)sid * n + k + c] = dk;
#pragma unroll
        for (int u = 0; u < NC; ++u)
          if (((warp - u) & (kPan - 1)) == c && u < chunks) {
            const bool on = rho[u] > c && rho[u] - c <= b;
            const double l = quotient(on ? v[u] : 1.0, by);
            if (on) {
              const int e = (c * lda + (32 * u + lane) / NP) * NP + part;
              ((double*)A)[e] = v[u];
              ((double*)L)[e] = l;
            }
          }
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < NC; ++u) {
        const int j = (warp - u) & (kPan - 1);
        if (j > c && u < chunks) {
          const bool on = rho[u] > c && rho[u] - c <= b;
          const T l = L[c * lda + (on ? (32 * u + lane) / NP : 0)], a = A[c * lda + j];
          double x;
          if constexpr (CPLX)
            x = sub_prod(v[u], l, a, part);
          else
            x = sub_prod(v[u], l, a);
          // (an update past the panel's end or above the diagonal changes only entries nothing reads;
          // the imaginary part of the diagonal is not read either)
          if (on) v[u] = x;
          if (NC > 1 && u == 0 && j == c + 1 && lane == (c + 1) * NP) sh_d = v[u];
        }
      }
      if (NC > 1) __syncthreads();
    }
    // ---- own rows' panel entries to every CTA
    if (G > 1) {
      for (int e = tid; e < (T0 * kPan << lg); e += kPanThreads) {
        const int g = e & (G - 1), c = (e >> lg) % kPan, t = (e >> lg) / kPan;
        if (kPan + off0 + t * G - c > b) continue;
        cl.map_shared_rank(Ap, g)[c * ldp + off0 + t * G] = A[c * lda + kPan + t];
      }
    }
    csync();
    // ---- the eight updates of the own rows' columns k+kPan .. i
    if (T0 > 0) {
      const int len0 = off0 + 1, lenT = off0 + (T0 - 1) * G + 1;
      const int width = (len0 + lenT) * NP;
      const int total = ((T0 + 1) / 2) * width;
      for (int e0 = tid & ~31; e0 < total; e0 += kPanThreads) {
        const int e = e0 + (tid & 31);
        bool on = e < total;
        int t = on ? e / width : 0;
        int x = on ? e - t * width : 0;
        const int lt = (off0 + t * G + 1) * NP;
        if (x >= lt) {
          x -= lt;
          if (2 * t == T0 - 1) on = false;  // an odd count: the middle row has no partner
          t = T0 - 1 - t;
        }
        const int part = x % NP, j = x / NP;  // column k + kPan + j
        const int ri = off0 + t * G;          // row k + kPan + ri
        if (CPLX && part == 1 && j == ri) on = false;
        const int c0 = on ? (ri + kPan - b > 0 ? ri + kPan - b : 0) : kPan;  // first column that reaches the row
        const int cs = __reduce_min_sync(0xffffffffu, c0);
        double* w = own(t) + NP * (ri - j) + part;
        double v = on ? *w : 0.0;
        const T* lp = L + kPan + t;
        const T* ap = Ap + j;
#pragma unroll
        for (int c = 0; c < kPan; ++c) {
          if (c < cs) continue;
          if (c < c0) continue;
          if constexpr (CPLX)
            v = sub_prod(v, lp[c * lda], ap[c * ldp], part);
          else
            v = sub_prod(v, lp[c * lda], ap[c * ldp]);
        }
        if (on) *w = v;
      }
    }
    finish_rows(new0, kPan);
    __syncthreads();
    if (k + kPan < n) send_triangle(k + kPan, s0);
    csync();
  }
  if (NC > 1) {
    if (tid == 0 && rank == 0) neg_out[sid] = neg;
  } else {  // every warp counted the pivots of its column
    long long* sums = (long long*)A;
    if (lane == 0) sums[warp] = neg;
    __syncthreads();
    if (tid == 0 && rank == 0) {
      long long total = 0;
      for (int w = 0; w < kPan; ++w) total += sums[w];
      neg_out[sid] = total;
    }
  }
}

static size_t window_bytes(int b, int cplx) {
  return (size_t)(b + 1) * (b + 2) / 2 * (cplx ? 16 : 8);
}
static size_t inertia_smem_base(int b, int cplx) {
  size_t npairs = (size_t)b * (b + 1) / 2;
  return ((npairs * 4 + 15) & ~size_t(15)) + (size_t)(b + 1) * (cplx ? 16 : 8) +
         (((size_t)(b + 1) * sizeof(int) + 15) & ~size_t(15));
}
static size_t single_smem(int b, int cplx) { return inertia_smem_base(b, cplx) + window_bytes(b, cplx); }
static bool window_in_smem(int b, int cplx) { return single_smem(b, cplx) <= 226 * 1024; }

// Workspace layout: amax bits, nonfinite flag, sigma[], neg[], global windows.
struct InertiaWs {
  unsigned long long* amax;
  int* nonfinite;
  double* sigma;
  int64_t* neg;
  char* gwin;
  size_t gwin_stride;
};

static InertiaWs plan_inertia(Arena& a, int b, int cplx, int nsigma) {
  InertiaWs w;
  w.amax = a.take<unsigned long long>(1);
  w.nonfinite = a.take<int>(1);
  w.sigma = a.take<double>(nsigma);
  w.neg = a.take<int64_t>(nsigma);
  w.gwin = nullptr;
  w.gwin_stride = 0;
  if (!window_in_smem(b, cplx)) {
    w.gwin_stride = (window_bytes(b, cplx) + 255) & ~size_t(255);
    w.gwin = a.take<char>(w.gwin_stride * nsigma);
  }
  return w;
}

// Computes amax (and the non-finite flag) of a band into ws.  Async.
int launch_band_amax(int64_t n, int b, int cplx, const void* band, int64_t ldab,
                     unsigned long long* amax, int* nonfinite, cudaStream_t st) {
  PD_CK(cudaMemsetAsync(amax, 0, sizeof(unsigned long long), st));
  PD_CK(cudaMemsetAsync(nonfinite, 0, sizeof(int), st));
  int64_t total = n * (int64_t)(b + 1);
  int blocks = (int)((total + 255) / 256);
  if (blocks > 152 * 8) blocks = 152 * 8;
  if (blocks < 1) blocks = 1;
  band_amax_kernel<<<blocks, 256, 0, st>>>(n, b, cplx, (const double*)band, ldab, amax, nonfinite);
  PD_CK_LAUNCH();
  return 0;
}

using PanelKernel = void (*)(int64_t, int, const double*, int64_t, const double*, const unsigned long long*, int64_t*,
                            double*, int, int, int);
template <bool CPLX>
static PanelKernel panel_kernel(int chunks) {
  return chunks <= 1   ? (PanelKernel)inertia_panel_kernel<CPLX, 1>
         : chunks <= 2 ? (PanelKernel)inertia_panel_kernel<CPLX, 2>
         : chunks <= 4 ? (PanelKernel)inertia_panel_kernel<CPLX, 4>
         : chunks <= 8 ? (PanelKernel)inertia_panel_kernel<CPLX, 8>
                       : nullptr;
}

static cudaLaunchConfig_t panel_config(int G, unsigned grid, size_t smem, cudaStream_t st, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kPanThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = G;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// Clusters of G CTAs of the panel kernel that run at once (0: this shape does not fit), cached per
// device and shape.
template <bool CPLX>
static int panel_clusters(int b, int G) {
  static std::mutex mu;
  static std::map<std::tuple<int, int, int>, int> known;
  const PanelShape s = panel_shape(b, CPLX, G);
  PanelKernel kern = panel_kernel<CPLX>(s.chunks);
  int dev = 0;
  if (!kern || s.smem > 226 * 1024 || cudaGetDevice(&dev) != cudaSuccess) return 0;
  std::lock_guard<std::mutex> lk(mu);
  const auto key = std::make_tuple(dev, b, G);
  auto it = known.find(key);
  if (it != known.end()) return it->second;
  int nc = 0;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cudaLaunchAttribute attr;
  const cudaLaunchConfig_t cfg = panel_config(G, (unsigned)G, s.smem, nullptr, &attr);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&nc, kern, &cfg);
  if (e != cudaSuccess) {
    cudaGetLastError();
    nc = 0;
  }
  if (known.size() > 4096) known.clear();
  known[key] = nc;
  return nc;
}

// CTAs of inertia_kernel that share an SM, cached per device and band.
template <bool CPLX>
static int single_per_sm(int b) {
  static std::mutex mu;
  static std::map<std::pair<int, int>, int> known;
  int dev = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  std::lock_guard<std::mutex> lk(mu);
  const auto it = known.find(std::make_pair(dev, b));
  if (it != known.end()) return it->second;
  cudaError_t e = cudaFuncSetAttribute(inertia_kernel<CPLX>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, inertia_kernel<CPLX>, 256, single_smem(b, CPLX));
  if (e != cudaSuccess) cudaGetLastError();
  if (known.size() > 4096) known.clear();
  return known[std::make_pair(dev, b)] = std::max(per, 1);
}

// The cluster size for nsigma shifts, or 0 for one CTA per shift and one column per step
// (inertia_kernel): the least estimated clocks per column of a fit to measured times.  Panel kernel:
// the panel's chain (a division and an update, in one warp per column or through two barriers), the
// rest of a round (barriers, row entry, triangle), the CTA's share of the updates at 76 clocks per
// warp instruction and FP64 pipe; CTAs that share an SM share its pipes.  `sms` is what clusters of G
// reach at one CTA per SM.  One CTA per shift runs in rounds of all that fit on the chip, the last one with fewer to
// an SM.  Checked on 605 calls (b = 0 .. 150, real and complex, 1 .. 2500 shifts, every G): the choice costs 1.5%
// over the best G on average and is at most 6% slower than one CTA per shift.  (Rounds counted in full, and
// at eight to an SM where registers allow five, sent calls of many shifts to the panel kernel, which has no
// advantage there: n = 1000, b = 32 complex, 1500 shifts 22.7 ms against 16.3, b = 40, 504 shifts 11.8 against 10.0.)  At
// b = 64 complex the measured times cross between 63 shifts (4.3 us per column in clusters of 4 or 2 against
// 6.6) and 110 (7.3 against 6.65).  A diagonal band has nothing to update.
// beside: the counts run on a side stream next to factorizations that need whole SMs, and nobody waits
// for them until two filter passes are done, so they keep to about 20 CTAs (9 shifts of n = 8192, b = 64
// complex on 112 SMs stretched a factorization of 64 systems from 6.4 to 18 ms).
constexpr int kBesideCtas = 20;
template <bool CPLX>
static int panel_cluster_size(int b, int nsigma, bool single_ok, bool beside) {
  static const int sms[5] = {152, 152, 144, 120, 112};
  const double np = CPLX ? 2.0 : 1.0, ops = CPLX ? 4.0 : 2.0;
  const double work = 0.5 * b * (b + 1.0) * np / 32.0 * ops * 19.0;  // all updates of one column
  int best = -1;
  double best_t = 0.0;
  if (single_ok) {
    if (b == 0) return 0;
    const double div = np * 221.0 * ceil_div(b, 32);
    const int per_sm = single_per_sm<CPLX>(b), rest = nsigma % (152 * per_sm);
    auto round = [&](double co) { return std::max(work + div + 2280.0 + 11.5 * ops, co * (1.09 * work + div + 395.0)); };
    best_t = 0.92 * (nsigma / (152 * per_sm) * round(per_sm) + (rest ? round((double)ceil_div(rest, 152)) : 0.0));
    best = 0;
  }
  for (int G = 1, q = 0; G <= 16; G *= 2, ++q) {
    const int nc = panel_clusters<CPLX>(b, G);
    if (nc < 1) continue;
    if (beside && best >= 0 && (int64_t)nsigma * G > kBesideCtas) break;
    const int chunks = panel_shape(b, CPLX, G).chunks;
    const int waves = (int)ceil_div(nsigma, nc);
    const double co = (double)ceil_div((int64_t)std::min(nsigma, nc) * G, sms[q]);
    const double upd = 1.01 * work / G + 38.0, pan = chunks * (6.85 + 2.19 * ops) * 19.0 + 122.0;
    const double chain = (chunks == 1 ? 525.0 + 82.5 * ops : 1660.0 + 227.0 * ops) + (G > 1 ? 547.0 : 375.0);
    const double shared = co > 1 ? (CPLX && chunks > 1 ? 1.55 : 1.35) : 1.0;
    const double t = (waves > 1 ? 1.02 : 1.0) * waves * std::max(shared * (chain + upd), co * (upd + pan));
    if (best < 0 || t < best_t) {
      best = G;
      best_t = t;
    }
  }
  return best;
}

template <bool CPLX>
static int launch_panel(int64_t n, int b, const void* band, int64_t ldab, int nsigma, const double* d_sigma,
                        const unsigned long long* amax, int64_t* d_neg, double* d_piv, int G, cudaStream_t st) {
  const PanelShape s = panel_shape(b, CPLX, G);
  PanelKernel kern = panel_kernel<CPLX>(s.chunks);
  PD_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024));
  if (G > 8) PD_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchAttribute attr;
  const cudaLaunchConfig_t cfg = panel_config(G, (unsigned)nsigma * (unsigned)G, s.smem, st, &attr);
  PD_CK(cudaLaunchKernelEx(&cfg, kern, n, b, (const double*)band, ldab, d_sigma, amax, d_neg, d_piv, s.nslot, s.rown,
                           s.chunks));
  count_launch();
  return 0;
}

// Batched inertia with sigma already on the device; results into d_neg.  Async.  gwin (the window in
// the workspace) serves only bands that no cluster's shared memory holds.
int launch_inertia(int64_t n, int b, int cplx, const void* band, int64_t ldab, int nsigma,
                   const double* d_sigma, const unsigned long long* amax, int64_t* d_neg,
                   double* d_piv, char* gwin, size_t gwin_stride, cudaStream_t st, bool beside = false) {
  if (nsigma <= 0) return 0;
  const bool single = window_in_smem(b, cplx);
  const int G = cplx ? panel_cluster_size<true>(b, nsigma, single, beside)
                     : panel_cluster_size<false>(b, nsigma, single, beside);
  if (G > 0)
    return cplx ? launch_panel<true>(n, b, band, ldab, nsigma, d_sigma, amax, d_neg, d_piv, G, st)
                : launch_panel<false>(n, b, band, ldab, nsigma, d_sigma, amax, d_neg, d_piv, G, st);
  const size_t smem = single ? single_smem(b, cplx) : inertia_smem_base(b, cplx);
  auto kern = cplx ? inertia_kernel<true> : inertia_kernel<false>;
  PD_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024));
  kern<<<nsigma, 256, smem, st>>>(n, b, (const double*)band, ldab, d_sigma, amax, d_neg, d_piv,
                                  single ? nullptr : gwin, gwin_stride);
  PD_CK_LAUNCH();
  return 0;
}

size_t inertia_ws_bytes(int b, int cplx, int nsigma) {
  Arena a;
  plan_inertia(a, b, cplx, nsigma);
  return a.used();
}

// Asynchronous counts beside other work: everything is enqueued on st; the counts (nsigma int64)
// and the non-finite flag (int) stay in the workspace at *d_neg / *d_bad.
int inertia_counts_async(int64_t n, int b, int cplx, const void* band, int64_t ldab, int nsigma,
                         const double* h_sigma, void* work, size_t wbytes, cudaStream_t st,
                         const int64_t** d_neg, const int** d_bad) {
  Arena a(work, wbytes);
  InertiaWs w = plan_inertia(a, b, cplx, nsigma);
  if (!a.fits()) return PDESHEP_WORKSPACE_TOO_SMALL;
  PD_TRY(launch_band_amax(n, b, cplx, band, ldab, w.amax, w.nonfinite, st));
  PD_CK(cudaMemcpyAsync(w.sigma, h_sigma, sizeof(double) * nsigma, cudaMemcpyHostToDevice, st));
  PD_TRY(launch_inertia(n, b, cplx, band, ldab, nsigma, w.sigma, w.amax, w.neg, nullptr, w.gwin,
                        w.gwin_stride, st, true));
  *d_neg = w.neg;
  *d_bad = w.nonfinite;
  return 0;
}

// Synchronous helper used by the host-side drivers (bisection, slicing).
int inertia_counts(int64_t n, int b, int cplx, const void* band, int64_t ldab, int nsigma,
                   const double* h_sigma, int64_t* h_neg, double* d_piv, void* work, size_t wbytes,
                   cudaStream_t st, bool* nonfinite_out) {
  Arena a(work, wbytes);
  InertiaWs w = plan_inertia(a, b, cplx, nsigma);
  if (!a.fits()) return PDESHEP_WORKSPACE_TOO_SMALL;
  PD_TRY(launch_band_amax(n, b, cplx, band, ldab, w.amax, w.nonfinite, st));
  PD_CK(cudaMemcpyAsync(w.sigma, h_sigma, sizeof(double) * nsigma, cudaMemcpyHostToDevice, st));
  PD_TRY(launch_inertia(n, b, cplx, band, ldab, nsigma, w.sigma, w.amax, w.neg, d_piv, w.gwin,
                        w.gwin_stride, st));
  int bad = 0;
  PD_CK(cudaMemcpyAsync(h_neg, w.neg, sizeof(int64_t) * nsigma, cudaMemcpyDeviceToHost, st));
  PD_CK(cudaMemcpyAsync(&bad, w.nonfinite, sizeof(int), cudaMemcpyDeviceToHost, st));
  PD_CK(cudaStreamSynchronize(st));
  if (nonfinite_out) *nonfinite_out = bad != 0;
  return 0;
}

// ---------------------------------------------------------------------------
// Gershgorin interval: per row, centre Re B(i,i), radius sum_{j != i} |B(i,j)|.
// ---------------------------------------------------------------------------
__global__ void gershgorin_kernel(int64_t n, int b, int cplx, const double* __restrict__ band,
                                  int64_t ldab, double* part_lo, double* part_hi) {
  double lo = INFINITY, hi = -INFINITY;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    // Row i of the Hermitian band in ascending column order, |b_ij| = sqrt(re^2 + im^2)
    // rounded step by step (no FMA): the interval is a fixed function of the band's bits,
    // so bin decisions taken against it (the proposer's histogram) are reproducible.
    double r = 0.0;
    const int64_t j0 = i - b < 0 ? 0 : i - b, j1 = i + b > n - 1 ? n - 1 : i + b;
    for (int64_t j = j0; j <= j1; ++j) {
      if (j == i) continue;
      // B(i, j) for j < i is stored in column j at row offset i - j; for j > i it is
      // conj(B(j, i)), stored in column i at offset j - i (the modulus ignores the conjugate)
      const int64_t e = j < i ? (i - j) + j * ldab : (j - i) + i * ldab;
      double a;
      if (cplx) {
        const double re = band[2 * e], im = band[2 * e + 1];
        a = __dsqrt_rn(__dadd_rn(__dmul_rn(re, re), __dmul_rn(im, im)));
      } else {
        const double re = band[e];
        a = __dsqrt_rn(__dmul_rn(re, re));
      }
      r = __dadd_rn(r, a);
    }
    double c = cplx ? band[2 * (i * ldab)] : band[i * ldab];
    lo = fmin(lo, __dsub_rn(c, r));
    hi = fmax(hi, __dadd_rn(c, r));
  }
  __shared__ double slo[32], shi[32];
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_down_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_down_sync(0xffffffffu, hi, o));
  }
  if ((threadIdx.x & 31) == 0) {
    slo[threadIdx.x >> 5] = lo;
    shi[threadIdx.x >> 5] = hi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
      lo = fmin(lo, slo[w]);
      hi = fmax(hi, shi[w]);
    }
    part_lo[blockIdx.x] = lo;
    part_hi[blockIdx.x] = hi;
  }
}

__global__ void minmax_final_kernel(int nparts, double* part_lo, double* part_hi) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    double lo = INFINITY, hi = -INFINITY;
    for (int p = 0; p < nparts; ++p) {
      lo = fmin(lo, part_lo[p]);
      hi = fmax(hi, part_hi[p]);
    }
    part_lo[0] = lo;
    part_hi[0] = hi;
  }
}

static const int kGershBlocks = 256;

int gershgorin_device(int64_t n, int b, int cplx, const void* band, int64_t ldab, double* d_lo,
                      double* d_hi, cudaStream_t st) {
  gershgorin_kernel<<<kGershBlocks, 256, 0, st>>>(n, b, cplx, (const double*)band, ldab, d_lo, d_hi);
  PD_CK_LAUNCH();
  minmax_final_kernel<<<1, 32, 0, st>>>(kGershBlocks, d_lo, d_hi);
  PD_CK_LAUNCH();
  return 0;
}
size_t gershgorin_ws_doubles() { return 2 * kGershBlocks; }

// ---------------------------------------------------------------------------
// Allocation-free variant.  Its scratch (the amax word, the non-finite flag,
// the shifts and the counts) lives in a fixed device array that every GPU
// loading this library holds until the process exits; the LDL^T window must
// then fit in shared memory.  Host code cannot use the array's name as a
// device address, so every call looks the address up on the current device
// with cudaGetSymbolAddress (cheap next to the synchronous inertia launch; no
// cached pointer can outlive a cudaDeviceReset or a change of context).
// ---------------------------------------------------------------------------
constexpr int kNoAllocMaxSigma = 1024;
constexpr size_t kNoAllocBytes = 20 * 1024;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

static int noalloc_scratch_address(void** out) {
  void* p = nullptr;
  PD_CK(cudaGetSymbolAddress(&p, g_noalloc_scratch));
  *out = p;
  return 0;
}

}  // namespace pdeshep

using namespace pdeshep;

extern "C" int pdeshep_inertia_noalloc(int64_t n, int32_t b, int32_t is_complex, const void* d_band,
                                       int64_t ldab, int32_t nsigma, const double* h_sigma,
                                       int64_t* h_neg, void* stream) {
  if (n < 0) return -1;
  const int cplx = is_complex ? 1 : 0;
  if (b < 0) {
    set_last_error_msg("pdeshep_inertia_noalloc: negative semi-bandwidth");
    return -2;
  }
  if (!window_in_smem(b, cplx)) {
    set_last_error_msg("pdeshep_inertia_noalloc: band too wide for the shared-memory window "
                       "(real b <= 194, complex b <= 149)");
    return -2;
  }
  if (!d_band && n > 0) return -4;
  if (ldab < b + 1) return -5;
  if (nsigma < 0 || nsigma > kNoAllocMaxSigma) {
    set_last_error_msg("pdeshep_inertia_noalloc: nsigma must be in [0, 1024]");
    return -6;
  }
  if (!h_sigma && nsigma > 0) return -7;
  if (!h_neg && nsigma > 0) return -8;
  if (n == 0 || nsigma == 0) {
    for (int s = 0; s < nsigma; ++s) h_neg[s] = 0;
    return 0;
  }
  void* base = nullptr;
  PD_TRY(noalloc_scratch_address(&base));
  char* p = (char*)base;
  unsigned long long* amax = (unsigned long long*)p;
  int* nonfinite = (int*)(p + 64);
  double* sigma = (double*)(p + 256);
  int64_t* neg = (int64_t*)(p + 256 + sizeof(double) * kNoAllocMaxSigma);
  cudaStream_t st = (cudaStream_t)stream;
  // amax and the flag are cleared here; sigma and neg are overwritten by this call
  PD_TRY(launch_band_amax(n, b, cplx, d_band, ldab, amax, nonfinite, st));
  PD_CK(cudaMemcpyAsync(sigma, h_sigma, sizeof(double) * nsigma, cudaMemcpyHostToDevice, st));
  PD_TRY(launch_inertia(n, b, cplx, d_band, ldab, nsigma, sigma, amax, neg, nullptr, nullptr, 0, st));
  int bad = 0;
  PD_CK(cudaMemcpyAsync(h_neg, neg, sizeof(int64_t) * nsigma, cudaMemcpyDeviceToHost, st));
  PD_CK(cudaMemcpyAsync(&bad, nonfinite, sizeof(int), cudaMemcpyDeviceToHost, st));
  PD_CK(cudaStreamSynchronize(st));
  return bad ? PDESHEP_NONFINITE_INPUT : 0;
}

extern "C" size_t pdeshep_inertia_workspace_size(int64_t n, int32_t b, int32_t is_complex,
                                                 int32_t nsigma) {
  (void)n;
  if (b < 0 || nsigma < 0) return 0;
  return inertia_ws_bytes(b, is_complex ? 1 : 0, nsigma);
}

extern "C" int pdeshep_inertia(int64_t n, int32_t b, int32_t is_complex, const void* d_band,
                               int64_t ldab, int32_t nsigma, const double* h_sigma, int64_t* h_neg,
                               double* d_pivots, void* d_work, size_t work_bytes, void* stream) {
  if (n < 0) return -1;
  if (b < 0 || b > 4096) return -2;
  if (!d_band && n > 0) return -4;
  if (ldab < b + 1) return -5;
  if (nsigma < 0) return -6;
  if (!h_sigma && nsigma > 0) return -7;
  if (!h_neg && nsigma > 0) return -8;
  if (n == 0 || nsigma == 0) {
    for (int s = 0; s < nsigma; ++s) h_neg[s] = 0;
    return 0;
  }
  if (!d_work) return -10;
  bool bad = false;
  int st = inertia_counts(n, b, is_complex ? 1 : 0, d_band, ldab, nsigma, h_sigma, h_neg, d_pivots,
                          d_work, work_bytes, (cudaStream_t)stream, &bad);
  if (st) return st;
  return bad ? PDESHEP_NONFINITE_INPUT : 0;
}

extern "C" int pdeshep_gershgorin(int64_t n, int32_t b, int32_t is_complex, const void* d_band,
                                  int64_t ldab, double* h_lo, double* h_hi, void* d_work,
                                  size_t work_bytes, void* stream) {
  if (n <= 0) return -1;
  if (b < 0) return -2;
  if (!d_band) return -4;
  if (ldab < b + 1) return -5;
  if (!h_lo) return -6;
  if (!h_hi) return -7;
  if (!d_work || work_bytes < sizeof(double) * gershgorin_ws_doubles()) return -8;
  cudaStream_t st = (cudaStream_t)stream;
  double* lo = (double*)d_work;
  double* hi = lo + kGershBlocks;
  PD_TRY(gershgorin_device(n, b, is_complex ? 1 : 0, d_band, ldab, lo, hi, st));
  PD_CK(cudaMemcpyAsync(h_lo, lo, sizeof(double), cudaMemcpyDeviceToHost, st));
  PD_CK(cudaMemcpyAsync(h_hi, hi, sizeof(double), cudaMemcpyDeviceToHost, st));
  PD_CK(cudaStreamSynchronize(st));
  return 0;
}
