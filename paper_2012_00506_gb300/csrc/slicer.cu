// slicer.cu -- learned slice proposal.  Cheap statistics of the band feed a
// small FP32 network that predicts where the equal-count slice boundaries lie;
// exact LDL^T inertia counts then validate every proposed boundary and a
// multisection on inertia re-places the ones that miss their target count.
//
// The paper partitions the spectrum by inertia counts (Section 3.2) and names
// density-of-states estimates as the tool when no earlier spectrum is known
// (Section 3.1); equal eigenvalue counts per slice is one of its partition
// objectives (Section 3.1).  The network only proposes: every count returned
// comes from the inertia kernel.
//
// Features (98 per band):
//   [0, 64)   histogram of diag(B) over the Gershgorin interval [lo, hi]
//             (64 equal bins, fractions of n; bin k = floor((d - lo)/w), w =
//             (hi - lo)/64, clamped to [0, 63], evaluated in FP64)
//   64, 65    Gershgorin centre c = (lo+hi)/2 and radius r = (hi-lo)/2, both
//             divided by s = max(|lo|, |hi|) (scale-free)
//   [66, 98)  Chebyshev moments mu_k = z^H T_k(Bs) z / (n P), k = 0..31, of
//             Bs = (B - c I)/r, averaged over P = 8 Rademacher probes z
//             (kernel polynomial method; mu_0 = 1), accumulated in FP64
// Probe entry i of probe p: +1 if bit 0 of splitmix64(seed + p n + i) is 0,
// else -1, where splitmix64 is Vigna's generator (golden-ratio increment
// 0x9e3779b97f4a7c15, then xor-shift-multiply by 0xbf58476d1ce4e5b9 and
// 0x94d049bb133111eb with shifts 30, 27, 31).
//
// Network: 98 -> 256 -> 256 -> 256 -> 64, ReLU after the hidden layers,
// softmax over 64 slice-mass fractions, cumulative sums = 63 boundaries in
// normalised [0, 1] coordinates of the Gershgorin interval, i.e. the inverse
// of the normalised eigenvalue counting function at the fractions j/64.
// Loss: mean over the batch and the 63 boundaries of the squared error.
// Optimiser: Adam (beta1 0.9, beta2 0.999, eps 1e-8, bias-corrected).
// Parameter vector: for each layer, W (out x in, row-major) then bias (out).
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "dense.cuh"

namespace pdeshep {

namespace cg = cooperative_groups;

// from inertia.cu
int gershgorin_device(int64_t n, int b, int cplx, const void* band, int64_t ldab, double* d_lo, double* d_hi,
                      cudaStream_t st);
size_t gershgorin_ws_doubles();
size_t inertia_ws_bytes(int b, int cplx, int nsigma);
int inertia_counts(int64_t n, int b, int cplx, const void* band, int64_t ldab, int nsigma, const double* h_sigma,
                   int64_t* h_neg, double* d_piv, void* work, size_t wbytes, cudaStream_t st, bool* nonfinite_out);

constexpr int kFeat = 98, kHid = 256, kOut = 64, kBins = 64, kMoments = 32, kProbes = 8;
constexpr int kNParams =
    kHid * kFeat + kHid + kHid * kHid + kHid + kHid * kHid + kHid + kOut * kHid + kOut;
constexpr int kChebBlocks = 64;
constexpr int kMaxSlices = 1024;


// ---------------------------------------------------------------------------
// features
// ---------------------------------------------------------------------------
__global__ void lohi_kernel(const double* glo, const double* ghi, double* lohi) {
  if (threadIdx.x == 0) {
    lohi[0] = glo[0];
    lohi[1] = ghi[0];
  }
}

__global__ void diag_hist_kernel(int64_t n, int cplx, const double* __restrict__ band, int64_t ldab,
                                 const double* __restrict__ lohi, unsigned int* __restrict__ hist) {
  __shared__ unsigned int h[kBins];
  for (int i = threadIdx.x; i < kBins; i += blockDim.x) h[i] = 0;
  __syncthreads();
  const double lo = lohi[0], hi = lohi[1];
  const double w = (hi - lo) / kBins;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double d = cplx ? band[2 * (i * ldab)] : band[i * ldab];
    int k = 0;
    if (w > 0.0) {
      const double t = floor((d - lo) / w);
      k = t < 0.0 ? 0 : (t > (double)(kBins - 1) ? kBins - 1 : (int)t);
    }
    atomicAdd(&h[k], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kBins; i += blockDim.x)
    if (h[i]) atomicAdd(&hist[i], h[i]);
}

__global__ void feat_head_kernel(int64_t n, const unsigned int* __restrict__ hist, const double* __restrict__ lohi,
                                 float* __restrict__ feat) {
  for (int i = threadIdx.x; i < kBins; i += blockDim.x) feat[i] = (float)((double)hist[i] / (double)n);
  if (threadIdx.x == 0) {
    const double lo = lohi[0], hi = lohi[1];
    double s = fmax(fabs(lo), fabs(hi));
    if (!(s > 0.0)) s = 1.0;
    feat[64] = (float)(0.5 * (lo + hi) / s);
    feat[65] = (float)(0.5 * (hi - lo) / s);
    feat[66] = 1.0f;
  }
}

// probes Z (n x P column-major, real values in the band's scalar type); T0 = Z
template <typename S>
__global__ void probe_kernel(int64_t n, uint64_t seed, S* __restrict__ Z, S* __restrict__ T0) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * kProbes;
       e += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t r = splitmix64(seed + (uint64_t)e);
    const double v = (r & 1ull) ? -1.0 : 1.0;
    Z[e] = sc<S>::from_re(v);
    T0[e] = sc<S>::from_re(v);
  }
}

// Tn = (Y - c T1)/r (first step) or 2 (Y - c T1)/r - T0 with Y = B T1; block
// partial sums of Re(conj(z) Tn) per probe into part[p * gridDim.x + block].
template <typename S>
__global__ void cheb_step_kernel(int64_t n, const double* __restrict__ lohi, int first, const S* __restrict__ Y,
                                 const S* __restrict__ T1, const S* __restrict__ T0, S* __restrict__ Tn,
                                 const S* __restrict__ Z, double* __restrict__ part) {
  const double c = 0.5 * (lohi[0] + lohi[1]);
  double r = 0.5 * (lohi[1] - lohi[0]);
  if (!(r > 0.0)) r = 1.0;
  const int p = blockIdx.y;
  double acc = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = (int64_t)p * n + i;
    S v = sc<S>::sub(Y[e], sc<S>::scale(T1[e], c));
    if (first)
      v = sc<S>::scale(v, 1.0 / r);
    else
      v = sc<S>::sub(sc<S>::scale(v, 2.0 / r), T0[e]);
    Tn[e] = v;
    acc += sc<S>::re(sc<S>::mul(sc<S>::conj(Z[e]), v));
  }
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    part[(int64_t)p * gridDim.x + blockIdx.x] = t;
  }
}

__global__ void moment_kernel(int64_t n, int nparts, const double* __restrict__ part, int k, float* feat) {
  __shared__ double red[32];
  double t = 0.0;
  for (int q = threadIdx.x; q < kProbes * nparts; q += blockDim.x) t += part[q];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    feat[66 + k] = (float)(s / ((double)n * kProbes));
  }
}

struct FeatWs {
  double *glo, *ghi, *lohi, *part;
  unsigned int* hist;
  void *Z, *T0, *T1, *T2, *Y;
};

static FeatWs plan_feat(Arena& a, int64_t n, size_t es) {
  FeatWs w;
  w.glo = a.take<double>(gershgorin_ws_doubles() / 2);
  w.ghi = a.take<double>(gershgorin_ws_doubles() / 2);
  w.lohi = a.take<double>(2);
  w.part = a.take<double>(kProbes * kChebBlocks);
  w.hist = a.take<unsigned int>(kBins);
  w.Z = a.take<char>(n * kProbes * es);
  w.T0 = a.take<char>(n * kProbes * es);
  w.T1 = a.take<char>(n * kProbes * es);
  w.T2 = a.take<char>(n * kProbes * es);
  w.Y = a.take<char>(n * kProbes * es);
  return w;
}

template <typename S>
static int features(int64_t n, int b, int cplx, const void* band, int64_t ldab, uint64_t seed, float* d_feat,
                    const FeatWs& w, cudaStream_t st) {
  PD_TRY(gershgorin_device(n, b, cplx, band, ldab, w.glo, w.ghi, st));
  lohi_kernel<<<1, 32, 0, st>>>(w.glo, w.ghi, w.lohi);
  PD_CK_LAUNCH();
  PD_CK(cudaMemsetAsync(w.hist, 0, sizeof(unsigned int) * kBins, st));
  diag_hist_kernel<<<64, 256, 0, st>>>(n, cplx, (const double*)band, ldab, w.lohi, w.hist);
  PD_CK_LAUNCH();
  feat_head_kernel<<<1, 64, 0, st>>>(n, w.hist, w.lohi, d_feat);
  PD_CK_LAUNCH();
  S* Z = (S*)w.Z;
  S* T[3] = {(S*)w.T0, (S*)w.T1, (S*)w.T2};
  S* Y = (S*)w.Y;
  probe_kernel<S><<<152, 256, 0, st>>>(n, seed, Z, T[0]);
  PD_CK_LAUNCH();
  // three-term recurrence T_{k} = 2 Bs T_{k-1} - T_{k-2}, vectors rotating through T[k % 3]
  for (int k = 1; k < kMoments; ++k) {
    S* tprev = T[(k - 1) % 3];
    S* tprev2 = T[(k + 1) % 3];
    S* tk = T[k % 3];
    PD_TRY(launch_band_matmul<S>(n, b, band, ldab, kProbes, tprev, Y, st));
    cheb_step_kernel<S><<<dim3(kChebBlocks, kProbes), 256, 0, st>>>(n, w.lohi, k == 1, Y, tprev, tprev2, tk, Z,
                                                                     w.part);
    PD_CK_LAUNCH();
    moment_kernel<<<1, 256, 0, st>>>(n, kChebBlocks, w.part, k, d_feat);
    PD_CK_LAUNCH();
  }
  return 0;
}

// ---------------------------------------------------------------------------
// network (FP32)
// ---------------------------------------------------------------------------
struct Layer {
  int in, out;
  int64_t w, b;  // offsets of W and bias in the parameter vector
};

static void layer_table(Layer L[4]) {
  const int dims[5] = {kFeat, kHid, kHid, kHid, kOut};
  int64_t off = 0;
  for (int l = 0; l < 4; ++l) {
    L[l].in = dims[l];
    L[l].out = dims[l + 1];
    L[l].w = off;
    off += (int64_t)dims[l] * dims[l + 1];
    L[l].b = off;
    off += dims[l + 1];
  }
}

// The layers are small (256 x 256 weights, a batch of at most a few hundred): what costs is latency, not
// arithmetic or bandwidth.  So one launch takes a pass through all layers and back: a cluster of 8 CTAs has 8
// rows of the batch, each CTA the weights of 32 units of every layer (both ways, 162 KB, on their way to shared
// memory from the start), and hands its activations to the other seven by distributed shared memory, a
// cluster barrier per layer.  The weight gradients, which sum over the whole batch, are a second launch, with
// the loss and Adam's step; it brings the parameters and moments before it waits for the first.  Sums run
// over ascending k in one chain of FMAs.
// Measured, batch 64, one Adam step: 14 launches of 32 x 32 tiles staged 32 k at a time took 127 us of
// device time and 158 us in all; 8 launches, a layer each, 46 us in all; these two 31 us
// (batches of 1, 120, 256: 25, 33, 72 us back to back; a layer a launch took 36, 50, 67), all with the same bits.
constexpr int kRows = 8;           // batch rows per cluster
constexpr int kUnits = kHid / 8;   // units of a hidden layer per CTA
constexpr int kPitch = kHid + 4;   // floats: 16-byte rows, 8 consecutive rows in different banks
constexpr int kPitch0 = kFeat + 2; // ... of the first layer's weights

// rows x cols floats (row stride ld) to shared memory (row stride pitch); rows at or past nrows are zero
__device__ __forceinline__ void stage_rows(float* dst, int pitch, const float* src, int64_t ld, int rows, int nrows,
                                           int cols) {
  if ((((uintptr_t)src | (uintptr_t)(ld * 4)) & 15) == 0 && (cols & 3) == 0) {
    const int c4 = cols >> 2;
#pragma unroll 8
    for (int e = threadIdx.x; e < rows * c4; e += blockDim.x) {
      const int r = e / c4, c = e - r * c4;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < nrows) v = *(const float4*)(src + r * ld + 4 * c);
      *(float4*)(dst + r * pitch + 4 * c) = v;
    }
  } else {
#pragma unroll 8
    for (int e = threadIdx.x; e < rows * cols; e += blockDim.x) {
      const int r = e / cols, c = e - r * cols;
      dst[r * pitch + c] = r < nrows ? src[r * ld + c] : 0.f;
    }
  }
}

// the same by asynchronous copies, of rows x cols floats that exist
__device__ __forceinline__ void request_rows(float* dst, int pitch, const float* src, int64_t ld, int rows, int cols) {
  const unsigned d0 = (unsigned)__cvta_generic_to_shared(dst);
  if ((((uintptr_t)src | (uintptr_t)(ld * 4)) & 15) == 0 && (cols & 3) == 0) {
    const int c4 = cols >> 2;
    for (int e = threadIdx.x; e < rows * c4; e += blockDim.x) {
      const int r = e / c4, c = e - r * c4;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d0 + 4 * (r * pitch + 4 * c)),
                   "l"(src + r * ld + 4 * c));
    }
  } else {
    for (int e = threadIdx.x; e < rows * cols; e += blockDim.x) {
      const int r = e / cols, c = e - r * cols;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d0 + 4 * (r * pitch + c)),
                   "l"(src + r * ld + c));
    }
  }
  asm volatile("cp.async.commit_group;\n" ::);
}
template <int PENDING>
__device__ __forceinline__ void arrived() {  // all but the last PENDING requests, for the whole CTA
  asm volatile("cp.async.wait_group %0;\n" ::"n"(PENDING) : "memory");
  __syncthreads();
}

struct PassBuffers {
  float* act[4];   // [1..3]: outputs of the hidden layers
  float* dact[5];  // [1..4]: gradients with respect to the layers' sums
};

constexpr int kPassThreads = 256;  // 8 warps copy; 4 of them sum (lane = unit, a warp two rows)
constexpr size_t kPassFloats = (size_t)kUnits * kPitch0 + 2 * kUnits * kPitch + (kOut / 8) * kPitch + kOut * kUnits +
                               2 * kHid * kUnits + 2 * kRows * kPitch;

// Forward pass (bounds) of the rows of each cluster, with a target also the loss shares and the gradients with
// respect to every layer's sums.  Y[o] = max(sum_i X[i] W[o][i] + bias[o], 0); softmax over the 64 outputs of
// the last layer, cumulative sums -> 63 boundaries; dX[i] = (sum_o dY[o] W[o][i]) * [X[i] > 0].
__global__ void __cluster_dims__(8) __launch_bounds__(kPassThreads)
    mlp_pass_kernel(int B, const float* __restrict__ params, const float* X, float* bounds, const float* target,
                    const PassBuffers io, float* loss_part) {
  extern __shared__ __align__(16) float ps[];
  __shared__ float zb[kOut];  // the logits of this CTA's row
  __shared__ __align__(16) float p_[4][kOut], cs_[4][kOut], dc_[4][kOut], dp_[4][kOut];
  __shared__ float red_[4][2];
  cg::cluster_group cl = cg::this_cluster();
  const int g = (int)cl.block_rank(), tid = threadIdx.x, tx = tid & 31, ty = tid >> 5, u0 = g * kUnits;
  constexpr int64_t w0 = 0, b0 = w0 + kHid * kFeat, w1 = b0 + kHid, b1 = w1 + kHid * kHid, w2 = b1 + kHid,
                    b2 = w2 + kHid * kHid, w3 = b2 + kHid, b3 = w3 + kOut * kHid;
  float* W0 = ps;                       // [units][kPitch0], then rows of W1, W2, of the last layer
  float* W1 = W0 + kUnits * kPitch0;    // [units][kPitch]
  float* W2 = W1 + kUnits * kPitch;
  float* W3 = W2 + kUnits * kPitch;     // [8][kPitch]
  float* V3 = W3 + (kOut / 8) * kPitch; // [64][units]: columns of the last layer's weights, then of W2, W1
  float* V2 = V3 + kOut * kUnits;       // [256][units]
  float* V1 = V2 + kHid * kUnits;
  float* buf = V1 + kHid * kUnits;      // [2][rows][kPitch]: a layer's input, all units
  request_rows(W0, kPitch0, params + w0 + (int64_t)u0 * kFeat, kFeat, kUnits, kFeat);
  request_rows(W1, kPitch, params + w1 + (int64_t)u0 * kHid, kHid, kUnits, kHid);
  request_rows(W2, kPitch, params + w2 + (int64_t)u0 * kHid, kHid, kUnits, kHid);
  request_rows(W3, kPitch, params + w3 + (int64_t)g * (kOut / 8) * kHid, kHid, kOut / 8, kHid);
  if (target) {
    request_rows(V3, kUnits, params + w3 + u0, kHid, kOut, kUnits);
    request_rows(V2, kUnits, params + w2 + u0, kHid, kHid, kUnits);
    request_rows(V1, kUnits, params + w1 + u0, kHid, kHid, kUnits);
  } else {  // (empty groups: the same counts below)
    for (int q = 0; q < 3; ++q) asm volatile("cp.async.commit_group;\n" ::);
  }
  const float bias[3] = {params[b0 + u0 + tx], params[b1 + u0 + tx], params[b2 + u0 + tx]};
  const float bias3 = params[b3 + g * (kOut / 8) + (tid & 7)];
  cudaTriggerProgrammaticLaunchCompletion();
  cl.sync();  // every CTA runs: its shared memory may be written
  // this thread's rows ty, ty + 4 of unit u0 + tx: to every CTA's buffer and to memory
  const bool sums = tid < kPassThreads / 2;
  auto give = [&](float* dst, float* out, int r0, float v0, float v1) {
    if (!sums) return;
    if (dst)
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        float* d = cl.map_shared_rank(dst, c) + u0 + tx;
        d[ty * kPitch] = v0;
        d[(ty + 4) * kPitch] = v1;
      }
    if (r0 + ty < B) out[(int64_t)(r0 + ty) * kHid + u0 + tx] = v0;
    if (r0 + ty + 4 < B) out[(int64_t)(r0 + ty + 4) * kHid + u0 + tx] = v1;
  };
  auto forward = [&](const float* W, int pitch, int in, const float* x, float& a0, float& a1) {
    a0 = a1 = 0.f;
    if (!sums) return;
    const float *w = W + tx * pitch, *x0 = x + ty * kPitch, *x1 = x + (ty + 4) * kPitch;
    int k = 0;
#pragma unroll 8
    for (; k + 4 <= in; k += 4) {
      const float4 wv = *(const float4*)(w + k), u = *(const float4*)(x0 + k), v = *(const float4*)(x1 + k);
      a0 = fmaf(u.x, wv.x, a0);
      a1 = fmaf(v.x, wv.x, a1);
      a0 = fmaf(u.y, wv.y, a0);
      a1 = fmaf(v.y, wv.y, a1);
      a0 = fmaf(u.z, wv.z, a0);
      a1 = fmaf(v.z, wv.z, a1);
      a0 = fmaf(u.w, wv.w, a0);
      a1 = fmaf(v.w, wv.w, a1);
    }
    for (; k < in; ++k) {
      a0 = fmaf(x0[k], w[k], a0);
      a1 = fmaf(x1[k], w[k], a1);
    }
  };
  auto backward = [&](const float* V, int out, const float* d, float& a0, float& a1) {
    a0 = a1 = 0.f;
    if (!sums) return;
    const float *d0 = d + ty * kPitch, *d1 = d + (ty + 4) * kPitch;
#pragma unroll 4
    for (int k = 0; k < out; k += 4) {
      const float4 u = *(const float4*)(d0 + k), v = *(const float4*)(d1 + k);
      const float v0 = V[k * kUnits + tx], v1 = V[(k + 1) * kUnits + tx], v2 = V[(k + 2) * kUnits + tx],
                  v3 = V[(k + 3) * kUnits + tx];
      a0 = fmaf(u.x, v0, a0);
      a1 = fmaf(v.x, v0, a1);
      a0 = fmaf(u.y, v1, a0);
      a1 = fmaf(v.y, v1, a1);
      a0 = fmaf(u.z, v2, a0);
      a1 = fmaf(v.z, v2, a1);
      a0 = fmaf(u.w, v3, a0);
      a1 = fmaf(v.w, v3, a1);
    }
  };
  float *A = buf, *Bf = buf + kRows * kPitch;
  for (int r0 = (blockIdx.x / 8) * kRows; r0 < B; r0 += (gridDim.x / 8) * kRows) {
    float h[3][2];
    stage_rows(A, kPitch, X + (int64_t)r0 * kFeat, kFeat, kRows, B - r0, kFeat);
    arrived<6>();
    forward(W0, kPitch0, kFeat, A, h[0][0], h[0][1]);
    for (int q = 0; q < 2; ++q) h[0][q] = fmaxf(h[0][q] + bias[0], 0.f);
    give(Bf, io.act[1], r0, h[0][0], h[0][1]);
    arrived<5>();
    cl.sync();
    forward(W1, kPitch, kHid, Bf, h[1][0], h[1][1]);
    for (int q = 0; q < 2; ++q) h[1][q] = fmaxf(h[1][q] + bias[1], 0.f);
    give(A, io.act[2], r0, h[1][0], h[1][1]);
    arrived<4>();
    cl.sync();
    forward(W2, kPitch, kHid, A, h[2][0], h[2][1]);
    for (int q = 0; q < 2; ++q) h[2][q] = fmaxf(h[2][q] + bias[2], 0.f);
    give(Bf, io.act[3], r0, h[2][0], h[2][1]);
    arrived<3>();
    cl.sync();
    // the last layer: 8 outputs of 8 rows, each row's to the CTA of its number
    if (tid < 64) {
      const int o = tid & 7, row = tid >> 3;
      const float *w = W3 + o * kPitch, *x = Bf + row * kPitch;
      float z = 0.f;
#pragma unroll 8
      for (int k = 0; k < kHid; k += 4) {
        const float4 wv = *(const float4*)(w + k), u = *(const float4*)(x + k);
        z = fmaf(u.x, wv.x, z);
        z = fmaf(u.y, wv.y, z);
        z = fmaf(u.z, wv.z, z);
        z = fmaf(u.w, wv.w, z);
      }
      cl.map_shared_rank(zb, row)[g * 8 + o] = z + bias3;
    }
    cl.sync();
    // head of row r0 + g (every 64 threads, the first ones write)
    const int bt = r0 + g, j = tid & 63, s2 = tid >> 6;
    const bool live = bt < B, writer = live && s2 == 0;
    float *p = p_[s2], *cs = cs_[s2], *dc = dc_[s2], *dp = dp_[s2], *red = red_[s2];
    const float z = zb[j];
    float m = z;
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((j & 31) == 0) red[j >> 5] = m;
    __syncthreads();
    m = fmaxf(red[0], red[1]);
    __syncthreads();
    const float e = expf(z - m);
    float s = e;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((j & 31) == 0) red[j >> 5] = s;
    __syncthreads();
    s = red[0] + red[1];
    p[j] = e / s;
    __syncthreads();
    if (j == 0) {
      float c = 0.f;
#pragma unroll
      for (int k = 0; k < kOut; ++k) {
        c += p[k];
        cs[k] = c;
      }
    }
    __syncthreads();
    if (writer && j < kOut - 1) bounds[(int64_t)bt * (kOut - 1) + j] = cs[j];
    if (target) {
      const float scale = 1.0f / ((float)B * (float)(kOut - 1));
      float l = 0.f;
      if (live && j < kOut - 1) {
        const float d = cs[j] - target[(int64_t)bt * (kOut - 1) + j];
        l = d * d * scale;
        dc[j] = 2.f * d * scale;
      } else {
        dc[j] = 0.f;
      }
      for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
      __syncthreads();
      if ((j & 31) == 0) red[j >> 5] = l;
      __syncthreads();
      if (j == 0) {
        if (writer) loss_part[bt] = red[0] + red[1];
        float acc = 0.f;  // dL/dp_k = sum_{i >= k} dL/dc_i
#pragma unroll
        for (int k = kOut - 1; k >= 0; --k) {
          acc += dc[k];
          dp[k] = acc;
        }
      }
      __syncthreads();
      float sdp = p[j] * dp[j];
      for (int o = 16; o > 0; o >>= 1) sdp += __shfl_xor_sync(0xffffffffu, sdp, o);
      if ((j & 31) == 0) red[j >> 5] = sdp;
      __syncthreads();
      sdp = red[0] + red[1];
      const float dz = p[j] * (dp[j] - sdp);
      for (int c = s2; c < 8; c += 4) cl.map_shared_rank(A, c)[g * kPitch + j] = dz;
      if (writer) io.dact[4][(int64_t)bt * kOut + j] = dz;
      arrived<2>();
      cl.sync();
      float d0, d1;
      backward(V3, kOut, A, d0, d1);
      d0 = h[2][0] > 0.f ? d0 : 0.f;
      d1 = h[2][1] > 0.f ? d1 : 0.f;
      give(Bf, io.dact[3], r0, d0, d1);
      arrived<1>();
      cl.sync();
      backward(V2, kHid, Bf, d0, d1);
      d0 = h[1][0] > 0.f ? d0 : 0.f;
      d1 = h[1][1] > 0.f ? d1 : 0.f;
      give(A, io.dact[2], r0, d0, d1);
      arrived<0>();
      cl.sync();
      backward(V1, kHid, A, d0, d1);
      give(nullptr, io.dact[1], r0, h[0][0] > 0.f ? d0 : 0.f, h[0][1] > 0.f ? d1 : 0.f);
    }
    cl.sync();  // the buffers are free, and nobody leaves while others write
  }
}

// Forward passes of large batches, a layer a launch: the clusters above are 8 rows each and 15 run at once, so from
// their ninth round on CTAs all over the chip with 32 x 32 tiles are faster (forward, us: 800 rows 64 against 79 in
// tiles, 1024 80 and 77, 2048 151 and 109, 65535 4777 and 1857; with a gradient the pass above always is:
// 65535 rows 14.7 ms in all against 35).  The same sums in the same order, so the same bits.
constexpr int kTiledRows = 8 * 15 * kRows;  // forward passes of more rows take the tiles

// Y[bt][o] = act(sum_i X[bt][i] W[o][i] + bias[o]); one CTA per 32 x 32 output tile
__global__ void __launch_bounds__(256) mlp_tile_kernel(int B, int in, int out, const float* __restrict__ X,
                                                       const float* __restrict__ W, const float* __restrict__ bias,
                                                       float* __restrict__ Y, int relu) {
  __shared__ float Xs[32][33], Ws[32][33];
  const int o0 = blockIdx.x * 32, b0 = blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int k0 = 0; k0 < in; k0 += 32) {
    for (int e = threadIdx.x; e < 32 * 32; e += 256) {
      const int r = e >> 5, c = e & 31;
      Xs[r][c] = (b0 + r < B && k0 + c < in) ? X[(int64_t)(b0 + r) * in + k0 + c] : 0.f;
      Ws[r][c] = (o0 + r < out && k0 + c < in) ? W[(int64_t)(o0 + r) * in + k0 + c] : 0.f;
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < 32; ++k) {
      const float wv = Ws[tx][k];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = fmaf(Xs[ty + 8 * q][k], wv, acc[q]);
    }
    __syncthreads();
  }
  const int o = o0 + tx;
  if (o >= out) return;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int bt = b0 + ty + 8 * q;
    if (bt >= B) continue;
    float v = acc[q] + bias[o];
    if (relu) v = fmaxf(v, 0.f);
    Y[(int64_t)bt * out + o] = v;
  }
}

// softmax over the 64 outputs of a row, cumulative sums -> 63 boundaries
__global__ void __launch_bounds__(kOut) mlp_head_kernel(const float* __restrict__ Z, float* __restrict__ bounds) {
  const int64_t bt = blockIdx.x;
  const int j = threadIdx.x;
  __shared__ float p[kOut], cs[kOut], red[4];
  const float z = Z[bt * kOut + j];
  float m = z;
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((j & 31) == 0) red[j >> 5] = m;
  __syncthreads();
  m = fmaxf(red[0], red[1]);
  const float e = expf(z - m);
  float s = e;
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((j & 31) == 0) red[2 + (j >> 5)] = s;
  __syncthreads();
  p[j] = e / (red[2] + red[3]);
  __syncthreads();
  if (j == 0) {
    float c = 0.f;
    for (int k = 0; k < kOut; ++k) {
      c += p[k];
      cs[k] = c;
    }
  }
  __syncthreads();
  if (j < kOut - 1) bounds[bt * (kOut - 1) + j] = cs[j];
}

// Adam's state and step (m null: write the gradient instead)
struct Adam {
  float *p, *m, *v;
  float lr, b1, b2, eps, c1, c2;
};

struct GradLayer {
  const float *dY, *X;
  int in, out, tiles_i, tile0;  // tile0: first CTA of the layer
  int64_t w, b;                 // offsets of W and bias in the parameter vector
};
struct GradLayers {
  GradLayer l[4];
  int tiles;
};

// All layers' dW[o][i] = sum_bt dY[bt][o] X[bt][i] and db[o] = sum_bt dY[bt][o] (by the CTAs of a layer's
// first column tile), written to g or taken into Adam's step at once; the last CTA sums the loss.
__global__ void __launch_bounds__(256) mlp_bwd_w_kernel(int B, const __grid_constant__ GradLayers L,
                                                        float* g, const Adam ad,
                                                        const float* part, float* loss) {
  constexpr int kChunk = 64;  // batch rows per stage
  __shared__ __align__(16) float Ds[kChunk * 36], Xs[kChunk * 36];
  if ((int)blockIdx.x == L.tiles) {
    cudaGridDependencySynchronize();
    float s = 0.f;
    for (int i = threadIdx.x; i < B; i += blockDim.x) s += part[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) Ds[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      float t = 0.f;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += Ds[w];
      *loss = t;
    }
    return;
  }
  int li = 0;
  while (li < 3 && (int)blockIdx.x >= L.l[li + 1].tile0) ++li;
  const GradLayer& l = L.l[li];
  const int tile = blockIdx.x - l.tile0;
  const int i0 = tile % l.tiles_i * 32, o0 = tile / l.tiles_i * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int i = i0 + tx;
  const bool bias = i0 == 0 && ty == 0;
  // parameters and moments of this thread's entries: 4 weights, a bias
  float pv[5], mv[5], vv[5];
  int64_t at[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    at[q] = q < 4 ? (i < l.in ? l.w + (int64_t)(o0 + ty + 8 * q) * l.in + i : -1) : bias ? l.b + o0 + tx : -1;
    if (ad.m && at[q] >= 0) {
      pv[q] = ad.p[at[q]];
      mv[q] = ad.m[at[q]];
      vv[q] = ad.v[at[q]];
    }
  }
  cudaGridDependencySynchronize();
  float acc[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
  for (int k0 = 0; k0 < B; k0 += kChunk) {
    const int nk = min(kChunk, B - k0);
    __syncthreads();
    stage_rows(Ds, 36, l.dY + (int64_t)k0 * l.out + o0, l.out, nk, nk, 32);
    stage_rows(Xs, 36, l.X + (int64_t)k0 * l.in + i0, l.in, nk, nk, min(32, l.in - i0));
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < nk; ++k) {
      const float xv = Xs[k * 36 + tx];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = fmaf(Ds[k * 36 + ty + 8 * q], xv, acc[q]);
    }
    if (bias)
#pragma unroll 8
      for (int k = 0; k < nk; ++k) acc[4] += Ds[k * 36 + tx];
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    if (at[q] < 0) continue;
    if (!ad.m) {
      g[at[q]] = acc[q];
      continue;
    }
    const float gi = acc[q];
    const float mi = ad.b1 * mv[q] + (1.f - ad.b1) * gi;
    const float vi = ad.b2 * vv[q] + (1.f - ad.b2) * gi * gi;
    ad.m[at[q]] = mi;
    ad.v[at[q]] = vi;
    ad.p[at[q]] = pv[q] - ad.lr * (mi / ad.c1) / (sqrtf(vi / ad.c2) + ad.eps);
  }
}

struct MlpWs {
  float* act[5];   // act[l] = input of layer l (act[0] unused: the caller's X)
  float* dact[5];  // dact[l] = dL/d(pre-activation feeding act[l])
  float* lpart;
};

static MlpWs plan_mlp(Arena& a, int B) {
  MlpWs w;
  const int dims[5] = {kFeat, kHid, kHid, kHid, kOut};
  for (int l = 0; l < 5; ++l) {
    w.act[l] = l == 0 ? nullptr : a.take<float>((size_t)B * dims[l]);
    w.dact[l] = l == 0 ? nullptr : a.take<float>((size_t)B * dims[l]);
  }
  w.lpart = a.take<float>(B);
  return w;
}

// launch that may start before the kernel in front has finished; the kernels above wait for it themselves
template <typename... P, typename... A>
static int launch_after(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  PD_CK(cudaLaunchKernelEx(&cfg, kernel, (P)args...));
  PD_CK_LAUNCH();
  return 0;
}

// forward (bounds); with target: loss and the full backward pass into grad, or into Adam's step (adam.m set)
static int mlp_run(int B, const float* params, const float* X, float* bounds, const float* target, float* grad,
                   const Adam& adam, float* loss, const MlpWs& w, cudaStream_t st) {
  Layer L[4];
  layer_table(L);
  if (!target && B > kTiledRows) {
    for (int l = 0; l < 4; ++l) {
      const dim3 g((unsigned)(L[l].out / 32), (unsigned)ceil_div(B, 32));
      mlp_tile_kernel<<<g, 256, 0, st>>>(B, L[l].in, L[l].out, l ? w.act[l] : X, params + L[l].w, params + L[l].b,
                                         w.act[l + 1], l < 3 ? 1 : 0);
      PD_CK_LAUNCH();
    }
    mlp_head_kernel<<<(unsigned)B, kOut, 0, st>>>(w.act[4], bounds);
    PD_CK_LAUNCH();
    return 0;
  }
  PassBuffers io = {};
  for (int l = 1; l < 4; ++l) io.act[l] = w.act[l];
  for (int l = 1; l < 5; ++l) io.dact[l] = w.dact[l];
  const size_t smem = sizeof(float) * kPassFloats;
  PD_CK(cudaFuncSetAttribute(mlp_pass_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  // 15 clusters of 8 CTAs run at once; they keep their weights over the rest of the batch
  const int clusters = (int)std::min<int64_t>(ceil_div(B, kRows), 15);
  mlp_pass_kernel<<<(unsigned)clusters * 8, kPassThreads, smem, st>>>(B, params, X, bounds, target, io, w.lpart);
  PD_CK_LAUNCH();
  if (!target) return 0;
  GradLayers G;
  G.tiles = 0;
  for (int l = 0; l < 4; ++l) {
    const int ti = (int)ceil_div(L[l].in, 32);
    G.l[l] = GradLayer{w.dact[l + 1], l == 0 ? X : w.act[l], L[l].in, L[l].out, ti, G.tiles, L[l].w, L[l].b};
    G.tiles += ti * (L[l].out / 32);
  }
  return launch_after(mlp_bwd_w_kernel, dim3((unsigned)(G.tiles + 1)), 256, 0, st, B, G, grad, adam, w.lpart, loss);
}

// ---------------------------------------------------------------------------
// proposal + validation + multisection fix-up
// ---------------------------------------------------------------------------
// Normalised position of count fraction f from the 63 predicted boundaries
// (grid fractions j/64, end points 0 -> 0 and 1 -> 1), piecewise linear.
static double inverse_cdf(const float* c63, double f) {
  if (!c63) return f;  // no network: uniform density over the Gershgorin interval
  f = std::min(1.0, std::max(0.0, f));
  const double x = f * kOut;
  int j = (int)floor(x);
  if (j >= kOut) j = kOut - 1;
  const double t = x - j;
  auto g = [&](int q) -> double {
    if (q <= 0) return 0.0;
    if (q >= kOut) return 1.0;
    return std::min(1.0, std::max(0.0, (double)c63[q - 1]));
  };
  return g(j) + t * (g(j + 1) - g(j));
}

struct Probe {
  double sigma;
  int64_t neg;
};

static int propose(int64_t n, int b, int cplx, const void* band, int64_t ldab, const float* c63, double lo,
                   double hi, double f0, double f1, int K, int count_tol, int fanout, double* bounds,
                   int32_t* counts, int32_t* used_fallback, int64_t* evals_out, int64_t* proposed_counts,
                   void* iw, size_t iws, cudaStream_t st) {
  const double span = hi - lo;
  const double pad = 1e-3 * (span > 0 ? span : 1.0) + 1e-300;
  const double below = lo - pad, above = hi + pad;  // count 0 and n by the Gershgorin theorem
  std::vector<int64_t> tgt(K + 1);
  std::vector<double> sig(K + 1);
  std::vector<int64_t> neg(K + 1, -1);
  for (int k = 0; k <= K; ++k) {
    const double f = f0 + (f1 - f0) * k / K;
    tgt[k] = std::min<int64_t>(n, std::max<int64_t>(0, (int64_t)floor(f * (double)n + 0.5)));
    if (tgt[k] == 0) {
      sig[k] = below;
      neg[k] = 0;
    } else if (tgt[k] == n) {
      sig[k] = above;
      neg[k] = n;
    } else {
      sig[k] = lo + span * inverse_cdf(c63, (double)tgt[k] / (double)n);
    }
  }
  std::vector<Probe> seen = {{below, 0}, {above, n}};
  int64_t evals = 0;
  auto evaluate = [&](const std::vector<double>& s, std::vector<int64_t>& out) -> int {
    out.assign(s.size(), 0);
    if (s.empty()) return 0;
    if (inertia_ws_bytes(b, cplx, (int)s.size()) > iws) return PDESHEP_WORKSPACE_TOO_SMALL;
    bool bad = false;
    PD_TRY(inertia_counts(n, b, cplx, band, ldab, (int)s.size(), s.data(), out.data(), nullptr, iw, iws, st, &bad));
    if (bad) return PDESHEP_NONFINITE_INPUT;
    evals += (int64_t)s.size();
    for (size_t e = 0; e < s.size(); ++e) seen.push_back({s[e], out[e]});
    return 0;
  };
  // 1. validate every proposed interior boundary in one inertia launch
  std::vector<double> s;
  std::vector<int> owner;
  std::vector<int64_t> r;
  for (int k = 0; k <= K; ++k)
    if (neg[k] < 0) {
      s.push_back(sig[k]);
      owner.push_back(k);
    }
  PD_TRY(evaluate(s, r));
  for (size_t e = 0; e < s.size(); ++e) neg[owner[e]] = r[e];
  auto ok = [&](int k) { return llabs(neg[k] - tgt[k]) <= count_tol; };
  std::vector<int> todo;
  for (int k = 0; k <= K; ++k)
    if (!ok(k)) todo.push_back(k);
  if (used_fallback) *used_fallback = (int32_t)todo.size();
  if (proposed_counts)
    for (int k = 0; k <= K; ++k) proposed_counts[k] = neg[k];
  // 2. multisection on the failed boundaries.  Every count evaluated so far
  // (for any boundary) is reused: a point inside a boundary's window is taken
  // at once, the others bracket it as [a, c] with count(a) < target - tol and
  // count(c) > target + tol (counts are monotone in sigma).
  auto closest_in_window = [&](int k) -> const Probe* {
    const Probe* best = nullptr;
    for (const Probe& q : seen)
      if (llabs(q.neg - tgt[k]) <= count_tol && (!best || llabs(q.neg - tgt[k]) < llabs(best->neg - tgt[k])))
        best = &q;
    return best;
  };
  for (int round = 0; round < 200 && !todo.empty(); ++round) {
    s.clear();
    owner.clear();
    std::vector<int> next;
    for (int k : todo) {
      if (const Probe* q = closest_in_window(k)) {
        sig[k] = q->sigma;
        neg[k] = q->neg;
        continue;
      }
      double a = below, c = above;
      int64_t na = 0, nc = n;
      for (const Probe& q : seen) {
        if (q.neg < tgt[k] - count_tol && q.sigma > a) {
          a = q.sigma;
          na = q.neg;
        }
        if (q.neg > tgt[k] + count_tol && q.sigma < c) {
          c = q.sigma;
          nc = q.neg;
        }
      }
      const double w = c - a;
      next.push_back(k);
      if (!(w > 4e-16 * std::max(1.0, std::max(fabs(a), fabs(c))))) continue;  // unsplittable cluster
      auto add = [&](double x) {
        if (x > a && x < c) {
          s.push_back(x);
          owner.push_back(k);
        }
      };
      if (fanout == 1) {
        add(a + 0.5 * w);  // plain bisection
      } else {
        // one point where the straight line through (a, count(a)) and
        // (c, count(c)) reaches the target (regula falsi on the counting
        // function), the others split [a, c] evenly so that the bracket
        // shrinks by fanout whatever the interpolation is worth
        add(a + w * ((double)(tgt[k] - na) / (double)(nc - na)));
        for (int f = 1; f < fanout; ++f) add(a + w * f / fanout);
      }
    }
    todo.swap(next);
    if (s.empty()) break;
    PD_TRY(evaluate(s, r));
  }
  for (size_t e = 0; e < todo.size();) {  // windows met by the last round's points
    const int k = todo[e];
    if (const Probe* q = closest_in_window(k)) {
      sig[k] = q->sigma;
      neg[k] = q->neg;
      todo.erase(todo.begin() + e);
    } else {
      ++e;
    }
  }
  // boundaries whose window could not be reached (a cluster wider than the
  // tolerance): the evaluated point with the closest count
  for (int k : todo) {
    const Probe* bestp = nullptr;
    for (const Probe& q : seen)
      if (!bestp || llabs(q.neg - tgt[k]) < llabs(bestp->neg - tgt[k])) bestp = &q;
    sig[k] = bestp->sigma;
    neg[k] = bestp->neg;
  }
  // order (sigma, count) pairs together; counts are monotone in sigma
  std::vector<Probe> fin(K + 1);
  for (int k = 0; k <= K; ++k) fin[k] = {sig[k], neg[k]};
  std::sort(fin.begin(), fin.end(), [](const Probe& x, const Probe& y) {
    return x.sigma < y.sigma || (x.sigma == y.sigma && x.neg < y.neg);
  });
  for (int k = 0; k <= K; ++k) bounds[k] = fin[k].sigma;
  for (int k = 0; k < K; ++k) counts[k] = (int32_t)(fin[k + 1].neg - fin[k].neg);
  if (evals_out) *evals_out = evals;
  return 0;
}

static size_t propose_inertia_bytes(int b, int cplx, int K, int fanout) {
  return std::max(inertia_ws_bytes(b, cplx, (K + 1) * std::max(1, fanout)), (size_t)4096);
}

}  // namespace pdeshep

using namespace pdeshep;

extern "C" int64_t pdeshep_mlp_param_count(void) { return kNParams; }

extern "C" size_t pdeshep_slice_features_workspace_size(int64_t n, int32_t is_complex) {
  if (n <= 0) return 0;
  Arena a;
  plan_feat(a, n, is_complex ? sizeof(double2) : sizeof(double));
  return a.used();
}

extern "C" int pdeshep_slice_features(int64_t n, int32_t b, int32_t is_complex, const void* d_band, int64_t ldab,
                                      uint64_t seed, float* d_features, void* d_work, size_t work_bytes,
                                      void* stream) {
  if (n <= 0) return -1;
  if (b < 0) return -2;
  if (!d_band) return -4;
  if (ldab < b + 1) return -5;
  if (!d_features) return -7;
  if (!d_work) return -8;
  Arena a(d_work, work_bytes);
  const FeatWs w = plan_feat(a, n, is_complex ? sizeof(double2) : sizeof(double));
  if (!a.fits()) return PDESHEP_WORKSPACE_TOO_SMALL;
  cudaStream_t st = (cudaStream_t)stream;
  if (is_complex) return features<double2>(n, b, 1, d_band, ldab, seed, d_features, w, st);
  return features<double>(n, b, 0, d_band, ldab, seed, d_features, w, st);
}

extern "C" size_t pdeshep_mlp_workspace_size(int32_t batch) {
  if (batch <= 0) return 0;
  Arena a;
  plan_mlp(a, batch);
  a.take<float>(kNParams);
  a.take<float>((size_t)batch * (kOut - 1));
  return a.used();
}

extern "C" int pdeshep_mlp_forward(const float* d_params, int32_t batch, const float* d_x, float* d_bounds,
                                   void* d_work, size_t work_bytes, void* stream) {
  if (!d_params) return -1;
  if (batch <= 0 || batch > 65535) return -2;
  if (!d_x) return -3;
  if (!d_bounds) return -4;
  if (!d_work) return -5;
  Arena a(d_work, work_bytes);
  const MlpWs w = plan_mlp(a, batch);
  if (!a.fits()) return PDESHEP_WORKSPACE_TOO_SMALL;
  return mlp_run(batch, d_params, d_x, d_bounds, nullptr, nullptr, Adam{}, nullptr, w, (cudaStream_t)stream);
}

extern "C" int pdeshep_mlp_grad(const float* d_params, int32_t batch, const float* d_x, const float* d_target,
                                float* d_grad, float* d_loss, void* d_work, size_t work_bytes, void* stream) {
  if (!d_params) return -1;
  if (batch <= 0 || batch > 65535) return -2;
  if (!d_x) return -3;
  if (!d_target) return -4;
  if (!d_grad) return -5;
  if (!d_loss) return -6;
  if (!d_work) return -7;
  Arena a(d_work, work_bytes);
  const MlpWs w = plan_mlp(a, batch);
  float* bounds = a.take<float>((size_t)batch * (kOut - 1));
  if (!a.fits()) return PDESHEP_WORKSPACE_TOO_SMALL;
  return mlp_run(batch, d_params, d_x, bounds, d_target, d_grad, Adam{}, d_loss, w, (cudaStream_t)stream);
}

extern "C" int pdeshep_mlp_train_step(float* d_params, float* d_adam_m, float* d_adam_v, int32_t step, float lr,
                                      int32_t batch, const float* d_x, const float* d_target, float* d_loss,
                                      void* d_work, size_t work_bytes, void* stream) {
  if (!d_params) return -1;
  if (!d_adam_m) return -2;
  if (!d_adam_v) return -3;
  if (step < 1) return -4;
  if (!(lr > 0.f)) return -5;
  if (batch <= 0 || batch > 65535) return -6;
  if (!d_x) return -7;
  if (!d_target) return -8;
  if (!d_loss) return -9;
  if (!d_work) return -10;
  Arena a(d_work, work_bytes);
  const MlpWs w = plan_mlp(a, batch);
  a.take<float>(kNParams);  // (the size the workspace query reports)
  float* bounds = a.take<float>((size_t)batch * (kOut - 1));
  if (!a.fits()) return PDESHEP_WORKSPACE_TOO_SMALL;
  cudaStream_t st = (cudaStream_t)stream;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  const Adam adam{d_params, d_adam_m, d_adam_v, lr, b1, b2, 1e-8f, c1, c2};
  return mlp_run(batch, d_params, d_x, bounds, d_target, nullptr, adam, d_loss, w, st);
}

extern "C" size_t pdeshep_propose_workspace_size(int64_t n, int32_t b, int32_t is_complex, int32_t nslices,
                                                 int32_t fanout) {
  if (n <= 0 || b < 0 || nslices < 1 || nslices > kMaxSlices || fanout < 1 || fanout > 64) return 0;
  Arena a;
  plan_feat(a, n, is_complex ? sizeof(double2) : sizeof(double));
  plan_mlp(a, 1);
  a.take<float>(kFeat);
  a.take<float>(kOut);
  a.take<char>(propose_inertia_bytes(b, is_complex ? 1 : 0, nslices, fanout));
  return a.used();
}

extern "C" int pdeshep_propose_slices(int64_t n, int32_t b, int32_t is_complex, const void* d_band, int64_t ldab,
                                      const float* d_params, uint64_t seed, double frac_lo, double frac_hi,
                                      int32_t nslices, int32_t count_tol, int32_t fanout, double* h_bounds,
                                      int32_t* h_counts, int32_t* h_used_fallback, int64_t* h_inertia_evals,
                                      int64_t* h_proposed_counts, void* d_work, size_t work_bytes,
                                      void* stream) {
  if (n <= 0) return -1;
  if (b < 0) return -2;
  if (!d_band) return -4;
  if (ldab < b + 1) return -5;
  if (!(frac_lo >= 0.0 && frac_lo < 1.0)) return -8;
  if (!(frac_hi > frac_lo && frac_hi <= 1.0)) return -9;
  if (nslices < 1 || nslices > kMaxSlices) return -10;
  if (count_tol < 0) return -11;
  if (fanout < 1 || fanout > 64) return -12;
  if (!h_bounds) return -13;
  if (!h_counts) return -14;
  if (!d_work) return -18;
  const int cplx = is_complex ? 1 : 0;
  cudaStream_t st = (cudaStream_t)stream;
  Arena a(d_work, work_bytes);
  const FeatWs fw = plan_feat(a, n, cplx ? sizeof(double2) : sizeof(double));
  const MlpWs mw = plan_mlp(a, 1);
  float* feat = a.take<float>(kFeat);
  float* bnd = a.take<float>(kOut);
  const size_t iws = propose_inertia_bytes(b, cplx, nslices, fanout);
  char* iw = a.take<char>(iws);
  if (!a.fits()) return PDESHEP_WORKSPACE_TOO_SMALL;
  double lohi[2];
  float c63[kOut - 1];
  if (d_params) {
    if (cplx)
      PD_TRY(features<double2>(n, b, 1, d_band, ldab, seed, feat, fw, st));
    else
      PD_TRY(features<double>(n, b, 0, d_band, ldab, seed, feat, fw, st));
    PD_TRY(mlp_run(1, d_params, feat, bnd, nullptr, nullptr, Adam{}, nullptr, mw, st));
    PD_CK(cudaMemcpyAsync(c63, bnd, sizeof(float) * (kOut - 1), cudaMemcpyDeviceToHost, st));
  } else {
    PD_TRY(gershgorin_device(n, b, cplx, d_band, ldab, fw.glo, fw.ghi, st));
    lohi_kernel<<<1, 32, 0, st>>>(fw.glo, fw.ghi, fw.lohi);
    PD_CK_LAUNCH();
  }
  PD_CK(cudaMemcpyAsync(lohi, fw.lohi, sizeof(double) * 2, cudaMemcpyDeviceToHost, st));
  PD_CK(cudaStreamSynchronize(st));
  if (!std::isfinite(lohi[0]) || !std::isfinite(lohi[1])) return PDESHEP_NONFINITE_INPUT;
  int32_t used = 0;
  int64_t evals = 0;
  PD_TRY(propose(n, b, cplx, d_band, ldab, d_params ? c63 : nullptr, lohi[0], lohi[1], frac_lo, frac_hi, nslices,
                 count_tol, fanout, h_bounds, h_counts, &used, &evals, h_proposed_counts, iw, iws, st));
  if (h_used_fallback) *h_used_fallback = used;
  if (h_inertia_evals) *h_inertia_evals = evals;
  return 0;
}

// ---------------------------------------------------------------------------
// Training labels of the proposer: the equal-count boundaries, each the
// midpoint between eigenvalues t_k - 1 and t_k (t_k = round(k n / nslices),
// k = 1..nslices-1, clipped to [1, n-1]) enclosed by bisection on inertia,
// normalised to the Gershgorin interval [lo, hi] and clipped to [0, 1].
// ---------------------------------------------------------------------------
extern "C" size_t pdeshep_equal_count_targets_workspace_size(int64_t n, int32_t b, int32_t is_complex,
                                                             int32_t nslices, int32_t fanout) {
  if (nslices < 2 || fanout < 1) return 0;
  const size_t bis = pdeshep_bisect_workspace_size(n, b, is_complex, 2 * (nslices - 1), fanout);
  return std::max(bis, sizeof(double) * gershgorin_ws_doubles());
}

extern "C" int pdeshep_equal_count_targets(int64_t n, int32_t b, int32_t is_complex, const void* d_band, int64_t ldab,
                                           int32_t nslices, double rtol, int32_t fanout, float* h_targets,
                                           void* d_work, size_t work_bytes, void* stream) {
  if (n < 2) return -1;
  if (b < 0) return -2;
  if (!d_band) return -4;
  if (ldab < b + 1) return -5;
  if (nslices < 2 || nslices > 65536) return -6;
  if (!(rtol > 0.0)) return -7;
  if (fanout < 1 || fanout > 64) return -8;
  if (!h_targets) return -9;
  if (!d_work || work_bytes < pdeshep_equal_count_targets_workspace_size(n, b, is_complex, nslices, fanout))
    return -10;
  double lo = 0.0, hi = 0.0;
  PD_TRY(pdeshep_gershgorin(n, b, is_complex, d_band, ldab, &lo, &hi, d_work, work_bytes, stream));
  const int nb = nslices - 1;
  std::vector<int64_t> t(nb), idx;
  for (int k = 1; k <= nb; ++k) {
    int64_t v = (2 * (int64_t)k * n + nslices) / (2 * (int64_t)nslices);
    t[k - 1] = std::min<int64_t>(std::max<int64_t>(v, 1), n - 1);
    idx.push_back(t[k - 1] - 1);
    idx.push_back(t[k - 1]);
  }
  std::sort(idx.begin(), idx.end());
  idx.erase(std::unique(idx.begin(), idx.end()), idx.end());
  std::vector<double> elo(idx.size()), ehi(idx.size());
  PD_TRY(pdeshep_bisect(n, b, is_complex, d_band, ldab, (int32_t)idx.size(), idx.data(), rtol, fanout, elo.data(),
                        ehi.data(), d_work, work_bytes, stream));
  auto mid = [&](int64_t k) {
    const size_t p = std::lower_bound(idx.begin(), idx.end(), k) - idx.begin();
    return 0.5 * (elo[p] + ehi[p]);
  };
  const double span = hi > lo ? hi - lo : 1.0;
  for (int k = 0; k < nb; ++k) {
    const double sig = 0.5 * (mid(t[k] - 1) + mid(t[k]));
    const double u = (sig - lo) / span;
    h_targets[k] = (float)(u < 0.0 ? 0.0 : (u > 1.0 ? 1.0 : u));
  }
  return 0;
}
