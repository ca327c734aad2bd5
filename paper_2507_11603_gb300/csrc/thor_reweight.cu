// thor_reweight.cu -- post-processing of a shell run (Sec. 5.1): the escaped photons of
// one radiative-transfer run are reweighted to other intrinsic line widths, equivalent
// widths and dust optical depths, using their emitted frequency X0, escaping frequency X
// and the HI column they traversed (dust following the gas).
//
// A weight costs two exponentials and a division, ~45 instructions; the floor is their issue
// (2e5 photons x 256 targets: 72e6 warp instructions, 60 us).  What is around them is kept
// below that: a CTA takes a chunk of up to 2048 photons, sorts it by (bin, photon) once in
// shared memory and then walks the sorted records with one target per lane, so a record is
// read by broadcast, its bin is the same for all lanes and its weights add up in a register.
// A bin's sum leaves the CTA by one FP64 atomic per target.  (One CTA per 256 photons and
// target, with an FP32 histogram in shared memory, took 703 us there: every target re-read
// the photons, shared FP32 atomics are compare-and-swap loops, and each CTA ended with an
// atomic per occupied bin, 38e6 of them.)  Weights add in FP32 over blocks of 256 photons and in
// two-float arithmetic (error-free sums) above that.  Few weights per photon do not pay for the
// sort: launch_reweight draws the lines between the three kernels.
#include <algorithm>

#include "thor_internal.h"

namespace thor {
namespace {

constexpr int kRwThreads = 256;
constexpr int kRwChunk = 2048;   // photons per CTA at most (a power of two, <= 2^11)
constexpr int kRwBlockBits = 8;  // FP32 sums run over blocks of 2^8 photons
constexpr uint32_t kRwNone = 0xffffffffu;

// Intrinsic spectrum p(X) = pl N(X; 0, sigma^2) + (1 - pl) U(X; -C, C), as
// {pl / (sqrt(2 pi) sigma), 1 / (2 sigma^2), (1 - pl) / (2C), C}.
struct Spectrum { float gn, gi, cd, C; };

__device__ __forceinline__ float pdf(const Spectrum& s, float X) {
  const float g = s.gn * expf(-s.gi * X * X);
  return (fabsf(X) <= s.C) ? g + s.cd : g;
}

// Running sum of one bin and target: hi + lo, the rounding error of every hi + v kept in lo.
struct TwoSum {
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void flush(double* o) {
    const double v = isfinite(hi) ? (double)hi + (double)lo : (double)hi;
    if (v != 0.0) atomicAdd(o, v);
    hi = 0.0f; lo = 0.0f;
  }
  __device__ __forceinline__ void add(float v, double* o) {
    const float t = __fadd_rn(hi, v);
    if (!(fabsf(t) <= 1e38f)) {  // near overflow, or not finite: the sums part in FP64
      flush(o);
      hi = v;
      return;
    }
    const float z = __fsub_rn(t, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(v, z)));
    hi = t;
  }
};

// A photon's weight for a target, and its bin (n_bins: below the range, n_bins + 1: above).
__device__ __forceinline__ float weight(const Spectrum& ps, const Spectrum& pt, float tau_d, float x0, float col) {
  const float s = pdf(ps, x0);
  return (s > 0.0f) ? __fmul_rn(__fdiv_rn(pdf(pt, x0), s), expf(-tau_d * col)) : 0.0f;
}
__device__ __forceinline__ int bin_of(float X, float X_min, float inv_dX, int n_bins) {
  const float f = (X - X_min) * inv_dX;
  if (!(f >= 0.0f)) return n_bins;
  return f >= (float)n_bins ? n_bins + 1 : (int)f;
}

// Few photons and targets: one CTA per 256 photons and target, weights added to an FP32 histogram
// in shared memory.
__global__ void __launch_bounds__(kRwThreads) reweight_few_kernel(int64_t n, const float* __restrict__ X0,
                                                                  const float* __restrict__ X,
                                                                  const float* __restrict__ col,
                                                                  const uint8_t* __restrict__ status,
                                                                  const float* __restrict__ params, int n_bins,
                                                                  float X_min, float inv_dX, double* __restrict__ out) {
  extern __shared__ float hist[];  // n_bins + 2
  const int t = blockIdx.y;
  for (int b = threadIdx.x; b < n_bins + 2; b += blockDim.x) hist[b] = 0.0f;
  const Spectrum ps{params[0], params[1], params[2], params[3]};
  const float* q = params + 5 * (t + 1);
  const Spectrum pt{q[0], q[1], q[2], q[3]};
  const float tau_d = q[4];
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * kRwThreads + threadIdx.x;
  if (i < n && status[i] == 1)
    atomicAdd(&hist[bin_of(X[i], X_min, inv_dX, n_bins)], weight(ps, pt, tau_d, X0[i], col[i]));
  __syncthreads();
  double* o = out + (size_t)t * (n_bins + 2);
  for (int b = threadIdx.x; b < n_bins + 2; b += blockDim.x)
    if (hist[b] != 0.0f) atomicAdd(&o[b], (double)hist[b]);
}

// Many photons, few targets: a CTA strides through the photons for one target.  Up to kFoldBins
// bins the weights add in FP32 and each bin's sum moves to FP64 after 256 photons (up to four
// times as many where they spread over more than 16 bins); with more bins that would cost more
// than the photons, and they are spread enough to add in FP64 at once (a compare-and-swap loop as
// in FP32, which few bins make slow: 1e7 photons, 50 bins 160 us, 84 with FP32 sums).
constexpr int kFoldBins = 1022;
template <bool kWide>
__global__ void __launch_bounds__(kRwThreads) reweight_long_kernel(int64_t n, const float* __restrict__ X0,
                                                                   const float* __restrict__ X,
                                                                   const float* __restrict__ col,
                                                                   const uint8_t* __restrict__ status,
                                                                   const float* __restrict__ params, int n_bins,
                                                                   float X_min, float inv_dX, double* __restrict__ out) {
  extern __shared__ double sum[];  // n_bins + 2, and as many FP32 sums behind them
  float* hist = reinterpret_cast<float*>(sum + n_bins + 2);
  const int t = blockIdx.y;
  for (int b = threadIdx.x; b < n_bins + 2; b += blockDim.x) {
    sum[b] = 0.0;
    if (!kWide) hist[b] = 0.0f;
  }
  const Spectrum ps{params[0], params[1], params[2], params[3]};
  const float* q = params + 5 * (t + 1);
  const Spectrum pt{q[0], q[1], q[2], q[3]};
  const float tau_d = q[4];
  __syncthreads();
  auto fold = [&]() {
    __syncthreads();
    for (int b = threadIdx.x; b < n_bins + 2; b += blockDim.x) {
      const float v = hist[b];
      if (v != 0.0f) { sum[b] += (double)v; hist[b] = 0.0f; }
    }
    __syncthreads();
  };
  const int most = min(max(n_bins / 16, 1), 4);
  int rounds = 0;
  for (int64_t base = (int64_t)blockIdx.x * kRwThreads; base < n; base += (int64_t)gridDim.x * kRwThreads) {
    const int64_t i = base + threadIdx.x;
    if (i < n && status[i] == 1) {
      const float w = weight(ps, pt, tau_d, X0[i], col[i]);
      const int b = bin_of(X[i], X_min, inv_dX, n_bins);
      if (kWide) atomicAdd(&sum[b], (double)w);
      else atomicAdd(&hist[b], w);
    }
    if (!kWide && ++rounds == most) { fold(); rounds = 0; }
  }
  if (!kWide) fold();
  else __syncthreads();
  double* o = out + (size_t)t * (n_bins + 2);
  for (int b = threadIdx.x; b < n_bins + 2; b += blockDim.x)
    if (sum[b] != 0.0) atomicAdd(&o[b], sum[b]);
}

// chunk: photons per CTA (a power of two in [256, kRwChunk]).  A CTA of blockIdx.y handles the
// target groups y, y + gridDim.y, ... of 2^group_log2 targets; its lanes split into
// 32 / 2^group_log2 parts per warp, and warps beyond the groups into further parts.
__global__ void __launch_bounds__(kRwThreads) reweight_kernel(int64_t n, const float* __restrict__ X0,
                                                              const float* __restrict__ X,
                                                              const float* __restrict__ col,
                                                              const uint8_t* __restrict__ status,
                                                              const float* __restrict__ params, int n_targets,
                                                              int group_log2, int chunk, int n_bins, float X_min,
                                                              float inv_dX, double* __restrict__ out) {
  __shared__ uint32_t key[kRwChunk];
  __shared__ float4 rec[kRwChunk];  // X0, p_s(X0), column, key
  __shared__ int n_valid;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const Spectrum ps{params[0], params[1], params[2], params[3]};
  const int group = 1 << group_log2, n_groups = (n_targets + group - 1) >> group_log2;
  const int sub = lane >> group_log2, subs = 32 >> group_log2;
  int mine = 0;  // target groups of this CTA
  for (int g = blockIdx.y; g < n_groups; g += gridDim.y) ++mine;
  const int splits = mine >= kRwThreads / 32 ? 1 : (kRwThreads / 32) / mine;  // warps per group
  const int parts = splits * subs;
  for (int64_t base = (int64_t)blockIdx.x * chunk; base < n; base += (int64_t)gridDim.x * chunk) {
    if (tid == 0) n_valid = 0;
    __syncthreads();
    int valid = 0;
    for (int j = tid; j < chunk; j += kRwThreads) {
      uint32_t k = kRwNone;
      if (base + j < n && status[base + j] == 1) {
        k = ((uint32_t)bin_of(X[base + j], X_min, inv_dX, n_bins) << 11) | (uint32_t)j;
        ++valid;
      }
      key[j] = k;
    }
    valid = __reduce_add_sync(0xffffffffu, valid);
    if (lane == 0 && valid) atomicAdd(&n_valid, valid);
    // bitonic sort of the keys
    for (int k = 2; k <= chunk; k <<= 1) {
      for (int d = k >> 1; d > 0; d >>= 1) {
        __syncthreads();
        for (int i = tid; i < chunk / 2; i += kRwThreads) {
          const int lo = 2 * i - (i & (d - 1)), hi = lo + d;
          const uint32_t a = key[lo], c = key[hi];
          if ((a > c) == ((lo & k) == 0)) { key[lo] = c; key[hi] = a; }
        }
      }
    }
    __syncthreads();
    const int nv = n_valid;
    for (int j = tid; j < nv; j += kRwThreads) {
      const uint32_t k = key[j];
      const int64_t i = base + (k & 2047u);
      const float x0 = X0[i];
      rec[j] = make_float4(x0, pdf(ps, x0), col[i], __uint_as_float(k));
    }
    __syncthreads();
    for (int task = warp; task < mine * splits; task += kRwThreads / 32) {
      const int g = blockIdx.y + (task / splits) * gridDim.y;
      const int t = (g << group_log2) + (lane & (group - 1));
      const int part = (task % splits) * subs + sub;
      const int j0 = (int)((int64_t)nv * part / parts), j1 = (int)((int64_t)nv * (part + 1) / parts);
      if (t < n_targets && j0 < j1) {
        const float* q = params + 5 * (t + 1);
        const Spectrum pt{q[0], q[1], q[2], q[3]};
        const float tau_d = q[4];
        double* o = out + (size_t)t * (n_bins + 2);
        TwoSum sum;
        float acc = 0.0f;
        uint32_t cur = __float_as_uint(rec[j0].w) >> kRwBlockBits;  // bin and block of 256 photons
        for (int j = j0; j < j1; ++j) {
          const float4 r = rec[j];
          const uint32_t k = __float_as_uint(r.w) >> kRwBlockBits;
          const float w = (r.y > 0.0f) ? __fmul_rn(__fdiv_rn(pdf(pt, r.x), r.y), expf(-tau_d * r.z)) : 0.0f;
          if (k != cur) {
            sum.add(acc, o + (cur >> 3));
            acc = 0.0f;
            if ((k >> 3) != (cur >> 3)) sum.flush(o + (cur >> 3));
            cur = k;
          }
          acc = __fadd_rn(acc, w);
        }
        sum.add(acc, o + (cur >> 3));
        sum.flush(o + (cur >> 3));
      }
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_reweight(int64_t n, const float* X0, const float* X, const float* col, const uint8_t* status,
                            const float* d_params, int n_targets, int n_bins, double X_min, double X_max,
                            double* d_out, int n_sm, cudaStream_t s) {
  const float lo = (float)X_min, inv = (float)(n_bins / (X_max - X_min));
  const bool wide = n_bins > kFoldBins;
  // Sorting a chunk costs a CTA some 8 us, whatever the targets: up to some 2^21 photon-targets
  // (of few photons; less of many, where an atomic per bin, target and 256 photons weighs more) a
  // CTA per 256 photons and target is done earlier.  us, few / chunks, 300 bins: 5000 x 1 7 / 10,
  // x 64 10 / 20, x 256 17 / 25; 2e4 x 64 16 / 24, x 256 44 / 43; 6e4 x 16 16 / 19, x 32 24 / 26,
  // x 64 41 / 38; 2e5 x 2 18 / 24, x 4 24 / 26, x 8 36 / 28, x 256 747 / 181; 50 bins: 6e4 x 36
  // 25 / 28, x 50 32 / 29; 2e5 x 5 23 / 33; 4000 bins: 2e5 x 4 26 / 20.
  const int64_t few = n <= 1 << 16   ? (n_bins < 100 ? (int64_t)1 << 21 : (int64_t)3 << 20)
                      : n <= 1 << 18 ? (wide ? (int64_t)3 << 18 : (int64_t)1 << 20)
                                     : n <= 1 << 19 ? (int64_t)3 << 18 : 0;
  if (n * n_targets <= few) {
    const dim3 grid((unsigned)((n + kRwThreads - 1) / kRwThreads), (unsigned)n_targets);
    reweight_few_kernel<<<grid, kRwThreads, (size_t)(n_bins + 2) * sizeof(float), s>>>(n, X0, X, col, status, d_params,
                                                                                       n_bins, lo, inv, d_out);
    return cudaGetLastError();
  }
  // Many photons, few targets: sorting a photon costs more than its few weights.  us, chunks /
  // striding CTAs: 50 bins, 1e7 x 1 446 / 84, x 3 444 / 232, x 6 462 / 448, x 8 460 / 594; 3e5 x 4
  // 49 / 30; 400 bins, 3e5 x 3 32 / 35, x 4 32 / 38, 1e6 x 4 74 / 66; 4000 bins, 1e6 x 3 80 / 59,
  // x 4 81 / 81, 1e7 x 6 672 / 523.  With fewer bins a chunk's sums collide more (4 bins, 3e5 x 4
  // 102 / 26), but the FP32 sums move to FP64 after every 256 photons (10 bins, 3e6 x 6 185 / 153,
  // 1e7 x 4 573 / 426, x 5 462 / 530), and with one or two bins the shared sums collide (1 bin, 1e7
  // x 3 679 / 1117).
  const bool many = n >= 1 << 20;
  const int strided = n_bins < 4      ? 2
                      : n_bins < 32   ? (!many ? 8 : n < 1 << 22 ? 6 : 4)
                      : n_bins <= 100 ? 6
                      : !wide         ? (many ? 6 : 3)
                                      : (n >= 1 << 21 ? 6 : many ? 3 : 2);
  if (n_targets <= strided) {
    const size_t smem = (size_t)(n_bins + 2) * (wide ? 8 : 12);
    const int64_t want = (n + kRwThreads - 1) / kRwThreads;
    const int64_t cap = n_sm * std::min<int64_t>(8, (200 << 10) / smem);  // resident CTAs
    (wide ? reweight_long_kernel<true> : reweight_long_kernel<false>)<<<
        dim3((unsigned)std::min(want, cap), (unsigned)n_targets), kRwThreads, smem, s>>>(n, X0, X, col, status, d_params,
                                                                                         n_bins, lo, inv, d_out);
    return cudaGetLastError();
  }
  // One target per lane: groups of 32 targets, or of the next power of two where there are
  // fewer (the lanes then split the records).
  int group_log2 = 0;
  while (group_log2 < 5 && (1 << group_log2) < n_targets) ++group_log2;
  const int n_groups = (n_targets + (1 << group_log2) - 1) >> group_log2;
  // Long chunks mean fewer atomics (one per bin and target of a chunk), short ones more CTAs:
  // the longest that still gives every SM two.  Where the chunks are too few for that, the
  // target groups are spread over CTAs that sort the same chunk (a few per cent of its work).
  int chunk = kRwChunk;
  while (chunk > 256 && (n + chunk - 1) / chunk * n_groups < 2 * n_sm) chunk >>= 1;
  const int64_t chunks = (n + chunk - 1) / chunk;
  const int64_t gx = chunks < 65536 ? chunks : 65536;
  int64_t gy = (4 * (int64_t)n_sm + gx - 1) / gx;
  if (gy > n_groups) gy = n_groups;
  const dim3 grid((unsigned)gx, (unsigned)gy);
  reweight_kernel<<<grid, kRwThreads, 0, s>>>(n, X0, X, col, status, d_params, n_targets, group_log2, chunk, n_bins, lo,
                                              inv, d_out);
  return cudaGetLastError();
}

}  // namespace thor
