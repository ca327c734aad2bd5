// thor_forest.cu -- synthetic Lyman-alpha forest optical depth (THOR Sec. 3.5.2, Eq. 11):
// tau(v_b) = sum_k n_k sigma_0(T_k) ds H(a_k, (v_b - v_k) / v_th,k) along periodic
// sightlines parallel to z, v_k = (k + 1/2) dv_cell + v_los,k, v_b = (b + 1/2) dv_bin,
// nearest periodic image in a box of width V = nz dv_cell = n_bins dv_bin.
//
// One CTA per sightline (several where there are few).  The sightline's cells are staged in
// shared memory (velocity, 1/v_th, a, a^2, amplitudes).  Velocities are 32-bit fixed point with
// the period V mapped onto 2^32 (unit V / 2^32): v_b - v_k wraps modulo 2^32, which is the
// nearest periodic image when read as a signed integer, exactly and without a branch.
//
// Evaluating every cell at every bin is bound by instruction issue (0.97 of the issue peak:
// 22 lane instructions per pair, 5.5 ms for 4096 sightlines of 1024 cells x 2048 bins), and most
// pairs lie far out in the Lorentzian wing, where a cell's profile is smooth on the scale of
// many bins.  So the spectrum is cut into intervals of at most 64 bins and 8 coarse ones:
//   far    a cell whose line centre is at least kFar half-widths from an interval's centre, with
//          the interval outside |x| < 6, contributes at the interval's 16 Chebyshev nodes instead
//          of at its bins -- on the coarse intervals where it is far from one, else on the fine
//          ones.  With kFar = 2.25 the interpolation error of the wing (t g(t), t = 1 / x^2) is
//          at most 1.2e-8 of the contribution, evaluated in FP64 over all half-widths and both
//          levels (largest where |x| = 6 decides, at 4.8 Doppler widths), under FP32's own
//          rounding; all contributions are positive, so it is the same for the sum;
//   near   the other cells (the core |x| < 6, the wing next to it, and the cells opposite the
//          interval, where the nearest image changes side) are evaluated at each bin.
// A chunk of cells most of whose pairs are near (hot gas, or a box narrower than some 12 Doppler
// widths) is evaluated at every bin without sorting its cells (kDirect).
// The node sums become Chebyshev coefficients once per interval and each bin evaluates them.
// FP32 accumulation in two levels (blocks of 32 cells, then the running total of the blocks in
// order), whatever the number of sightlines of a call: a sightline has the same bits alone, in a
// sub-range, in staged rows and in the whole box.
#include "thor_device.cuh"
#include "thor_internal.h"

namespace thor {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kForestThreads = 256;
constexpr int kForestWarps = kForestThreads / 32;
constexpr int kCellChunk = 1024;  // cells staged per pass
constexpr int kMaxBins = 2048;
constexpr int kIvBins = 64;       // bins per interval at most (two per lane)
constexpr int kMaxIv = kMaxBins / kIvBins;
constexpr int kCoarse = 8;        // coarse intervals
constexpr int kNodes = 16;        // Chebyshev nodes per interval
constexpr float kFar = 2.25f;
// Share of near pairs from which on a chunk is evaluated directly, all its cells at up to eight
// bins per lane.  Sorted, a near pair costs some 14% more (one read of the cell per two bins, the
// walk through the mask), a far pair about a quarter.  2048 sightlines of 1024 cells x 2048 bins,
// ms, sorted / direct: cells around 1e6 K 4.6 / 4.8, 2e6 K 5.7 / 5.4, 1e7 K 7.6 / 6.7.
constexpr float kDirect = 0.6f;

// Wing (|x| >= 6) without the a/sqrt(pi) factor: t g(t), t = 1/(x^2 + a^2), g the
// degree-4 fit of thor_device.cuh (one polynomial for the whole wing, no branch).  MUFU
// reciprocal (relative error ~1 ulp, well inside the 1e-5 budget).
__device__ __forceinline__ float wing_tP(float a2, float x2) {
  const float t = rcp_approx(x2 + a2);
  return t * wing_g(t);
}

// Interval iv of 2^iv_log2 holds the bins whose centres lie in it: from first_bin(iv) to first_bin(iv + 1).
__device__ __forceinline__ int first_bin(int iv, int iv_log2, int n_bins) {
  return (2 * iv * n_bins + (1 << iv_log2) - 1) >> (iv_log2 + 1);
}
__device__ __forceinline__ int interval_of(int b, int iv_log2, int n_bins) {
  return ((2 * b + 1) << iv_log2) / (2 * n_bins);
}
// The bin centre's velocity in fixed point.
__device__ __forceinline__ uint32_t bin_fix(int b, double dv_bin, double to_fix) {
  return (uint32_t)(unsigned long long)llrint(((double)b + 0.5) * dv_bin * to_fix);
}

struct ForestCells {
  float4 p[kCellChunk];        // (v as fixed point bits, unit / v_th, a, a^2)
  float2 amp[kCellChunk];      // (n sigma_0 ds, n sigma_0 ds a / sqrt(pi))
  uint32_t core[kCellChunk];   // |x| = 6 in fixed point, rounded up; 2^32 - 1: always near
};

// Distance from an interval's centre (half-width h) from which on a cell is far.
__device__ __forceinline__ uint32_t far_from(uint32_t h, uint32_t core) {
  return max((uint32_t)(kFar * (float)h), core + min(h, ~core));
}
// A cell's line centre d from an interval's centre (fixed point, wrapped), half-width h: far?
// The interval must also lie on one side of the cell's antipode (nearest image).
__device__ __forceinline__ bool is_far(uint32_t d, uint32_t h, uint32_t core) {
  const uint32_t ad = (d & 0x80000000u) ? 0u - d : d;
  return ad >= far_from(h, core) && ad <= 0x80000000u - h - 2u;
}

// One wing term at a node or bin at fixed-point velocity v.
__device__ __forceinline__ float wing_at(uint32_t v, const float4& c, float ampw) {
  const float x = (float)(int32_t)(v - __float_as_uint(c.x)) * c.y;
  return ampw * wing_tP(c.w, x * x);
}
__device__ __forceinline__ float profile_at(uint32_t v, const float4& c, const float2& am, const float* sK, float sum) {
  const float x = (float)(int32_t)(v - __float_as_uint(c.x)) * c.y;  // nearest image, in Doppler widths
  const float x2 = x * x;
  if (x2 >= 36.0f) return __fmaf_rn(am.y, wing_tP(c.w, x2), sum);
  return __fmaf_rn(am.x, voigt_core<true>(c.z, fabsf(x), x2, sK), sum);
}

// Cells of the mask (bit k: cell j0 + k) at the interval's nodes, two cells at a time: lanes
// 0-15 and 16-31 hold the 16 nodes each.
__device__ __forceinline__ float node_terms(const ForestCells& sc, int j0, unsigned mask, uint32_t vnode, float sum) {
  const bool upper = (threadIdx.x & 16u) != 0u;
  while (mask) {
    int k = __ffs(mask) - 1;
    mask &= mask - 1u;
    bool on = true;
    if (upper) {
      on = mask != 0u;
      k = on ? __ffs(mask) - 1 : k;
    }
    mask &= mask - 1u;  // 0 stays 0
    const float w = wing_at(vnode, sc.p[j0 + k], sc.amp[j0 + k].y);
    sum += on ? w : 0.0f;
  }
  return sum;
}

// Cells [0, nk) at N bins per lane (v[q]), in the order of the near cells' sums: blocks of 32
// cells, then the blocks.
template <int N>
__device__ __forceinline__ void direct_terms(const ForestCells& sc, int nk, const float* sK, const uint32_t (&v)[8],
                                             float (&acc)[8]) {
#pragma unroll 1
  for (int j0 = 0; j0 < nk; j0 += 32) {
    const int je = min(nk, j0 + 32);
    float p[N];
#pragma unroll
    for (int q = 0; q < N; ++q) p[q] = 0.0f;
#pragma unroll 4
    for (int j = j0; j < je; ++j) {
      const float4 c = sc.p[j];
      const float2 am = sc.amp[j];
#pragma unroll
      for (int q = 0; q < N; ++q) p[q] = profile_at(v[q], c, am, sK, p[q]);
    }
#pragma unroll
    for (int q = 0; q < N; ++q) acc[q] += p[q];
  }
}

// The chunk's cells at all bins of the CTA (intervals iv0 .. iv0 + iv_cta), added to sAcc.  Out of
// line, so that the interval code keeps its registers (inlined, cold boxes took 3% longer).
__device__ __noinline__ void direct_chunk(const ForestCells* sc, int nk, const float* sK, float* sAcc, int iv0,
                                          int iv_cta, int iv_log2, int n_bins, double dv_bin, double to_fix) {
  __builtin_assume(__isShared(sc));
  __builtin_assume(__isShared(sK));
  __builtin_assume(__isShared(sAcc));
  const int b0 = first_bin(iv0, iv_log2, n_bins), nb = first_bin(iv0 + iv_cta, iv_log2, n_bins) - b0;
  const int n = (nb + kForestThreads - 1) / kForestThreads;  // bins per lane: 1 to 8
  uint32_t v[8];
  float acc[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    v[q] = q < n ? bin_fix(b0 + q * kForestThreads + (int)threadIdx.x, dv_bin, to_fix) : 0u;
    acc[q] = 0.0f;
  }
  if (n > 6) direct_terms<8>(*sc, nk, sK, v, acc);
  else if (n > 4) direct_terms<6>(*sc, nk, sK, v, acc);
  else if (n > 2) direct_terms<4>(*sc, nk, sK, v, acc);
  else if (n == 2) direct_terms<2>(*sc, nk, sK, v, acc);
  else if ((int)(threadIdx.x & ~31u) < nb) direct_terms<1>(*sc, nk, sK, v, acc);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int b = q * kForestThreads + (int)threadIdx.x;
    if (b < nb) {
      const int iv = interval_of(b0 + b, iv_log2, n_bins);
      sAcc[(iv - iv0) * kIvBins + b0 + b - first_bin(iv, iv_log2, n_bins)] += acc[q];
    }
  }
}

// Chebyshev coefficient k of node values f: (2/16) sum_n f_n cos(k pi (n + 1/2) / 16).
__device__ __forceinline__ float cheb_coef(const float* f, int k, const float* cosT) {
  float s = 0.0f;
#pragma unroll
  for (int n = 0; n < kNodes; ++n) s = __fmaf_rn(f[n], cosT[(k * (2 * n + 1)) & 63], s);
  return s * (2.0f / kNodes);
}
__device__ __forceinline__ float cheb_eval(const float* c, float xi) {  // Clenshaw
  const float x2 = 2.0f * xi;
  float b1 = 0.0f, b2 = 0.0f;
#pragma unroll
  for (int k = kNodes - 1; k >= 1; --k) {
    const float b = __fmaf_rn(x2, b1, c[k] - b2);
    b2 = b1;
    b1 = b;
  }
  return __fmaf_rn(xi, b1, __fmaf_rn(0.5f, c[0], -b2));
}

// n_iv = 2^iv_log2 intervals; the CTA's blockIdx.y takes the iv_cta intervals from iv_cta
// blockIdx.y on.  Where there are fewer intervals than warps, `splits` warps share an interval's
// blocks of 32 cells: kPartBlocks / iv_cta blocks of each interval at a time go to shared memory
// (`part`), and their partial sums are added in order (all blocks of a chunk at once leave two
// CTAs per SM instead of four: a call of 60 sightlines of 1024 cells x 2048 bins 212 instead of 158 us).
constexpr int kPartBlocks = 32;
struct BlockSums {  // of one interval's bins and nodes (lanes 0-15 and 16-31 as node_terms has them)
  float bins[kIvBins], nodes[32];
};

template <bool kSplit>
__global__ void __launch_bounds__(kForestThreads, 4) forest_kernel(
    const float* __restrict__ nHI, const float* __restrict__ T, const float* __restrict__ vlos, int nx, int ny,
    int nz, int64_t first, double ds_cm, double dv_cell, int n_bins, double dv_bin, int iv_log2, int iv_cta,
    float* __restrict__ tau, const float* __restrict__ gK) {
  __shared__ __align__(16) float sK[THOR_VOIGT_NINT * THOR_VOIGT_NCOEF];
  __shared__ ForestCells sc;
  constexpr int kIv = kSplit ? kForestWarps / 2 : kMaxIv;
  __shared__ float sAcc[kIv * kIvBins];          // direct sums: interval, bin
  __shared__ float sFine[kIv * kNodes];          // node sums, then coefficients
  __shared__ float sCoarse[kCoarse][kNodes];     // node sums, then coefficients
  __shared__ float sCos[64];                     // cos(pi m / 32)
  __shared__ uint32_t sV[kSplit ? kIv * kIvBins : 1];
  __shared__ BlockSums part[kSplit ? kPartBlocks : 1];
  load_ktab(sK, gK);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t sl = first + blockIdx.x;
  const int ix = (int)(sl % nx), iy = (int)(sl / nx);
  const double V = (double)nz * dv_cell;
  const double to_fix = 4294967296.0 / V;  // fixed-point units per km/s
  const double to_x = 1.0 / (THOR_VTH1 * to_fix);
  const double amp1 = THOR_SIG1 * ds_cm;
  const int64_t plane = (int64_t)nx * ny;
  const int n_iv = 1 << iv_log2, iv0 = blockIdx.y * iv_cta;
  const int splits = kSplit ? kForestWarps / iv_cta : 1, n_task = iv_cta * splits;
  const int batch = kSplit ? kPartBlocks / iv_cta : kCellChunk / 32;  // blocks of 32 cells at a time
  const uint32_t h = iv_log2 ? 1u << (31 - iv_log2) : 0x80000000u;  // half-width of an interval
  const bool far_on = iv_log2 >= 3, coarse_on = iv_log2 >= 4;
  constexpr uint32_t hc = 0x80000000u / kCoarse;
  const int coarse_shift = iv_log2 - 3;
  if (tid < 64) sCos[tid] = cospif((float)tid / 32.0f);
  for (int j = tid; j < iv_cta * kIvBins; j += kForestThreads) sAcc[j] = 0.0f;
  for (int j = tid; j < iv_cta * kNodes; j += kForestThreads) sFine[j] = 0.0f;
  if (tid < kCoarse * kNodes) sCoarse[tid / kNodes][tid % kNodes] = 0.0f;
  __syncthreads();
  const float xi_node = sCos[2 * (lane & 15) + 1];
  const int32_t off_fine = __float2int_rn(xi_node * (float)h), off_coarse = __float2int_rn(xi_node * (float)hc);

  // kSplit: the bins' velocities (FP64 arithmetic) once for the warps that share an interval
  if (kSplit && tid < iv_cta * kIvBins)
    sV[tid] = bin_fix(first_bin(iv0 + tid / kIvBins, iv_log2, n_bins) + tid % kIvBins, dv_bin, to_fix);
  for (int k0 = 0; k0 < nz; k0 += kCellChunk) {
    const int nk = min(kCellChunk, nz - k0);
    uint32_t near_sum = 0u, cells = 0u;  // near share of this thread's pairs, 2^-16 each
    __syncthreads();
    for (int j = tid; j < nk; j += kForestThreads) {
      const int64_t c = (int64_t)(k0 + j) * plane + (int64_t)iy * nx + ix;
      const double rT = rsqrt((double)__ldg(T + c));
      const double vk = ((double)(k0 + j) + 0.5) * dv_cell + (double)__ldg(vlos + c);
      const uint32_t vfix = (uint32_t)(unsigned long long)llrint(vk * to_fix);  // modulo the period
      const double amp = (double)__ldg(nHI + c) * amp1 * rT;
      const double a = THOR_A1 * rT;
      const float iv = (float)(rT * to_x), ampw = (float)(amp * a * 0.5641895835477563);
      sc.p[j] = make_float4(__uint_as_float(vfix), iv, (float)a, (float)(a * a));
      sc.amp[j] = make_float2((float)amp, ampw);
      // cells that are not finite (or near overflow) stay near everywhere: each bin then gets
      // the plain sum
      const float w = __fdividef(6.00002f, iv);
      sc.core[j] = (w < 2.0e9f && w > 0.0f && fabsf(ampw) < 1e30f) ? (uint32_t)w + 2u : 0xffffffffu;
      near_sum += min((min(far_from(h, sc.core[j]), 0x80000000u) >> 15) + (h >> 15), 65536u);
      ++cells;
    }
    // (every CTA of a sightline decides alike: the votes are over all its cells)
    const int votes = __syncthreads_count(far_on && cells && (float)near_sum >= kDirect * 65536.0f * (float)cells);
    const bool direct = 2 * votes > min(nk, kForestThreads);
    if (!kSplit && direct) {
      direct_chunk(&sc, nk, sK, sAcc, iv0, iv_cta, iv_log2, n_bins, dv_bin, to_fix);
      continue;
    }
    if (coarse_on && !direct) {  // one coarse interval per warp
      const int c = warp;
      if ((((c + 1) << coarse_shift) > iv0) && ((c << coarse_shift) < iv0 + iv_cta)) {
        const uint32_t vc = (uint32_t)c * (2u * hc) + hc;
        float sum = 0.0f;
        for (int j0 = 0; j0 < nk; j0 += 32) {
          const int j = j0 + lane;
          bool far = false;
          if (j < nk) far = is_far(vc - __float_as_uint(sc.p[j].x), hc, sc.core[j]);
          sum += node_terms(sc, j0, __ballot_sync(kFull, far), vc + (uint32_t)off_coarse, 0.0f);
        }
        sum += __shfl_down_sync(kFull, sum, 16);
        if (lane < kNodes) sCoarse[c][lane] += sum;
      }
    }
    float acc = 0.0f, nodes = 0.0f;  // kSplit: totals of one bin per thread, one interval's nodes per warp
    for (int jb = 0; jb < nk; jb += 32 * batch) {
      const int je = min(nk, jb + 32 * batch);
      for (int task = warp; task < n_task; task += kForestWarps) {
        const int i = task / splits, iv = iv0 + i, split = task % splits;
        const uint32_t vc = (uint32_t)iv * (2u * h) + h;  // interval centre
        const uint32_t vcc = (uint32_t)(iv >> (coarse_on ? coarse_shift : 0)) * (2u * hc) + hc;
        const int b0 = first_bin(iv, iv_log2, n_bins), nb = first_bin(iv + 1, iv_log2, n_bins) - b0;
        const uint32_t v0 = kSplit ? sV[i * kIvBins + lane] : bin_fix(b0 + lane, dv_bin, to_fix);
        const uint32_t v1 = kSplit ? sV[i * kIvBins + lane + 32] : bin_fix(b0 + lane + 32, dv_bin, to_fix);
        const bool two = nb > 32;
        float acc0 = 0.0f, acc1 = 0.0f, sum = 0.0f;
        for (int j0 = jb + 32 * split; j0 < je; j0 += 32 * splits) {
          const int j = j0 + lane;
          bool near = false, fine = false;
          if (j < nk) {
            const uint32_t vk = __float_as_uint(sc.p[j].x), core = sc.core[j];
            const bool coarse = coarse_on && !direct && is_far(vcc - vk, hc, core);
            fine = far_on && !direct && !coarse && is_far(vc - vk, h, core);
            near = !fine && !coarse;
          }
          unsigned mask = __ballot_sync(kFull, near);
          const float node = node_terms(sc, j0, __ballot_sync(kFull, fine), vc + (uint32_t)off_fine, 0.0f);
          float p0 = 0.0f, p1 = 0.0f;
          while (mask) {
            const int k = j0 + __ffs(mask) - 1;
            mask &= mask - 1u;
            const float4 c = sc.p[k];
            const float2 am = sc.amp[k];
            p0 = profile_at(v0, c, am, sK, p0);
            if (two) p1 = profile_at(v1, c, am, sK, p1);
          }
          if (!kSplit) {
            acc0 += p0;
            acc1 += p1;
            sum += node;
          } else {
            BlockSums& o = part[i * batch + ((j0 - jb) >> 5)];
            o.bins[lane] = p0;
            o.bins[lane + 32] = p1;
            o.nodes[lane] = node;
          }
        }
        if (!kSplit) {
          sum += __shfl_down_sync(kFull, sum, 16);
          if (lane < kNodes) sFine[i * kNodes + lane] += sum;
          sAcc[i * kIvBins + lane] += acc0;
          sAcc[i * kIvBins + lane + 32] += acc1;
        }
      }
      if (kSplit) {
        __syncthreads();
        const int n = (je - jb + 31) >> 5;
        if (tid < iv_cta * kIvBins) {
          const BlockSums* o = part + tid / kIvBins * batch;
#pragma unroll 4
          for (int b = 0; b < n; ++b) acc += o[b].bins[tid % kIvBins];
        }
        if (warp < iv_cta) {
          const BlockSums* o = part + warp * batch;
#pragma unroll 4
          for (int b = 0; b < n; ++b) nodes += o[b].nodes[lane];
        }
        if (je < nk) __syncthreads();
      }
    }
    if (kSplit) {
      if (tid < iv_cta * kIvBins) sAcc[tid] += acc;
      if (warp < iv_cta) {
        nodes += __shfl_down_sync(kFull, nodes, 16);
        if (lane < kNodes) sFine[warp * kNodes + lane] += nodes;
      }
    }
  }
  __syncthreads();
  // node sums to coefficients: coarse first, then each interval's own nodes plus the coarse sum there
  if (coarse_on) {
    const float c = cheb_coef(sCoarse[warp], lane & 15, sCos);
    __syncwarp();
    if (lane < kNodes) sCoarse[warp][lane] = c;
  }
  __syncthreads();
  for (int i = warp; i < iv_cta; i += kForestWarps) {
    const int iv = iv0 + i;
    if (far_on) {
      float f = sFine[i * kNodes + (lane & 15)];
      if (coarse_on) {
        const int c = iv >> coarse_shift;
        const uint32_t v = (uint32_t)iv * (2u * h) + h + (uint32_t)off_fine, vc = (uint32_t)c * (2u * hc) + hc;
        f += cheb_eval(sCoarse[c], (float)(int32_t)(v - vc) * (1.0f / (float)hc));
      }
      __syncwarp();
      float* row = sFine + i * kNodes;
      if (lane < kNodes) row[lane] = f;
      __syncwarp();
      const float c = cheb_coef(row, lane & 15, sCos);
      __syncwarp();
      if (lane < kNodes) row[lane] = c;
      __syncwarp();
    }
    const int b0 = first_bin(iv, iv_log2, n_bins), nb = first_bin(iv + 1, iv_log2, n_bins) - b0;
    const uint32_t vc = (uint32_t)iv * (2u * h) + h;
    for (int q = lane; q < nb; q += 32) {
      float t = sAcc[i * kIvBins + q];
      if (far_on) {
        const uint32_t v = kSplit ? sV[i * kIvBins + q] : bin_fix(b0 + q, dv_bin, to_fix);
        t += cheb_eval(sFine + i * kNodes, (float)(int32_t)(v - vc) * (1.0f / (float)h));
      }
      tau[(size_t)blockIdx.x * n_bins + b0 + q] = t;
    }
  }
}

}  // namespace

cudaError_t launch_forest(const float* nHI, const float* T, const float* vlos, int nx, int ny, int nz, int64_t first,
                          int64_t count, double ds_cm, double dv_cell, int n_bins, double dv_bin, float* tau,
                          const float* d_ktab, cudaStream_t s) {
  // Intervals of at most 64 bins, a power of two of them.  From 8 on the far cells pay (a far
  // cell costs 16 node terms per interval; up to 128 bins nearly every cell is near anyway).
  int iv_log2 = 0;
  while ((kIvBins << iv_log2) < n_bins) ++iv_log2;
  if (n_bins > 128 && iv_log2 < 3) iv_log2 = 3;
  // Few sightlines: several CTAs share one, each with some of its intervals (and its own copy of
  // the cells), until there are two per SM.
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int iv_cta = 1 << iv_log2;
  while (iv_cta > 1 && count * ((1 << iv_log2) / iv_cta) < 2 * (int64_t)sms) iv_cta >>= 1;
  int64_t done = 0;
  while (done < count) {  // grid.x limit
    const int64_t n = count - done < (int64_t)0x7fffffff ? count - done : (int64_t)0x7fffffff;
    const dim3 grid((unsigned)n, (unsigned)((1 << iv_log2) / iv_cta));
    (iv_cta < kForestWarps ? forest_kernel<true> : forest_kernel<false>)<<<grid, kForestThreads, 0, s>>>(
        nHI, T, vlos, nx, ny, nz, first + done, ds_cm, dv_cell, n_bins, dv_bin, iv_log2, iv_cta,
        tau + (size_t)done * n_bins, d_ktab);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    done += n;
  }
  return cudaSuccess;
}

}  // namespace thor
