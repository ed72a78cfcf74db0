// Posterior summaries from the stored samples (Sec. 3.5 uncertainty
// quantification, Sec. 4.1 calibration against synthetic truth, Sec. 5 effective
// sample size), one warp per (event, coordinate) series of the n stored samples:
//   - effective sample size n / tau, tau = 1 + 2 sum_{t >= 1} rho_t over the
//     lags while the autocorrelation rho_t stays positive (time order);
//   - median and the half-length of the [lo, hi] percentile interval, linear
//     interpolation between order statistics at rank (n - 1) p / 100 (sorted
//     in shared memory, bitonic);
//   - the fraction of samples below the true value.
// FP64 arithmetic on the FP32 stored offsets from theta_0.
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.h"
#include "view.h"

namespace spider {
namespace {

constexpr int kUqWarps = 8;

__device__ __forceinline__ double warp_sum_d(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

__device__ __forceinline__ double pct_sorted(const float* a, int n, double p) {
  const double pos = (double)(n - 1) * p / 100.0;
  int lo = (int)floor(pos);
  if (lo < 0) lo = 0;
  if (lo > n - 1) lo = n - 1;
  const int hi = lo + 1 < n ? lo + 1 : n - 1;
  const double f = pos - (double)lo;
  return (double)a[lo] + f * ((double)a[hi] - (double)a[lo]);
}

// Sums of four lags at once: after the five exchange steps lane l holds the sum
// of c[l / 8] over the lanes.  Each step adds the two halves of the lanes that a
// butterfly over the same offsets would add, so every sum has the bits of that
// butterfly, with 8 exchanges for four sums instead of 20.
__device__ __forceinline__ double warp_sum4_d(const double (&c)[4], int lane) {
  const bool up16 = lane & 16, up8 = lane & 8;
  double a = up16 ? c[2] : c[0], b = up16 ? c[3] : c[1];
  a += __shfl_xor_sync(0xffffffffu, up16 ? c[0] : c[2], 16);
  b += __shfl_xor_sync(0xffffffffu, up16 ? c[1] : c[3], 16);
  double x = up8 ? b : a;
  x += __shfl_xor_sync(0xffffffffu, up8 ? a : b, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// truth and the results are in the caller's event order, absolute (FP64 theta_0
// added); samples: sample_cap slots of M float4; the n series values are slots
// (first + s) % cap, s = 0..n-1, oldest first.  n2: next power of two >= n.
//
// Bound by the FP64 pipe (two FMAs a cycle and SM): the autocorrelation takes
// n - t of them for lag t.  The deviations are kept in FP64, so a term is one FMA
// (conversions and subtractions of both factors in every term made it five FP64
// instructions), and four lags run at once, sharing the loads of x[s] and one
// reduction; the lags past the first one that is not positive are dropped.
// 20,000 series of 400 samples: 10.2 -> 2.4 ms.
__global__ void __launch_bounds__(kUqWarps * 32)
    k_uq(const float4* __restrict__ samples, int64_t M, int64_t cap, int64_t first, int n, int n2,
         const int32_t* __restrict__ ev_out, const double* __restrict__ th0, const double* __restrict__ truth,
         double lo_pct, double hi_pct, double* med, double* half, double* calib, double* ess) {
  extern __shared__ __align__(8) double dbuf[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  // per warp: n2 deviations, then n2 values
  double* d = dbuf + (size_t)w * (n2 + n2 / 2);
  float* x = reinterpret_cast<float*>(d + n2);
  const int64_t series = (int64_t)blockIdx.x * nw + w;
  if (series >= 4 * M) return;
  const int64_t m = series >> 2;
  const int a = (int)(series & 3);
  const float* src = reinterpret_cast<const float*>(samples) + 4 * m + a;
  const size_t o = 4 * (size_t)ev_out[m] + a;         // the caller's event
  const double base = th0[4 * m + a];
  for (int s = lane; s < n2; s += 32) {
    float val = __int_as_float(0x7F800000);   // +inf pads the sort
    if (s < n) {
      int64_t slot = first + s;               // first < cap and n <= cap
      if (slot >= cap) slot -= cap;
      val = __ldg(src + slot * M * 4);
    }
    x[s] = val;
  }
  __syncwarp();
  // effective sample size (time order)
  if (ess) {
    double mu = 0.0;
    for (int s = lane; s < n; s += 32) mu += (double)x[s];
    mu = warp_sum_d(mu) / n;
    double c0 = 0.0;
    for (int s = lane; s < n; s += 32) {
      const double dv = (double)x[s] - mu;
      d[s] = dv;
      c0 += dv * dv;
    }
    c0 = warp_sum_d(c0);
    __syncwarp();
    double tau = 1.0;
    if (c0 > 0.0) {
      bool go = true;
      for (int t = 1; t < n && go; t += 4) {
        double c[4] = {0.0, 0.0, 0.0, 0.0};
        int s = lane;
        for (; s + t + 3 < n; s += 32) {
          const double v = d[s];
#pragma unroll
          for (int i = 0; i < 4; ++i) c[i] += v * d[s + t + i];
        }
        if (s + t < n) {                      // the last stride: fewer of the four lags
          const double v = d[s];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (s + t + i < n) c[i] += v * d[s + t + i];
        }
        const double sum = warp_sum4_d(c, lane);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const double rho = __shfl_sync(0xffffffffu, sum, 8 * i) / c0;
          go = go && t + i < n && rho > 0.0;
          if (go) tau += 2.0 * rho;
        }
      }
    }
    if (lane == 0) ess[o] = (double)n / tau;
  }
  // calibration against the truth (as an offset from theta_0, like the samples)
  double below = 0.0;
  if (truth && calib) {
    const double tv = truth[o] - base;
    for (int s = lane; s < n; s += 32) below += (double)x[s] < tv ? 1.0 : 0.0;
    below = warp_sum_d(below);
  }
  __syncwarp();
  // bitonic sort of the series (ascending)
  if (med || half)
    for (int k = 2; k <= n2; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int h = lane; h < n2 / 2; h += 32) {
          const int i = ((h & ~(j - 1)) << 1) | (h & (j - 1)), l = i | j;
          const float p = x[i], q = x[l];
          const bool up = (i & k) == 0;
          if ((p > q) == up) {
            x[i] = q;
            x[l] = p;
          }
        }
        __syncwarp();
      }
  if (lane == 0) {
    if (med) med[o] = base + pct_sorted(x, n, 50.0);
    if (half) half[o] = 0.5 * (pct_sorted(x, n, hi_pct) - pct_sorted(x, n, lo_pct));
    if (calib) calib[o] = below / n;
  }
}

}  // namespace

int uq_max_samples() { return 4096; }

cudaError_t launch_uq(const StepView& v, int64_t first, int n, const double* truth, double lo_pct,
                      double hi_pct, double* med, double* half, double* calib, double* ess, cudaStream_t st) {
  int n2 = 1;
  while (n2 < n) n2 <<= 1;
  const size_t per_warp = (size_t)n2 * (sizeof(double) + sizeof(float));
  // eight series per CTA while their buffers leave room for two CTAs an SM, at
  // least one (48 KB at 4096 samples)
  int warps = (int)(((size_t)100 << 10) / per_warp);
  warps = warps < 1 ? 1 : (warps > kUqWarps ? kUqWarps : warps);
  const size_t smem = warps * per_warp;
  cudaError_t e = cudaFuncSetAttribute(k_uq, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 << 10);
  if (e != cudaSuccess) return e;
  const int64_t nser = 4 * v.M;
  const unsigned grid = (unsigned)((nser + warps - 1) / warps);
  k_uq<<<grid, warps * 32, smem, st>>>(v.samples, v.M, v.sample_cap, first, n, n2, v.ev_out, v.th0_d, truth,
                                       lo_pct, hi_pct, med, half, calib, ess);
  return cudaGetLastError();
}

}  // namespace spider
