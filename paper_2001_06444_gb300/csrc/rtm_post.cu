// rtm_post.cu — per-shot normalisation and stacking, the Laplacian filter of
// the brute stack, and the ensemble statistics of stage 3 (sm_103a).
#include <cuda_runtime.h>

#include <cmath>

#include "rtm_common.h"
#include "rtm_launch.h"

namespace rtm {

// Source-normalised image of each item (Eq. 5; eps max(den) keeps the
// division finite, a pixel with zero illumination contributes 0), added in
// item order to its sample's stack with Kahan compensation; num and den are
// cleared for the next batch.  One thread per 4 consecutive pixels.
__global__ void k_norm_stack(float *num, float *den, const unsigned *dmax,
                             const int *item_sample, int B, float eps, long long pplane,
                             float *stack_all, float *comp_all, int nsample, int *err) {
  const long long e = 4 * (blockIdx.x * (long long)blockDim.x + threadIdx.x);
  if (e >= pplane) return;
  (void)nsample;
  (void)err;
  int cur = -1;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f), cmp = acc;
  for (int b = 0; b < B; ++b) {
    const int smp = item_sample[b];
    if (!RTM_IN(smp, nsample, err) || !RTM_IN(e + 3, pplane, err)) continue;
    if (smp != cur) {
      if (cur >= 0) {
        *reinterpret_cast<float4 *>(stack_all + cur * pplane + e) = acc;
        *reinterpret_cast<float4 *>(comp_all + cur * pplane + e) = cmp;
      }
      acc = *reinterpret_cast<const float4 *>(stack_all + smp * pplane + e);
      cmp = *reinterpret_cast<const float4 *>(comp_all + smp * pplane + e);
      cur = smp;
    }
    const float add = eps * __uint_as_float(dmax[b]);
    float4 *pn = reinterpret_cast<float4 *>(num + b * pplane + e);
    float4 *pd = reinterpret_cast<float4 *>(den + b * pplane + e);
    const float4 nu = *pn, de = *pd;
    const float nv[4] = {nu.x, nu.y, nu.z, nu.w};
    const float dv[4] = {de.x, de.y, de.z, de.w};
    float a[4] = {acc.x, acc.y, acc.z, acc.w};
    float c[4] = {cmp.x, cmp.y, cmp.z, cmp.w};
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const float dd = dv[l] + add;
      // eps < 0: the numerator as it is (the adjoint of Born modelling)
      const float img = eps < 0.f ? nv[l] : (dd > 0.f ? nv[l] / dd : 0.f);
      const float y = img - c[l];
      const float t = a[l] + y;
      c[l] = (t - a[l]) - y;
      a[l] = t;
    }
    acc = make_float4(a[0], a[1], a[2], a[3]);
    cmp = make_float4(c[0], c[1], c[2], c[3]);
    *pn = make_float4(0.f, 0.f, 0.f, 0.f);
    *pd = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  if (cur >= 0) {
    *reinterpret_cast<float4 *>(stack_all + cur * pplane + e) = acc;
    *reinterpret_cast<float4 *>(comp_all + cur * pplane + e) = cmp;
  }
}

// Laplacian filter of §3 on the stack: -(D_zz + D_xx) with 3-point second
// differences and the border value repeated outside; out is compact [nz][nx].
__global__ void k_filter(const float *stack_all, const float *comp_all, int nz, int nx, int SX,
                         float rdz2, float rdx2, int laplacian, float *out) {
  const int smp = blockIdx.z, i = blockIdx.y;
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nx) return;
  const long long base = (long long)smp * nz * SX;
  auto at = [&](int ii, int jj) {
    ii = min(max(ii, 0), nz - 1);
    jj = min(max(jj, 0), nx - 1);
    const long long o = base + (long long)ii * SX + jj;
    return stack_all[o] - comp_all[o];
  };
  const float c = at(i, j);
  float r = c;
  if (laplacian) {
    const float dzz = (at(i - 1, j) - 2.f * c) + at(i + 1, j);
    const float dxx = (at(i, j - 1) - 2.f * c) + at(i, j + 1);
    r = -(dzz * rdz2 + dxx * rdx2);
  }
  out[(long long)smp * nz * nx + (long long)i * nx + j] = r;
}

// Per-pixel statistics over n images: mean and standard deviation (divisor
// n-1) in FP64, and the 5% / 95% quantiles (linear interpolation at h = (n-1)
// p).  A block stages PB pixels x n values in shared memory, pixel-fastest, so
// global loads are coalesced and shared accesses are conflict-free.
//
// Two forms.  The general one sums in FP64, two passes, and sorts each pixel's
// column (bitonic).  It is bound by FP64 arithmetic, which this device runs at
// about 1/64 of the FP32 rate (5 FP64 operations a value), and by the sort:
// 0.70 ms for 64 x 597,051.  The other (3 to kFastN images, every value of the
// block finite) takes one pixel per thread and no FP64 operation per value:
//   - each value becomes an integer X on a grid 2^55 below the pixel's largest
//     power of two, so sum X is exact in 64 bits (a pixel with a value more than
//     2^31 times smaller than its largest, which the grid would cut, sums in FP64);
//   - with M the rounded mean of the X, sum (X - M)^2 is exact in three 64-bit
//     sums of products of 28-bit digits, and sum (X - mean)^2 = sum (X - M)^2 -
//     R^2 / n with R = sum X - n M: no cancellation, at most one rounding each
//     in FP64 per pixel;
//   - the quantiles need the few smallest and largest values only: sorted lists
//     of L in registers, 2 L minima and maxima a value.
constexpr int kFastN = 128;

// Quantile p of the sorted column from its two order statistics: separately
// rounded multiply and add (no FMA contraction), so the FP64 value, and hence
// its float rounding, is the textbook formula's.
__device__ __forceinline__ float interpolate(float xl, float xh, double f) {
  return (float)__dadd_rn((double)xl, __dmul_rn(f, __dsub_rn((double)xh, (double)xl)));
}

// The float with bits b as an integer on the grid 2^(emax - 181).
__device__ __forceinline__ long long grid_value(unsigned b, int emax) {
  const int e = (b >> 23) & 0xff;
  const unsigned long long m = (unsigned long long)((b & 0x7fffffu) | (e ? 0x800000u : 0u)) << 31;
  const long long x = (long long)(m >> min(emax - max(e, 1), 63));
  return (int)b < 0 ? -x : x;
}

// a / n correctly rounded from inv = 1 / n rounded (Markstein's correction)
__device__ __forceinline__ double div_by(double a, double n, double inv) {
  const double q = a * inv;
  return __fma_rn(__fma_rn(-q, n, a), inv, q);
}

template <int L>
__device__ __forceinline__ void fast_stats(const float *col, int n, int PB, int emax, double inv_n,
                                           double inv_n1, int lo5, int lo95, double f5, double f95,
                                           double &mean, double &sd, float &q5, float &q95) {
  float lowest[L], highest[L];  // sorted: lowest[0] the smallest, highest[0] the largest
#pragma unroll
  for (int i = 0; i < L; ++i) {
    lowest[i] = INFINITY;
    highest[i] = -INFINITY;
  }
  long long sum = 0;
#pragma unroll 4
  for (int k = 0; k < n; ++k) {
    const float v = col[k * PB];
    sum += grid_value(__float_as_uint(v), emax);
    float a = v, b = v;
#pragma unroll
    for (int i = 0; i < L; ++i) {
      const float c = fminf(lowest[i], a), d = fmaxf(highest[i], b);
      if (i + 1 < L) {
        a = fmaxf(lowest[i], a);
        b = fminf(highest[i], b);
      }
      lowest[i] = c;
      highest[i] = d;
    }
  }
  const double scale = __hiloint2double((emax - 181 + 1023) << 20, 0);  // of the grid
  const double mu = div_by((double)sum, (double)n, inv_n);
  mean = mu * scale;
  const long long M = __double2ll_rn(mu);
  unsigned long long s00 = 0, s10 = 0, s11 = 0;
#pragma unroll 4
  for (int k = 0; k < n; ++k) {
    const long long d = grid_value(__float_as_uint(col[k * PB]), emax) - M;
    const unsigned long long a = (unsigned long long)(d < 0 ? -d : d);
    const unsigned a0 = (unsigned)a & 0xfffffffu, a1 = (unsigned)(a >> 28);
    s00 += (unsigned long long)a0 * a0;
    s10 += (unsigned long long)a1 * a0;
    s11 += (unsigned long long)a1 * a1;
  }
  // (s10 < 2^63 and s11 <= 2^63 for n <= 128)
  double q = __fma_rn((double)s11, 72057594037927936.0,
                      __fma_rn((double)s10, 536870912.0, (double)s00));
  const double R = (double)(sum - n * M);
  q = __fma_rn(-R, R * inv_n, q);
  sd = n > 1 ? sqrt(div_by(q, (double)(n - 1), inv_n1)) * scale : 0.0;
  float a = lowest[0], b = lowest[0], c = highest[0], d = highest[0];
  const int hi5 = min(lo5 + 1, n - 1), hi95 = min(lo95 + 1, n - 1);
#pragma unroll
  for (int i = 1; i < L; ++i) {
    a = lo5 == i ? lowest[i] : a;
    b = hi5 == i ? lowest[i] : b;
    c = n - 1 - lo95 == i ? highest[i] : c;
    d = n - 1 - hi95 == i ? highest[i] : d;
  }
  q5 = interpolate(a, b, f5);
  q95 = interpolate(c, d, f95);
}

// Mean and standard deviation of one column in FP64, two passes, as sorted_stats
// takes them.
__device__ __forceinline__ void column_moments(const float *col, int n, int PB, double &mean,
                                               double &sd) {
  double s = 0.0;
  for (int k = 0; k < n; ++k) s += (double)col[k * PB];
  const double m = s / n;
  double q = 0.0;
  for (int k = 0; k < n; ++k) {
    const double d = (double)col[k * PB] - m;
    q += d * d;
  }
  mean = m;
  sd = n > 1 ? sqrt(q / (n - 1)) : 0.0;
}

// The general form on the column block in shared memory [npad][PB]: sums in FP64,
// two passes, and a bitonic sort of each column.
__device__ __forceinline__ void sorted_stats(float *sv, int n, int npad, int PB, long long p0,
                                             long long npix, double *mean, double *std_, float *q05,
                                             float *q95) {
  double mu[2] = {0.0, 0.0}, sd[2] = {0.0, 0.0};
  for (int p = threadIdx.x, t = 0; p < PB && t < 2; p += blockDim.x, ++t) {
    double s = 0.0;
    for (int k = 0; k < n; ++k) s += (double)sv[k * PB + p];
    const double m = s / n;
    double q = 0.0;
    for (int k = 0; k < n; ++k) {
      const double d = (double)sv[k * PB + p] - m;
      q += d * d;
    }
    mu[t] = m;
    sd[t] = n > 1 ? sqrt(q / (n - 1)) : 0.0;
  }
  __syncthreads();
  const int half = npad / 2;
  for (int k = 2; k <= npad; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < PB * half; t += blockDim.x) {
        const int p = t % PB, q = t / PB;
        const int i = ((q & ~(j - 1)) << 1) | (q & (j - 1));
        const int l = i | j;
        const float a = sv[i * PB + p], c = sv[l * PB + p];
        const bool up = (i & k) == 0;
        if ((a > c) == up) {
          sv[i * PB + p] = c;
          sv[l * PB + p] = a;
        }
      }
      __syncthreads();
    }
  }
  for (int p = threadIdx.x, t = 0; p < PB && t < 2; p += blockDim.x, ++t) {
    const long long pix = p0 + p;
    if (pix >= npix) continue;
    mean[pix] = mu[t];
    std_[pix] = sd[t];
    const double ps[2] = {0.05, 0.95};
    float qo[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const double h = __dmul_rn((double)(n - 1), ps[u]);  // (h - lo must not contract into one rounding)
      const int lo = (int)floor(h);
      qo[u] = interpolate(sv[lo * PB + p], sv[min(lo + 1, n - 1) * PB + p], h - lo);
    }
    q05[pix] = qo[0];
    q95[pix] = qo[1];
  }
}

// (A kernel of its own: as an instance of the fast one, which computes the
// quantiles' positions first and in every thread, it took 3 % longer, 129 images
// of 597,051 pixels 3433 -> 3538 us.)
__global__ void k_ens_stats(const float *images, int n, int npad, int PB, long long npix,
                            double *mean, double *std_, float *q05, float *q95) {
  extern __shared__ float sv[];  // [npad][PB]
  const long long p0 = (long long)blockIdx.x * PB;
  for (int idx = threadIdx.x; idx < npad * PB; idx += blockDim.x) {
    const int k = idx / PB, p = idx - k * PB;
    float x = INFINITY;
    if (k < n) x = (p0 + p < npix) ? images[(long long)k * npix + p0 + p] : 0.f;
    sv[idx] = x;
  }
  __syncthreads();
  sorted_stats(sv, n, npad, PB, p0, npix, mean, std_, q05, q95);
}

// One pixel per thread (blockDim.x >= PB); a block with a value that is not finite
// takes the general form.  L: length of the lists.
template <int L>
__global__ void k_ens_stats_fast(const float *images, int n, int npad, int PB, long long npix,
                                 double *mean, double *std_, float *q05, float *q95) {
  extern __shared__ float sv[];  // [npad][PB]
  const long long p0 = (long long)blockIdx.x * PB;
  const int p = threadIdx.x;
  const bool in = p < PB && p0 + p < npix;
  unsigned top = 0, low = 0xffffffffu;  // bits of the largest magnitude, of the smallest but 0 (less 1)
  if (p < PB) {
    const float *src = images + p0 + p;
#pragma unroll 8
    for (int k = 0; k < n; ++k) {
      const float v = in ? __ldcs(src + (long long)k * npix) : 0.f;
      sv[k * PB + p] = v;
      const unsigned mag = __float_as_uint(v) & 0x7fffffffu;
      top = max(top, mag);
      low = min(low, mag - 1u);  // (0 becomes the largest)
    }
  }
  if (!__syncthreads_or(top >= 0x7f800000u)) {  // all finite
    if (!in) return;
    const double h5 = __dmul_rn((double)(n - 1), 0.05), h95 = __dmul_rn((double)(n - 1), 0.95);
    const int lo5 = (int)floor(h5), lo95 = (int)floor(h95);
    double m, s;
    float a, b;
    const int emax = max((int)(top >> 23), 1);
    fast_stats<L>(sv + p, n, PB, emax, 1.0 / n, n > 1 ? 1.0 / (n - 1) : 0.0, lo5, lo95, h5 - lo5,
                  h95 - lo95, m, s, a, b);
    // a value too small for the pixel's grid was cut: where the large ones cancel,
    // it is the mean
    if (emax - max((int)((low + 1u) >> 23), 1) > 31 && low != 0xffffffffu)
      column_moments(sv + p, n, PB, m, s);
    mean[p0 + p] = m;
    std_[p0 + p] = s;
    q05[p0 + p] = a;
    q95[p0 + p] = b;
    return;
  }
  for (int idx = n * PB + threadIdx.x; idx < npad * PB; idx += blockDim.x) sv[idx] = INFINITY;
  __syncthreads();
  sorted_stats(sv, n, npad, PB, p0, npix, mean, std_, q05, q95);
}

__global__ void k_init_range(unsigned long long *mm) {
  mm[0] = 0ull;                    // max of a non-negative map
  mm[1] = 0x7FF0000000000000ull;  // +inf: min
}

// Extremes of the map: one pair of atomics per block (a pair per warp on the
// same two words took longer than the read).
constexpr int kRangeThreads = 256, kRangeLoads = 4;
__global__ void __launch_bounds__(kRangeThreads) k_std_range(const double *std_, long long npix,
                                                             unsigned long long *mm) {
  __shared__ double s_mx[kRangeThreads / 32], s_mn[kRangeThreads / 32];
  double mx = 0.0, mn = INFINITY;
  const long long stride = (long long)gridDim.x * kRangeThreads;
  for (long long e = blockIdx.x * (long long)kRangeThreads + threadIdx.x; e < npix;
       e += kRangeLoads * stride) {
    double x[kRangeLoads];
#pragma unroll
    for (int k = 0; k < kRangeLoads; ++k) x[k] = std_[e + k * stride < npix ? e + k * stride : e];
#pragma unroll
    for (int k = 0; k < kRangeLoads; ++k) {
      mx = fmax(mx, x[k]);
      mn = fmin(mn, x[k]);
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
  }
  if ((threadIdx.x & 31) == 0) {
    s_mx[threadIdx.x >> 5] = mx;
    s_mn[threadIdx.x >> 5] = mn;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kRangeThreads / 32; ++w) {
      mx = fmax(mx, s_mx[w]);
      mn = fmin(mn, s_mn[w]);
    }
    atomicMax(&mm[0], (unsigned long long)__double_as_longlong(mx));
    atomicMin(&mm[1], (unsigned long long)__double_as_longlong(mn));
  }
}

// Eq. 6: c = (s_max - s) / (s_max - s_min), 1 if the map is flat;
// Eq. 7: r = s / mean, 0 where the mean is 0.
__global__ void k_unc_maps(const double *mean, const double *std_, long long npix,
                           const unsigned long long *mm, double *conf, double *ratio) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= npix) return;
  const double smax = __longlong_as_double((long long)mm[0]);
  const double smin = __longlong_as_double((long long)mm[1]);
  const double s = std_[e], m = mean[e];
  conf[e] = smax > smin ? (smax - s) / (smax - smin) : 1.0;
  ratio[e] = m != 0.0 ? s / m : 0.0;
}

// ------------------------------------------------------------ launchers --

cudaError_t launch_norm_stack(float *num, float *den, const unsigned *dmax,
                              const int *item_sample, int B, float eps, long long pplane,
                              float *stack_all, float *comp_all, int nsample, int *err,
                              cudaStream_t st) {
  const long long n4 = pplane / 4;
  k_norm_stack<<<(unsigned)((n4 + 255) / 256), 256, 0, st>>>(
      num, den, dmax, item_sample, B, eps, pplane, stack_all, comp_all, nsample, err);
  return cudaGetLastError();
}

cudaError_t launch_filter(const float *stack_all, const float *comp_all, int nsample, int nz,
                          int nx, int SX, float rdz2, float rdx2, int laplacian, float *out,
                          cudaStream_t st) {
  dim3 grid((nx + 127) / 128, nz, nsample);
  k_filter<<<grid, 128, 0, st>>>(stack_all, comp_all, nz, nx, SX, rdz2, rdx2, laplacian, out);
  return cudaGetLastError();
}

int ens_stats_max_n() { return 32768; }

cudaError_t launch_ens_stats(const float *images, int n, long long npix, double *mean,
                             double *std_, float *q05, float *q95, cudaStream_t st) {
  int npad = 1;
  while (npad < n) npad <<= 1;
  if (npad < 2) npad = 2;
  int PB = (48 * 1024) / (4 * npad);
  if (PB > 256) PB = 256;
  if (PB < 1) PB = 1;
  const size_t smem = (size_t)PB * npad * sizeof(float);
  const long long blocks = (npix + PB - 1) / PB;
  auto go = [&](auto kernel, int threads) -> cudaError_t {
    if (smem > 48 * 1024) {
      const cudaError_t e = allow_shared_memory(kernel);
      if (e != cudaSuccess) return e;
    }
    kernel<<<(unsigned)blocks, threads, smem, st>>>(images, n, npad, PB, npix, mean, std_, q05, q95);
    return cudaGetLastError();
  };
  // the fast form's lists hold the order statistics up to floor(0.05 (n-1)) + 1
  // from either end: 3 for n <= 40, 5 for n <= 80, 8 for n <= 140
  const int threads = (PB + 31) / 32 * 32;
  // (one and two images: the general form's 72 and 97 us against 81 and 102 for
  // 597,051 pixels, where the fast form's FP64 operations per pixel outweigh it)
  if (n <= 2) return go(k_ens_stats, 256);
  if (n <= 40) return go(k_ens_stats_fast<3>, threads);
  if (n <= 80) return go(k_ens_stats_fast<5>, threads);
  if (n <= kFastN) return go(k_ens_stats_fast<8>, threads);
  return go(k_ens_stats, 256);
}

cudaError_t launch_unc_maps(const double *mean, const double *std_, long long npix,
                            double *conf, double *ratio, unsigned long long *scratch,
                            cudaStream_t st) {
  k_init_range<<<1, 1, 0, st>>>(scratch);
  long long blocks = (npix + 255) / 256;
  long long rb = (npix + kRangeThreads * kRangeLoads - 1) / (kRangeThreads * kRangeLoads);
  if (rb > 4 * 152) rb = 4 * 152;
  k_std_range<<<(unsigned)(rb < 1 ? 1 : rb), kRangeThreads, 0, st>>>(std_, npix, scratch);
  k_unc_maps<<<(unsigned)(blocks < 1 ? 1 : blocks), 256, 0, st>>>(mean, std_, npix, scratch,
                                                                  conf, ratio);
  return cudaGetLastError();
}

}  // namespace rtm
