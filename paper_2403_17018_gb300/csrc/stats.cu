// MLMC level statistics on the device (arxiv 2403.17018, section 3: Def. of
// Y_l and V_l, Eq. A). Every reduction has a fixed order, so the result
// depends only on the batch contents and B. What bounds these kernels on
// GB300 is FP64 latency and throughput, not memory, so none of them divides
// per sample: the QoI moments take two passes over the batch (mean, then
// squared deviations), the fields one pass about a shift close to the mean.
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "henry_device.cuh"

namespace henry {

constexpr int kStatThreads = 256;

// Block sum of a double, the same result in every thread (fixed order).
__device__ __forceinline__ double stat_sum(double v, double* sh) {
  const double s = block_sum(v, sh);
  __syncthreads();
  if (threadIdx.x == 0) sh[0] = s;
  __syncthreads();
  const double t = sh[0];
  __syncthreads();
  return t;
}

// Sum of squared deviations from the mean, given the sums f1 of deviations
// and f2 of squared deviations from a shift close to the mean and inv = 1 / n.
// Rounding of the difference must not leave a negative variance (a NaN stays).
__device__ __forceinline__ double centred_m2(double f1, double f2, double inv) {
  const double v = fma(-f1 * inv, f1, f2);
  return v < 0.0 ? 0.0 : v;
}

// Moments of one QoI (blockIdx.x) over the valid samples of the batch, two
// passes: out[0] = n, then mean_f, m2_f, mean_d, m2_d [kNQ] of g = q_fine
// and d = q_fine - q_coarse. The first pass sums the distances from the first
// valid sample, so that the mean of a constant batch (counted cells, empty
// boxes) is its value and its variance zero, exactly; the second the
// deviations from that mean (centred_m2). Grid kNQ blocks: 600
// samples take 8 us, where one block that ran Welford's update (two
// divisions per sample and QoI) took 387 us.
__global__ void __launch_bounds__(kStatThreads)
k_level_stats(unsigned long long* ctr, int B, const double* __restrict__ qf,
              const double* __restrict__ qc, const int* __restrict__ status,
              double* __restrict__ out) {
  HENRY_COUNT_LAUNCH(ctr);
  __shared__ double sh[kStatThreads / 32];
  __shared__ int first;
  const int k = blockIdx.x;
  if (threadIdx.x == 0) first = B;
  __syncthreads();
  int b0 = threadIdx.x;
  while (b0 < B && status && status[b0] != 0) b0 += kStatThreads;
  b0 = __reduce_min_sync(0xffffffffu, b0);
  if ((threadIdx.x & 31) == 0 && b0 < B) atomicMin(&first, b0);
  __syncthreads();
  double xf = 0.0, xd = 0.0;                // the first valid sample's g and d
  if (first < B) {
    xf = qf[(int64_t)first * kNQ + k];
    xd = qc ? xf - qc[(int64_t)first * kNQ + k] : xf;
  }
  double cnt = 0.0, sf = 0.0, sd = 0.0;
  auto each = [&](auto&& f) {
    for (int b = threadIdx.x; b < B; b += kStatThreads) {
      if (status && status[b] != 0) continue;
      const double g = qf[(int64_t)b * kNQ + k];
      f(g, qc ? g - qc[(int64_t)b * kNQ + k] : g);
    }
  };
  each([&](double g, double d) {
    cnt += 1.0;
    sf += g - xf;
    if (qc) sd += d - xd;
  });
  const double n = stat_sum(cnt, sh);
  const double inv = n > 0.0 ? 1.0 / n : 0.0;
  const double mf = fma(stat_sum(sf, sh), inv, xf);
  const double md = qc ? fma(stat_sum(sd, sh), inv, xd) : mf;
  double f1 = 0.0, f2 = 0.0, d1 = 0.0, d2 = 0.0;
  each([&](double g, double d) {
    const double e = g - mf;
    f1 += e;
    f2 = fma(e, e, f2);
    if (qc) {
      const double h = d - md;
      d1 += h;
      d2 = fma(h, h, d2);
    }
  });
  f1 = stat_sum(f1, sh);
  f2 = stat_sum(f2, sh);
  if (qc) {
    d1 = stat_sum(d1, sh);
    d2 = stat_sum(d2, sh);
  } else {
    d1 = f1;
    d2 = f2;
  }
  if (threadIdx.x == 0) {
    if (k == 0) out[0] = n;
    out[1 + k] = fma(f1, inv, mf);
    out[1 + kNQ + k] = centred_m2(f1, f2, inv);
    out[1 + 2 * kNQ + k] = fma(d1, inv, md);
    out[1 + 3 * kNQ + k] = centred_m2(d1, d2, inv);
  }
}

// Count, mean and sum of squared deviations of one group of samples.
struct Moments {
  double n, mean, m2;
};

// Chan's merge of b into a.
__device__ __forceinline__ void chan_merge(Moments& a, const Moments& b) {
  if (b.n == 0.0) return;
  if (a.n == 0.0) {
    a = b;
    return;
  }
  const double n = a.n + b.n, d = b.mean - a.mean, w = b.n / n;
  a.mean = fma(d, w, a.mean);
  a.m2 = a.m2 + b.m2 + d * d * (a.n * w);
  a.n = n;
}

// Per-cell statistics of c_l and c_l - P0 c_{l-1} over the batch, merged into
// the running state held in device memory. A block takes 32 cells and G
// groups of consecutive samples; each thread sums the deviations and their
// squares of its cell over its group's valid samples about a shift, the mean
// of eight samples from the group's first valid one on (which stands in for
// failed ones, summed in pairs: the shift of a constant cell is its value) or
// of fewer where the group has no more, so that nothing cancels: three FP64
// instructions per sample (and quantity). The groups are merged by a
// fixed tree (Chan). 600 samples of 8192 cells: 1028 us with a thread per cell running
// Welford's update, 61 us so.
constexpr int kShift = 8;

__global__ void __launch_bounds__(1024)
k_field_stats(unsigned long long* ctr, int nx, int ny, int B,
                              const double* __restrict__ cf, const double* __restrict__ cc,
                              const int* __restrict__ status, int64_t* __restrict__ n,
                              double* __restrict__ mean_f, double* __restrict__ m2_f,
                              double* __restrict__ mean_d, double* __restrict__ m2_d) {
  HENRY_COUNT_LAUNCH(ctr);
  extern __shared__ Moments mom[];          // [2][G][32], G a power of two
  const int G = blockDim.y, x = threadIdx.x, y = threadIdx.y;
  const int ncell = nx * ny;
  const int cell = blockIdx.x * 32 + x;
  const int b0 = (int)((int64_t)B * y / G), b1 = (int)((int64_t)B * (y + 1) / G);
  Moments f = {0.0, 0.0, 0.0}, d = {0.0, 0.0, 0.0};
  if (cell < ncell) {
    const int j = cell / nx, i = cell - j * nx;
    const int ncc = (nx / 2) * (ny / 2);
    const int ccell = (j >> 1) * (nx / 2) + (i >> 1);
    const double* pf = cf + cell;
    const double* pc = cc ? cc + ccell : nullptr;
    double kf = 0.0, kd = 0.0;
    int bs = b0;                              // the first valid sample
    while (bs < b1 && status && status[bs] != 0) ++bs;
    if (bs < b1 && b1 - bs < kShift) {        // a short group: its mean, from the first one's distance
      const double x0 = pf[(int64_t)bs * ncell], y0 = pc ? x0 - pc[(int64_t)bs * ncc] : 0.0;
      int c = 1;
      for (int b = bs + 1; b < b1; ++b) {
        if (status && status[b] != 0) continue;
        const double g = pf[(int64_t)b * ncell];
        kf += g - x0;
        if (pc) kd += (g - pc[(int64_t)b * ncc]) - y0;
        ++c;
      }
      const double w = c > 1 ? 1.0 / (double)c : 0.0;
      kf = fma(kf, w, x0);
      kd = fma(kd, w, y0);
    } else if (bs < b1) {
      double g[kShift], u[kShift];
#pragma unroll
      for (int m = 0; m < kShift; ++m) {
        const int b = bs + m < b1 && (!status || status[bs + m] == 0) ? bs + m : bs;
        g[m] = pf[(int64_t)b * ncell];
        u[m] = pc ? g[m] - pc[(int64_t)b * ncc] : 0.0;
      }
#pragma unroll
      for (int w = kShift / 2; w > 0; w >>= 1)
#pragma unroll
        for (int m = 0; m < w; ++m) {
          g[m] += g[m + w];
          u[m] += u[m + w];
        }
      kf = g[0] * (1.0 / kShift);
      kd = u[0] * (1.0 / kShift);
    }
    double f1 = 0.0, f2 = 0.0, d1 = 0.0, d2 = 0.0;
    int cnt = 0;
#pragma unroll 8
    for (int b = b0; b < b1; ++b) {
      const bool ok = !status || status[b] == 0;
      const double g = pf[(int64_t)b * ncell];
      const double h = pc ? pc[(int64_t)b * ncc] : 0.0;
      if (!ok) continue;
      ++cnt;
      const double e = g - kf;
      f1 += e;
      f2 = fma(e, e, f2);
      if (pc) {
        const double u = (g - h) - kd;
        d1 += u;
        d2 = fma(u, u, d2);
      }
    }
    if (cnt > 0) {
      const double w = 1.0 / (double)cnt;
      f = {(double)cnt, fma(f1, w, kf), centred_m2(f1, f2, w)};
      d = pc ? Moments{(double)cnt, fma(d1, w, kd), centred_m2(d1, d2, w)} : f;
    }
  }
  mom[y * 32 + x] = f;
  mom[(G + y) * 32 + x] = d;
  __syncthreads();
  // merge the groups pairwise, fine field and difference in different warps
  for (int h = G >> 1; h > 0; h >>= 1) {
    const int q = y / h, g = y - q * h;
    if (q < 2) chan_merge(mom[(q * G + g) * 32 + x], mom[(q * G + g + h) * 32 + x]);
    __syncthreads();
  }
  // and into the running state; its counts change once both have read them
  const int q = G > 1 ? y : 0;
  double total = 0.0;
  if (y < 2 && cell < ncell) {
    for (int r = q; r < (G > 1 ? q + 1 : 2); ++r) {
      double* mean = r ? mean_d : mean_f;
      double* m2 = r ? m2_d : m2_f;
      Moments t = {(double)n[cell], mean[cell], m2[cell]};
      chan_merge(t, mom[r * G * 32 + x]);
      mean[cell] = t.mean;
      m2[cell] = t.m2;
      total = t.n;
    }
  }
  __syncthreads();
  if (y == 0 && cell < ncell) n[cell] = (int64_t)total;
}

// Per-cell exceedance counts (section 4: probability that the salt mass
// fraction at a location exceeds a threshold): count[cell] += number of
// valid samples b with c_b[cell] > threshold (exact, independent of
// batching). 32 cells and G groups of samples per block; the comparison is
// one of 64-bit integers ordered like the doubles, not an FP64 instruction
// (112 us with a thread per cell, 12 us so, for 600 samples of 8192 cells).
__device__ __forceinline__ long long order_key(double v) {
  const long long b = __double_as_longlong(v);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

__global__ void __launch_bounds__(1024)
k_field_exceed(unsigned long long* ctr, int ncell, int B,
                               const double* __restrict__ c, const int* __restrict__ status,
                               double threshold, int64_t* __restrict__ count) {
  HENRY_COUNT_LAUNCH(ctr);
  extern __shared__ int cnt_sh[];           // [G][32]
  const int G = blockDim.y, x = threadIdx.x, y = threadIdx.y;
  const int cell = blockIdx.x * 32 + x;
  const int b0 = (int)((int64_t)B * y / G), b1 = (int)((int64_t)B * (y + 1) / G);
  // +0 stands for both zeros; a NaN (above infinity's key, or below
  // -infinity's) exceeds nothing
  const long long t = order_key(threshold == 0.0 ? 0.0 : threshold), inf = order_key(INFINITY);
  int k = 0;
  if (cell < ncell) {
#pragma unroll 8
    for (int b = b0; b < b1; ++b) {
      const long long v = order_key(c[(int64_t)b * ncell + cell]);
      k += (!status || status[b] == 0) && v > t && v <= inf ? 1 : 0;
    }
  }
  cnt_sh[y * 32 + x] = k;
  __syncthreads();
  if (y > 0 || cell >= ncell) return;
  int64_t s = 0;
  for (int g = 0; g < G; ++g) s += cnt_sh[g * 32 + x];
  count[cell] += s;
}

// Sample groups per block: enough that the blocks of a small grid, with at
// most 1024 threads each, still fill the GPU, and no more than samples.
static int sample_groups(int ncell, int B) {
  int G = (ncell + 31) / 32 < 152 ? 32 : 8;
  while (G > 1 && G > B) G /= 2;
  return G;
}

cudaError_t launch_field_exceed(unsigned long long* ctr, int ncell, int B, const double* c,
                                const int* status, double threshold, int64_t* count,
                                cudaStream_t s) {
  const int G = sample_groups(ncell, B);
  k_field_exceed<<<(ncell + 31) / 32, dim3(32, G), G * 32 * sizeof(int), s>>>(ctr, ncell, B, c, status,
                                                                              threshold, count);
  return cudaGetLastError();
}

cudaError_t launch_level_stats(unsigned long long* ctr, int B, const double* qf, const double* qc,
                               const int* status, double* out, cudaStream_t s) {
  k_level_stats<<<kNQ, kStatThreads, 0, s>>>(ctr, B, qf, qc, status, out);
  return cudaGetLastError();
}

cudaError_t launch_field_stats(unsigned long long* ctr, int nx, int ny, int B, const double* cf,
                               const double* cc, const int* status, int64_t* n, double* mean_f,
                               double* m2_f, double* mean_d, double* m2_d, cudaStream_t s) {
  const int ncell = nx * ny;
  const int G = sample_groups(ncell, B);
  k_field_stats<<<(ncell + 31) / 32, dim3(32, G), 2 * G * 32 * sizeof(Moments), s>>>(
      ctr, nx, ny, B, cf, cc, status, n, mean_f, m2_f, mean_d, m2_d);
  return cudaGetLastError();
}

}  // namespace henry
