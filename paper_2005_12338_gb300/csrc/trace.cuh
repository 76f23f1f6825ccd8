// Eq. 26's traces: sum_ij X_ij Y_ji per tau point, and their weighted sum over tau.
// Shared by the energies of rssri_sigma and by rssri_energy_static, so that both
// add in the same order.
//
// A tau point's matrix is dealt out as 32 x 32 tiles to `parts` blocks (Y's
// tile transposed through shared memory, so that both are read along rows).
// rssri_energy_static at n = 40, 32 tau points: 8.2 us a call, most of it the
// host's; 10.6 to 12.3 with one block per tau point, strided reads of Y and a
// second launch for the sum over tau.
#pragma once

#include <algorithm>

#include "common.cuh"

namespace rssri {

constexpr int TRACE_SLOTS = 4096;  // partial traces of a call at most (n_tau if that is more)

// Blocks per tau point.
inline int trace_parts(int n, int nt) {
  const long long t = (n + 31) / 32;
  return (int)std::max<long long>(1, std::min<long long>({t * t, TRACE_SLOTS / nt, 456 / nt + 1}));
}

__device__ __forceinline__ double trace_block_sum(double v, double *sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += sh[k];
  return s;
}

// Part p of `parts` of sum_ij x_ij y_ji (256 threads; every thread returns it).
__device__ __forceinline__ double trace_part(const double *__restrict__ x,
                                             const double *__restrict__ y, int n, int p, int parts) {
  __shared__ double sy[32][33];
  __shared__ double sh[8];
  const int T = (n + 31) / 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  double s = 0.0;
  for (int q = p; q < T * T; q += parts) {
    const int i0 = q / T * 32, j0 = q % T * 32;
    double xv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = ty + 8 * u;
      xv[u] = i0 + r < n && j0 + tx < n ? x[(long long)(i0 + r) * n + j0 + tx] : 0.0;
      sy[r][tx] = j0 + r < n && i0 + tx < n ? y[(long long)(j0 + r) * n + i0 + tx] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) s = fma(xv[u], sy[tx][ty + 8 * u], s);
    __syncthreads();
  }
  return trace_block_sum(s, sh);
}

// sum_t w_t tr_t, tr_t the sum of its parts in order, t in order: the products are
// formed by all threads (256), thread 0 adds them; valid in thread 0.
__device__ __forceinline__ double trace_weighted(const double *w, const double *part, int parts,
                                                 int nt) {
  __shared__ double sh[256];
  double a = 0.0;
  for (int t0 = 0; t0 < nt; t0 += 256) {
    const int t = t0 + threadIdx.x;
    if (t < nt && threadIdx.x < 256) {
      double s = 0.0;
      for (int p = 0; p < parts; ++p) s += part[(long long)t * parts + p];
      sh[threadIdx.x] = w[t] * s;
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int k = 0; k < min(256, nt - t0); ++k) a += sh[k];
    __syncthreads();
  }
  return a;
}

}  // namespace rssri
