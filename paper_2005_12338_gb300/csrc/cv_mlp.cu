// Learned control variate: per-element statistics of the stochastic terms,
// orbital-pair features, and a small MLP (10 -> 256 -> 256 -> 256 -> 1, SiLU)
// trained and evaluated by the kernels in this file.
//
// With E[F(R^L, R'^L)] = Sigma_DD exactly, Sigma_c = mean F(R,R') -
// c o (mean F(R^L,R'^L) - Sigma_DD) is unbiased for any c fixed independently
// of the draws it is used with, and per element its variance is smallest at
// c* = Cov(F, F^L) / Var(F^L).  The network maps features of (i, j, tau) to
// c = 1 + y and is fitted on an independent training run by minimising
// sum w (c - c*)^2 / sum w with w = Var(F^L).  The products of the two hidden
// 256 x 256 layers, forward and backward, run on the tensor cores with bf16
// operands and fp32 accumulation (tcgen05); the 10-wide input layer, the
// 1-wide output layer, activations, loss and Adam are fp32.  Fixed-order
// reductions throughout.
//
// A training step of 2,048 rows is small work in a long chain of launches: 17
// launches, each as wide as the shape allows, where element-wise passes join
// the product or the transposes next to them and the sums over rows (biases,
// input and output layer) run side by side in one launch.  100 steps with the
// statistics run at N = 64 take 21 ms; one launch per operation with the sums
// over rows on one or two blocks took 92 ms (the column sums ~150 us each).
#include <cuda_bf16.h>

#include "cv_mlp.cuh"
#include "tc_gemm.cuh"

namespace rssri {
namespace {

int grid_cap(long long work, int threads) {
  long long b = (work + threads - 1) / threads;
  return (int)(b < 1 ? 1 : (b > 152 * 32 ? 152 * 32 : b));
}

__global__ void sreduce_kernel(const float *__restrict__ part, int ks, int M, int N,
                               float *__restrict__ C, long long ldc, float alpha) {
  const long long mn = (long long)M * N;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < mn;
       e += (long long)gridDim.x * blockDim.x) {
    float s = 0.f;
    for (int k = 0; k < ks; ++k) s += part[k * mn + e];
    const long long i = e / N, j = e - i * N;
    C[i * ldc + j] = alpha * s;
  }
}

__device__ __forceinline__ float silu(float z) { return z / (1.f + __expf(-z)); }

// Layer 0 (10 inputs, fp32): Z = X W0^T + b, h = bf16(silu(Z)), A = silu(Z).  One
// thread per output; the ten products are added in ascending order.
__global__ void __launch_bounds__(256) layer0_kernel(const float *__restrict__ X,
                                                     const float *__restrict__ W,
                                                     const float *__restrict__ b, int m,
                                                     float *__restrict__ Z, float *__restrict__ A,
                                                     __nv_bfloat16 *__restrict__ h) {
  // block: 256 outputs of a row group; this thread's weights stay in registers
  const int j = threadIdx.x;
  float w[CV_NFEAT];
#pragma unroll
  for (int k = 0; k < CV_NFEAT; ++k) w[k] = W[j * CV_NFEAT + k];
  const float bj = b[j];
  for (long long r = blockIdx.x; r < m; r += gridDim.x) {
    float acc = 0.f;
#pragma unroll
    for (int k = 0; k < CV_NFEAT; ++k) acc = fmaf(X[r * CV_NFEAT + k], w[k], acc);
    const float z = acc + bj, av = silu(z);
    const long long e = r * CV_HIDDEN + j;
    Z[e] = z;
    A[e] = av;
    h[e] = __float2bfloat16_rn(av);
  }
}

// Z += b, A = silu(Z), h = bf16(A), four elements per thread (256 columns).
__global__ void __launch_bounds__(256) bias_silu_kernel(float *__restrict__ Z,
                                                        const float *__restrict__ b, long long total,
                                                        float *__restrict__ A,
                                                        __nv_bfloat16 *__restrict__ h) {
  for (long long e = 4 * (blockIdx.x * (long long)blockDim.x + threadIdx.x); e < total;
       e += 4LL * gridDim.x * blockDim.x) {
    float4 z = *reinterpret_cast<float4 *>(Z + e);
    const float4 bv = *reinterpret_cast<const float4 *>(b + (e & (CV_HIDDEN - 1)));
    z.x += bv.x;
    z.y += bv.y;
    z.z += bv.z;
    z.w += bv.w;
    const float4 a = make_float4(silu(z.x), silu(z.y), silu(z.z), silu(z.w));
    *reinterpret_cast<float4 *>(Z + e) = z;
    *reinterpret_cast<float4 *>(A + e) = a;
    const __nv_bfloat162 lo = __floats2bfloat162_rn(a.x, a.y), hi = __floats2bfloat162_rn(a.z, a.w);
    *reinterpret_cast<uint2 *>(h + e) = make_uint2(*reinterpret_cast<const uint32_t *>(&lo),
                                                   *reinterpret_cast<const uint32_t *>(&hi));
  }
}

// The last hidden layer's bias and silu, and the output layer: Z += b, A = silu(Z),
// y = sum_k A_k w_k + b3, k ascending.  32 rows per block through shared memory; a
// lane owns a row, so that the sum runs in order at register speed.
__global__ void __launch_bounds__(256) output_kernel(float *__restrict__ Z, const float *__restrict__ b,
                                                     const float *__restrict__ w3,
                                                     const float *__restrict__ b3, int m,
                                                     float *__restrict__ A, float *__restrict__ y) {
  __shared__ float s[32][CV_HIDDEN + 1];
  __shared__ float w[CV_HIDDEN];
  const long long r0 = (long long)blockIdx.x * 32;
  const int c = threadIdx.x;
  w[c] = w3[c];
  const float bc = b[c];
#pragma unroll 8
  for (int r = 0; r < 32; ++r) {
    if (r0 + r >= m) break;
    const long long e = (r0 + r) * CV_HIDDEN + c;
    const float z = Z[e] + bc, a = silu(z);
    Z[e] = z;
    A[e] = a;
    s[r][c] = a;
  }
  __syncthreads();
  if (threadIdx.x < 32 && r0 + threadIdx.x < m) {
    float acc = 0.f;
#pragma unroll 16
    for (int k = 0; k < CV_HIDDEN; ++k) acc = fmaf(s[threadIdx.x][k], w[k], acc);
    y[r0 + threadIdx.x] = acc + b3[0];
  }
}

// d = dA silu'(Z) for one element.
__device__ __forceinline__ float silu_back(float dA, float z) {
  const float s = 1.f / (1.f + __expf(-z));
  return dA * s * (1.f + z * (1.f - s));
}

// Z <- dA silu'(Z) with dA given, or dA = dy w3^T (w3 non-null); h = bf16(Z) (may be
// null); and with t0: bf16 transposes t0 of the new Z and t1 of A, [256][ldt] with
// columns m..ldt-1 zero.  32 x 32 tiles through shared memory.
__global__ void __launch_bounds__(256) back_kernel(const float *__restrict__ dA,
                                                   const float *__restrict__ dy,
                                                   const float *__restrict__ w3, float *__restrict__ Z,
                                                   const float *__restrict__ A, int m,
                                                   __nv_bfloat16 *__restrict__ h,
                                                   __nv_bfloat16 *__restrict__ t0,
                                                   __nv_bfloat16 *__restrict__ t1, long long ldt) {
  __shared__ float sz[32][33], sa[32][33];
  const long long r0 = (long long)blockIdx.x * 32;
  const int c0 = blockIdx.y * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
  for (int k = ty; k < 32; k += 8) {
    const long long r = r0 + k;
    float d = 0.f, a = 0.f;
    if (r < m) {
      const long long e = r * CV_HIDDEN + c0 + tx;
      // dy w3 as a product of one term: fma(dy, w3, 0)
      d = silu_back(w3 ? fmaf(dy[r], w3[c0 + tx], 0.f) : dA[e], Z[e]);
      Z[e] = d;
      if (h) h[e] = __float2bfloat16_rn(d);
      if (t0) a = A[e];
    }
    sz[k][tx] = d;
    sa[k][tx] = a;
  }
  if (!t0) return;
  __syncthreads();
#pragma unroll
  for (int k = ty; k < 32; k += 8) {
    const long long r = r0 + tx;
    if (r < ldt) {
      t0[(long long)(c0 + k) * ldt + r] = __float2bfloat16_rn(sz[tx][k]);
      t1[(long long)(c0 + k) * ldt + r] = __float2bfloat16_rn(sa[tx][k]);
    }
  }
}

// bf16 copies of W1, W2 and their transposes (32 x 32 tiles; blockIdx.z: which).
__global__ void __launch_bounds__(256) weights_kernel(const float *__restrict__ W1,
                                                      const float *__restrict__ W2,
                                                      __nv_bfloat16 *__restrict__ w) {
  constexpr int H = CV_HIDDEN;
  __shared__ float t[32][33];
  const float *W = blockIdx.z ? W2 : W1;
  __nv_bfloat16 *o = w + (long long)blockIdx.z * H * H, *ot = w + (2LL + blockIdx.z) * H * H;
  const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int k = ty; k < 32; k += 8) {
    const float v = W[(r0 + k) * H + c0 + tx];
    o[(r0 + k) * H + c0 + tx] = __float2bfloat16_rn(v);
    t[k][tx] = v;
  }
  __syncthreads();
  for (int k = ty; k < 32; k += 8) ot[(c0 + k) * H + r0 + tx] = __float2bfloat16_rn(t[tx][k]);
}

// Per warp of the loss sum: thread t of 1024 adds the elements t, t + 1024, ... in
// order, then the warp its 32 sums; block b is warp b.  sums [2][32].
constexpr int LOSS_T = 1024;
__global__ void loss_sums_kernel(const float *__restrict__ y, const float *__restrict__ t,
                                 const float *__restrict__ w, int M, double *__restrict__ sums) {
  double sw = 0, sl = 0;
  for (int i = blockIdx.x * 32 + threadIdx.x; i < M; i += LOSS_T) {
    sw += w[i];
    const double r = 1.0 + y[i] - t[i];
    sl += w[i] * r * r;
  }
  for (int o = 16; o > 0; o >>= 1) {
    sw += __shfl_down_sync(0xffffffffu, sw, o);
    sl += __shfl_down_sync(0xffffffffu, sl, o);
  }
  if (threadIdx.x == 0) {
    sums[blockIdx.x] = sw;
    sums[32 + blockIdx.x] = sl;
  }
}
// dy = 2 w (1 + y - t) / sum w (dy may be null); loss = sum w (1 + y - t)^2 / sum w
__global__ void loss_kernel(const float *__restrict__ y, const float *__restrict__ t,
                            const float *__restrict__ w, int M, const double *__restrict__ sums,
                            float *__restrict__ dy, float *__restrict__ loss) {
  double swt = 0, slt = 0;
  for (int k = 0; k < 32; ++k) {
    swt += sums[k];
    slt += sums[32 + k];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0 && loss) loss[0] = (float)(slt / swt);
  if (!dy) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < M; i += gridDim.x * blockDim.x)
    dy[i] = (float)(2.0 * w[i] * (1.0 + y[i] - t[i]) / swt);
}

// The sums over the m rows that the parameter gradients need, one launch, each in
// ascending row order within its chunk of kc rows (ks chunks; the biases in one):
//   block roles  [0, 24)              db of layer 2, 1, 0: column sums of dZ2, dZ1, dZ0
//                [24, 24 + 8 ks)      dW3 = dy^T A2 (32 columns, one chunk)
//                [.., + 8 ks)         dW0 = dZ0^T X (32 rows, one chunk)
//                last                 db3 = sum dy
// Rows are staged through shared memory in double-buffered pieces, so that the
// chain of dependent adds (4 cycles each) is what a block waits for, not memory:
// one thread per column straight from memory took ~150 us for 2,048 rows.
struct SumArgs {
  const float *dz[3], *dy, *a2, *x;
  float *db[3], *db3, *w3, *w0;  // w3, w0: results (ks = 1) or [ks] partials
  int m, ks, kc;
};
constexpr int SROWS = 128;
__global__ void __launch_bounds__(320) sums_kernel(const SumArgs g) {
  __shared__ float buf[2][SROWS][33];
  __shared__ float aux[2][SROWS][CV_NFEAT];
  const int role = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float *src;
  int c0, kbeg = 0, kend = g.m, kind, z = 0;  // kind: 0 column sum, 1 dW3, 2 dW0, 3 sum of dy
  if (role < 24) {
    kind = 0;
    src = g.dz[role >> 3];
    c0 = (role & 7) * 32;
  } else if (role < 24 + 16 * g.ks) {
    const int q = role - 24;
    kind = q < 8 * g.ks ? 1 : 2;
    const int u = kind == 1 ? q : q - 8 * g.ks;
    src = kind == 1 ? g.a2 : g.dz[2];
    c0 = (u & 7) * 32;
    z = u >> 3;
    kbeg = z * g.kc;
    kend = min(g.m, kbeg + g.kc);
  } else {
    kind = 3;
    src = g.dy;
    c0 = 0;
  }
  // a piece: 128 rows x 32 columns (kind 3: 128 values of dy in column 0)
  constexpr int PER = (SROWS * 32 + 319) / 320;
  constexpr int PAX = (SROWS * CV_NFEAT + 319) / 320;
  float v[PER], ax[PAX];
  auto load = [&](int k0) {
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int e = tid + p * 320, r = e >> 5, c = e & 31;
      v[p] = 0.f;
      if (e < SROWS * 32 && k0 + r < kend) {
        if (kind != 3) v[p] = src[(long long)(k0 + r) * CV_HIDDEN + c0 + c];
        else if (c == 0) v[p] = src[k0 + r];
      }
    }
#pragma unroll
    for (int p = 0; p < PAX; ++p) {
      const int e = tid + p * 320;
      ax[p] = 0.f;
      if (kind == 2 && e < SROWS * CV_NFEAT && k0 + e / CV_NFEAT < kend)
        ax[p] = g.x[(long long)k0 * CV_NFEAT + e];
      if (kind == 1 && e < SROWS && k0 + e < kend) ax[p] = g.dy[k0 + e];
    }
  };
  auto store = [&](int bsel) {
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int e = tid + p * 320;
      if (e < SROWS * 32) buf[bsel][e >> 5][e & 31] = v[p];
    }
#pragma unroll
    for (int p = 0; p < PAX; ++p) {
      const int e = tid + p * 320;
      if (kind == 2 && e < SROWS * CV_NFEAT) aux[bsel][e / CV_NFEAT][e % CV_NFEAT] = ax[p];
      if (kind == 1 && e < SROWS) aux[bsel][e][0] = ax[p];
    }
  };
  float acc = 0.f;
  int bsel = 0;
  load(kbeg);
  store(0);
  __syncthreads();
  for (int k0 = kbeg; k0 < kend; k0 += SROWS) {
    const bool more = k0 + SROWS < kend;
    if (more) load(k0 + SROWS);
    const int cnt = min(SROWS, kend - k0);
    if (kind == 2) {
#pragma unroll 16
      for (int r = 0; r < cnt; ++r) acc = fmaf(buf[bsel][r][lane], aux[bsel][r][warp], acc);
    } else if (warp == 0 && kind == 1) {
#pragma unroll 16
      for (int r = 0; r < cnt; ++r) acc = fmaf(aux[bsel][r][0], buf[bsel][r][lane], acc);
    } else if (warp == 0) {
#pragma unroll 16
      for (int r = 0; r < cnt; ++r) acc += buf[bsel][r][lane];
    }
    if (more) {
      store(bsel ^ 1);
      __syncthreads();
      bsel ^= 1;
    }
  }
  if (kind == 0 && warp == 0) g.db[role >> 3][c0 + lane] = acc;
  if (kind == 1 && warp == 0) g.w3[(long long)z * CV_HIDDEN + c0 + lane] = acc;
  if (kind == 2) g.w0[((long long)z * CV_HIDDEN + c0 + lane) * CV_NFEAT + warp] = acc;
  if (kind == 3 && tid == 0) g.db3[0] = acc;
}

// The chunks' partial sums of dW3 and dW0, added in order.
__global__ void sums_reduce_kernel(const float *__restrict__ p3, const float *__restrict__ p0, int ks,
                                   float *__restrict__ w3, float *__restrict__ w0) {
  const int n3 = CV_HIDDEN, n0 = CV_HIDDEN * CV_NFEAT;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n3 + n0; e += gridDim.x * blockDim.x) {
    const bool a = e < n3;
    const float *p = a ? p3 + e : p0 + (e - n3);
    const int st = a ? n3 : n0;
    float s = 0.f;
    for (int k = 0; k < ks; ++k) s += p[(long long)k * st];
    (a ? w3[e] : w0[e - n3]) = s;
  }
}

__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g,
                            float *__restrict__ m, float *__restrict__ v, int n, float lr, float b1,
                            float b2, float eps, float bc1, float bc2) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const float gi = g[e];
    const float mi = b1 * m[e] + (1.f - b1) * gi;
    const float vi = b2 * v[e] + (1.f - b2) * gi * gi;
    m[e] = mi;
    v[e] = vi;
    p[e] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
  }
}

// stats[0..4][e] += F, F^L, F^2, (F^L)^2, F F^L with F = BC[x], F^L = -BC[nh + x]
__global__ void cv_stats_kernel(const double *__restrict__ BC, int nh, long long nn,
                                double *__restrict__ stats) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nn;
       e += (long long)gridDim.x * blockDim.x) {
    double s0 = 0, s1 = 0, s2 = 0, s3 = 0, s4 = 0;
    for (int x = 0; x < nh; ++x) {
      const double f = BC[(long long)x * nn + e], fl = -BC[(long long)(nh + x) * nn + e];
      s0 += f;
      s1 += fl;
      s2 += f * f;
      s3 += fl * fl;
      s4 += f * fl;
    }
    stats[e] += s0;
    stats[nn + e] += s1;
    stats[2 * nn + e] += s2;
    stats[3 * nn + e] += s3;
    stats[4 * nn + e] += s4;
  }
}

// c* = Cov(F, F^L) / Var(F^L) (1 where Var = 0), weight Var(F^L)
__global__ void cv_targets_kernel(const double *__restrict__ stats, long long nn, int nt, int ns,
                                  float *__restrict__ target, float *__restrict__ weight) {
  const long long total = nn * nt;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long t = e / nn, r = e - t * nn;
    const double *s = stats + t * 5 * nn;
    const double sf = s[r], sl = s[nn + r], sll = s[3 * nn + r], sfl = s[4 * nn + r];
    const double var = (sll - sl * sl / ns) / (ns - 1);
    const double cov = (sfl - sf * sl / ns) / (ns - 1);
    const bool ok = var > 0.0;
    target[e] = ok ? (float)(cov / var) : 1.f;
    weight[e] = ok ? (float)var : 0.f;
  }
}

// per tau: mx[t] = {max |sdd(t)|, max_k |G_kk(t)|, max_k |Gb_kk(t)|}
__global__ void cv_maxima_kernel(const double *__restrict__ sdd, const double *__restrict__ G,
                                 const double *__restrict__ Gb, int n, double *__restrict__ mx) {
  __shared__ double sh[3][32];
  const int t = blockIdx.x;
  const long long nn = (long long)n * n;
  double a = 0, b = 0, c = 0;
  for (long long e = threadIdx.x; e < nn; e += blockDim.x) a = fmax(a, fabs(sdd[t * nn + e]));
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    b = fmax(b, fabs(G[t * nn + (long long)k * n + k]));
    c = fmax(c, fabs(Gb[t * nn + (long long)k * n + k]));
  }
  for (int o = 16; o > 0; o >>= 1) {
    a = fmax(a, __shfl_down_sync(0xffffffffu, a, o));
    b = fmax(b, __shfl_down_sync(0xffffffffu, b, o));
    c = fmax(c, __shfl_down_sync(0xffffffffu, c, o));
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (l == 0) {
    sh[0][w] = a;
    sh[1][w] = b;
    sh[2][w] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < nw; ++k) {
      sh[0][0] = fmax(sh[0][0], sh[0][k]);
      sh[1][0] = fmax(sh[1][0], sh[1][k]);
      sh[2][0] = fmax(sh[2][0], sh[2][k]);
    }
    mx[3 * t] = sh[0][0];
    mx[3 * t + 1] = sh[1][0];
    mx[3 * t + 2] = sh[2][0];
  }
}

// rn[i] = Frobenius norm of row i of [K]^L (sum over its kept pairs and Q)
__global__ void cv_rownorm_kernel(const double *__restrict__ KP, const int *__restrict__ rowptr,
                                  int naux, double *__restrict__ rn) {
  const int i = blockIdx.x;
  double s = 0;
  const long long beg = (long long)rowptr[i] * naux, end = (long long)rowptr[i + 1] * naux;
  for (long long e = beg + threadIdx.x; e < end; e += blockDim.x) s += KP[e] * KP[e];
  __shared__ double sh[32];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) v += sh[k];
    rn[i] = sqrt(v);
  }
}

// out[0] = max x[0..n)
__global__ void max_small_kernel(const double *__restrict__ x, int n, double *__restrict__ out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double m = 0;
  for (int i = 0; i < n; ++i) m = fmax(m, x[i]);
  out[0] = m;
}

__global__ void cv_features_kernel(const double *__restrict__ sdd, const double *__restrict__ G,
                                   const double *__restrict__ Gb, const double *__restrict__ tau,
                                   double lnbeta, const double *__restrict__ rn,
                                   const double *__restrict__ rmaxp, const double *__restrict__ mx,
                                   int n, int nt, float *__restrict__ X) {
  const double rmax = rmaxp[0];
  const long long nn = (long long)n * n, total = nn * nt;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long t = e / nn, r = e - t * nn;
    const int i = (int)(r / n), j = (int)(r - (long long)i * n);
    const double *g = G + t * nn, *gb = Gb + t * nn;
    const double sm = mx[3 * t], gm = mx[3 * t + 1], gbm = mx[3 * t + 2];
    float *f = X + e * CV_NFEAT;
    f[0] = (float)((double)abs(i - j) / n);
    f[1] = (float)(log(tau[t]) / lnbeta);
    f[2] = sm > 0 ? (float)(sdd[t * nn + r] / sm) : 0.f;
    f[3] = (float)(g[(long long)i * n + i] / gm);
    f[4] = (float)(g[(long long)j * n + j] / gm);
    f[5] = (float)(gb[(long long)i * n + i] / gbm);
    f[6] = (float)(gb[(long long)j * n + j] / gbm);
    f[7] = rmax > 0 ? (float)(rn[i] / rmax) : 0.f;
    f[8] = rmax > 0 ? (float)(rn[j] / rmax) : 0.f;
    f[9] = (i == j) ? 1.f : 0.f;
  }
}

// Rows (start + k stride) mod total, k < m, of the features, targets and weights.
__global__ void gather_batch_kernel(const float *__restrict__ X, const float *__restrict__ T,
                                    const float *__restrict__ W, long long total, long long start,
                                    long long stride, int m, float *__restrict__ bx,
                                    float *__restrict__ bt, float *__restrict__ bw) {
  constexpr int C = CV_NFEAT + 2;
  const long long n = (long long)m * C;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const long long k = e / C;
    const int c = (int)(e - k * C);
    const long long row = (start + k * stride) % total;
    if (c < CV_NFEAT) bx[k * CV_NFEAT + c] = X[row * CV_NFEAT + c];
    else if (c == CV_NFEAT) bt[k] = T[row];
    else bw[k] = W[row];
  }
}

__global__ void add_one_kernel(const float *__restrict__ y, long long m, double *__restrict__ c) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < m;
       e += (long long)gridDim.x * blockDim.x)
    c[e] = 1.0 + (double)y[e];
}

// sig = (init ? c o base : sig) + sum_x (BC[x] + c o BC[nh + x]) / ns   (BC[nh+x] = -F^L)
__global__ void cv_accumulate_kernel(const double *__restrict__ BC, int nh, long long nn,
                                     double ns, const double *__restrict__ base,
                                     const double *__restrict__ c, int init,
                                     double *__restrict__ sig) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nn;
       e += (long long)gridDim.x * blockDim.x) {
    const double ce = c[e];
    double acc = 0.0;
    for (int x = 0; x < nh; ++x)
      acc += BC[(long long)x * nn + e] + ce * BC[(long long)(nh + x) * nn + e];
    sig[e] = (init ? ce * base[e] : sig[e]) + acc / ns;
  }
}

// e_st[x] += -w ((2 t^2 - s2) - Tr((c o F^L) Gb)) / ne, block per pair x
__global__ void cv_pair_energy_kernel(const double *__restrict__ BC, int nh, int n,
                                      const double *__restrict__ c, const double *__restrict__ gb,
                                      const double *__restrict__ t, const double *__restrict__ s2,
                                      double w, double ne, double *__restrict__ e_st) {
  __shared__ double sh[32];
  const int x = blockIdx.x;
  const long long nn = (long long)n * n;
  const double *FL = BC + (long long)(nh + x) * nn;  // -F^L
  double q = 0;
  for (long long e = threadIdx.x; e < nn; e += blockDim.x) {
    const long long i = e / n, j = e - i * n;
    q += c[e] * FL[e] * gb[j * n + i];
  }
  for (int o = 16; o > 0; o >>= 1) q += __shfl_down_sync(0xffffffffu, q, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = q;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) v += sh[k];
    const double de = (2.0 * t[x] * t[x] - s2[x]) + v;
    e_st[x] += -w * de / ne;
  }
}

// out[t] = sum_ij W[t][i][j] X[t][i][j] Y[t][j][i]
__global__ void trace_prod_w_kernel(const double *__restrict__ X, const double *__restrict__ Y,
                                    const double *__restrict__ W, int n, double *__restrict__ out) {
  __shared__ double sh[32];
  const int ti = blockIdx.x;
  const long long nn = (long long)n * n;
  const double *x = X + ti * nn, *y = Y + ti * nn, *w = W + ti * nn;
  double s = 0.0;
  for (long long e = threadIdx.x; e < nn; e += blockDim.x) {
    const long long i = e / n, j = e - i * n;
    s += w[e] * x[e] * y[j * n + i];
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) v += sh[k];
    out[ti] = v;
  }
}

}  // namespace

// ------------------------------------------------------------ launchers --
#define RS_L()                  \
  do {                          \
    ++launch_counter();         \
    RS_TRY(cudaGetLastError()); \
  } while (0)

// Parameter layout (floats): W0 [256][10], b0, W1 [256][256], b1, W2, b2, W3 [1][256], b3.
namespace {
constexpr long long O_W0 = 0, O_B0 = O_W0 + CV_HIDDEN * CV_NFEAT, O_W1 = O_B0 + CV_HIDDEN,
                    O_B1 = O_W1 + CV_HIDDEN * CV_HIDDEN, O_W2 = O_B1 + CV_HIDDEN,
                    O_B2 = O_W2 + CV_HIDDEN * CV_HIDDEN, O_W3 = O_B2 + CV_HIDDEN,
                    O_B3 = O_W3 + CV_HIDDEN;
static_assert(O_B3 + 1 == CV_NPARAM, "parameter layout");
}  // namespace

// Split of a contraction over the m rows into g chunks of kc (a multiple of
// 64): the tensor-core weight-gradient products take the chunks as batch
// entries of strided views of one transposed buffer of row stride g kc.
void tc_split(int m, int *g, int *kc) {
  int gg = std::max(1, std::min(8, m / 2048));
  int k = (ceil_div(m, gg) + 63) / 64 * 64;
  *g = gg;
  *kc = k;
}

long long tc_ldt(int m) {
  int g, kc;
  tc_split(m, &g, &kc);
  return (long long)g * kc;
}

// act layout (floats): Z0 A0 Z1 A1 Z2 A2 [m][256] fp32, y [m], dy [m], 2 spare,
// then bf16: H0, H1 [m][256] (bf16 activations / gradient rows), T0, T1
// [256][ldt] (transposes for the weight gradients)
size_t cv_act_floats(int m) {
  // tc_ldt(m) <= m + 8 * 63: sized with m + 512 so that the size grows with m
  return (size_t)m * (6 * CV_HIDDEN + 4) + (size_t)m * CV_HIDDEN +
         (size_t)CV_HIDDEN * ((size_t)m + 512);
}

// work layout (floats): bf16 W1, W2, W1^T, W2^T (4 x 256 x 256), the weight
// gradient partials [8][256][256] fp32, then the fp32 products' split-K scratch
size_t cv_tc_work_floats() {
  return 2LL * CV_HIDDEN * CV_HIDDEN + 8LL * CV_HIDDEN * CV_HIDDEN;
}

namespace {
struct Bf16Bufs {
  __nv_bfloat16 *h0, *h1, *t0, *t1, *w[2], *wt[2];
  float *part;
  float *work;  // fp32 split-K scratch
  long long ldt;
};

Bf16Bufs bf16_bufs(const float *params, float *act, float *work, int m) {
  const int H = CV_HIDDEN;
  Bf16Bufs b;
  float *base = act + (long long)m * (6 * H + 4);
  b.h0 = reinterpret_cast<__nv_bfloat16 *>(base);
  b.h1 = b.h0 + (long long)m * H;
  b.ldt = tc_ldt(m);
  b.t0 = b.h1 + (long long)m * H;
  b.t1 = b.t0 + (long long)H * b.ldt;
  __nv_bfloat16 *wb = reinterpret_cast<__nv_bfloat16 *>(work);
  b.w[0] = wb;
  b.w[1] = wb + H * H;
  b.wt[0] = wb + 2 * H * H;
  b.wt[1] = wb + 3 * H * H;
  b.part = work + 2 * H * H;
  b.work = b.part + 8 * H * H;
  (void)params;
  return b;
}

TcOperand tco(const void *p, long long ld, long long sb, int rows) {
  TcOperand t;
  t.ptr = p;
  t.ld = ld;
  t.sb = sb;
  t.rows = rows;
  return t;
}

// C [M][N] fp32 = A [M][K] B^T, A and B bf16 K-contiguous (tensor cores)
cudaError_t tc_mm(const __nv_bfloat16 *A, long long lda, const __nv_bfloat16 *B, long long ldb,
                  int M, int N, int K, float *C, cudaStream_t s) {
  TcGemm g;
  g.kind = TC_BF16;
  g.M = M;
  g.N = N;
  g.K[0] = K;
  g.A[0] = tco(A, lda, 0, M);
  g.B[0] = tco(B, ldb, 0, N);
  g.c32 = C;
  return tc_gemm(g, s);
}

// dW [N][M]... : out[o][i] = sum_r At[o][r] Bt[i][r] over r < m, split into g
// chunks (batch entries of strided views), partials reduced in order
cudaError_t tc_wgrad(const __nv_bfloat16 *At, const __nv_bfloat16 *Bt, long long ldt, int m,
                     float *part, float *out, cudaStream_t s) {
  const int H = CV_HIDDEN;
  int g, kc;
  tc_split(m, &g, &kc);
  TcGemm t;
  t.kind = TC_BF16;
  t.M = H;
  t.N = H;
  t.batch = g;
  t.bpc = 1;
  t.K[0] = kc;
  t.A[0] = tco(At, ldt, kc, H);
  t.B[0] = tco(Bt, ldt, kc, H);
  t.c32 = g == 1 ? out : part;
  RS_TRY(tc_gemm(t, s));
  if (g == 1) return cudaSuccess;
  sreduce_kernel<<<grid_cap((long long)H * H, 256), 256, 0, s>>>(part, g, H, H, out, H, 1.f);
  ++launch_counter();
  return cudaGetLastError();
}

}  // namespace

cudaError_t cv_forward(const float *params, const float *X, int m, float *act, float *work,
                       cudaStream_t s) {
  const int H = CV_HIDDEN;
  const long long mh = (long long)m * H;
  float *Z0 = act, *A0 = Z0 + mh, *Z1 = A0 + mh, *A1 = Z1 + mh, *Z2 = A1 + mh, *A2 = Z2 + mh,
        *y = A2 + mh;
  Bf16Bufs b = bf16_bufs(params, act, work, m);
  // bf16 copies of the hidden weights W1, W2 (the B operands: rows = outputs) and
  // of their transposes (the backward pass: rows = inputs)
  weights_kernel<<<dim3(H / 32, H / 32, 2), 256, 0, s>>>(params + O_W1, params + O_W2, b.w[0]);
  RS_L();
  // layer 0 (10 inputs): fp32
  layer0_kernel<<<std::min(m, 152 * 8), H, 0, s>>>(X, params + O_W0, params + O_B0, m, Z0, A0, b.h0);
  RS_L();
  // layers 1, 2: tensor cores on bf16 activations
  RS_TRY(tc_mm(b.h0, H, b.w[0], H, m, H, H, Z1, s));
  bias_silu_kernel<<<grid_cap(mh / 4, 256), 256, 0, s>>>(Z1, params + O_B1, mh, A1, b.h1);
  RS_L();
  RS_TRY(tc_mm(b.h1, H, b.w[1], H, m, H, H, Z2, s));
  // the last bias and the output layer (1 output): fp32
  output_kernel<<<ceil_div(m, 32), 256, 0, s>>>(Z2, params + O_B2, params + O_W3, params + O_B3, m,
                                                A2, y);
  RS_L();
  return cudaSuccess;
}

namespace {
// The loss after cv_forward, and with dy its derivative.
cudaError_t loss_pass(const float *y, int m, const float *target, const float *weight, double *sums,
                      float *dy, float *loss, cudaStream_t s) {
  loss_sums_kernel<<<32, 32, 0, s>>>(y, target, weight, m, sums);
  RS_L();
  loss_kernel<<<dy ? std::min(152, ceil_div(m, 32)) : 1, 32, 0, s>>>(y, target, weight, m, sums, dy,
                                                                     loss);
  RS_L();
  return cudaSuccess;
}
}  // namespace

cudaError_t cv_loss(int m, const float *target, const float *weight, float *act, float *loss,
                    float *work, cudaStream_t s) {
  Bf16Bufs b = bf16_bufs(nullptr, act, work, m);
  return loss_pass(act + 6LL * m * CV_HIDDEN, m, target, weight, reinterpret_cast<double *>(b.work),
                   nullptr, loss, s);
}

cudaError_t cv_backward(const float *params, const float *X, int m, const float *target,
                        const float *weight, float *act, float *grad, float *loss, float *work,
                        cudaStream_t s) {
  const int H = CV_HIDDEN;
  const long long mh = (long long)m * H;
  float *Z0 = act, *A0 = Z0 + mh, *Z1 = A0 + mh, *A1 = Z1 + mh, *Z2 = A1 + mh, *A2 = Z2 + mh,
        *y = A2 + mh, *dy = y + m;
  Bf16Bufs b = bf16_bufs(params, act, work, m);
  double *sums = reinterpret_cast<double *>(b.work);
  RS_TRY(loss_pass(y, m, target, weight, sums, dy, loss, s));
  const dim3 gt((unsigned)((b.ldt + 31) / 32), H / 32), gm((unsigned)ceil_div(m, 32), H / 32);
  // layer 3: dA2 = dy W3, dZ2 = dA2 silu'(Z2) (in Z2's place)
  back_kernel<<<gt, 256, 0, s>>>(nullptr, dy, params + O_W3, Z2, A1, m, b.h1, b.t0, b.t1, b.ldt);
  RS_L();
  // layer 2: dW2 = dZ2^T A1; dA1 = dZ2 W2 (in A1's place); dZ1 = dA1 silu'(Z1)
  RS_TRY(tc_wgrad(b.t0, b.t1, b.ldt, m, b.part, grad + O_W2, s));
  RS_TRY(tc_mm(b.h1, H, b.wt[1], H, m, H, H, A1, s));
  back_kernel<<<gt, 256, 0, s>>>(A1, nullptr, nullptr, Z1, A0, m, b.h0, b.t0, b.t1, b.ldt);
  RS_L();
  // layer 1: dW1 = dZ1^T A0; dA0 = dZ1 W1; dZ0 = dA0 silu'(Z0)
  RS_TRY(tc_wgrad(b.t0, b.t1, b.ldt, m, b.part, grad + O_W1, s));
  RS_TRY(tc_mm(b.h0, H, b.wt[0], H, m, H, H, A0, s));
  back_kernel<<<gm, 256, 0, s>>>(A0, nullptr, nullptr, Z0, nullptr, m, nullptr, nullptr, nullptr, 0);
  RS_L();
  // the sums over the rows: db2, db1, db0, dW3 = dy^T A2, db3, dW0 = dZ0^T X (fp32)
  SumArgs g;
  cv_row_chunks(m, &g.ks, &g.kc);
  float *p3 = b.work + 128, *p0 = p3 + (long long)g.ks * H;
  g.dz[0] = Z2; g.dz[1] = Z1; g.dz[2] = Z0;
  g.dy = dy; g.a2 = A2; g.x = X;
  g.db[0] = grad + O_B2; g.db[1] = grad + O_B1; g.db[2] = grad + O_B0;
  g.db3 = grad + O_B3;
  g.w3 = g.ks > 1 ? p3 : grad + O_W3;
  g.w0 = g.ks > 1 ? p0 : grad + O_W0;
  g.m = m;
  sums_kernel<<<24 + 16 * g.ks + 1, 320, 0, s>>>(g);
  RS_L();
  if (g.ks > 1) {
    sums_reduce_kernel<<<11, 256, 0, s>>>(p3, p0, g.ks, grad + O_W3, grad + O_W0);
    RS_L();
  }
  return cudaSuccess;
}

cudaError_t cv_adam(float *p, const float *g, float *m, float *v, int n, float lr, int step,
                    cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float bc1 = 1.f - powf(b1, (float)step), bc2 = 1.f - powf(b2, (float)step);
  adam_kernel<<<grid_cap(n, 256), 256, 0, s>>>(p, g, m, v, n, lr, b1, b2, 1e-8f, bc1, bc2);
  RS_L();
  return cudaSuccess;
}

cudaError_t cv_stats(const double *BC, int nh, int n, double *stats, cudaStream_t s) {
  const long long nn = (long long)n * n;
  cv_stats_kernel<<<grid_cap(nn, 256), 256, 0, s>>>(BC, nh, nn, stats);
  RS_L();
  return cudaSuccess;
}

cudaError_t cv_targets(const double *stats, int n, int nt, int ns, float *target, float *weight,
                       cudaStream_t s) {
  const long long nn = (long long)n * n;
  cv_targets_kernel<<<grid_cap(nn * nt, 256), 256, 0, s>>>(stats, nn, nt, ns, target, weight);
  RS_L();
  return cudaSuccess;
}

cudaError_t cv_features(const double *sdd, const double *G, const double *Gb, const double *tau,
                        double beta, const double *KP, const int *rowptr, int naux, int n, int nt,
                        double *scratch, float *X, cudaStream_t s) {
  double *mx = scratch, *rn = scratch + 3 * nt;
  cv_maxima_kernel<<<nt, 256, 0, s>>>(sdd, G, Gb, n, mx);
  RS_L();
  cv_rownorm_kernel<<<n, 256, 0, s>>>(KP, rowptr, naux, rn);
  RS_L();
  max_small_kernel<<<1, 32, 0, s>>>(rn, n, rn + n);
  RS_L();
  cv_features_kernel<<<grid_cap((long long)n * n * nt, 256), 256, 0, s>>>(
      sdd, G, Gb, tau, log(beta), rn, rn + n, mx, n, nt, X);
  RS_L();
  return cudaSuccess;
}

cudaError_t cv_gather(const float *X, const float *T, const float *W, long long total,
                      long long start, long long stride, int m, float *bx, float *bt, float *bw,
                      cudaStream_t s) {
  gather_batch_kernel<<<grid_cap((long long)m * (CV_NFEAT + 2), 256), 256, 0, s>>>(
      X, T, W, total, start, stride, m, bx, bt, bw);
  RS_L();
  return cudaSuccess;
}

cudaError_t cv_accumulate(const double *BC, int nh, int n, double ns, const double *base,
                          const double *c, int init, double *sig, cudaStream_t s) {
  const long long nn = (long long)n * n;
  cv_accumulate_kernel<<<grid_cap(nn, 256), 256, 0, s>>>(BC, nh, nn, ns, base, c, init, sig);
  RS_L();
  return cudaSuccess;
}

cudaError_t cv_pair_energy(const double *BC, int nh, int n, const double *c, const double *gb,
                           const double *t, const double *s2, double w, double ne, double *e_st,
                           cudaStream_t s) {
  cv_pair_energy_kernel<<<nh, 256, 0, s>>>(BC, nh, n, c, gb, t, s2, w, ne, e_st);
  RS_L();
  return cudaSuccess;
}

cudaError_t trace_prod_w(const double *X, const double *Y, const double *W, int n, int nt,
                         double *out, cudaStream_t s) {
  trace_prod_w_kernel<<<nt, 256, 0, s>>>(X, Y, W, n, out);
  RS_L();
  return cudaSuccess;
}

cudaError_t cv_coefficients(const float *y, long long m, double *c, cudaStream_t s) {
  add_one_kernel<<<grid_cap(m, 256), 256, 0, s>>>(y, m, c);
  RS_L();
  return cudaSuccess;
}

}  // namespace rssri
