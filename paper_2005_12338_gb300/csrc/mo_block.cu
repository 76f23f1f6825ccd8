// The deterministic block on the orbitals (S7, see mo.cuh): U from V_i,abc, the
// weights of its contraction index per tau point, and the Gram matrices.
//
// Bound by the fp64 (or fp32) pipe.  Whole calls, the contraction over the kept
// pairs before and this after: N = 20, 32 tau points, fp64 19.7 -> 2.7 ms (32
// tau points in one launch instead of nine launches each); N = 100, 32 tau
// points, fp64 350.5 -> 85.2 ms; N = 150, 24 tau points, double-float 293.8 ->
// 128.0 ms (93.6 and 138.5 before 16-wide tiles, which waste the least on the
// diagonal).  With the setup's narrow tiles too: 1.5, 80.7 and 125 ms.
#include "mo_tile.cuh"

namespace rssri {
namespace {

template <class P>
__global__ void mo_weights_kernel(const double *__restrict__ gv, const double *__restrict__ go,
                                  int nv, int no, int c0, int nc, int nt,
                                  const int *__restrict__ texp, long long ldw,
                                  typename P::V *__restrict__ w) {
  const long long kk = (long long)nc * nv * nv, total = kk * nt;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long t = e / kk, k = e - t * kk;
    const int c = (int)(k / ((long long)nv * nv)), ab = (int)(k - (long long)c * nv * nv);
    const int a = ab / nv, b = ab - a * nv;
    double v = go[t * no + c0 + c] * gv[t * nv + a] * gv[t * nv + b];
    if (texp) v = scalbn(v, -texp[t]);
    w[t * ldw + k] = P::from_double(v);
  }
}

// Tiles (a block, b block) with a block <= b block; both transposes are staged,
// so that reads (contiguous in a) and writes (contiguous in b) are coalesced.
template <class P>
__global__ void __launch_bounds__(256) mo_pack_kernel(const double *__restrict__ V, int n, int nv,
                                                      int nc, int T, double scale, long long ldu,
                                                      typename P::V *__restrict__ U) {
  __shared__ double x[32][33], y[32][33];
  int ta, tb;
  tri_tile(blockIdx.x, T, ta, tb);
  const int i = blockIdx.y, c = blockIdx.z;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const double *Vc = V + (long long)c * nv * n * nv;
  // x[bb][aa] = V(a = 32 ta + aa, b = 32 tb + bb), y[aa][bb] = V(a = 32 tb + bb, b = 32 ta + aa)
  for (int r = ty; r < 32; r += 8) {
    const int a = ta * 32 + tx, b = tb * 32 + r;
    x[r][tx] = a < nv && b < nv ? Vc[((long long)b * n + i) * nv + a] : 0.0;
    const int a2 = tb * 32 + tx, b2 = ta * 32 + r;
    y[r][tx] = a2 < nv && b2 < nv ? Vc[((long long)b2 * n + i) * nv + a2] : 0.0;
  }
  __syncthreads();
  const long long kc = (long long)c * nv * nv;
  auto at = [&](int a, int b) {
    const long long k = kc + (long long)a * nv + b;
    return ldu ? i * ldu + k : ((k >> 4) * n + i) * 16 + (k & 15);
  };
  const double rs = scale * 0.70710678118654752440, ra = scale * 1.2247448713915890491;  // 1/sqrt 2, sqrt(3/2)
  for (int r = ty; r < 32; r += 8) {
    // row a of slot (a, b), a in block ta, b in block tb
    int a = ta * 32 + r, b = tb * 32 + tx;
    if (a < nv && b < nv) {
      const double ab = x[tx][r], ba = y[r][tx];
      const double v = a == b ? scale * ab : (a < b ? (ab + ba) * rs : (ba - ab) * ra);
      U[at(a, b)] = P::from_double(v);
    }
    if (ta != tb) {  // the mirrored slot (a in block tb, b in block ta): a > b
      a = tb * 32 + r;
      b = ta * 32 + tx;
      if (a < nv && b < nv) {
        const double ab = y[tx][r], ba = x[r][tx];
        U[at(a, b)] = P::from_double((ba - ab) * ra);
      }
    }
  }
}

// out[a] = sum_q x[a][q]^2, one warp per row.
__global__ void mo_row_norm2_kernel(const double *__restrict__ x, int rows, int cols,
                                    double *__restrict__ out) {
  const int r = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (r >= rows) return;
  double v = 0.0;
  for (int q = lane; q < cols; q += 32) {
    const double u = x[(long long)r * cols + q];
    v = fma(u, u, v);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if (lane == 0) out[r] = v;
}

// Split of the Gram contraction: enough CTAs that the last ones to finish
// leave the chip idle for a few percent of the time only, chunks of at least
// 128 terms (512 left the chip half idle at N = 20); independent of the tile, so that the tile never changes a result.
void gram_plan(const MoGram &g, int *ks, long long *kc) {
  const long long tiles = tile_count(32, g.n, g.n, 1) * g.nt;
  long long k = (152LL * 24 + tiles - 1) / tiles;
  k = std::max<long long>(1, std::min<long long>({k, g.K / 128, 1024}));
  const long long c = ((g.K + k - 1) / k + 15) / 16 * 16;
  *kc = std::max<long long>(c, 16);
  *ks = (int)std::max<long long>(1, (g.K + *kc - 1) / *kc);
}
}  // namespace

size_t mo_gram_work(const MoGram &g) {
  int ks;
  long long kc;
  gram_plan(g, &ks, &kc);
  return (size_t)g.nt * ks * g.n * g.n;
}

double mo_gram_flops(const MoGram &g) {
  const int e = tile_edge(g.df, pick_tile(g.df, g.n, g.n, 1));
  double f = 0.0;
  for (int i = 0; i < g.n; i += e)
    for (int j = i; j < g.n; j += e)
      f += 2.0 * std::min(e, g.n - i) * (double)std::min(e, g.n - j);
  return f * (double)g.K * g.nt;
}

cudaError_t mo_gram(const MoGram &g, double *work, cudaStream_t s) {
  if (g.n <= 0 || g.nt <= 0) return cudaSuccess;
  int ks;
  NtArgs a{};
  gram_plan(g, &ks, &a.kchunk);
  a.M = a.N = g.n; a.K = g.K;
  a.nb = 1; a.ksplit = ks; a.sym = 1;
  a.A = a.B = g.U; a.ks = g.w;
  a.lda = a.ldb = g.ldu; a.sks = g.K;
  a.out = work;
  RS_TRY(nt_dispatch<1>(g.df, a, (long long)g.nt * ks, s));
  mo_reduce_kernel<<<grid_cap((long long)g.nt * g.n * g.n, 256), 256, 0, s>>>(
      work, ks, g.n, g.nt, -1.0, g.wexp, 1, g.accumulate, g.out);
  ++launch_counter();
  return cudaGetLastError();
}

cudaError_t mo_weights(int df, const double *gv, const double *go, int nv, int no, int c0, int nc,
                       int nt, const int *exps, long long ldw, void *w, cudaStream_t s) {
  const long long total = (long long)nt * nc * nv * nv;
  if (df)
    mo_weights_kernel<DF><<<grid_cap(total, 256), 256, 0, s>>>(gv, go, nv, no, c0, nc, nt, exps, ldw,
                                                              static_cast<float2 *>(w));
  else
    mo_weights_kernel<F64><<<grid_cap(total, 256), 256, 0, s>>>(gv, go, nv, no, c0, nc, nt, nullptr,
                                                               ldw, static_cast<double *>(w));
  ++launch_counter();
  return cudaGetLastError();
}

cudaError_t mo_pack(int df, const double *V, int n, int nv, int nc, double scale, long long ldu,
                    void *U, cudaStream_t s) {
  const int T = ceil_div(nv, 32);
  dim3 grid(T * (T + 1) / 2, n, nc);
  if (df)
    mo_pack_kernel<DF><<<grid, 256, 0, s>>>(V, n, nv, nc, T, scale, ldu, static_cast<float2 *>(U));
  else
    mo_pack_kernel<F64><<<grid, 256, 0, s>>>(V, n, nv, nc, T, scale, ldu, static_cast<double *>(U));
  ++launch_counter();
  return cudaGetLastError();
}

cudaError_t mo_row_norm2(const double *x, int rows, int cols, double *out, cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  mo_row_norm2_kernel<<<ceil_div((long long)rows * 32, 256), 256, 0, s>>>(x, rows, cols, out);
  ++launch_counter();
  return cudaGetLastError();
}

}  // namespace rssri
