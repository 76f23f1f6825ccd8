// fp64 matrix products for the RS-SRI-GF2 path.
//
// On GB300 the fp64 ceiling is the scalar DFMA pipe (two fp64 FMAs per clock
// per SM, about 1.2 TFLOP/s for the GPU; the fp64 mma.sync path is slower),
// so these are register-tiled SIMT kernels: an output tile per block (64, 40,
// 48, 100, 24 or 16 wide, 2x2 to 5x5 outputs per thread), K slabs double-buffered
// through shared memory with coalesced global loads for either operand
// layout.  Since the DFMA pipe is the bound, the work that matters is the
// zero-padded part of the edge tiles; the tile is chosen per problem shape.
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "common.cuh"

namespace rssri {
namespace {

// Tile shape: BM x BN outputs per block, BK-deep K slabs, TM x TN outputs per
// thread.  Every shape accumulates each output over k in ascending order with
// one fma per k, so all shapes give bitwise-identical results; the launcher
// picks the shape that is fastest for each problem shape (padded work on the
// DFMA pipe is what differs: 200-wide operands waste 39% of 64-wide tiles).
template <int BM_, int BN_, int BK_, int TM_, int TN_>
struct Tile {
  static constexpr int BM = BM_, BN = BN_, BK = BK_, TM = TM_, TN = TN_;
  static constexpr int TX = BN / TN, TY = BM / TM, NT = TX * TY;
};
using T64 = Tile<64, 64, 16, 4, 4>;
using T40 = Tile<40, 40, 8, 4, 4>;
using T48 = Tile<48, 48, 16, 4, 4>;
using T100 = Tile<100, 100, 8, 5, 5>;
// small products (the metric root of a small N_aux, a few hundred outputs): one
// 64-wide tile would keep the fp64 pipe of one SM busy for tens of microseconds
// (N = 20, N_aux = 60: setup and sampling 2.67 -> 1.47 ms; N = 100: 85.2 -> 80.7)
using T24 = Tile<24, 24, 16, 3, 3>;
using T16 = Tile<16, 16, 16, 2, 2>;
constexpr int kNumTiles = 6;
constexpr int kTileEdge[kNumTiles] = {64, 40, 48, 100, 24, 16};
constexpr int kTileDepth[kNumTiles] = {16, 8, 16, 8, 16, 16};
// split-K planning always uses the 64-wide reference tile, so the chunking of
// K (and therefore the result) does not depend on the tile shape chosen.
constexpr int RBM = 64, RBN = 64, RBK = 16;
constexpr int PAD = 1;

// MODE 0: strided operands (transA/transB per TA/TB).
// MODE 1: segmented: A(m,kk) = A[col[s0+kk]*lda + m], B(kk,q) = B[(s0+kk)*ldb + q],
//         with s0 = seg[b] and K_b = seg[b+1] - seg[b].
template <class TL, int MODE, int TA, int TB>
__global__ void __launch_bounds__(TL::NT) dgemm_kernel(
    int M, int N, int K, int kchunk, int ksplit, const double *__restrict__ A, long long lda,
    long long sA, const double *__restrict__ B, long long ldb, long long sB,
    double *__restrict__ C, long long ldc, long long sC, double alpha, double beta,
    int partial, const int *__restrict__ seg, const int *__restrict__ col) {
  constexpr int BM = TL::BM, BN = TL::BN, BK = TL::BK, TM = TL::TM, TN = TL::TN, NT = TL::NT;
  constexpr int LA = (BM * BK + NT - 1) / NT, LB = (BN * BK + NT - 1) / NT;
  constexpr bool AK = (MODE == 0 && TA == 0);  // A tile loaded along k
  constexpr bool BKc = (MODE == 0 && TB == 1); // B tile loaded along k
  __shared__ double As[2][BK][BM + PAD];
  __shared__ double Bs[2][BK][BN + PAD];

  const int z = blockIdx.z;
  const int b = z / ksplit, ks = z % ksplit;
  int kbeg, kend;
  long long s0 = 0;
  if (MODE == 1) {
    s0 = seg[b];
    kbeg = 0;
    kend = seg[b + 1] - seg[b];
  } else {
    kbeg = ks * kchunk;
    kend = min(K, kbeg + kchunk);
    A += (long long)b * sA;
    B += (long long)b * sB;
  }
  double *Cb = partial ? C + (long long)z * M * N : C + (long long)b * sC;
  const long long ldcb = partial ? N : ldc;

  const int row0 = blockIdx.y * BM, col0 = blockIdx.x * BN;
  const int tid = threadIdx.x, tx = tid % TL::TX, ty = tid / TL::TX;
  double acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.0;

  double ra[LA], rb[LB];
  auto load = [&](int kt) {
#pragma unroll
    for (int r = 0; r < LA; ++r) {
      const int e = tid + r * NT;
      double v = 0.0;
      if (e < BM * BK) {
        const int i = AK ? e / BK : e % BM, k = AK ? e % BK : e / BM;
        const int gi = row0 + i, gk = kt + k;
        if (gi < M && gk < kend) {
          if (MODE == 1) v = A[(long long)col[s0 + gk] * lda + gi];
          else if (TA == 0) v = A[(long long)gi * lda + gk];
          else v = A[(long long)gk * lda + gi];
        }
      }
      ra[r] = v;
    }
#pragma unroll
    for (int r = 0; r < LB; ++r) {
      const int e = tid + r * NT;
      double v = 0.0;
      if (e < BN * BK) {
        const int j = BKc ? e / BK : e % BN, k = BKc ? e % BK : e / BN;
        const int gj = col0 + j, gk = kt + k;
        if (gj < N && gk < kend) {
          if (MODE == 1) v = B[(s0 + gk) * ldb + gj];
          else if (TB == 0) v = B[(long long)gk * ldb + gj];
          else v = B[(long long)gj * ldb + gk];
        }
      }
      rb[r] = v;
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int r = 0; r < LA; ++r) {
      const int e = tid + r * NT;
      if (e < BM * BK) {
        const int i = AK ? e / BK : e % BM, k = AK ? e % BK : e / BM;
        As[buf][k][i] = ra[r];
      }
    }
#pragma unroll
    for (int r = 0; r < LB; ++r) {
      const int e = tid + r * NT;
      if (e < BN * BK) {
        const int j = BKc ? e / BK : e % BN, k = BKc ? e % BK : e / BN;
        Bs[buf][k][j] = rb[r];
      }
    }
  };

  if (kbeg < kend) {
    load(kbeg);
    store(0);
    __syncthreads();
    int buf = 0;
    for (int kt = kbeg; kt < kend; kt += BK) {
      const bool more = kt + BK < kend;
      if (more) load(kt + BK);
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        double a[TM], bb[TN];
#pragma unroll
        for (int i = 0; i < TM; ++i) a[i] = As[buf][kk][ty * TM + i];
#pragma unroll
        for (int j = 0; j < TN; ++j) bb[j] = Bs[buf][kk][tx * TN + j];
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], bb[j], acc[i][j]);
      }
      if (more) {
        store(buf ^ 1);
        __syncthreads();
        buf ^= 1;
      }
    }
  }

#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int gi = row0 + ty * TM + i;
    if (gi >= M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int gj = col0 + tx * TN + j;
      if (gj >= N) continue;
      double *p = Cb + (long long)gi * ldcb + gj;
      if (partial) *p = acc[i][j];
      else *p = (beta != 0.0) ? fma(alpha, acc[i][j], beta * *p) : alpha * acc[i][j];
    }
  }
}

// C[b] = alpha * sum_{ks} part[b][ks] + beta * C[b], fixed order over ks.
__global__ void splitk_reduce_kernel(int M, int N, int batch, int ksplit,
                                     const double *__restrict__ part, double *__restrict__ C,
                                     long long ldc, long long sC, double alpha, double beta) {
  const long long mn = (long long)M * N;
  const long long total = mn * batch;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int b = (int)(e / mn);
    const long long r = e - (long long)b * mn;
    const int i = (int)(r / N), j = (int)(r - (long long)i * N);
    const double *p = part + (long long)b * ksplit * mn + r;
    double s = 0.0;
    for (int k = 0; k < ksplit; ++k) s += p[k * mn];
    double *c = C + (long long)b * sC + (long long)i * ldc + j;
    *c = (beta != 0.0) ? fma(alpha, s, beta * *c) : alpha * s;
  }
}

template <class TL, int TA, int TB>
cudaError_t launch_strided_t(const GemmArgs &g, int ksplit, int kchunk, int b0, int nb,
                             double *work, cudaStream_t s) {
  const bool part = ksplit > 1;
  // a launch has 65,535 rows of tiles at most: taller products ([K]^L of a million kept
  // pairs under 16-wide tiles) in several; those with split K have a few rows only
  constexpr int ROWS = 65535 * TL::BM;
  for (int m0 = 0; m0 < g.M; m0 += std::min(ROWS, g.M - m0)) {
    const int m = std::min(ROWS, g.M - m0);
    dim3 grid(ceil_div(g.N, TL::BN), ceil_div(m, TL::BM), nb * ksplit);
    dgemm_kernel<TL, 0, TA, TB><<<grid, TL::NT, 0, s>>>(
        m, g.N, g.K, kchunk, ksplit, g.A + (long long)b0 * g.sA + (long long)m0 * (TA ? 1 : g.lda),
        g.lda, g.sA, g.B + (long long)b0 * g.sB, g.ldb, g.sB,
        part ? work : g.C + (long long)b0 * g.sC + (long long)m0 * g.ldc, g.ldc, g.sC, g.alpha,
        g.beta, part ? 1 : 0, nullptr, nullptr);
    ++launch_counter();
    RS_TRY(cudaGetLastError());
  }
  if (part) {
    const long long total = (long long)g.M * g.N * nb;
    const int blocks = (int)std::min<long long>((total + 255) / 256, 152 * 16);
    splitk_reduce_kernel<<<blocks, 256, 0, s>>>(g.M, g.N, nb, ksplit, work,
                                                 g.C + (long long)b0 * g.sC, g.ldc, g.sC,
                                                 g.alpha, g.beta);
    ++launch_counter();
    RS_TRY(cudaGetLastError());
  }
  return cudaSuccess;
}

template <class TL>
cudaError_t launch_strided(const GemmArgs &g, int ks, int kc, int b0, int nb, double *work,
                           cudaStream_t s) {
  if (!g.transA && !g.transB) return launch_strided_t<TL, 0, 0>(g, ks, kc, b0, nb, work, s);
  if (!g.transA && g.transB) return launch_strided_t<TL, 0, 1>(g, ks, kc, b0, nb, work, s);
  if (g.transA && !g.transB) return launch_strided_t<TL, 1, 0>(g, ks, kc, b0, nb, work, s);
  return launch_strided_t<TL, 1, 1>(g, ks, kc, b0, nb, work, s);
}

cudaError_t launch_tile(int tile, const GemmArgs &g, int ks, int kc, int b0, int nb,
                        double *work, cudaStream_t s) {
  switch (tile) {
    case 1: return launch_strided<T40>(g, ks, kc, b0, nb, work, s);
    case 2: return launch_strided<T48>(g, ks, kc, b0, nb, work, s);
    case 3: return launch_strided<T100>(g, ks, kc, b0, nb, work, s);
    case 4: return launch_strided<T24>(g, ks, kc, b0, nb, work, s);
    case 5: return launch_strided<T16>(g, ks, kc, b0, nb, work, s);
    default: return launch_strided<T64>(g, ks, kc, b0, nb, work, s);
  }
}

void split_plan(const GemmArgs &g, int *ksplit, int *kchunk) {
  const long long tiles = (long long)ceil_div(g.M, RBM) * ceil_div(g.N, RBN) * g.batch;
  int ks = 1;
  if (tiles < 2 * 152 && g.K >= 1024) {
    ks = (int)std::min<long long>((4 * 152 + tiles - 1) / tiles, g.K / 256);
    ks = std::max(1, std::min(ks, 256));
  }
  int kc = ceil_div(g.K, ks);
  kc = ceil_div(kc, RBK) * RBK;
  ks = std::max(1, ceil_div(g.K, kc));
  *ksplit = ks;
  *kchunk = std::max(kc, RBK);
}

// ------------------------------------------------------------ autotuner ----
// The tile shape of each distinct problem shape is chosen once per process:
// by timing every shape on the first call (when the product does not read C,
// so repeating it is harmless), else by a model of the padded work.  Large
// products are timed on a part of the result that holds a dozen of the largest tiles
// per SM, so that a first call does not run all of them six times more.  First calls of
// a process, fp64: setup at N = 300, N_aux = 900: 1,955 -> 1,554 ms (532 again); sampling
// with a caller's G at N = 200, which forms D: 1,013 -> 866 ms (391 again).
struct ShapeKey {
  int M, N, K, batch, ta, tb, mode;
  bool operator<(const ShapeKey &o) const {
    return std::tie(M, N, K, batch, ta, tb, mode) <
           std::tie(o.M, o.N, o.K, o.batch, o.ta, o.tb, o.mode);
  }
};
std::mutex g_tune_mutex;
std::map<ShapeKey, int> g_tune;

// The part of a product that its tiles are timed on: whole batch entries, then whole rows
// or columns, the other dimension cut to a multiple of every tile's edge.
GemmArgs tune_part(const GemmArgs &g, int ks) {
  constexpr long long OUTPUTS = 152LL * 12 * 100 * 100;
  constexpr long long EDGES = 4800;  // the tile edges' least common multiple
  GemmArgs t = g;
  if (ks > 1) return t;
  const long long mn = (long long)g.M * g.N;
  t.batch = (int)std::min<long long>(g.batch, (OUTPUTS + mn - 1) / mn);
  if (mn > OUTPUTS) {
    int &cut = g.N >= g.M ? t.N : t.M;
    const long long other = std::min(g.M, g.N), want = (OUTPUTS + other - 1) / other;
    cut = (int)std::min<long long>(cut, (want + EDGES - 1) / EDGES * EDGES);
  }
  return t;
}

int model_tile(int M, int N, int K, int batch) {
  int best = 0;
  double best_cost = 0;
  for (int t = 0; t < kNumTiles; ++t) {
    const int e = kTileEdge[t], d = kTileDepth[t];
    const double padded = (double)ceil_div(M, e) * e * ceil_div(N, e) * e * ceil_div(K, d) * d;
    const double blocks = (double)ceil_div(M, e) * ceil_div(N, e) * batch;
    const double fill = std::min(1.0, blocks / (2.0 * 152));
    const double cost = padded / fill;
    if (t == 0 || cost < best_cost * 0.97) {
      best = t;
      best_cost = cost;
    }
  }
  return best;
}

}  // namespace

int dgemm_ksplit(const GemmArgs &g) {
  int ks, kc;
  split_plan(g, &ks, &kc);
  return ks;
}

size_t dgemm_work_elems(const GemmArgs &g) {
  const int ks = dgemm_ksplit(g);
  if (ks <= 1) return 0;
  const int per = std::max(1, 65535 / ks);
  const int nb = std::min(g.batch, per);
  return (size_t)ks * nb * g.M * g.N;
}

cudaError_t dgemm(const GemmArgs &g, double *work, size_t work_elems, cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return cudaSuccess;
  int ks, kc;
  split_plan(g, &ks, &kc);
  if (ks > 1 && work_elems < dgemm_work_elems(g)) return cudaErrorInvalidValue;
  const int per = std::max(1, 65535 / ks);
  const ShapeKey key{g.M, g.N, g.K, g.batch, g.transA, g.transB, 0};
  int tile = -1;
  {
    std::lock_guard<std::mutex> lock(g_tune_mutex);
    auto it = g_tune.find(key);
    if (it != g_tune.end()) tile = it->second;
  }
  auto run = [&](int t, const GemmArgs &a) -> cudaError_t {
    for (int b0 = 0; b0 < a.batch; b0 += per) {
      const int nb = std::min(per, a.batch - b0);
      RS_TRY(launch_tile(t, a, ks, kc, b0, nb, work, s));
    }
    return cudaSuccess;
  };
  if (tile < 0) {
    tile = model_tile(g.M, g.N, g.K, g.batch);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    RS_TRY(cudaStreamIsCapturing(s, &cap));
    if (g.beta == 0.0 && cap == cudaStreamCaptureStatusNone) {
      cudaEvent_t e0 = nullptr, e1 = nullptr;
      RS_TRY(cudaEventCreate(&e0));
      RS_TRY(cudaEventCreate(&e1));
      float best_ms = 0;
      const GemmArgs part = tune_part(g, ks);
      cudaError_t err = cudaSuccess;
      for (int t = 0; t < kNumTiles && err == cudaSuccess; ++t) {
        float ms = 0;
        err = cudaEventRecord(e0, s);
        if (err == cudaSuccess) err = run(t, part);
        if (err == cudaSuccess) err = cudaEventRecord(e1, s);
        if (err == cudaSuccess) err = cudaEventSynchronize(e1);
        if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, e0, e1);
        if (err == cudaSuccess && (t == 0 || ms < best_ms)) {
          best_ms = ms;
          tile = t;
        }
      }
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
      RS_TRY(err);
    }
    std::lock_guard<std::mutex> lock(g_tune_mutex);
    g_tune[key] = tile;
  }
  return run(tile, g);
}

int dgemm_tile_edge(const GemmArgs &g) {
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  auto it = g_tune.find(ShapeKey{g.M, g.N, g.K, g.batch, g.transA, g.transB, 0});
  return it == g_tune.end() ? -1 : kTileEdge[it->second];
}

namespace {
template <class TL>
cudaError_t launch_segmented(int nb, int M, int N, const int *seg, const int *col,
                             const double *A, long long lda, const double *B, long long ldb,
                             double *C, long long ldc, long long sC, cudaStream_t s) {
  dim3 grid(ceil_div(N, TL::BN), ceil_div(M, TL::BM), nb);
  dgemm_kernel<TL, 1, 1, 0><<<grid, TL::NT, 0, s>>>(M, N, 0, 0, 1, A, lda, 0, B, ldb, 0, C, ldc,
                                                    sC, 1.0, 0.0, 0, seg, col);
  ++launch_counter();
  return cudaGetLastError();
}
}  // namespace

cudaError_t dgemm_segmented(int batch, int M, int N, const int *seg, const int *col,
                            const double *A, long long lda, const double *B, long long ldb,
                            double *C, long long ldc, long long sC, cudaStream_t s) {
  if (batch <= 0 || M <= 0 || N <= 0) return cudaSuccess;
  // segment lengths vary; plan the tile on a typical depth of 40
  const int tile = model_tile(M, N, 40, batch);
  for (int b0 = 0; b0 < batch; b0 += 65535) {
    const int nb = std::min(65535, batch - b0);
    double *Cb = C + (long long)b0 * sC;
    const int *sg = seg + b0;
    cudaError_t e;
    switch (tile) {
      case 1: e = launch_segmented<T40>(nb, M, N, sg, col, A, lda, B, ldb, Cb, ldc, sC, s); break;
      case 2: e = launch_segmented<T48>(nb, M, N, sg, col, A, lda, B, ldb, Cb, ldc, sC, s); break;
      case 3: e = launch_segmented<T100>(nb, M, N, sg, col, A, lda, B, ldb, Cb, ldc, sC, s); break;
      case 4: e = launch_segmented<T24>(nb, M, N, sg, col, A, lda, B, ldb, Cb, ldc, sC, s); break;
      case 5: e = launch_segmented<T16>(nb, M, N, sg, col, A, lda, B, ldb, Cb, ldc, sC, s); break;
      default: e = launch_segmented<T64>(nb, M, N, sg, col, A, lda, B, ldb, Cb, ldc, sC, s);
    }
    RS_TRY(e);
  }
  return cudaSuccess;
}

}  // namespace rssri
