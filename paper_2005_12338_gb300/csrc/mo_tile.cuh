// Register-tiled products of the orbital-basis path (mo.cuh): the two kinds of
// arithmetic, the tile shapes and their choice, and the kernel
// out = A diag(ks) B^T that the chain and the deterministic block share.
//
// The products run on the fp64 pipe (IEEE form) or on
// the fp32 pipes (double-float form: each value a pair of floats, about a
// dozen fp32 operations per multiply-add).  Either way one multiply-add of a
// warp occupies its pipe for so long (16 cycles for fp64, 3 for a
// double-float one on four schedulers) that shared-memory reads and global
// loads hide behind it; what is left to choose is the share of tile work
// spent on padding, so the tile edge is picked per shape by padded work over
// lane use, and scaling the contraction index (one multiply per loaded
// element of A, against BN multiply-adds per element) costs about 1%.
#pragma once

#include <algorithm>

#include "dd_arith.cuh"
#include "mo.cuh"

namespace rssri {
namespace {

inline int grid_cap(long long work, int threads) {
  long long b = (work + threads - 1) / threads;
  return (int)(b < 1 ? 1 : (b > 152 * 32 ? 152 * 32 : b));
}

__device__ __forceinline__ float2 split_pair(double v) {
  const float hi = __double2float_rn(v);
  return make_float2(hi, __double2float_rn(v - (double)hi));
}
// ------------------------------------------------------- arithmetic kinds --
struct F64 {
  using V = double;
  struct Acc {
    double s;
  };
  static __device__ __forceinline__ V zero() { return 0.0; }
  static __device__ __forceinline__ void clear(Acc &a) { a.s = 0.0; }
  static __device__ __forceinline__ V mul(V a, V b) { return a * b; }
  static __device__ __forceinline__ void mac(Acc &c, V a, V b) { c.s = fma(a, b, c.s); }
  static __device__ __forceinline__ void renorm(Acc &, bool) {}
  static __device__ __forceinline__ double value(const Acc &a) { return a.s; }
  static __device__ __forceinline__ V store(const Acc &a) { return a.s; }
  static __device__ __forceinline__ double to_double(V v) { return v; }
  static __device__ __forceinline__ V from_double(double v) { return v; }
};
// Running pair (s, e) renormalised after every slab and added into the total
// (th, tl) every 256 terms (see dd_arith.cuh).
struct DF {
  using V = float2;
  struct Acc {
    float s, e, th, tl;
  };
  static __device__ __forceinline__ V zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ void clear(Acc &a) { a.s = a.e = a.th = a.tl = 0.f; }
  static __device__ __forceinline__ V mul(V a, V b) {
    const float p = __fmul_rn(a.x, b.x);
    float e = __fmaf_rn(a.x, b.x, -p);
    e = __fmaf_rn(a.x, b.y, e);
    e = __fmaf_rn(a.y, b.x, e);
    const float h = __fadd_rn(p, e);
    return make_float2(h, __fsub_rn(e, __fsub_rn(h, p)));
  }
  static __device__ __forceinline__ void mac(Acc &c, V a, V b) { df_mac(c.s, c.e, a, b); }
  static __device__ __forceinline__ void renorm(Acc &c, bool total) {
    const float sn = __fadd_rn(c.s, c.e);
    c.e = __fsub_rn(c.e, __fsub_rn(sn, c.s));
    c.s = sn;
    if (total) {
      df_acc(c.th, c.tl, c.s, c.e);
      c.s = c.e = 0.f;
    }
  }
  static __device__ __forceinline__ double value(const Acc &a) {
    return (double)a.th + (double)a.tl;
  }
  static __device__ __forceinline__ V store(const Acc &a) { return make_float2(a.th, a.tl); }
  static __device__ __forceinline__ double to_double(V v) { return (double)v.x + (double)v.y; }
  static __device__ __forceinline__ V from_double(double v) { return split_pair(v); }
};

// Tile: TY x TX threads, each owning TI x TJ outputs at strides TY and TX; K in
// slabs of BK, double-buffered; KU k steps of a slab unrolled (a fully unrolled
// slab of double-float multiply-adds outgrows the instruction cache).
template <int TY_, int TX_, int TI_, int TJ_, int BK_, int MINB_, int KU_>
struct Geo {
  static constexpr int TY = TY_, TX = TX_, TI = TI_, TJ = TJ_, BK = BK_, MINB = MINB_, KU = KU_;
  static constexpr int BM = TY * TI, BN = TX * TJ, NT = TY * TX;
};

struct NtArgs {
  int M, N;
  long long K, kchunk;
  int nb, ksplit, sym, tn, ntiles;
  const void *A, *B, *ks;
  long long lda, ldb, sA, sB, sks;
  void *out;  // [z][M][N]
};

// Position of a tile in the upper triangle (ti <= tj) of a T x T tile grid.
__device__ __forceinline__ void tri_tile(int q, int T, int &ti, int &tj) {
  ti = 0;
  while (q >= T - ti) {
    q -= T - ti;
    ++ti;
  }
  tj = ti + q;
}

// out[z] = A_b diag(ks_t) B_b^T over one K chunk, z = (t nb + b) ksplit + split.
// RAW: the result as fp64 (a partial sum), else of the operands' type.
template <class P, class G, int RAW>
__global__ void __launch_bounds__(G::NT, G::MINB) mo_nt_kernel(const NtArgs g) {
  using V = typename P::V;
  constexpr int BM = G::BM, BN = G::BN, BK = G::BK, NT = G::NT;
  constexpr int LA = (BM * BK + NT - 1) / NT, LB = (BN * BK + NT - 1) / NT;
  __shared__ V As[2][BK][BM + 1];
  __shared__ V Bs[2][BK][BN + 1];
  const int tile = blockIdx.x % g.ntiles, z = blockIdx.x / g.ntiles;
  int ti, tj;
  if (g.sym) {
    tri_tile(tile, g.tn, ti, tj);
  } else {
    ti = tile / g.tn;
    tj = tile - ti * g.tn;
  }
  const int split = z % g.ksplit, zb = z / g.ksplit, b = zb % g.nb, t = zb / g.nb;
  const V *A = static_cast<const V *>(g.A) + b * g.sA;
  const V *B = static_cast<const V *>(g.B) + b * g.sB;
  const V *ks = static_cast<const V *>(g.ks) + t * g.sks;
  const long long kbeg = split * g.kchunk, kend = min(g.K, kbeg + g.kchunk);
  const int row0 = ti * BM, col0 = tj * BN;
  const int tid = threadIdx.x, tx = tid % G::TX, ty = tid / G::TX;
  typename P::Acc acc[G::TI][G::TJ];
#pragma unroll
  for (int i = 0; i < G::TI; ++i)
#pragma unroll
    for (int j = 0; j < G::TJ; ++j) P::clear(acc[i][j]);
  V ra[LA], rb[LB];
  auto load = [&](long long kt) {
#pragma unroll
    for (int r = 0; r < LA; ++r) {
      const int e = tid + r * NT, i = e / BK, k = e % BK;
      V v = P::zero();
      if (e < BM * BK && row0 + i < g.M && kt + k < kend)
        v = P::mul(A[(long long)(row0 + i) * g.lda + kt + k], ks[kt + k]);
      ra[r] = v;
    }
#pragma unroll
    for (int r = 0; r < LB; ++r) {
      const int e = tid + r * NT, j = e / BK, k = e % BK;
      V v = P::zero();
      if (e < BN * BK && col0 + j < g.N && kt + k < kend)
        v = B[(long long)(col0 + j) * g.ldb + kt + k];
      rb[r] = v;
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int r = 0; r < LA; ++r) {
      const int e = tid + r * NT;
      if (e < BM * BK) As[buf][e % BK][e / BK] = ra[r];
    }
#pragma unroll
    for (int r = 0; r < LB; ++r) {
      const int e = tid + r * NT;
      if (e < BN * BK) Bs[buf][e % BK][e / BK] = rb[r];
    }
  };
  constexpr int FOLD = 256 / BK;
  if (kbeg < kend) {
    load(kbeg);
    store(0);
    __syncthreads();
    int buf = 0, slab = 0;
    for (long long kt = kbeg; kt < kend; kt += BK) {
      const bool more = kt + BK < kend;
      if (more) load(kt + BK);
#pragma unroll G::KU
      for (int kk = 0; kk < BK; ++kk) {
        V a[G::TI], bb[G::TJ];
#pragma unroll
        for (int i = 0; i < G::TI; ++i) a[i] = As[buf][kk][ty + G::TY * i];
#pragma unroll
        for (int j = 0; j < G::TJ; ++j) bb[j] = Bs[buf][kk][tx + G::TX * j];
#pragma unroll
        for (int i = 0; i < G::TI; ++i)
#pragma unroll
          for (int j = 0; j < G::TJ; ++j) P::mac(acc[i][j], a[i], bb[j]);
      }
      const bool total = ++slab == FOLD || !more;
      if (total) slab = 0;
#pragma unroll
      for (int i = 0; i < G::TI; ++i)
#pragma unroll
        for (int j = 0; j < G::TJ; ++j) P::renorm(acc[i][j], total);
      if (more) {
        store(buf ^ 1);
        __syncthreads();
        buf ^= 1;
      }
    }
  }
  const long long o0 = (long long)z * g.M * g.N;
#pragma unroll
  for (int i = 0; i < G::TI; ++i) {
    const int gi = row0 + ty + G::TY * i;
    if (gi >= g.M) continue;
#pragma unroll
    for (int j = 0; j < G::TJ; ++j) {
      const int gj = col0 + tx + G::TX * j;
      if (gj >= g.N) continue;
      const long long o = o0 + (long long)gi * g.N + gj;
      if (RAW) static_cast<double *>(g.out)[o] = P::value(acc[i][j]);
      else static_cast<V *>(g.out)[o] = P::store(acc[i][j]);
    }
  }
}

// out[t][e] (+)= sign 2^e_t sum_s part[t][s][src(e)], s in order; sym: (i > j) reads (j, i).
__global__ void mo_reduce_kernel(const double *__restrict__ part, int ns, int n, int nt, double sign,
                                 const int *__restrict__ texp, int sym, int accumulate,
                                 double *__restrict__ out) {
  const long long nn = (long long)n * n, total = nn * nt;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long t = e / nn, r = e - t * nn;
    long long src = r;
    if (sym) {
      const long long i = r / n, j = r - i * n;
      if (i > j) src = j * n + i;
    }
    const double *p = part + t * ns * nn + src;
    double s = 0.0;
    for (int k = 0; k < ns; ++k) s += p[k * nn];
    s *= sign;
    if (texp) s = scalbn(s, texp[t]);
    out[e] = accumulate ? out[e] + s : s;
  }
}

// ------------------------------------------------------------ tile choice --
// fp64: 64-thread tiles of edge 16, 24, 32, 40, 48 (2 to 6 outputs per thread and
// side), 256 threads for 64 and 400 (of 416 lanes) for 100.  Every tile sums k
// in ascending order, so the choice does not change a result.
using D16 = Geo<8, 8, 2, 2, 16, 12, 8>;
using D24 = Geo<8, 8, 3, 3, 16, 8, 8>;
using D32 = Geo<8, 8, 4, 4, 16, 8, 8>;
using D40 = Geo<8, 8, 5, 5, 8, 8, 8>;
using D48 = Geo<8, 8, 6, 6, 8, 6, 8>;
using D64 = Geo<16, 16, 4, 4, 16, 2, 8>;
using D100 = Geo<20, 20, 5, 5, 8, 1, 8>;
// double-float: 64-thread tiles of 16, 24, 32, 40, 256-thread tile of 64
using S16 = Geo<8, 8, 2, 2, 16, 12, 4>;
using S24 = Geo<8, 8, 3, 3, 16, 8, 2>;
using S32 = Geo<8, 8, 4, 4, 16, 6, 2>;
using S40 = Geo<8, 8, 5, 5, 8, 6, 1>;
using S64 = Geo<16, 16, 4, 4, 16, 2, 4>;

struct TileInfo {
  int edge;
  double cost;  // relative time per padded output and k step
};
// Measured on Gram matrices of n = 64 to 200 (padded multiply-adds, TFLOP/s): fp64
// 1.14-1.18 for edges 24 to 48, 1.20 for 64, 1.03 for 100; double-float 4.15, 3.75,
// 3.8, 4.67 for 24, 32, 40, 64.
constexpr TileInfo kD[] = {{16, 1.06}, {24, 1.03}, {32, 1.03}, {40, 1.04}, {48, 1.03}, {64, 1.0}, {100, 1.14}};
constexpr TileInfo kS[] = {{16, 1.25}, {24, 1.13}, {32, 1.24}, {40, 1.22}, {64, 1.0}};
constexpr int kND = sizeof(kD) / sizeof(kD[0]), kNS = sizeof(kS) / sizeof(kS[0]);

// The tile of least padded work (sym: tiles on and above the diagonal).
int pick(const TileInfo *t, int cnt, int M, int N, int sym) {
  int best = 0;
  double bc = 0;
  for (int k = 0; k < cnt; ++k) {
    const double tm = ceil_div(M, t[k].edge), tn = ceil_div(N, t[k].edge);
    const double c = (sym ? tm * (tm + 1) / 2 : tm * tn) * t[k].edge * t[k].edge * t[k].cost;
    if (k == 0 || c < bc) {
      best = k;
      bc = c;
    }
  }
  return best;
}
int pick_tile(int df, int M, int N, int sym) {
  return df ? pick(kS, kNS, M, N, sym) : pick(kD, kND, M, N, sym);
}
int tile_edge(int df, int k) { return df ? kS[k].edge : kD[k].edge; }
long long tile_count(int edge, int M, int N, int sym) {
  const long long tm = ceil_div(M, edge), tn = ceil_div(N, edge);
  return sym ? tm * (tm + 1) / 2 : tm * tn;
}

template <class P, class G, int RAW>
cudaError_t launch_nt(NtArgs a, long long z, cudaStream_t s) {
  a.tn = ceil_div(a.N, G::BN);
  a.ntiles = (int)tile_count(G::BM, a.M, a.N, a.sym);
  const long long blocks = (long long)a.ntiles * z;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  mo_nt_kernel<P, G, RAW><<<(unsigned)blocks, G::NT, 0, s>>>(a);
  ++launch_counter();
  return cudaGetLastError();
}
template <int RAW> cudaError_t nt_dispatch(int df, const NtArgs &a, long long z, cudaStream_t s) {
  const int k = pick_tile(df, a.M, a.N, a.sym);
  if (df) {
    switch (k) {
      case 0: return launch_nt<DF, S16, RAW>(a, z, s);
      case 1: return launch_nt<DF, S24, RAW>(a, z, s);
      case 2: return launch_nt<DF, S32, RAW>(a, z, s);
      case 3: return launch_nt<DF, S40, RAW>(a, z, s);
      default: return launch_nt<DF, S64, RAW>(a, z, s);
    }
  }
  switch (k) {
    case 0: return launch_nt<F64, D16, RAW>(a, z, s);
    case 1: return launch_nt<F64, D24, RAW>(a, z, s);
    case 2: return launch_nt<F64, D32, RAW>(a, z, s);
    case 3: return launch_nt<F64, D40, RAW>(a, z, s);
    case 4: return launch_nt<F64, D48, RAW>(a, z, s);
    case 5: return launch_nt<F64, D64, RAW>(a, z, s);
    default: return launch_nt<F64, D100, RAW>(a, z, s);
  }
}

}  // namespace
}  // namespace rssri
