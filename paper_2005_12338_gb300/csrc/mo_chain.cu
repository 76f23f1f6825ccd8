// The chain on the orbitals (S8, see mo.cuh): M = Z_X gv Z_Y^T per sample pair
// and tau point, its traces, and the sum over pairs of M_(:,o) go M_(o,:) - 2 t M.
//
// Bound by the fp64 pipe (or the fp32 pipes, double-float): at N = 200, 64
// pairs, 16 tau points the fp64 sampling call takes 41.2 ms with these
// products, 146 ms with the four general ones per factor pair (137 of them
// in those products), the pipe busy all along either way.
#include "mo_tile.cuh"

namespace rssri {
namespace {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
__device__ double block_sum(double v) {
  __shared__ double sh[32];
  __syncthreads();
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
  if (l == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    double x = (l < nw) ? sh[l] : 0.0;
    x = warp_sum(x);
    if (l == 0) sh[0] = x;
  }
  __syncthreads();
  return sh[0];
}

struct SumArgs {
  int n, no, cnt, nkind, per, groups, tn, ntiles;
  const void *M, *go;
  long long sgo;
  const double *tr;
  double *out;  // [t][group][n][n]
};

// One group of sample pairs of one tau point: out = sum over its pairs x and
// kinds k of sgn_k (M_(:,o) go M_(o,:) - 2 t M), the products of all pairs one
// running contraction over (x, k, o); the kinds of a pair follow one another,
// as they cancel to the small stochastic part.
template <class P, class G>
__global__ void __launch_bounds__(G::NT, G::MINB) mo_sum_kernel(const SumArgs g) {
  using V = typename P::V;
  constexpr int BM = G::BM, BN = G::BN, BK = G::BK, NT = G::NT;
  constexpr int LA = (BM * BK + NT - 1) / NT, LB = (BN * BK + NT - 1) / NT;
  __shared__ V As[2][BK][BM + 1];
  __shared__ V Bs[2][BK][BN + 1];
  const int tile = blockIdx.x % g.ntiles, z = blockIdx.x / g.ntiles;
  const int ti = tile / g.tn, tj = tile - ti * g.tn;
  const int grp = z % g.groups, t = z / g.groups;
  const long long nn = (long long)g.n * g.n;
  const V *Mt = static_cast<const V *>(g.M) + (long long)t * g.nkind * g.cnt * nn;
  const V *go = static_cast<const V *>(g.go) + t * g.sgo;
  const double *tr = g.tr + (long long)t * g.nkind * g.cnt;
  const int x0 = grp * g.per, x1 = min(g.cnt, x0 + g.per);
  const int row0 = ti * BM, col0 = tj * BN;
  const int tid = threadIdx.x, tx = tid % G::TX, ty = tid / G::TX;
  typename P::Acc acc[G::TI][G::TJ];
#pragma unroll
  for (int i = 0; i < G::TI; ++i)
#pragma unroll
    for (int j = 0; j < G::TJ; ++j) P::clear(acc[i][j]);
  V ra[LA], rb[LB];
  auto load = [&](int x, int k0, int kt) {
    const V *Mb = Mt + (long long)(k0 * g.cnt + x) * nn;
#pragma unroll
    for (int r = 0; r < LA; ++r) {
      const int e = tid + r * NT, i = e / BK, k = e % BK;
      V v = P::zero();
      if (e < BM * BK && row0 + i < g.n && kt + k < g.no) {
        V s = go[kt + k];
        if (k0) s = P::mul(s, P::from_double(-1.0));
        v = P::mul(Mb[(long long)(row0 + i) * g.n + kt + k], s);
      }
      ra[r] = v;
    }
#pragma unroll
    for (int r = 0; r < LB; ++r) {
      const int e = tid + r * NT, j = e % BN, k = e / BN;
      V v = P::zero();
      if (e < BN * BK && col0 + j < g.n && kt + k < g.no)
        v = Mb[(long long)(kt + k) * g.n + col0 + j];
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
      if (e < BN * BK) Bs[buf][e / BN][e % BN] = rb[r];
    }
  };
  constexpr int FOLD = 256 / BK;
  int x = x0, kind = 0, kt = 0;
  if (x < x1) {
    load(x, kind, kt);
    store(0);
    __syncthreads();
    int buf = 0, slab = 0;
    for (;;) {
      int nx = x, nkd = kind, nk = kt + BK;
      if (nk >= g.no) {
        nk = 0;
        if (++nkd == g.nkind) {
          nkd = 0;
          ++nx;
        }
      }
      const bool more = nx < x1;
      if (more) load(nx, nkd, nk);
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
      if (nk == 0) {  // the last slab of this product: - sgn 2 t M
        const V *Mb = Mt + (long long)(kind * g.cnt + x) * nn;
        const V f = P::from_double((kind ? 2.0 : -2.0) * tr[kind * g.cnt + x]);
#pragma unroll
        for (int i = 0; i < G::TI; ++i) {
          const int gi = row0 + ty + G::TY * i;
#pragma unroll
          for (int j = 0; j < G::TJ; ++j) {
            const int gj = col0 + tx + G::TX * j;
            if (gi < g.n && gj < g.n) P::mac(acc[i][j], f, Mb[(long long)gi * g.n + gj]);
          }
        }
      }
      const bool total = ++slab == FOLD || !more;
      if (total) slab = 0;
#pragma unroll
      for (int i = 0; i < G::TI; ++i)
#pragma unroll
        for (int j = 0; j < G::TJ; ++j) P::renorm(acc[i][j], total);
      if (!more) break;
      store(buf ^ 1);
      __syncthreads();
      buf ^= 1;
      x = nx;
      kind = nkd;
      kt = nk;
    }
  }
  double *out = g.out + (long long)z * nn;
#pragma unroll
  for (int i = 0; i < G::TI; ++i) {
    const int gi = row0 + ty + G::TY * i;
    if (gi >= g.n) continue;
#pragma unroll
    for (int j = 0; j < G::TJ; ++j) {
      const int gj = col0 + tx + G::TX * j;
      if (gj < g.n) out[(long long)gi * g.n + gj] = P::value(acc[i][j]);
    }
  }
}

// One block per matrix: the trace and the quadratic trace over the occupied
// block, whose transposed reads go through 32 x 32 shared tiles.
template <class P>
__global__ void __launch_bounds__(256) mo_traces_kernel(const typename P::V *__restrict__ M, int nb,
                                                        int n, int no,
                                                        const typename P::V *__restrict__ go,
                                                        long long sgo, double *__restrict__ tr,
                                                        double *__restrict__ s2) {
  __shared__ double ta[32][33], tb[32][33];
  const long long z = blockIdx.x, nn = (long long)n * n;
  const typename P::V *m = M + z * nn;
  const typename P::V *g = go + (z / nb) * sgo;
  double tl = 0.0;
  for (int i = threadIdx.x; i < no; i += blockDim.x)
    tl += P::to_double(m[(long long)i * n + i]) * P::to_double(g[i]);
  const double t = block_sum(tl);
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, T = (no + 31) / 32;
  double sl = 0.0;
  for (int bi = 0; bi < T; ++bi)
    for (int bj = bi; bj < T; ++bj) {
      __syncthreads();
      for (int r = ty; r < 32; r += 8) {
        const int i = bi * 32 + r, j = bj * 32 + tx, i2 = bj * 32 + r, j2 = bi * 32 + tx;
        ta[r][tx] = i < no && j < no ? P::to_double(m[(long long)i * n + j]) *
                                           P::to_double(g[j])
                                     : 0.0;
        tb[r][tx] = i2 < no && j2 < no ? P::to_double(m[(long long)i2 * n + j2]) *
                                             P::to_double(g[j2])
                                       : 0.0;
      }
      __syncthreads();
      double v = 0.0;
      for (int r = ty; r < 32; r += 8) v += ta[r][tx] * tb[tx][r];
      sl += bi == bj ? v : 2.0 * v;
    }
  const double s = block_sum(sl);
  if (threadIdx.x == 0) {
    tr[z] = t;
    s2[z] = s;
  }
}

__global__ void mo_energy_kernel(const double *__restrict__ tr, const double *__restrict__ s2, int nt,
                                 int nkind, int cnt, const double *__restrict__ tau_w,
                                 const int *__restrict__ eexp, int fexp, double ne,
                                 double *__restrict__ e_st) {
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < cnt; x += gridDim.x * blockDim.x) {
    double e = e_st[x];
    for (int t = 0; t < nt; ++t) {
      double de = 0.0;
      for (int k = 0; k < nkind; ++k) {
        const long long z = ((long long)t * nkind + k) * cnt + x;
        const double v = 2.0 * tr[z] * tr[z] - s2[z];
        de += k == 0 ? v : -v;
      }
      if (eexp) de = scalbn(de, 2 * eexp[t] + fexp);
      e += -tau_w[t] * de / ne;
    }
    e_st[x] = e;
  }
}

// One block per tau point.
__global__ void __launch_bounds__(256) mo_tables_kernel(const double *__restrict__ e, int n, int no,
                                                        double mu, const double *__restrict__ tau,
                                                        const MoTab tab) {
  __shared__ int mx[4];
  const int t = blockIdx.x, nv = n - no;
  if (threadIdx.x < 4) mx[threadIdx.x] = -100000;
  __syncthreads();
  const double tt = tau[t];
  double *gv = tab.gv + (long long)t * nv, *go = tab.go + (long long)t * no;
  double *hv = tab.hv + (long long)t * nv, *ho = tab.ho + (long long)t * no;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const bool occ = i < no;
    const double x = occ ? (e[i] - mu) * tt : -(e[i] - mu) * tt;
    const double v = exp(x), h = exp(0.5 * x);
    (occ ? go[i] : gv[i - no]) = v;
    (occ ? ho[i] : hv[i - no]) = h;
    // largest exponents (zero and non-finite values: none)
    if (v > 0.0 && isfinite(v)) atomicMax(&mx[occ ? 1 : 0], ilogb(v));
    if (h > 0.0 && isfinite(h)) atomicMax(&mx[occ ? 3 : 2], ilogb(h));
  }
  __syncthreads();
  const int ev = mx[0] > -100000 ? mx[0] : 0, eo = mx[1] > -100000 ? mx[1] : 0;
  if (threadIdx.x == 0) {
    tab.texp[t] = 2 * ev + eo;
    tab.eexp[t] = ev + eo;
    tab.hexp[t] = 2 * (mx[2] > -100000 ? mx[2] : 0) + (mx[3] > -100000 ? mx[3] : 0);
  }
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    if (i < no) tab.gohl[(long long)t * no + i] = split_pair(scalbn(go[i], -eo));
    else tab.gvhl[(long long)t * nv + i - no] = split_pair(scalbn(gv[i - no], -ev));
  }
}

__global__ void mo_orth_kernel(const double *__restrict__ m, int n, double tol, int *__restrict__ flag) {
  const long long nn = (long long)n * n;
  int bad = 0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nn;
       e += (long long)gridDim.x * blockDim.x) {
    const double d = fabs(m[e] - (e / n == e % n ? 1.0 : 0.0));
    bad |= (d <= tol ? 0 : 1) | (d <= 0.5 ? 0 : 2);
  }
  if (bad) atomicOr(flag, bad);
}

__global__ void __launch_bounds__(256) mo_range_kernel(const double *__restrict__ x, long long len,
                                                       int *__restrict__ range) {
  __shared__ int smax;
  if (threadIdx.x == 0) smax = 0;
  __syncthreads();
  int mx = 0;
  const double *p = x + (long long)blockIdx.x * len;
  for (long long e = threadIdx.x; e < len; e += blockDim.x)
    mx = max(mx, (int)((__double_as_longlong(p[e]) >> 52) & 0x7FF));
  atomicMax(&smax, mx);
  __syncthreads();
  if (threadIdx.x == 0 && smax != 0 && (smax < 1023 - 40 || smax > 1023 + 40)) atomicOr(&range[0], 1);
}

template <class P, class G> cudaError_t launch_sum(SumArgs a, int nt, cudaStream_t s) {
  a.tn = ceil_div(a.n, G::BN);
  a.ntiles = (int)tile_count(G::BM, a.n, a.n, 0);
  const long long blocks = (long long)a.ntiles * a.groups * nt;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  mo_sum_kernel<P, G><<<(unsigned)blocks, G::NT, 0, s>>>(a);
  ++launch_counter();
  return cudaGetLastError();
}
// Sample pairs per partial sum, and how many partial sums.
void sum_plan(const MoSum &g, int *groups, int *per) {
  const long long tiles = tile_count(32, g.n, g.n, 0) * g.nt;
  const long long want = std::max<long long>(1, (152LL * 24 + tiles - 1) / tiles);
  *per = (int)std::max<long long>(1, (g.cnt + want - 1) / want);
  *groups = ceil_div(g.cnt, *per);
}

}  // namespace

cudaError_t mo_nt(const MoNt &g, cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0 || g.nb <= 0 || g.nt <= 0) return cudaSuccess;
  NtArgs a{};
  a.M = g.M; a.N = g.N; a.K = g.K; a.kchunk = g.K;
  a.nb = g.nb; a.ksplit = 1;
  a.A = g.A; a.B = g.B; a.ks = g.ks;
  a.lda = g.lda; a.ldb = g.ldb; a.sA = g.sA; a.sB = g.sB; a.sks = g.sks;
  a.out = g.out;
  return nt_dispatch<0>(g.df, a, (long long)g.nb * g.nt, s);
}

size_t mo_sum_work(const MoSum &g) {
  int groups, per;
  sum_plan(g, &groups, &per);
  return (size_t)g.nt * groups * g.n * g.n;
}

cudaError_t mo_sum(const MoSum &g, double *work, cudaStream_t s) {
  if (g.n <= 0 || g.nt <= 0 || g.cnt <= 0) return cudaSuccess;
  SumArgs a{};
  sum_plan(g, &a.groups, &a.per);
  a.n = g.n; a.no = g.no; a.cnt = g.cnt; a.nkind = g.nkind;
  a.M = g.M; a.go = g.go; a.sgo = g.sgo; a.tr = g.tr;
  a.out = work;
  const int k = pick_tile(g.df, g.n, g.n, 0);
  cudaError_t e;
  if (g.df) {
    switch (k) {
      case 0: e = launch_sum<DF, S16>(a, g.nt, s); break;
      case 1: e = launch_sum<DF, S24>(a, g.nt, s); break;
      case 2: e = launch_sum<DF, S32>(a, g.nt, s); break;
      case 3: e = launch_sum<DF, S40>(a, g.nt, s); break;
      default: e = launch_sum<DF, S64>(a, g.nt, s);
    }
  } else {
    switch (k) {
      case 0: e = launch_sum<F64, D16>(a, g.nt, s); break;
      case 1: e = launch_sum<F64, D24>(a, g.nt, s); break;
      case 2: e = launch_sum<F64, D32>(a, g.nt, s); break;
      case 3: e = launch_sum<F64, D40>(a, g.nt, s); break;
      case 4: e = launch_sum<F64, D48>(a, g.nt, s); break;
      case 5: e = launch_sum<F64, D64>(a, g.nt, s); break;
      default: e = launch_sum<F64, D100>(a, g.nt, s);
    }
  }
  RS_TRY(e);
  mo_reduce_kernel<<<grid_cap((long long)g.nt * g.n * g.n, 256), 256, 0, s>>>(
      work, a.groups, g.n, g.nt, 1.0, g.texp, 0, g.accumulate, g.acc);
  ++launch_counter();
  return cudaGetLastError();
}

cudaError_t mo_traces(int df, const void *M, int nt, int nb, int n, int no, const void *go,
                      long long sgo, double *tr, double *s2, cudaStream_t s) {
  const long long z = (long long)nt * nb;
  if (z <= 0) return cudaSuccess;
  if (z > 0x7fffffffLL) return cudaErrorInvalidValue;
  if (df)
    mo_traces_kernel<DF><<<(unsigned)z, 256, 0, s>>>(static_cast<const float2 *>(M), nb, n, no,
                                                     static_cast<const float2 *>(go), sgo, tr, s2);
  else
    mo_traces_kernel<F64><<<(unsigned)z, 256, 0, s>>>(static_cast<const double *>(M), nb, n, no,
                                                      static_cast<const double *>(go), sgo, tr,
                                                      s2);
  ++launch_counter();
  return cudaGetLastError();
}

cudaError_t mo_energy(const double *tr, const double *s2, int nt, int nkind, int cnt,
                      const double *tau_w, const int *texp, int fexp, double ne, double *e_st,
                      cudaStream_t s) {
  mo_energy_kernel<<<grid_cap(cnt, 128), 128, 0, s>>>(tr, s2, nt, nkind, cnt, tau_w, texp, fexp, ne,
                                                      e_st);
  ++launch_counter();
  return cudaGetLastError();
}

cudaError_t mo_tables(const double *orb_e, int n, int no, double mu, const double *tau, int nt,
                      const MoTab &t, cudaStream_t s) {
  mo_tables_kernel<<<nt, 256, 0, s>>>(orb_e, n, no, mu, tau, t);
  ++launch_counter();
  return cudaGetLastError();
}

cudaError_t mo_orth_check(const double *CtC, int n, double tol, int *flag, cudaStream_t s) {
  mo_orth_kernel<<<grid_cap((long long)n * n, 256), 256, 0, s>>>(CtC, n, tol, flag);
  ++launch_counter();
  return cudaGetLastError();
}

cudaError_t mo_range_check(const double *x, int segments, long long len, int *range,
                           cudaStream_t s) {
  if (segments <= 0 || len <= 0) return cudaSuccess;
  mo_range_kernel<<<segments, 256, 0, s>>>(x, len, range);
  ++launch_counter();
  return cudaGetLastError();
}

}  // namespace rssri
