// Sigma(tau) for a G given by its orbitals (Eq. 17), evaluated on the orbitals:
// with G = -C_v gv C_v^T and Gb = -C_o go C_o^T, gv and go diagonal, every
// product with G or Gb is a scaling of the contraction index, and that index
// runs over the virtual or the occupied orbitals only.
//
// Chain (S8).  With Z_X = C^T X C_v and Z_Y = C^T Y C_v (X, Y symmetric; once
// per sample pair, not per tau) and M = Z_X gv Z_Y^T [n x n, orbitals]:
//   C = X G Y = -M,  t = Tr(C Gb) = sum_o M_oo go_o,  Tr(B B) = sum M_oo' go_o' M_o'o go_o,
//   F = 2 t C - C Gb C = M_(:,o) go M_(o,:) - 2 t M
// in the orbital basis: 2 n^3 flops per factor pair and tau point against
// 8 n^3 for the four products X G, (X G) Y, C Gb, (2 t I - B) C.
#pragma once

#include "common.cuh"

namespace rssri {

// A product of the two kernels below, in fp64 (V = double) or double-float
// (V = float2, pairs).
//
// mo_nt: out[z] = A_b diag(ks_t) B_b^T for z = (t nb + b) (one product per inner
// batch b < nb and tau t < nt): A_b = A + b sA [M x K, row stride lda], B_b
// [N x K], ks_t = ks + t sks.
struct MoNt {
  int df = 0;  // 0: fp64, 1: double-float pairs
  int M = 0, N = 0, K = 0, nb = 1, nt = 1;
  const void *A = nullptr, *B = nullptr, *ks = nullptr;
  long long lda = 0, ldb = 0, sA = 0, sB = 0, sks = 0;
  void *out = nullptr;  // [nt][nb][M][N], of the operands' type
};
cudaError_t mo_nt(const MoNt &g, cudaStream_t s);

// Sum over sample pairs x < cnt and kinds k < nkind (k = 0: sign +, else -) of
// sgn (M_(:,o) go M_(o,:) - 2 t M) per tau: M [nt][nkind][cnt][n][n], go
// [nt][no] at stride sgo, tr [nt][nkind][cnt] the traces t; acc[t] [n][n] (+)=
// 2^e_t that sum (e_t = texp[t], null: 0).  The pairs are dealt to `groups`
// partial sums, added in a fixed order; work: mo_sum_work() doubles.
struct MoSum {
  int df = 0;
  int n = 0, no = 0, cnt = 0, nkind = 1, nt = 1;
  const void *M = nullptr, *go = nullptr;
  long long sgo = 0;
  const double *tr = nullptr;
  const int *texp = nullptr;
  double *acc = nullptr;  // [nt][n][n]
  int accumulate = 0;
};
size_t mo_sum_work(const MoSum &g);
cudaError_t mo_sum(const MoSum &g, double *work, cudaStream_t s);

// Per matrix z of M [nt][nb][n][n]: tr[z] = sum_o M_oo go_o and
// s2[z] = sum_oo' M_oo' go_o' M_o'o go_o (fp64), go_t at go + t sgo.
cudaError_t mo_traces(int df, const void *M, int nt, int nb, int n, int no, const void *go,
                      long long sgo, double *tr, double *s2, cudaStream_t s);
// e_st[x] += -(1 / ne) sum_t tau_w[t] 2^(2 e_t) sum_k (+-)(2 tr^2 - s2), tau in order; tau_w on the
// device, e_t = texp[t] (null: 0).
cudaError_t mo_energy(const double *tr, const double *s2, int nt, int nkind, int cnt,
                      const double *tau_w, const int *texp, double ne, double *e_st,
                      cudaStream_t s);

// The diagonals gv[t][a] = exp(-(e_(no+a) - mu) tau_t), go[t][c] = exp((e_c - mu) tau_t) in fp64,
// and, with df, as pairs of gv 2^-ev_t and go 2^-eo_t, the largest entry of each tau point
// in [1, 2): pairs keep their precision only well inside fp32's exponent range.  texp[t] =
// 2 ev_t + eo_t (the power of two that a term quadratic in gv and linear in go carries),
// eexp[t] = ev_t + eo_t.
cudaError_t mo_tables(const double *orb_e, int n, int no, double mu, const double *tau, int nt,
                      int df, double *gv, double *go, float2 *gvhl, float2 *gohl, int *texp,
                      int *eexp, cudaStream_t s);
// flag |= 1 when some |CtC - I| element exceeds tol.
cudaError_t mo_orth_check(const double *CtC, int n, double tol, int *flag, cudaStream_t s);
// The range rule of to_df64 (dd_df64.cuh) on each of `segments` matrices of len values, without
// converting them.
cudaError_t mo_range_check(const double *x, int segments, long long len, int *range,
                           cudaStream_t s);

}  // namespace rssri
