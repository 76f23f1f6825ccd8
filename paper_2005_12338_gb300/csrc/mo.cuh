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
//
// Deterministic block (S7).  Eq. 20 on v^L = sum_Q K^Q K^Q is
//   Sigma_DD,ij = -sum_abc gv_a gv_b go_c V_i,abc (2 V_j,abc - V_j,bac),
//   V_i,abc = sum_Q K^Q_ia K^Q_bc  (a, b virtual, c occupied, i an AO),
// and with U = the symmetric (a <= b, weight sqrt(2 - delta_ab)) and
// antisymmetric (sqrt(6)) parts of V in (a, b) it is minus a Gram matrix,
//   Sigma_DD,ij = -sum_k w_k(tau) U_ik U_jk,  w_k = gv_a gv_b go_c > 0,
// whose U does not depend on tau.  n^2 n_v^2 n_o flops per tau point
// (half of the symmetric product), against 2 N_aux P^2 + ~4 N_aux n^3 for the
// contraction over the P kept pairs.
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

// Gram matrices out[t] (+)= -2^e_t U diag(w_t) U^T for t < nt, U [n x K] row
// stride ldu, w [nt][K], e_t = wexp[t] (null: 0); symmetric, fp64 results.  K is
// split over CTAs; the partial sums go to `work` (mo_gram_work() doubles) and
// are added in a fixed order.
struct MoGram {
  int df = 0;
  int n = 0, nt = 1;
  long long K = 0;
  const void *U = nullptr, *w = nullptr;
  long long ldu = 0;
  const int *wexp = nullptr;
  double *out = nullptr;  // [nt][n][n]
  int accumulate = 0;
};
size_t mo_gram_work(const MoGram &g);
cudaError_t mo_gram(const MoGram &g, double *work, cudaStream_t s);
// Flops of the tiles mo_gram computes.
double mo_gram_flops(const MoGram &g);

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

// Whether the block on the orbitals is the cheaper one for P > 0 kept pairs.
// fp64 and double-float, by flops: n^2 n_v^2 n_o (and a fifth for the tiles on the diagonal)
// per tau point plus U once, against D once plus 2 N_aux P^2 and the dense products per tau
// point.  Both run at the same rate of the fp64 (or fp32) pipe.  At N = 100, N_aux = 300,
// eps = 1e-3 (P = 3,560) a tau point is 1.5 against 9.5 GFLOP; the lines cross near N = 270.
inline bool mo_block_pays(int n_, int n_occ, int n_aux, int P_, int n_tau) {
  const double n = n_, no = n_occ, nv = n - no, na = n_aux, P = P_, nt = n_tau;
  const double pairs = 2.0 * P * P * na +
                       nt * (2.0 * na * P * P + 2.0 * P * n * na + 4.0 * na * n * n * n +
                             4.0 * P * na * na);
  const double orbitals = 2.0 * P * nv * na + 2.0 * no * n * nv * na + 2.0 * n * nv * nv * no * na +
                          nt * 1.2 * n * n * nv * nv * no;
  return orbitals < pairs;
}
// Sliced (n <= 1024), by time, fitted to 122 sizes with both forms timed: N = 60 to 450, N_aux =
// 3N, 0.3 to 0.55 of the orbitals occupied, eps = 1e-3 to 0.1, 2 to 64 tau points (setup in ms,
// orbitals against pairs: N = 110, eps = 0.1, 8 tau points 4.3 : 7.0; N = 131, eps = 0.1, 64: 31 : 69;
// N = 230, eps = 1e-2, 64: 204 : 261; N = 257, eps = 1e-3, 64: 420 : 576; N = 272, eps = 1e-2, 64:
// 503 : 444; N = 400, eps = 1e-3, 16: 821 : 534).  The fit is within 21% of every time, and the
// form it takes was the slower one at 3 sizes, by at most 6%.  Terms: V and U once, and per tau
// point the Gram matrix's 128 x 128 tiles (with the digit products that its levels leave to do on
// a gapped system's grid, about 0.6 of all) and the digits; the exchange, the dense products over
// whole tiles, the passes over [n][n][N_aux], and the launches.
inline bool mo_block_pays_sliced(int n, int n_occ, int n_aux, int P_, int n_tau) {
  if (n > 1024) return false;
  auto tiles = [](double x) { return (double)((long long)(x + 127) / 128 * 128); };
  const double no = n_occ, nv = n - n_occ, na = n_aux, P = P_, nt = n_tau, K = nv * nv * no;
  const double T = tiles(n) / 128.0, area = 128.0 * 128.0 * T * (T + 1.0) / 2.0;
  const double orbitals = 2.0 * n * nv * no * tiles(nv) * na / 90e12 + 30e-12 * n * K +
                          nt * (2.0 * area * K / 128e12 + 3e-12 * n * K);
  const double pairs = nt * (2.0 * tiles(na) * P * P / 43e12 +
                             2.0 * na * n * tiles(n) * (n + tiles(n)) / 40e12 +
                             27e-12 * n * (double)n * na + 0.43e-3);
  return orbitals < pairs;
}

// Per matrix z of M [nt][nb][n][n]: tr[z] = sum_o M_oo go_o and
// s2[z] = sum_oo' M_oo' go_o' M_o'o go_o (fp64), go_t at go + t sgo.
cudaError_t mo_traces(int df, const void *M, int nt, int nb, int n, int no, const void *go,
                      long long sgo, double *tr, double *s2, cudaStream_t s);
// e_st[x] += -(1 / ne) sum_t tau_w[t] 2^(2 e_t + fexp) sum_k (+-)(2 tr^2 - s2), tau in order; tau_w
// on the device, e_t = texp[t] (texp null: neither).
cudaError_t mo_energy(const double *tr, const double *s2, int nt, int nkind, int cnt,
                      const double *tau_w, const int *texp, int fexp, double ne, double *e_st,
                      cudaStream_t s);

// The diagonals gv[t][a] = exp(-(e_(no+a) - mu) tau_t), go[t][c] = exp((e_c - mu) tau_t) in fp64,
// and, with df, as pairs of gv 2^-ev_t and go 2^-eo_t, the largest entry of each tau point
// in [1, 2): pairs keep their precision only well inside fp32's exponent range.  texp[t] =
// 2 ev_t + eo_t (the power of two that a term quadratic in gv and linear in go carries),
// eexp[t] = ev_t + eo_t.  hv, ho: the square roots of gv and go; hexp[t] = the exponent of the
// largest hv hv ho.
struct MoTab {
  double *gv, *go, *hv, *ho;
  float2 *gvhl, *gohl;
  int *texp, *eexp, *hexp;
};
cudaError_t mo_tables(const double *orb_e, int n, int no, double mu, const double *tau, int nt,
                      const MoTab &t, cudaStream_t s);
// w[t][((c - c0) nv + a) nv + b] = go[t][c] gv[t][a] gv[t][b], c0 <= c < c0 + nc, for nt tau
// points, rows at stride ldw; df: pairs of the same times 2^-exps[t].
cudaError_t mo_weights(int df, const double *gv, const double *go, int nv, int no, int c0, int nc,
                       int nt, const int *exps, long long ldw, void *w, cudaStream_t s);
// U_ik, k = (c nv + a) nv + b, from V[c][b][i][a] (fp64, nc x nv x n x nv): slot a < b holds
// (V_ab + V_ba) / sqrt 2, a = b holds V_aa, a > b holds (V_ba - V_ab) sqrt(3/2), all times
// scale; df: pairs.  U_ik is at U[i ldu + k], or with ldu = 0 at U[((k / 16) n + i) 16 + k % 16].
cudaError_t mo_pack(int df, const double *V, int n, int nv, int nc, double scale, long long ldu,
                    void *U, cudaStream_t s);

// out[a] = sum_q x[a][q]^2 (the diagonal of v^L on the kept pairs, where its largest magnitude is).
cudaError_t mo_row_norm2(const double *x, int rows, int cols, double *out, cudaStream_t s);

// flag |= 1 when some |CtC - I| element exceeds tol, |= 2 when one exceeds 1/2.
cudaError_t mo_orth_check(const double *CtC, int n, double tol, int *flag, cudaStream_t s);
// The range rule of to_df64 (dd_df64.cuh) on each of `segments` matrices of len values, without
// converting them.
cudaError_t mo_range_check(const double *x, int segments, long long len, int *range,
                           cudaStream_t s);

}  // namespace rssri
