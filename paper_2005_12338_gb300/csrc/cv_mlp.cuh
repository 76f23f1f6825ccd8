// Learned control variate kernels (see cv_mlp.cu).
#pragma once

#include <algorithm>

#include "common.cuh"

namespace rssri {

constexpr int CV_NFEAT = 10, CV_HIDDEN = 256;
constexpr long long CV_NPARAM =
    (long long)CV_HIDDEN * CV_NFEAT + CV_HIDDEN + 2LL * (CV_HIDDEN * CV_HIDDEN + CV_HIDDEN) +
    CV_HIDDEN + 1;

// Activations of m rows: [Z0 A0 Z1 A1 Z2 A2] (m x 256 each), y (m), dy (m),
// then the bf16 operands of the tensor-core hidden layers.
size_t cv_act_floats(int m);
// Floats of `work` that the tensor-core hidden layers use (bf16 weights and
// weight-gradient partials); the row sums' partials (cv_sum_floats(m)) follow them.
size_t cv_tc_work_floats();
// Chunks of the m rows that dW3 and dW0 are summed in: at most cv_max_chunks(m), *ks of
// *kc rows.
inline int cv_max_chunks(int m) { return m < 2048 ? 1 : std::min(76, m / 512); }
inline void cv_row_chunks(int m, int *ks, int *kc) {
  const int k = cv_max_chunks(m);
  *kc = k > 1 ? (ceil_div(m, k) + 15) / 16 * 16 : m;
  *ks = ceil_div(m, *kc);
}
// Their partials, and the loss sums (64 doubles), for any number of rows up to m: from the
// most chunks, which grow with m (*ks does not: 34 at 17,408 rows, 33 at 17,409).
inline size_t cv_sum_floats(int m) {
  return (size_t)cv_max_chunks(m) * (CV_HIDDEN + CV_HIDDEN * CV_NFEAT) + 128;
}
// Forward: y = MLP(X) - 1 in act (see cv_act_floats), X [m][10].
cudaError_t cv_forward(const float *params, const float *X, int m, float *act, float *work,
                       cudaStream_t s);
// After cv_forward: loss = sum w (1 + y - t)^2 / sum w alone.
cudaError_t cv_loss(int m, const float *target, const float *weight, float *act, float *loss,
                    float *work, cudaStream_t s);
// After cv_forward: loss = sum w (1 + y - t)^2 / sum w and its gradient.
cudaError_t cv_backward(const float *params, const float *X, int m, const float *target,
                        const float *weight, float *act, float *grad, float *loss, float *work,
                        cudaStream_t s);
cudaError_t cv_adam(float *p, const float *g, float *m, float *v, int n, float lr, int step,
                    cudaStream_t s);
// stats [5][n*n] += sums over the pair batch of F, F^L, F^2, (F^L)^2, F F^L.
cudaError_t cv_stats(const double *BC, int nh, int n, double *stats, cudaStream_t s);
// target c* and weight Var(F^L) per (tau, i, j) from stats [nt][5][n*n].
cudaError_t cv_targets(const double *stats, int n, int nt, int ns, float *target, float *weight,
                       cudaStream_t s);
// Feature rows X [nt*n*n][10]; scratch of 3*nt + n + 1 doubles.
cudaError_t cv_features(const double *sdd, const double *G, const double *Gb, const double *tau,
                        double beta, const double *KP, const int *rowptr, int naux, int n, int nt,
                        double *scratch, float *X, cudaStream_t s);
// Rows (start + k stride) mod total, k < m, of X [total][10], T and W [total].
cudaError_t cv_gather(const float *X, const float *T, const float *W, long long total,
                      long long start, long long stride, int m, float *bx, float *bt, float *bw,
                      cudaStream_t s);
// sig = (init ? c o base : sig) + sum_x (BC[x] + c o BC[nh+x]) / ns.
cudaError_t cv_accumulate(const double *BC, int nh, int n, double ns, const double *base,
                          const double *c, int init, double *sig, cudaStream_t s);
// e_st[x] += -w ((2 t_x^2 - s2_x) - Tr((c o F^L_x) Gb)) / ne with BC[nh+x] = -F^L_x.
cudaError_t cv_pair_energy(const double *BC, int nh, int n, const double *c, const double *gb,
                           const double *t, const double *s2, double w, double ne, double *e_st,
                           cudaStream_t s);
// out[t] = sum_ij W[t][i][j] X[t][i][j] Y[t][j][i]
cudaError_t trace_prod_w(const double *X, const double *Y, const double *W, int n, int nt,
                         double *out, cudaStream_t s);
// c = 1 + y in fp64.
cudaError_t cv_coefficients(const float *y, long long m, double *c, cudaStream_t s);

}  // namespace rssri
