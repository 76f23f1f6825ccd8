// Element-wise kernels of the tensor-core chain (see chain_tc.cu).  Operand
// buffers hold the product kind's type (TcKind: bf16, or fp32 rounded to tf32).
#pragma once

#include "common.cuh"

namespace rssri {

// From fac = [set][kind R, R^L][x][n][n] fp64: xsl = [R^S; R^L] and
// y3 = [R'; R'^S; R'^L], each [ns][n][ldp] (zero columns n..ldp-1).
cudaError_t chain_factors(int kind, const double *fac, int ns, int n, int ldp, void *xsl,
                          void *y3, cudaStream_t s);
// dst[c][i][j] = src[c][i][j] in the operand type with row stride ldp (zero padding).
cudaError_t chain_matrices(int kind, const double *src, int cnt, int n, int ldp, void *dst,
                           cudaStream_t s);
// Per sample pair and tau point j of a chunk of c: from xy [c][X: ns, Y: ns] the
// traces (part: scratch of c * ns * ceil(n/32) * 4 doubles), the energy increments
// (weights w[j], host; N_e = ne), and the diagonals 2 dt - X_ii, 2 t^L - Y_ii of
// a6 [c][2 ns][n][ldp], which holds -X and -Y.
constexpr int TC_CHUNK = 12;  // tau points per chunk at most
cudaError_t fold_tc(int kind, const float *xy, int ns, int n, int ldp, int c, const double *w,
                    double ne, void *a6, double *e_st, double *part, cudaStream_t s);
// The learned control variate on the tensor-core chain (Eq. 25 with the large
// part weighted element-wise by c): with fl[x] = F(R^L, R'^L) of pair x (fp32),
//   sig += (1 - c) o (mean_x fl[x] - sdd)           (fixed order over x),
//   e_st[x] += -(w / ne) sum_ij (1 - c_ij) fl[x]_ij gb_ji.
cudaError_t cv_tc_apply(const float *fl, int ns, int n, const double *c, const double *sdd,
                        const double *gb, double w, double ne, double *sig, double *e_st,
                        cudaStream_t s);
// sig[j] = base[j] + (sum over groups of part[j]) / ns for c tau points, groups summed in
// order.
cudaError_t reduce_tc(const float *part, int groups, int n, int c, const double *base, double ns,
                      double *sig, cudaStream_t s);

}  // namespace rssri
