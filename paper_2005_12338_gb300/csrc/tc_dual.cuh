// Stage 1 of the reduced-precision chain in one pass (see tc_dual.cu).
#pragma once

#include "tc_gemm.cuh"

namespace rssri {

// For c tau points j and ns sample pairs x, with operands of ld columns per row
// (n valid), n rows each:
//   dC  = P_S R' + P_L R'^S   (P: [c][2 ns], P_S = entry x, P_L = entry ns + x)
//   C^L = P_L R'^L            (y3: [3 ns], R', R'^S, R'^L = entries x, ns + x, 2 ns + x)
// accumulated in fp32, and written in the operand type only:
//   dcl [c][2 ns]: dC and C^L;  ct [c][ns]: (C^L + dC)^T;  dct: dC^T;  clt (or null): (C^L)^T.
struct TcDual {
  int n = 0, ns = 0, c = 0;
  long long ld = 0;
  const void *P = nullptr, *y3 = nullptr;
  void *dcl = nullptr, *ct = nullptr, *dct = nullptr, *clt = nullptr;
  int *err = nullptr;
  int wait_polls = 0;  // testing only (see TcGemm)
};
cudaError_t tc_dual(int kind, const TcDual &g, cudaStream_t s);
// One-time per-device launch attributes; call before capturing launches.
cudaError_t tc_dual_prepare();

}  // namespace rssri
