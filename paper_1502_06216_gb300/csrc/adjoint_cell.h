// adjoint_cell.h -- arithmetic of the adjoint solve at one cell that both of its forms share
// (jko_adjoint.cu, strip_adjoint.cu).  Plain C++ for both sides.
#pragma once

#include <cmath>

#ifndef JKO_HD
#ifdef __CUDACC__
#define JKO_HD __host__ __device__ __forceinline__
#else
#define JKO_HD inline
#endif
#endif

namespace jko {

// |change of lambda| at a cell in an iteration, which the solve's stop adds: in FP64 whatever the
// working precision (256^2 FP32, the ten-step gradient: 2-3 % against FP32 differences; with
// the conversions and the difference split off to other pipes the same).
template <typename T>
JKO_HD double lambda_change(T now, T before) {
  return fabs((double)now - (double)before);
}

}  // namespace jko
