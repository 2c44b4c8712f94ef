// Shared by the clustered S lists' forward (cluster.cu) and adjoint
// (cluster_adjoint.cu).
#pragma once
#include "launch.h"

namespace scatter {

constexpr double kClEps = 2e-6;   // columns with a largest term below this are left out
constexpr int kClMaxK = 320;      // columns of an instance
constexpr int kClMaxExp = 15;     // largest exponent of an axis

__device__ __forceinline__ float cl_rmax2(const ClArgs& a, int inst) { return __uint_as_float(a.rmax2[inst]); }

// Columns that a crystal of this call's radius needs, 0 if it is larger than
// the plan's X (the direct kernels then do the instance).
__device__ __forceinline__ int cl_columns(const ClArgs& a, const ClInst& in, int inst) {
  const float r2 = cl_rmax2(a, inst);
  if (!(r2 <= in.lim2)) return 0;
  const float rho = sqrtf(r2 / in.lim2) * 1.0001f;
  int lo = 0, hi = in.K;  // columns are sorted by the radius from which they matter
  while (lo < hi) {
    const int m = (lo + hi) >> 1;
    if (a.rho[in.col0 + m] < rho)
      lo = m + 1;
    else
      hi = m;
  }
  return lo;
}

}  // namespace scatter
