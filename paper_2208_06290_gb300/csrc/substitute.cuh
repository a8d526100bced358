// Substitution with one diagonal block of a leaf LU, by a warp.
#pragma once

#include "hodlr_internal.cuh"

namespace hodlr {

// x <- op(A)^{-1} x for the n x n (n <= 32) triangle at A (leading dimension m) and KC
// columns, lane = row: its unit lower part (useL) or its upper part, transposed or not;
// sweep 0 goes downwards, 1 upwards. Divisions by a pivot are multiplications by its
// reciprocal. The loads do not depend on x: they are in flight ahead of the steps.
template <int KC>
__device__ __forceinline__ void substitute(const double* __restrict__ A, int m, int n, int sweep, bool useL, int trans,
                                           int lane, double (&x)[KC]) {
  const double rcp = lane < n ? 1.0 / A[(size_t)lane * m + lane] : 0.0;
#pragma unroll 4
  for (int q = 0; q < n; ++q) {
    const int c = sweep == 0 ? q : n - 1 - q;
    const bool rest = lane < n && (sweep == 0 ? lane > c : lane < c);
    const double a = rest ? (trans ? A[(size_t)lane * m + c] : A[(size_t)c * m + lane]) : 0.0;
    const double r = __shfl_sync(0xffffffffu, rcp, c);
#pragma unroll
    for (int cc = 0; cc < KC; ++cc) {
      double v = __shfl_sync(0xffffffffu, x[cc], c);
      if (!useL) {
        v *= r;
        if (lane == c) x[cc] = v;
      }
      if (rest) x[cc] = fma(-a, v, x[cc]);
    }
  }
}

}  // namespace hodlr
