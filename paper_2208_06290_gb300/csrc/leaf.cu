// Leaf stage: batched triangular solves with the leaf LUs (Alg. 1 leaf loop;
// Alg. 3 second step; Alg. 2 / Alg. 4 leaf step) and the leaf products.
#include <type_traits>

#include "hodlr_internal.cuh"

namespace hodlr {

// ---------------------------------------------------------------------------
// K2 / K6 / K8-leaf: X_b <- D_b^{-1} X_b (trans 0) or D_b^{-T} X_b (trans 1) with the
// FP32 LUs, up to eight columns.
// One warp owns CPW right-hand-side columns of one leaf; lane l holds rows
// l, l+32, ... in registers, so the substitutions need no block barrier: the
// pivot row value moves by warp shuffle and each L / U column is read once
// per warp (coalesced, through L1/L2) for CPW columns at a time.
// The divisions by the pivots u_kk are multiplications by their reciprocals,
// formed once per CTA (within an ulp of the quotient).
template <typename TIN, typename TOUT, int RPL, int CPW>
__global__ void __launch_bounds__(256) leaf_solve_kernel(int m, const float* __restrict__ LU,
                                                         const int* __restrict__ perm, const TIN* in,
                                                         int64_t ldin, TOUT* out, int64_t ldout, int ncols,
                                                         int trans) {
  const int b = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nwarps = blockDim.x >> 5;
  const float* A = LU + (size_t)b * m * m;
  const int* pb = perm + (size_t)b * m;
  __shared__ float s_rcp[256];  // 1 / u_kk (m <= 256)
  for (int e = threadIdx.x; e < m; e += blockDim.x) s_rcp[e] = float(1) / A[(size_t)e * m + e];
  __syncthreads();
  const int64_t row0 = (int64_t)b * m;
  const int col0 = (blockIdx.y * nwarps + warp) * CPW;
  if (col0 >= ncols) return;
  float x[CPW][RPL];
#pragma unroll
  for (int s = 0; s < RPL; ++s) {
    const int i = lane + 32 * s;
    const int src = (i < m) ? (trans ? i : pb[i]) : 0;
#pragma unroll
    for (int c = 0; c < CPW; ++c) {
      const int col = col0 + c;
      x[c][s] = (i < m && col < ncols) ? conv<float>(in[(int64_t)col * ldin + row0 + src]) : float(0);
    }
  }
  if (!trans) {
    // forward: unit lower L
#pragma unroll
    for (int kb = 0; kb < RPL; ++kb) {
      for (int kk = 0; kk < 32; ++kk) {
        const int k = kb * 32 + kk;
        if (k >= m) break;
        float xk[CPW];
#pragma unroll
        for (int c = 0; c < CPW; ++c) xk[c] = __shfl_sync(0xffffffffu, x[c][kb], kk);
#pragma unroll
        for (int s = kb; s < RPL; ++s) {
          const int i = lane + 32 * s;
          if (i > k && i < m) {
            const float l = A[(size_t)k * m + i];
#pragma unroll
            for (int c = 0; c < CPW; ++c) x[c][s] -= l * xk[c];
          }
        }
      }
    }
    // backward: upper U
#pragma unroll
    for (int kb = RPL - 1; kb >= 0; --kb) {
      for (int kk = 31; kk >= 0; --kk) {
        const int k = kb * 32 + kk;
        if (k >= m) continue;
        const float rk = s_rcp[k];
        float xk[CPW];
#pragma unroll
        for (int c = 0; c < CPW; ++c) {
          const float v = __shfl_sync(0xffffffffu, x[c][kb], kk) * rk;
          if (lane == kk) x[c][kb] = v;
          xk[c] = v;
        }
#pragma unroll
        for (int s = 0; s <= kb; ++s) {
          const int i = lane + 32 * s;
          if (i < k) {
            const float u = A[(size_t)k * m + i];
#pragma unroll
            for (int c = 0; c < CPW; ++c) x[c][s] -= u * xk[c];
          }
        }
      }
    }
#pragma unroll
    for (int s = 0; s < RPL; ++s) {
      const int i = lane + 32 * s;
      if (i < m) {
#pragma unroll
        for (int c = 0; c < CPW; ++c)
          if (col0 + c < ncols) out[(int64_t)(col0 + c) * ldout + row0 + i] = conv<TOUT>(x[c][s]);
      }
    }
  } else {
    // D = P^T L U, so D^T = U^T L^T P: forward with U^T (non-unit lower),
    // backward with L^T (unit upper), then scatter by the permutation.
#pragma unroll
    for (int kb = 0; kb < RPL; ++kb) {
      for (int kk = 0; kk < 32; ++kk) {
        const int k = kb * 32 + kk;
        if (k >= m) break;
        const float rk = s_rcp[k];
        float xk[CPW];
#pragma unroll
        for (int c = 0; c < CPW; ++c) {
          const float v = __shfl_sync(0xffffffffu, x[c][kb], kk) * rk;
          if (lane == kk) x[c][kb] = v;
          xk[c] = v;
        }
#pragma unroll
        for (int s = kb; s < RPL; ++s) {
          const int i = lane + 32 * s;
          if (i > k && i < m) {
            const float u = A[(size_t)i * m + k];  // U(k, i) = U^T(i, k)
#pragma unroll
            for (int c = 0; c < CPW; ++c) x[c][s] -= u * xk[c];
          }
        }
      }
    }
#pragma unroll
    for (int kb = RPL - 1; kb >= 0; --kb) {
      for (int kk = 31; kk >= 0; --kk) {
        const int k = kb * 32 + kk;
        if (k >= m) continue;
        float xk[CPW];
#pragma unroll
        for (int c = 0; c < CPW; ++c) xk[c] = __shfl_sync(0xffffffffu, x[c][kb], kk);
#pragma unroll
        for (int s = 0; s <= kb; ++s) {
          const int i = lane + 32 * s;
          if (i < k) {
            const float l = A[(size_t)i * m + k];  // L(k, i) = L^T(i, k)
#pragma unroll
            for (int c = 0; c < CPW; ++c) x[c][s] -= l * xk[c];
          }
        }
      }
    }
#pragma unroll
    for (int s = 0; s < RPL; ++s) {
      const int i = lane + 32 * s;
      if (i < m) {
        const int dst = pb[i];
#pragma unroll
        for (int c = 0; c < CPW; ++c)
          if (col0 + c < ncols) out[(int64_t)(col0 + c) * ldout + row0 + dst] = conv<TOUT>(x[c][s]);
      }
    }
  }
}

template <typename TIN, typename TOUT, int RPL, int CPW>
static cudaError_t leaf_solve_cpw(const Factor& F, const TIN* in, int64_t ldin, TOUT* out, int64_t ldout,
                                  int ncols, int trans, cudaStream_t s) {
  const int nleaf = 1 << F.d.L;
  const int m = F.d.m;
  const int cols_per_cta = 8 * CPW;
  const double Nd = (double)nleaf * m;
  note_work((sizeof(TIN) + sizeof(TOUT)) * Nd * ncols + sizeof(float) * Nd * m + 4.0 * Nd, 2.0 * m * Nd * ncols);
  dim3 grid(nleaf, (ncols + cols_per_cta - 1) / cols_per_cta);
  leaf_solve_kernel<TIN, TOUT, RPL, CPW><<<grid, 256, 0, s>>>(m, static_cast<const float*>(F.lu), F.perm, in, ldin,
                                                                  out, ldout, ncols, trans);
  note_launches(1);
  return cudaGetLastError();
}

// Columns per warp: eight, fewer when the right-hand side is narrower, so no FLOPs
// go to padding columns. (These leaves have 129 to 256 rows: eight per lane.)
template <typename TIN, typename TOUT, int RPL>
static cudaError_t leaf_solve_rpl(const Factor& F, const TIN* in, int64_t ldin, TOUT* out, int64_t ldout,
                                  int ncols, int trans, cudaStream_t s) {
  if (ncols == 1) return leaf_solve_cpw<TIN, TOUT, RPL, 1>(F, in, ldin, out, ldout, ncols, trans, s);
  if (ncols == 2) return leaf_solve_cpw<TIN, TOUT, RPL, 2>(F, in, ldin, out, ldout, ncols, trans, s);
  if (ncols <= 4) return leaf_solve_cpw<TIN, TOUT, RPL, 4>(F, in, ldin, out, ldout, ncols, trans, s);
  return leaf_solve_cpw<TIN, TOUT, RPL, 8>(F, in, ldin, out, ldout, ncols, trans, s);
}

template <typename TIN, typename TOUT>
cudaError_t launch_leaf_solve(const Factor& F, const TIN* in, int64_t ldin, TOUT* out, int64_t ldout,
                              int ncols, int trans, cudaStream_t s) {
  ProfScope prof_(KC_LEAF_SOLVE, s);
  if (ncols <= 0) return cudaSuccess;
  if (leaf_uses_inverse(F)) return launch_leaf_apply_inv<TIN, TOUT>(F, in, ldin, out, ldout, ncols, trans, s);
  if constexpr (std::is_same<TIN, double>::value && std::is_same<TOUT, double>::value) {
    if (F.prec == HODLR_PREC_FP64)
      return ncols <= kSmallSolveCols ? launch_leaf_solve_small(F, in, ldin, out, ldout, ncols, trans, s)
                                      : launch_leaf_solve_split(F, in, ldin, out, ldout, ncols, trans, s);
  }
  if (ncols > 8) return launch_leaf_solve_f32<TIN, TOUT>(F, in, ldin, out, ldout, ncols, trans, s);
  return leaf_solve_rpl<TIN, TOUT, 8>(F, in, ldin, out, ldout, ncols, trans, s);
}

template cudaError_t launch_leaf_solve<double, double>(const Factor&, const double*, int64_t, double*, int64_t,
                                                       int, int, cudaStream_t);
template cudaError_t launch_leaf_solve<double, float>(const Factor&, const double*, int64_t, float*, int64_t,
                                                      int, int, cudaStream_t);
template cudaError_t launch_leaf_solve<double, __nv_bfloat16>(const Factor&, const double*, int64_t,
                                                              __nv_bfloat16*, int64_t, int, int, cudaStream_t);
template cudaError_t launch_leaf_solve<float, float>(const Factor&, const float*, int64_t, float*, int64_t,
                                                     int, int, cudaStream_t);

// ---------------------------------------------------------------------------
// Leaf part of the FP64 matvec: Y_b = D_b X_b. Thread i of the CTA owns row i
// of the leaf; KC columns of X_b are staged in shared memory per CTA.
template <int KC>
__global__ void __launch_bounds__(256) leaf_matvec_kernel(int m, const double* __restrict__ D,
                                                          const double* __restrict__ X, int64_t ldx,
                                                          double* __restrict__ Y, int64_t ldy, int k) {
  extern __shared__ double sx[];  // m x KC, [j][c]
  const int b = blockIdx.x;
  const int c0 = blockIdx.y * KC;
  const int kc = min(KC, k - c0);
  const double* Db = D + (size_t)b * m * m;
  const int64_t row0 = (int64_t)b * m;
  for (int e = threadIdx.x; e < m * KC; e += blockDim.x) {
    const int j = e % m, c = e / m;
    sx[j * KC + c] = (c < kc) ? X[(int64_t)(c0 + c) * ldx + row0 + j] : 0.0;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    double acc[KC];
#pragma unroll
    for (int c = 0; c < KC; ++c) acc[c] = 0.0;
    for (int j = 0; j < m; ++j) {
      const double d = Db[(size_t)j * m + i];
#pragma unroll
      for (int c = 0; c < KC; ++c) acc[c] += d * sx[j * KC + c];
    }
#pragma unroll
    for (int c = 0; c < KC; ++c)
      if (c < kc) Y[(int64_t)(c0 + c) * ldy + row0 + i] = acc[c];
  }
}

template <int KC>
static void leaf_matvec_go(const hodlr_desc& d, const double* D, const double* X, int64_t ldx, double* Y,
                           int64_t ldy, int k, cudaStream_t s) {
  const int m = d.m;
  const int nleaf = 1 << d.L;
  const int threads = m >= 256 ? 256 : ((m + 31) / 32) * 32;
  dim3 grid(nleaf, (k + KC - 1) / KC);
  const size_t sm = (size_t)m * KC * sizeof(double);
  if (sm > 48 * 1024) cudaFuncSetAttribute(leaf_matvec_kernel<KC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  { leaf_matvec_kernel<KC><<<grid, threads, sm, s>>>(m, D, X, ldx, Y, ldy, k); note_launches(1); }
}

cudaError_t launch_leaf_matvec(const hodlr_desc& d, const double* D, const double* X, int64_t ldx, double* Y,
                               int64_t ldy, int k, cudaStream_t s) {
  ProfScope prof_(KC_LEAF_MATVEC, s);
  const int m = d.m;
  const int nleaf = 1 << d.L;
  note_work(8.0 * ((double)m * m * nleaf + 2.0 * (double)d.N * k), 2.0 * m * (double)d.N * k);
  if (k >= 2) return launch_leaf_matvec_split(d, D, X, ldx, Y, ldy, k, s);
  leaf_matvec_go<1>(d, D, X, ldx, Y, ldy, k, s);
  return cudaGetLastError();
}

}  // namespace hodlr
