// Leaf solves of the low-precision factors whose leaves are FP32 LUs (m > 128),
// for more than eight columns.
#include "hodlr_internal.cuh"

namespace hodlr {

// X_b <- D_b^{-1} X_b (trans 0) or D_b^{-T} X_b (trans 1) by blocked right-looking
// substitution. CTA = one leaf x 64 columns, held in shared memory; per block of 32
// unknowns the panel of the triangular factor is staged, the block solved with one
// thread per column, and the remaining rows updated by a product (thread = 8 rows
// x 4 columns, 12 words of shared memory per 32 FMAs). The one-warp-per-eight-columns
// form (leaf.cu) moves every pivot by a shuffle and reads the factor from L2 for each
// eight columns; here it is read once per 64, and the FP32 pipe does the rest.
// Panels are loaded one block ahead; two CTAs share an SM, so that one's small solves run
// under the other's products. One launch of 640 columns and two of 16, 1024 leaves of
// 256 rows: 11.5 -> 4.6 ms.
template <typename TIN, typename TOUT>
__global__ void __launch_bounds__(256, 2) leaf_solve_f32_kernel(int m, const float* __restrict__ LU,
                                                                const int* __restrict__ perm, const TIN* in,
                                                                int64_t ldin, TOUT* out, int64_t ldout, int ncols,
                                                                int trans) {
  constexpr int PX = 68;
  extern __shared__ __align__(16) float sm[];
  const int mp = (m + 31) / 32 * 32;
  const int PA = mp + 4;
  float* sX = sm;             // [row][PX]
  float* sA = sX + mp * PX;   // [unknown of the block][PA rows]
  __shared__ float s_rcp[256];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t b = blockIdx.x;
  const float* A = LU + (size_t)b * m * m;
  const int* pb = perm + (size_t)b * m;
  const int64_t row0 = b * m;
  const int j0 = blockIdx.y * 64;
  s_rcp[tid] = tid < m ? 1.f / A[(size_t)tid * m + tid] : 1.f;
  for (int i = lane; i < mp; i += 32) {
    const int src = i < m ? (trans ? i : pb[i]) : 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int col = warp + 8 * u;
      sX[i * PX + col] = (i < m && j0 + col < ncols) ? conv<float>(in[(int64_t)(j0 + col) * ldin + row0 + src]) : 0.f;
    }
  }
  const int tx = tid & 15, ty = tid >> 4;
  // the panel of a block (32 unknowns from k0, rows it reaches) in registers, one block
  // ahead: value u of a thread is column warp + 8 (u / 8), row lane + 32 (u % 8) of the
  // eight 32-row groups, or transposed, row warp + 8 u of column `lane`
  float pre[32];
  auto fetch = [&](int sweep, int k0) {
    const int first = sweep == 0 ? k0 : 0, last = sweep == 0 ? mp : k0 + 32;
#pragma unroll
    for (int u = 0; u < 32; ++u) {
      const int c = trans ? lane : warp + 8 * (u >> 3), i = trans ? warp + 8 * u : lane + 32 * (u & 7);
      pre[u] = 0.f;
      if (i >= first && i < last && i < m && k0 + c < m)
        pre[u] = trans ? A[(size_t)i * m + k0 + c] : A[(size_t)(k0 + c) * m + i];
    }
  };
  fetch(0, 0);
  for (int sweep = 0; sweep < 2; ++sweep) {
    const bool unit = (sweep == 0) == (trans == 0);  // op(A) = L U, or U^T L^T
    for (int kb = 0; kb < mp; kb += 32) {
      const int k0 = sweep == 0 ? kb : mp - 32 - kb;
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 32; ++u) {
        const int c = trans ? lane : warp + 8 * (u >> 3), i = trans ? warp + 8 * u : lane + 32 * (u & 7);
        if (i < mp) sA[c * PA + i] = pre[u];
      }
      __syncthreads();
      if (kb + 32 < mp) fetch(sweep, sweep == 0 ? k0 + 32 : k0 - 32);
      else if (sweep == 0) fetch(1, mp - 32);
      if (tid < 64) {
        float x[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) x[i] = sX[(k0 + i) * PX + tid];
        if (sweep == 0) {
#pragma unroll
          for (int c = 0; c < 32; ++c) {
            if (!unit) x[c] *= s_rcp[k0 + c];
#pragma unroll
            for (int i = (c + 1) / 4 * 4; i < 32; i += 4) {
              const float4 a = *reinterpret_cast<const float4*>(sA + c * PA + k0 + i);
              if (i > c) x[i] = fmaf(-a.x, x[c], x[i]);
              if (i + 1 > c) x[i + 1] = fmaf(-a.y, x[c], x[i + 1]);
              if (i + 2 > c) x[i + 2] = fmaf(-a.z, x[c], x[i + 2]);
              if (i + 3 > c) x[i + 3] = fmaf(-a.w, x[c], x[i + 3]);
            }
          }
        } else {
#pragma unroll
          for (int c = 31; c >= 0; --c) {
            if (!unit) x[c] *= s_rcp[k0 + c];
#pragma unroll
            for (int i = 0; i < c; i += 4) {
              const float4 a = *reinterpret_cast<const float4*>(sA + c * PA + k0 + i);
              x[i] = fmaf(-a.x, x[c], x[i]);
              if (i + 1 < c) x[i + 1] = fmaf(-a.y, x[c], x[i + 1]);
              if (i + 2 < c) x[i + 2] = fmaf(-a.z, x[c], x[i + 2]);
              if (i + 3 < c) x[i + 3] = fmaf(-a.w, x[c], x[i + 3]);
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 32; ++i) sX[(k0 + i) * PX + tid] = x[i];
      }
      __syncthreads();
      const int g0 = sweep == 0 ? k0 + 32 : 0, g1 = sweep == 0 ? mp : k0;  // rows to update, multiples of 32
      for (int i0 = g0 + 8 * ty; i0 < g1; i0 += 128) {
        float acc[8][4];
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[a][q] = 0.f;
#pragma unroll 8
        for (int c = 0; c < 32; ++c) {
          float av[8], xv[4];
          *reinterpret_cast<float4*>(av) = *reinterpret_cast<const float4*>(sA + c * PA + i0);
          *reinterpret_cast<float4*>(av + 4) = *reinterpret_cast<const float4*>(sA + c * PA + i0 + 4);
          *reinterpret_cast<float4*>(xv) = *reinterpret_cast<const float4*>(sX + (k0 + c) * PX + 4 * tx);
#pragma unroll
          for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[a][q] = fmaf(av[a], xv[q], acc[a][q]);
        }
#pragma unroll
        for (int a = 0; a < 8; ++a) {
          float4* p = reinterpret_cast<float4*>(sX + (i0 + a) * PX + 4 * tx);
          float4 v = *p;
          v.x -= acc[a][0];
          v.y -= acc[a][1];
          v.z -= acc[a][2];
          v.w -= acc[a][3];
          *p = v;
        }
      }
    }
  }
  __syncthreads();
  for (int i = lane; i < m; i += 32) {
    const int dst = trans ? pb[i] : i;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int col = warp + 8 * u;
      if (j0 + col < ncols) out[(int64_t)(j0 + col) * ldout + row0 + dst] = conv<TOUT>(sX[i * PX + col]);
    }
  }
}

template <typename TIN, typename TOUT>
cudaError_t launch_leaf_solve_f32(const Factor& F, const TIN* in, int64_t ldin, TOUT* out, int64_t ldout, int ncols,
                                  int trans, cudaStream_t s) {
  const int m = F.d.m, mp = (m + 31) / 32 * 32;
  const double Nd = (double)((int64_t)1 << F.d.L) * m;
  note_work((sizeof(TIN) + sizeof(TOUT)) * Nd * ncols + 4.0 * Nd * m + 4.0 * Nd, 2.0 * m * Nd * ncols);
  const size_t sm = ((size_t)mp * 68 + (size_t)32 * (mp + 4)) * sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(leaf_solve_f32_kernel<TIN, TOUT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sm);
  if (e != cudaSuccess) return e;
  dim3 grid(1u << F.d.L, (unsigned)((ncols + 63) / 64));
  leaf_solve_f32_kernel<TIN, TOUT><<<grid, 256, sm, s>>>(m, static_cast<const float*>(F.lu), F.perm, in, ldin, out,
                                                         ldout, ncols, trans);
  note_launches(1);
  return cudaGetLastError();
}

#define HODLR_INST(TIN, TOUT)                                                                                   \
  template cudaError_t launch_leaf_solve_f32<TIN, TOUT>(const Factor&, const TIN*, int64_t, TOUT*, int64_t, int, \
                                                        int, cudaStream_t);
HODLR_INST(double, double)
HODLR_INST(double, float)
HODLR_INST(double, __nv_bfloat16)
HODLR_INST(float, float)
#undef HODLR_INST

}  // namespace hodlr
