// Coupling matrices with FP64 products (every factor but the BF16 one), one CTA per
// parent. K~ = [[I, T_b], [T_a, I]] (Eq. e:k) has identity diagonal blocks, so with
// S = I - T_a T_b
//   K~^{-1} = [[I + T_b S^{-1} T_a, -T_b S^{-1}], [-S^{-1} T_a, S^{-1}]],
//   det K~ = det S.
// S is inverted by Gauss-Jordan with partial pivoting in FP64 (LU's pivots), which
// also gives log|det S| and its sign. The four products are split-operand products on
// the tensor cores (fp64_split.cuh): on the FP64 pipe of the one SM that has the
// parent they took two thirds of the time at r = 32 and four fifths at r = 64.
// What is left is the inversion's r dependent steps. A level of up to 152 parents: 60 ->
// 46 us at r = 16 (the inversion also ends at r instead of 32), 500 -> 330 us at r = 64.
#include "fp64_split.cuh"
#include "gj.cuh"

namespace hodlr {
using namespace split;

namespace {

// out(i, j, sum_k a(i, k) b(k, j)) for the RT x RT matrices a, b (shared memory), by the
// whole CTA: a is split into sA (digits in fragment order, 32-term blocks) by eight
// lanes per row and block, column tiles of b by the warps. All reads of a and b end
// before the first out.
template <int RT, class A, class B, class Out>
__device__ __forceinline__ void cta_gemm(unsigned char* sA, int* sE, A a, B b, Out out) {
  constexpr int KB = RT / 32, MT = RT / 16, NT = RT == 64 ? 256 : 128;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  __syncthreads();
#pragma unroll
  for (int v = 0; v < RT * RT / 4 / NT; ++v) {
    const int task = v * NT + tid;
    const int grp = task & 7, kb = (task >> 3) % KB, row = (task >> 3) / KB;
    double y[1][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) y[0][q] = a(row, kb * 32 + grp * 4 + q);
    const int e = shared_exp<1, 7>(y);
    if (grp == 0) sE[kb * RT + row] = e;
    uint2 d[kDigits];
    split4(y[0], e, d);
    unsigned char* dst = sA + (((row >> 4) * KB + kb) * 2 + (grp >> 2)) * (kPlanes * 512) +
                         ((row & 7) * 4 + (grp & 3)) * 16 + ((row >> 3) & 1) * 8;
    store_planes(dst, d);
  }
  __syncthreads();
  const int j0 = warp * 8;  // RT / 8 warps
  double acc[MT][4];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[mt][u] = 0.0;
#pragma unroll 1
  for (int kb = 0; kb < KB; ++kb) {
    uint2 bf[2][kDigits];
    double x[2][4];
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int q = 0; q < 4; ++q) x[s][q] = b(kb * 32 + 16 * s + 4 * t + q, j0 + g);
    const int e = shared_exp<2, 3>(x);
#pragma unroll
    for (int s = 0; s < 2; ++s) split4(x[s], e, bf[s]);
    const int eb0 = __shfl_sync(0xffffffffu, e, 8 * t), eb1 = __shfl_sync(0xffffffffu, e, 8 * t + 4);
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
      const uint4* fa = reinterpret_cast<const uint4*>(sA + (mt * KB + kb) * 2 * (kPlanes * 512)) + lane;
      const int* ea = sE + kb * RT + mt * 16 + g;
      double v[4];
      tile<true>(StagedA<2>{fa, bf}, ea[0], ea[8], eb0, eb1, v, [&](int u) {
        double d = 0.0;
        for (int k = kb * 32; k < kb * 32 + 32; ++k)
          d = fma(a(mt * 16 + g + (u >> 1) * 8, k), b(k, j0 + 2 * t + (u & 1)), d);
        return d;
      });
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[mt][u] += v[u];
    }
  }
  __syncthreads();
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int u = 0; u < 4; ++u) out(mt * 16 + g + (u >> 1) * 8, j0 + 2 * t + (u & 1), acc[mt][u]);
}

// Lane of the unused row with the largest |x|, the lowest on ties, compared as
// integers (the FP64 pipe is left to the elimination); NaN above every number.
__device__ __forceinline__ int pivot_row(double x, bool used) {
  const uint64_t bits = (uint64_t)__double_as_longlong(x) & 0x7fffffffffffffffull;
  const uint32_t hi = used ? 0u : (uint32_t)(bits >> 32) + 1u, lo = used ? 0u : (uint32_t)bits;
  const uint32_t H = __reduce_max_sync(0xffffffffu, hi);
  const uint32_t Lo = __reduce_max_sync(0xffffffffu, hi == H ? lo : 0u);
  return __ffs(__ballot_sync(0xffffffffu, hi == H && lo == Lo)) - 1;
}

}  // namespace

template <int RT>
__global__ void __launch_bounds__(RT == 64 ? 256 : 128) coupling_split_kernel(
    int64_t cpn, int r, int c, const double* __restrict__ P, double* __restrict__ Kinv,
    double* __restrict__ node_ld, DevStatus* st, int64_t heap_first, float* __restrict__ Kf) {
  constexpr int NT = RT == 64 ? 256 : 128;
  constexpr int LD = RT + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* sA = smem_raw;                                               // planes, RT^2 16-bit each
  double* Ta = reinterpret_cast<double*>(smem_raw + (size_t)RT * RT * 2 * kPlanes);  // column-major, ld LD
  double* Tb = Ta + RT * LD;
  double* Si = Tb + RT * LD;  // S, then S^{-1}
  double* M1 = Si + RT * LD;  // S^{-1} T_a
  int* sE = reinterpret_cast<int*>(M1 + RT * LD);  // RT / 32 x RT
  __shared__ double s_la;
  __shared__ int s_neg, s_sing;
  const int64_t j = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t slot = (size_t)r * r * c;
  const int anc = r * (c - 1);
  const int64_t qa = 2 * j * cpn, qb = (2 * j + 1) * cpn;
  for (int e = tid; e < RT * RT; e += NT) {
    const int row = e % RT, col = e / RT;
    double a = 0.0, b = 0.0;
    if (row < r && col < r) {
      a = P[qa * slot + (size_t)(anc + col) * r + row];
      b = P[qb * slot + (size_t)(anc + col) * r + row];
    }
    Ta[col * LD + row] = a;
    Tb[col * LD + row] = b;
  }
  auto ta = [&](int i, int k) { return Ta[k * LD + i]; };
  auto tb = [&](int i, int k) { return Tb[k * LD + i]; };
  auto m1 = [&](int i, int k) { return M1[k * LD + i]; };
  // S^{-1} less the identity's rows (columns) where it has them: with weak coupling S^{-1}
  // is close to I, and the digits of what is left reach as far down as a sum needs. A
  // diagonal entry below 1/2 keeps its row and column as they are: with |T_a T_b| >> 1 the
  // products are as small as S^{-1} is, and T_a + (S^{-1} - I) T_a would cancel (roundings of
  // size |T| in results of size 1 / |T|). From 1/2 on, the two terms that are added are at
  // most twice the terms of the plain product.
  auto has_one = [&](int i) { return Si[i * LD + i] >= 0.5; };
  auto off = [&](int i, int k) { return Si[k * LD + i] - (i == k && has_one(i) ? 1.0 : 0.0); };
  cta_gemm<RT>(sA, sE, ta, tb, [&](int i, int k, double v) { Si[k * LD + i] = (i == k ? 1.0 : 0.0) - v; });
  __syncthreads();
  if constexpr (RT == 64) {
    double* scr = reinterpret_cast<double*>(sA);  // free until the next product
    double *spv = scr, *scol = scr + RT, *srow = scr + 2 * RT;
    int* spiv = reinterpret_cast<int*>(scr + 3 * RT);
    int* spos = spiv + RT;
    gj_invert_smem<double>(Si, r, LD, spiv, spv, scol, srow, spos, &s_la, &s_neg, &s_sing);
    for (int e = tid; e < r * r; e += NT) M1[e / r * LD + e % r] = Si[(size_t)spos[e / r] * LD + e % r];
    __syncthreads();
    for (int e = tid; e < r * r; e += NT) Si[e / r * LD + e % r] = M1[e / r * LD + e % r];
  } else {
    // lane = row, warp w columns 8w .. 8w + 7 in registers; rows are not moved: the
    // warp that owns column k finds the pivot and publishes it, double buffered, one
    // barrier per step
    __shared__ double sh_f[2][32], sh_piv[2];
    __shared__ int sh_p[2];
    const int c0 = warp * 8;
    double s[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) s[q] = Si[(c0 + q) * LD + lane];
    bool used = false;
    double mypiv = 1.0;
    int mypos = lane, mystep = lane, ninv = 0;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      if (k < r) {  // beyond r the matrix is the identity
        const int buf = k & 1;
        const int ow = k >> 3, kk = k & 7;
        if (warp == ow) {
          const int idx = pivot_row(s[kk], used);
          const double pv = __shfl_sync(0xffffffffu, s[kk], idx);
          sh_f[buf][lane] = s[kk];
          if (lane == 0) {
            sh_p[buf] = idx;
            sh_piv[buf] = pv;
          }
        }
        __syncthreads();
        const int p = sh_p[buf];
        const double piv = sh_piv[buf];
        const double rp = piv != 0.0 ? 1.0 / piv : 0.0;
        if (lane < k) ninv += p < mypos ? 1 : 0;
        if (lane == k) {
          mypiv = piv;
          mypos = p;
        }
        const bool isp = lane == p;
        if (isp) {
          used = true;
          mystep = k;
        }
        const double coef = isp ? rp : -sh_f[buf][lane] * rp;
        if (c0 < r) {
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const double pvq = __shfl_sync(0xffffffffu, s[q], p);
            s[q] = (warp == ow && q == kk) ? coef : fma(coef, pvq, isp ? 0.0 : s[q]);
          }
        }
      }
    }
    double la = lane < r ? log(fabs(mypiv)) : 0.0;
    int neg = ((lane < r && mypiv < 0.0) ? 1 : 0) ^ (ninv & 1);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      la += __shfl_xor_sync(0xffffffffu, la, o);
      neg ^= __shfl_xor_sync(0xffffffffu, neg, o);
    }
    const unsigned zero = __ballot_sync(0xffffffffu, lane < r && mypiv == 0.0);
    if (tid == 0) {
      s_la = la;
      s_neg = neg;
      s_sing = zero ? __ffs(zero) - 1 : -1;
    }
    // S^{-1}(k, i) = tableau(p_k, step of row i)
#pragma unroll
    for (int q = 0; q < 8; ++q) M1[(c0 + q) * LD + lane] = s[q];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 8; ++q) Si[(c0 + q) * LD + lane] = M1[__shfl_sync(0xffffffffu, mystep, c0 + q) * LD + mypos];
  }
  // M1 = S^{-1} T_a
  cta_gemm<RT>(sA, sE, off, ta, [&](int i, int k, double v) { M1[k * LD + i] = has_one(i) ? ta(i, k) + v : v; });
  const int n = 2 * r;
  double* out = Kinv + (size_t)j * n * n;  // column-major
  float* kf0 = Kf ? Kf + (size_t)(2 * j) * r * (n + 4) : nullptr;  // rows facing each child, FP32, pitch 2r + 4
  float* kf1 = Kf ? Kf + (size_t)(2 * j + 1) * r * (n + 4) : nullptr;
  // [11] = I + T_b M1
  cta_gemm<RT>(sA, sE, tb, m1, [&](int i, int k, double v) {
    if (i >= r || k >= r) return;
    const double w = v + (i == k ? 1.0 : 0.0);
    out[(size_t)k * n + i] = w;
    if (Kf) kf0[i * (n + 4) + k] = (float)w;
  });
  // [12] = -T_b S^{-1}
  cta_gemm<RT>(sA, sE, tb, off, [&](int i, int k, double v) {
    if (i >= r || k >= r) return;
    const double w = -(has_one(k) ? tb(i, k) + v : v);
    out[(size_t)(r + k) * n + i] = w;
    if (Kf) kf0[i * (n + 4) + r + k] = (float)w;
  });
  // [21] = -M1, [22] = S^{-1}
  for (int e = tid; e < r * r; e += NT) {
    const int i = e % r, k = e / r;
    const double a = -M1[k * LD + i], b = Si[k * LD + i];
    out[(size_t)k * n + r + i] = a;
    out[(size_t)(r + k) * n + r + i] = b;
    if (Kf) {
      kf1[i * (n + 4) + k] = (float)a;
      kf1[i * (n + 4) + r + k] = (float)b;
    }
  }
  if (tid == 0) {
    node_ld[2 * j] = s_la;
    node_ld[2 * j + 1] = (s_sing >= 0) ? 0.0 : (s_neg ? -1.0 : 1.0);
    if (s_sing >= 0) set_status(st, HODLR_ERR_SINGULAR_COUPLING, heap_first + j, r + s_sing);
  }
}

template <int RT>
static cudaError_t coupling_split_go(const Factor& F, int c, float* Kf, cudaStream_t s) {
  const int r = F.d.r, n = 2 * r;
  const int64_t parents = (int64_t)1 << (c - 1);
  const size_t sm = (size_t)RT * RT * 2 * kPlanes + 4 * (size_t)RT * (RT + 1) * sizeof(double) +
                    (size_t)RT * (RT / 32) * sizeof(int);
  cudaError_t e = cudaFuncSetAttribute(coupling_split_kernel<RT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sm);
  if (e != cudaSuccess) return e;
  coupling_split_kernel<RT><<<(unsigned)parents, RT == 64 ? 256 : 128, sm, s>>>(
      F.cpn, r, c, F.P, F.K + F.Koff[c] * n * n, F.node_ld + 2 * F.Koff[c], F.status, parents, Kf);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_coupling_factor_split(const Factor& F, int c, float* Kf, cudaStream_t s) {
  return F.d.r <= 32 ? coupling_split_go<32>(F, c, Kf, s) : coupling_split_go<64>(F, c, Kf, s);
}

}  // namespace hodlr
