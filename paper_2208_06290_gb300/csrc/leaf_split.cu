// FP64 leaf products and leaf solves for several columns on the FP16 tensor
// cores (fp64_split.cuh).
#include "fp64_split.cuh"
#include "substitute.cuh"

namespace hodlr {
using namespace split;

namespace {

// Digits of a 32 x 32 block as an A operand: [row tile of 16][k16][plane][lane] 16 B,
// with the rows' exponents in sE. Four warps, w4 = 0 .. 3, hold eight rows each: lane
// (g, t) terms 16 s + 4 t .. + 3 of row w4 8 + g.
constexpr int kBlockFrag = 2 * 2 * kPlanes * 512;
__device__ __forceinline__ void put_block(const double (&x)[2][4], unsigned char* dst, int* sE, int w4, int lane) {
  const int e = shared_exp<2, 3>(x);
  if ((lane & 3) == 0) sE[w4 * 8 + (lane >> 2)] = e;
  unsigned char* d0 = dst + (w4 >> 1) * (2 * kPlanes * 512) + lane * 16 + (w4 & 1) * 8;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    uint2 d[kDigits];
    split4(x[s], e, d);
    store_planes(d0 + s * kPlanes * 512, d);
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// Inverses of the 32 x 32 diagonal blocks of the leaf LUs, for the blocked
// substitutions below: L_kk^{-1} (unit lower) in the strict lower triangle and
// U_kk^{-1} in the upper one of a column-major block of the same size (tinv_elems). One
// warp per block and triangle, lane j = column j.
// x = T b instead of a substitution leaves a residual of up to u |A| |T| |A| |x|: as good as
// substitution's u |A| |x| unless |A| |T| is large, which is when the pivots fall by orders
// of magnitude within the block. Blocks whose |A| |T| or |T| |A| (the transposed solve)
// exceeds kTinvMost in the 1-norm, or that have a zero pivot, are marked in `sub` for
// plain substitution. (Random blocks have 1e2 to 1e3, kernel matrices with a nugget of
// 1e-3 2e3, smooth ones of condition 3e7 7e6, where solves lost a digit and more:
// backward error 4e-16 against 5e-17.)
// (One warp for both triangles and a division per column were 42 us of latency.)
constexpr float kTinvMost = 4096.f;

__device__ __forceinline__ float abs_f32(double x) { return __uint_as_float(f64_to_f32_trunc_bits(x) & 0x7fffffffu); }

__global__ void __launch_bounds__(128) leaf_tinv_kernel(int m, int64_t nblocks, const double* __restrict__ LU,
                                                        double* __restrict__ tinv, uint8_t* __restrict__ sub) {
  __shared__ double sB[2][32][33];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t id = (int64_t)blockIdx.x * 2 + (warp >> 1);
  const int nb = (m + 31) / 32;
  const int k0 = (int)(id % nb) * 32;
  const int n = min(32, m - k0);
  double(*B)[33] = sB[warp >> 1];  // B[col][row]
  if (id < nblocks) {
    const double* A = LU + (size_t)(id / nb) * m * m + (size_t)k0 * m + k0;
    for (int j = warp & 1; j < n; j += 2) B[j][lane] = lane < n ? A[(size_t)j * m + lane] : 0.0;
  }
  __syncthreads();
  if (id >= nblocks) return;  // whole warp
  const bool upper = (warp & 1) != 0;
  double* out = tinv + (size_t)(id / nb) * tinv_elems(m) + (size_t)k0 * 32;
  double x[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) x[i] = i == lane ? 1.0 : 0.0;
  if (!upper) {
    // unit lower: column `lane` of the inverse, rows below the diagonal
#pragma unroll
    for (int k = 0; k < 31; ++k) {
      if (k < n) {
#pragma unroll
        for (int i = k + 1; i < 32; ++i)
          if (i < n) x[i] = fma(-B[k][i], x[k], x[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < 32; ++i)
      if (i > lane && i < n) out[lane * n + i] = x[i];
  } else {
    // upper: column `lane`, rows up to the diagonal
    const double rcp = lane < n ? 1.0 / B[lane][lane] : 1.0;
#pragma unroll
    for (int k = 31; k >= 0; --k) {
      const double rk = __shfl_sync(0xffffffffu, rcp, k);
      if (k < n) {
        x[k] *= rk;
#pragma unroll
        for (int i = 0; i < k; ++i) x[i] = fma(-B[k][i], x[k], x[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < 32; ++i)
      if (i <= lane && lane < n) out[lane * n + i] = x[i];
  }
  // column sums of |A| and |T|, then those of |A| |T| and |T| |A|, in FP32
  const int mine = lane < n ? lane : 0;
  float fa[32], sa = 0.f, st = 0.f;
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    fa[i] = abs_f32(B[mine][i]);
    if (!upper && i == lane) fa[i] = 1.f;
    if (i >= n || (upper ? i > lane : i < lane)) fa[i] = 0.f;
    sa += fa[i];
  }
#pragma unroll
  for (int i = 0; i < 32; ++i) st += abs_f32(x[i]);
  float at = 0.f, ta = 0.f;
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    at += __shfl_sync(0xffffffffu, sa, i) * abs_f32(x[i]);
    ta += __shfl_sync(0xffffffffu, st, i) * fa[i];
  }
  const bool most = lane < n && !(at <= kTinvMost && ta <= kTinvMost);  // true for NaN
  const bool any = __any_sync(0xffffffffu, most);
  if (lane == 0) sub[2 * id + (upper ? 1 : 0)] = any ? 1 : 0;
}

cudaError_t launch_leaf_tinv(const Factor& F, cudaStream_t s) {
  const int nb = (F.d.m + 31) / 32;
  const int64_t blocks = ((int64_t)1 << F.d.L) * nb;
  leaf_tinv_kernel<<<(unsigned)((blocks + 1) / 2), 128, 0, s>>>(F.d.m, blocks, static_cast<const double*>(F.lu),
                                                                F.tinv, F.tsub);
  note_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// X_b <- D_b^{-1} X_b (trans 0) or D_b^{-T} X_b (trans 1) by blocked
// substitution with the leaf LUs. CTA = one leaf x 64 columns; every warp owns
// eight columns in shared memory (FP64) and runs right-looking over 32-row
// blocks: x_k <- T_k x_k with the inverted diagonal block, then x_j -= A_jk x_k.
// The A blocks are split by four of the CTA's warps into a double buffer (one
// barrier per block) from registers that were loaded one block ahead: with one or two
// CTAs of eight warps an SM, nothing else hides that load. The solved x_k is split
// into registers; all products are digit products, the subtractions FP64. A diagonal
// block's own diagonal is left out of its digits and applied in FP64: a row's other
// entries then have all of them (as one product, x_i alone in a row of zeros is small
// beside the block's largest entry too often, and FP64 FMAs for those took longer
// than all the digits). Marked diagonal blocks (leaf_tinv_kernel) are substituted.
// N = 2^18, leaf 256, 64 columns, both ways: 18.4 ms on the FP64 pipe, 4.2 now, of which 0.1
// are the accuracy of small sums and the diagonal in FP64.
template <int W, int MINB>
__global__ void __launch_bounds__(32 * W, MINB) leaf_solve_split_kernel(int m, const double* __restrict__ LU,
                                                                     const double* __restrict__ tinv,
                                                                     const uint8_t* __restrict__ tsub,
                                                                     const int* __restrict__ perm, const double* in,
                                                                     int64_t ldin, double* out, int64_t ldout,
                                                                     int ncols, int trans) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nb = (m + 31) / 32;
  const int S = nb * 32 + 2;  // rows of a column in shared memory: 16-byte aligned, staggered banks
  unsigned char* sA = smem_raw;                                        // two blocks
  int* sE = reinterpret_cast<int*>(smem_raw + 2 * kBlockFrag);         // 2 x 32
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  double* sD = reinterpret_cast<double*>(smem_raw + 2 * kBlockFrag + 256);  // 2 x 32: diagonal of a diagonal block
  double* sX = sD + 64 + (size_t)warp * 8 * S;                              // [column][row]
  const int64_t b = blockIdx.x;
  const double* A = LU + (size_t)b * m * m;
  const double* T = tinv + (size_t)b * tinv_elems(m);
  const unsigned marked = __ballot_sync(0xffffffffu, lane < 2 * nb && tsub[(size_t)b * 2 * nb + (lane < 2 * nb ? lane : 0)] != 0);
  const int* pb = perm + (size_t)b * m;
  const int64_t row0 = b * m;
  const int j0 = (blockIdx.y * W + warp) * 8;
  for (int cc = 0; cc < 8; ++cc) {
    const bool ok = j0 + cc < ncols;
    const double* src = in + (int64_t)(ok ? j0 + cc : 0) * ldin + row0;
    for (int i = lane; i < nb * 32; i += 32)
      sX[cc * S + i] = (ok && i < m) ? src[trans ? i : pb[i]] : 0.0;
  }
  __syncwarp();
  int buf = 0;
  // sweep 0: the lower-triangular factor of op(A), blocks downwards; sweep 1: the
  // upper one, upwards. op(A) = L U, or U^T L^T.
  const int helper = W == 8 ? (warp >> 2) : 0;
  // this lane's entries of block (sweep, kk, st): the diagonal block's inverse T_k (L_kk^{-1}
  // or U_kk^{-1}, transposed or not) for st 0, else the block of op(A) in row block j
  double pre[2][4], dg = 0.0;
  auto fetch = [&](int sweep, int kk, int st) {
    const bool useL = (sweep == 0) == (trans == 0);
    const int k = sweep == 0 ? kk : nb - 1 - kk, j = sweep == 0 ? k + st : k - st;
    const int nr = min(32, m - j * 32), nk = min(32, m - k * 32);
    const int row = (warp & 3) * 8 + g;
    const double* Aj = trans ? A + (size_t)(j * 32 + row) * m + k * 32 : A + (size_t)(k * 32) * m + j * 32 + row;
    const size_t cs = trans ? 1 : m;
    if (st == 0 && t == 0) dg = row >= nk ? 0.0 : useL ? 1.0 : T[k * 1024 + row * nk + row];
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int kc = 16 * s + 4 * t + q;
        double v = 0.0;
        if (row < nr && kc < nk) {
          if (st > 0) {
            v = Aj[kc * cs];
          } else {
            const int i = trans ? kc : row, c = trans ? row : kc;  // element (i, c) of L^{-1} or U^{-1}
            if (useL ? i > c : i < c) v = T[k * 1024 + c * nk + i];
          }
        }
        pre[s][q] = v;
      }
  };
  if (W < 8 || helper == 0) fetch(0, 0, 0);
  for (int sweep = 0; sweep < 2; ++sweep) {
    const bool useL = (sweep == 0) == (trans == 0);
    for (int kk = 0; kk < nb; ++kk) {
      const int k = sweep == 0 ? kk : nb - 1 - kk;
      uint2 bf[2][kDigits];
      int eb0 = 0, eb1 = 0;
      const int steps = nb - kk;  // the diagonal block, then the remaining ones
      for (int st = 0; st < steps; ++st) {
        const int j = sweep == 0 ? k + st : k - st;
        unsigned char* sAb = sA + buf * kBlockFrag;
        int* sEb = sE + buf * 32;
        if (W < 8 || helper == buf) {
          put_block(pre, sAb, sEb, warp & 3, lane);
          if (st == 0 && t == 0) sD[buf * 32 + (warp & 3) * 8 + g] = dg;
        }
        __syncthreads();
        if (W < 8 || helper != buf) {  // the next block's warps
          if (st + 1 < steps) fetch(sweep, kk, st + 1);
          else if (kk + 1 < nb) fetch(sweep, kk + 1, 0);
          else if (sweep == 0) fetch(1, 0, 0);
        }
        if (j0 < ncols && st == 0 && (marked >> (2 * k + (useL ? 0 : 1)) & 1u)) {
          double x[8];
#pragma unroll
          for (int cc = 0; cc < 8; ++cc) x[cc] = sX[cc * S + k * 32 + lane];
          substitute<8>(A + (size_t)k * 32 * (m + 1), m, min(32, m - k * 32), sweep, useL, trans, lane, x);
#pragma unroll
          for (int cc = 0; cc < 8; ++cc) sX[cc * S + k * 32 + lane] = x[cc];
          __syncwarp();
        } else if (j0 < ncols) {
          double* xk = sX + k * 32;
          double* xj = sX + j * 32;
          if (st <= 1) {
            // digits of x_k: the right-hand side of the diagonal block, then the solved block
            double x[2][4];
#pragma unroll
            for (int s = 0; s < 2; ++s) load4(xk + g * S + 16 * s + 4 * t, x[s]);
            const int e = shared_exp<2, 3>(x);
#pragma unroll
            for (int s = 0; s < 2; ++s) split4(x[s], e, bf[s]);
            eb0 = __shfl_sync(0xffffffffu, e, 8 * t);
            eb1 = __shfl_sync(0xffffffffu, e, 8 * t + 4);
          }
          double v[2][4];
#pragma unroll
          for (int mt = 0; mt < 2; ++mt) {
            const uint4* fa = reinterpret_cast<const uint4*>(sAb + mt * (2 * kPlanes * 512)) + lane;
            const int ea0 = sEb[mt * 16 + g], ea1 = sEb[mt * 16 + g + 8];
            tile<true>(StagedA<2>{fa, bf}, ea0, ea1, eb0, eb1, v[mt], [&](int u) {
              const int i = mt * 16 + g + (u >> 1) * 8;
              const double* xc = xk + (2 * t + (u & 1)) * S;
              const int ri = j * 32 + i, nk = min(32, m - k * 32);
              double a = 0.0;
              if (ri >= m) return a;
              if (st == 0) {  // the strict triangle's terms: mostly rows with one or two
                const int c1 = sweep == 0 ? i : nk;
                for (int c = sweep == 0 ? 0 : i + 1; c < c1; ++c)
                  a = fma(T[k * 1024 + (trans ? i * nk + c : c * nk + i)], xc[c], a);
              } else {
#pragma unroll 8
                for (int c = 0; c < nk; ++c)
                  a = fma(trans ? A[(size_t)ri * m + k * 32 + c] : A[(size_t)(k * 32 + c) * m + ri], xc[c], a);
              }
              return a;
            });
          }
          __syncwarp();
#pragma unroll
          for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              double* p = xj + (2 * t + (u & 1)) * S + mt * 16 + g + (u >> 1) * 8;
              *p = st == 0 ? fma(sD[buf * 32 + mt * 16 + g + (u >> 1) * 8], *p, v[mt][u]) : *p - v[mt][u];
            }
          __syncwarp();
        }
        buf ^= 1;
      }
    }
  }
  for (int cc = 0; cc < 8; ++cc) {
    if (j0 + cc >= ncols) break;
    double* dst = out + (int64_t)(j0 + cc) * ldout + row0;
    for (int i = lane; i < m; i += 32) dst[trans ? pb[i] : i] = sX[cc * S + i];
  }
}

template <int W, int MINB>
static cudaError_t leaf_solve_split_go(const Factor& F, const double* in, int64_t ldin, double* out, int64_t ldout,
                                       int ncols, int trans, cudaStream_t s) {
  const int m = F.d.m, nb = (m + 31) / 32;
  const size_t sm = 2 * kBlockFrag + 256 + 64 * sizeof(double) + (size_t)W * 8 * (nb * 32 + 2) * sizeof(double);
  cudaError_t e = cudaFuncSetAttribute(leaf_solve_split_kernel<W, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sm);
  if (e != cudaSuccess) return e;
  dim3 grid(1u << F.d.L, (unsigned)((ncols + 8 * W - 1) / (8 * W)));
  leaf_solve_split_kernel<W, MINB><<<grid, 32 * W, sm, s>>>(m, static_cast<const double*>(F.lu), F.tinv, F.tsub, F.perm,
                                                            in, ldin, out, ldout, ncols, trans);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_leaf_solve_split(const Factor& F, const double* in, int64_t ldin, double* out, int64_t ldout,
                                    int ncols, int trans, cudaStream_t s) {
  const int m = F.d.m;
  const double Nd = (double)((int64_t)1 << F.d.L) * m;
  note_work(16.0 * Nd * ncols + 8.0 * Nd * m + 4.0 * Nd, 2.0 * m * Nd * ncols);
  if (ncols <= 32) return leaf_solve_split_go<4, 2>(F, in, ldin, out, ldout, ncols, trans, s);
  if (m <= 128) return leaf_solve_split_go<8, 2>(F, in, ldin, out, ldout, ncols, trans, s);
  return leaf_solve_split_go<8, 1>(F, in, ldin, out, ldout, ncols, trans, s);
}

// ---------------------------------------------------------------------------
// Small batched products C = A B on 16 W rows x 8 NT columns per CTA (W warps,
// 16 rows each): the B operand is split by the CTA into shared memory, 128
// terms at a time; every warp splits its own A entries in registers (so A is
// read and split once per 8 NT columns). `Op` names the batch's matrices. C may
// overlay B's columns where a CTA has all rows and at most 128 terms.
template <class Op, int NT, int W>
__global__ void __launch_bounds__(32 * W, W == 4 ? 3 : 1) gemm_split_kernel(Op op) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* sB = smem_raw;                                             // [block][NT][plane][lane] 16 B
  int* sE = reinterpret_cast<int*>(smem_raw + 4 * NT * kPlanes * 512);      // [block][8 NT]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int rtiles = (op.rows + 16 * W - 1) / (16 * W);
  const int64_t batch = blockIdx.x / rtiles;
  const int i0 = (int)(blockIdx.x % rtiles) * (16 * W) + warp * 16 + 2 * g;  // rows i0, i0 + 1
  const int j0 = blockIdx.y * 8 * NT;
  double acc[NT][4];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[nt][u] = op.init(batch, i0 + (u >> 1), j0 + nt * 8 + 2 * t + (u & 1));
  const int rest = min(NT, (op.cols - j0 + 7) / 8);  // column tiles in use
  for (int k0 = 0; k0 < op.terms; k0 += 128) {
    const int nkb = min(4, (op.terms - k0 + 31) / 32);
    __syncthreads();
    for (int task = tid; task < nkb * NT * 64; task += 32 * W) {
      const int kb = task / (NT * 64), j = (task / 8) % (8 * NT), grp = task % 8;
      double y[1][4];
      op.load_b(batch, k0 + kb * 32 + grp * 4, j0 + j, y[0]);
      const int e = shared_exp<1, 7>(y);
      if (grp == 0) sE[kb * 8 * NT + j] = e;
      uint2 d[kDigits];
      split4(y[0], e, d);
      unsigned char* dst = sB + ((size_t)(kb * NT + (j >> 3)) * kPlanes * 32 + (j & 7) * 4 + (grp & 3)) * 16 +
                           (grp >> 2) * 8;
      store_planes(dst, d);
    }
    __syncthreads();
    for (int kb = 0; kb < nkb; ++kb) {
      const int kk = k0 + kb * 32;
      uint2 af[2][2][kDigits];
      int ea[2];
      {
        double x[2][2][4];
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
          for (int q = 0; q < 4; ++q) op.load_a(batch, i0, kk + 16 * s + 4 * t + q, x[0][s][q], x[1][s][q]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          ea[h] = shared_exp<2, 3>(x[h]);
#pragma unroll
          for (int s = 0; s < 2; ++s) split4(x[h][s], ea[h], af[s][h]);
        }
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        if (nt >= rest) break;
        const int eb0 = sE[kb * 8 * NT + nt * 8 + 2 * t], eb1 = sE[kb * 8 * NT + nt * 8 + 2 * t + 1];
        const uint4* fb = reinterpret_cast<const uint4*>(sB) + (size_t)(kb * NT + nt) * kPlanes * 32 + lane;
        double v[4];
        tile<true>(StagedB<1>{af, fb}, ea[0], ea[1], eb0, eb1, v, [&](int u) {
          double d = 0.0;
#pragma unroll 4
          for (int k = kk; k < kk + 32 && k < op.terms; ++k) {
            double a0, a1;
            op.load_a(batch, i0, k, a0, a1);
            d = fma((u >> 1) ? a1 : a0, op.b(batch, k, j0 + nt * 8 + 2 * t + (u & 1)), d);
          }
          return d;
        });
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[nt][u] += v[u];
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int u = 0; u < 2; ++u)
      op.store(batch, i0, j0 + nt * 8 + 2 * t + u, acc[nt][u], acc[nt][2 + u]);
}

template <class Op, int NT, int W>
static cudaError_t gemm_split_nt(const Op& op, int64_t batches, cudaStream_t s) {
  const size_t sm = (size_t)4 * NT * kPlanes * 512 + 4 * 8 * NT * sizeof(int);
  cudaError_t e = cudaFuncSetAttribute(gemm_split_kernel<Op, NT, W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sm);
  if (e != cudaSuccess) return e;
  dim3 grid((unsigned)(batches * ((op.rows + 16 * W - 1) / (16 * W))),
            (unsigned)((op.cols + 8 * NT - 1) / (8 * NT)));
  gemm_split_kernel<Op, NT, W><<<grid, 32 * W, sm, s>>>(op);
  note_launches(1);
  return cudaGetLastError();
}

template <class Op, int W = 4>
static cudaError_t gemm_split(const Op& op, int64_t batches, cudaStream_t s) {
  if (op.cols <= 8) return gemm_split_nt<Op, 1, W>(op, batches, s);
  if (op.cols <= 16) return gemm_split_nt<Op, 2, W>(op, batches, s);
  return gemm_split_nt<Op, 4, W>(op, batches, s);
}

// Y_b = D_b X_b.
struct LeafMatvecOp {
  int rows, cols, terms;
  const double* D;
  const double* X;
  int64_t ldx;
  double* Y;
  int64_t ldy;
  __device__ double init(int64_t, int, int) const { return 0.0; }
  __device__ void load_a(int64_t b, int i, int k, double& a0, double& a1) const {
    const double* p = D + (size_t)b * rows * rows + (size_t)k * rows + i;
    a0 = (k < terms && i < rows) ? p[0] : 0.0;
    a1 = (k < terms && i + 1 < rows) ? p[1] : 0.0;
  }
  __device__ double b(int64_t b, int k, int j) const { return j < cols ? X[(int64_t)j * ldx + b * rows + k] : 0.0; }
  __device__ void load_b(int64_t bt, int k, int j, double (&y)[4]) const {
#pragma unroll
    for (int q = 0; q < 4; ++q) y[q] = (k + q < terms) ? b(bt, k + q, j) : 0.0;
  }
  __device__ void store(int64_t b, int i, int j, double v0, double v1) const {
    if (j >= cols) return;
    double* p = Y + (int64_t)j * ldy + b * rows + i;
    if (i < rows) p[0] = v0;
    if (i + 1 < rows) p[1] = v1;
  }
};

cudaError_t launch_leaf_matvec_split(const hodlr_desc& d, const double* D, const double* X, int64_t ldx, double* Y,
                                     int64_t ldy, int k, cudaStream_t s) {
  return gemm_split(LeafMatvecOp{d.m, k, d.m, D, X, ldx, Y, ldy}, (int64_t)1 << d.L, s);
}

// Out = K~^{-1} Rhs (or its transpose) of every parent of child level c, over
// the children's first chunk slots: the right-hand side's rows 0 .. r-1 are the
// sum of one child's chunk partials, rows r .. 2r-1 the other's; the result's
// rows go to the first child and the second. Rows of K~^{-1} whose diagonal entry is
// at least 1/2 are taken as the identity's row plus the rest, Rhs + (K~^{-1} - I) Rhs: with
// weak coupling the rest is much smaller, and its digits reach as far down as the result
// needs. The other rows are multiplied as they are: with strong coupling K~^{-1} is small,
// and the two terms would cancel.
struct CouplingOp {
  int rows, cols, terms;  // 2r, right-hand sides, 2r
  int r, trans;
  const double* K;
  double* P;
  size_t slot;
  int64_t cpn, cpn_read;
  int64_t first, second;  // chunk offsets of the right-hand side's halves within the parent
  __device__ void load_a(int64_t b, int i, int k, double& a0, double& a1) const {
    const double* p = K + (size_t)b * rows * rows + (trans ? (size_t)i * rows + k : (size_t)k * rows + i);
    a0 = (k < terms && i < rows) ? p[0] : 0.0;
    a1 = (k < terms && i + 1 < rows) ? p[trans ? rows : 1] : 0.0;
    if (i == k && a0 >= 0.5) a0 -= 1.0;
    if (i + 1 == k && a1 >= 0.5) a1 -= 1.0;
  }
  __device__ double init(int64_t bt, int i, int j) const {
    return i < rows && K[(size_t)bt * rows * rows + (size_t)i * (rows + 1)] >= 0.5 ? b(bt, i, j) : 0.0;
  }
  __device__ double b(int64_t bt, int k, int j) const {
    if (j >= cols) return 0.0;
    const double* p = P + (2 * bt * cpn + (k < r ? first : second)) * slot + (size_t)j * r + (k < r ? k : k - r);
    double v = 0.0;
    for (int64_t q = 0; q < cpn_read; ++q) v += p[q * slot];
    return v;
  }
  __device__ void load_b(int64_t bt, int k, int j, double (&y)[4]) const {
    if (cpn_read == 1) {  // four loads in flight
      const double* p = P + 2 * bt * cpn * slot + (size_t)(j < cols ? j : 0) * r;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const bool low = k + q < r;
        y[q] = (j < cols && k + q < terms) ? p[(low ? first : second) * slot + (low ? k + q : k + q - r)] : 0.0;
      }
      return;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) y[q] = (k + q < terms) ? b(bt, k + q, j) : 0.0;
  }
  __device__ void put(int64_t b, int i, int j, double v) const {
    if (i < rows) P[(2 * b * cpn + (i < r ? 0 : cpn)) * slot + (size_t)j * r + (i < r ? i : i - r)] = v;
  }
  __device__ void store(int64_t b, int i, int j, double v0, double v1) const {
    if (j >= cols) return;
    put(b, i, j, v0);
    put(b, i + 1, j, v1);
  }
};

cudaError_t launch_coupling_apply_split(int64_t cpn, int r, int c, double* P, int64_t sw, int nrhs, const double* Kinv,
                                        int first_is_beta, int trans, int64_t cpn_read, cudaStream_t s) {
  const CouplingOp op{2 * r, nrhs, 2 * r, r, trans, Kinv, P, (size_t)r * sw, cpn, cpn_read,
                      first_is_beta ? cpn : 0, first_is_beta ? 0 : cpn};
  if (r <= 32) return gemm_split<CouplingOp, 4>(op, (int64_t)1 << (c - 1), s);
  return gemm_split<CouplingOp, 8>(op, (int64_t)1 << (c - 1), s);
}

// out_b = beta out_b + alpha A_b B_b^T (+ Tadd_b^T) of every leaf b, A_b and B_b
// the leaf's rows of two tall matrices.
template <typename TB>
struct LeafOuterOp {
  int rows, cols, terms;  // m, m, columns of A and B
  int64_t N;
  const double* A;
  int64_t lda;
  const TB* B;
  int64_t ldb;
  double alpha, beta;
  const double* Tadd;
  double* out;
  __device__ double init(int64_t, int, int) const { return 0.0; }
  __device__ void load_a(int64_t b, int i, int k, double& a0, double& a1) const {
    const double* p = A + (int64_t)k * lda + b * rows + i;
    a0 = (k < terms && i < rows) ? p[0] : 0.0;
    a1 = (k < terms && i + 1 < rows) ? p[1] : 0.0;
  }
  __device__ double b(int64_t b, int k, int j) const { return j < cols ? to_d(B[(int64_t)k * ldb + b * cols + j]) : 0.0; }
  __device__ void load_b(int64_t bt, int k, int j, double (&y)[4]) const {
#pragma unroll
    for (int q = 0; q < 4; ++q) y[q] = (k + q < terms) ? b(bt, k + q, j) : 0.0;
  }
  __device__ void put(int64_t b, int i, int j, double acc) const {
    if (i >= rows) return;
    double* p = out + ((size_t)b * cols + j) * rows + i;
    double v = alpha * acc;
    if (beta != 0.0) v += beta * *p;
    if (Tadd) v += Tadd[(int64_t)i * N + b * rows + j];
    *p = v;
  }
  __device__ void store(int64_t b, int i, int j, double v0, double v1) const {
    if (j >= cols) return;
    put(b, i, j, v0);
    put(b, i + 1, j, v1);
  }
};

template <typename TB>
cudaError_t launch_leaf_outer_split(int64_t N, int m, int K, const double* A, int64_t lda, const TB* B, int64_t ldb,
                                    double alpha, double beta, const double* Tadd, double* out, cudaStream_t s) {
  return gemm_split(LeafOuterOp<TB>{m, m, K, N, A, lda, B, ldb, alpha, beta, Tadd, out}, N / m, s);
}
template cudaError_t launch_leaf_outer_split<double>(int64_t, int, int, const double*, int64_t, const double*,
                                                     int64_t, double, double, const double*, double*, cudaStream_t);
template cudaError_t launch_leaf_outer_split<float>(int64_t, int, int, const double*, int64_t, const float*, int64_t,
                                                    double, double, const double*, double*, cudaStream_t);

}  // namespace hodlr
