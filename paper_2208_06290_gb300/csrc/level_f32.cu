// FP32 projections and rank-r updates of the level stage for more than eight
// columns (low-precision factors, their solves of several right-hand sides).
#include "hodlr_internal.cuh"

namespace hodlr {

namespace {

// Entries p[0 .. 3] as FP32, those at or beyond `left` zero.
template <typename T>
__device__ __forceinline__ void load_run(const T* p, int64_t left, bool vec, float (&x)[4]) {
  if (vec && left >= 4) {
    load4(p, x);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) x[q] = q < left ? conv<float>(p[q]) : 0.f;
  }
}

template <typename T>
bool vec4_ok(const T* p, int64_t ld, int64_t step) {  // four rows at a multiple of four rows
  return reinterpret_cast<uintptr_t>(p) % (4 * sizeof(T)) == 0 && ld % 4 == 0 && step % 4 == 0;
}

}  // namespace

// ---------------------------------------------------------------------------
// Projection partials P[q] = Bas(rows_q, block)^T R(rows_q, 0:ncols), q a row
// chunk, FP32 sums in row order, stored in FP64. CTA = (chunk, 64 WC columns of R,
// 32 WR basis columns); a warp takes a 32 x 64 tile, a lane 8 x 8 of it (16 loads
// of four words from shared memory per 64 FMAs: the FP32 pipe is the bound, not
// shared memory as with the 4 x 4 tiles before). Narrow right-hand sides leave
// warps over: WK groups of them take every WK-th block of 8 or 16 rows, and their sums
// are added in order at the end. Blocks are transposed into a double buffer from
// registers loaded one block ahead. FP32 factor and refinement, N = 2^18, r = 64:
// 11.0 -> 5.6 ms in 30 launches; a third of the FP32 pipe's rate, the rest is the
// latency of a few blocks per SM.
template <typename TB, typename TR, int WR, int WC, int WK>
__global__ void __launch_bounds__(256, 2) project_f32_kernel(int64_t N, int r, int c, const TB* __restrict__ Bas,
                                                             int64_t ldb, int bas_block, bool vecb,
                                                             const TR* __restrict__ R, int64_t ldr, bool vecr,
                                                             int ncols, double* __restrict__ P) {
  static_assert(WR * WC * WK == 8, "eight warps");
  constexpr int RT = 32 * WR, TN = 64 * WC;
  constexpr int KB = WK > 2 ? 8 : 16, KQ = KB / 4;  // rows of a block and their runs of four
  constexpr int PB = RT + 4, PR = TN + 4;           // pitches
  constexpr int LB = WK * KQ * RT / 256, LR = WK * KQ * TN / 256;  // runs of four rows per thread and block
  constexpr int kStage = WK * KB * (PB + PR);
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wr = warp % WR, wc = warp / WR % WC, wk = warp / (WR * WC);
  const int64_t ch = chunk_rows(N, c);
  const int64_t q = blockIdx.x, row0 = q * ch;
  const int j0 = blockIdx.y * TN;
  const TB* B0 = Bas + (int64_t)bas_block * r * ldb + row0;
  const TR* R0 = R + row0;
  const int tx = lane & 7, ty = lane >> 3;  // columns 4 tx (+ 32), basis columns 4 ty (+ 16)
  float acc[8][8];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 8; ++b) acc[a][b] = 0.f;
  float xb[LB][4], xr[LR][4];
  const int blocks = (int)((ch + KB * WK - 1) / (KB * WK));
  // run e of a block: row quad e % KQ, column e / KQ % width, row group e / (KQ width)
  auto fetch = [&](int it) {
#pragma unroll
    for (int u = 0; u < LB; ++u) {
      const int e = u * 256 + tid;
      const int col = e / KQ % RT;
      const int64_t k = (int64_t)(it * WK + e / (KQ * RT)) * KB + e % KQ * 4;
      load_run(B0 + (int64_t)(col < r ? col : 0) * ldb + k, col < r ? ch - k : 0, vecb, xb[u]);
    }
#pragma unroll
    for (int u = 0; u < LR; ++u) {
      const int e = u * 256 + tid;
      const int col = j0 + e / KQ % TN;
      const int64_t k = (int64_t)(it * WK + e / (KQ * TN)) * KB + e % KQ * 4;
      load_run(R0 + (int64_t)(col < ncols ? col : 0) * ldr + k, col < ncols ? ch - k : 0, vecr, xr[u]);
    }
  };
  fetch(0);
  for (int it = 0; it < blocks; ++it) {
    float* sB = sm + (it & 1) * kStage;
    float* sR = sB + WK * KB * PB;
#pragma unroll
    for (int u = 0; u < LB; ++u) {
      const int e = u * 256 + tid;
#pragma unroll
      for (int w = 0; w < 4; ++w) sB[(e / (KQ * RT) * KB + e % KQ * 4 + w) * PB + e / KQ % RT] = xb[u][w];
    }
#pragma unroll
    for (int u = 0; u < LR; ++u) {
      const int e = u * 256 + tid;
#pragma unroll
      for (int w = 0; w < 4; ++w) sR[(e / (KQ * TN) * KB + e % KQ * 4 + w) * PR + e / KQ % TN] = xr[u][w];
    }
    __syncthreads();  // one per block: the other buffer is written next
    if (it + 1 < blocks) fetch(it + 1);
    const float* pb = sB + wk * KB * PB + wr * 32 + 4 * ty;
    const float* pr = sR + wk * KB * PR + wc * 64 + 4 * tx;
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      float b[8], x[8];
      *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(pb + k * PB);
      *reinterpret_cast<float4*>(b + 4) = *reinterpret_cast<const float4*>(pb + k * PB + 16);
      *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(pr + k * PR);
      *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(pr + k * PR + 32);
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int w = 0; w < 8; ++w) acc[a][w] = fmaf(b[a], x[w], acc[a][w]);
    }
  }
  if (WK > 1) {
    // group by group through shared memory, in order
    __syncthreads();
    float* mine = sm + (warp % (WR * WC)) * 2048 + lane;
    for (int g = 1; g < WK; ++g) {
      if (wk == g) {
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int w = 0; w < 8; ++w) mine[(a * 8 + w) * 32] = acc[a][w];
      }
      __syncthreads();
      if (wk == 0) {
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int w = 0; w < 8; ++w) acc[a][w] += mine[(a * 8 + w) * 32];
      }
      __syncthreads();
    }
    if (wk > 0) return;
  }
  double* Pq = P + (size_t)q * r * ncols;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    const int col = j0 + wc * 64 + 4 * tx + (w & 3) + (w >> 2) * 32;
    if (col >= ncols) continue;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const int row = wr * 32 + 4 * ty + (a & 3) + (a >> 2) * 16;
      if (row < r) Pq[(size_t)col * r + row] = (double)acc[a][w];
    }
  }
}

// ---------------------------------------------------------------------------
// R(rows, 0:ncols) += alpha Bas(rows, block) W(node'). CTA = 16 MR rows of one node
// x 16 NR columns, thread = MR x NR (both in fours); the whole inner dimension r is
// staged once, so the FMAs run without a barrier. Rows run along the lanes, so the
// panel is read and written 16 bytes a lane, coalesced. The same case: 9.0 -> 6.7 ms.
template <typename TB, typename TR, int MR, int NR>
__global__ void __launch_bounds__(256, 2) update_f32_kernel(int64_t N, int r, int c, const TB* __restrict__ Bas,
                                                            int64_t ldb, int bas_block, bool vecb,
                                                            TR* __restrict__ R, int64_t ldr, bool vecr, int ncols,
                                                            const double* __restrict__ Wbase, int64_t wstride,
                                                            int swap_sibling, double alpha) {
  constexpr int TM = 16 * MR, TN = 16 * NR;
  constexpr int PW = TN + 4;
  extern __shared__ __align__(16) float sm[];
  float* sB = sm;           // [k][TM]
  float* sW = sm + r * TM;  // [k][PW]
  const int64_t n = N >> c;
  const int64_t tpn = (n + TM - 1) / TM;
  const int64_t node = blockIdx.x / tpn;
  const int64_t t0 = (blockIdx.x % tpn) * TM;
  const int rt = (int)(n - t0 < TM ? n - t0 : TM);
  const int64_t row0 = node * n + t0;
  const double* W = Wbase + (node ^ swap_sibling) * wstride;
  const int j0 = blockIdx.y * TN;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const TB* B0 = Bas + (int64_t)bas_block * r * ldb + row0;
  for (int e = tid; e < r * (TM / 4); e += 256) {
    const int i = e % (TM / 4) * 4, k = e / (TM / 4);
    float x[4];
    load_run(B0 + (int64_t)k * ldb + i, rt - i, vecb, x);
    *reinterpret_cast<float4*>(sB + k * TM + i) = make_float4(x[0], x[1], x[2], x[3]);
  }
  for (int e = tid; e < r * TN; e += 256) {
    const int k = e % r, col = e / r;
    sW[k * PW + col] = j0 + col < ncols ? (float)(alpha * W[(size_t)(j0 + col) * r + k]) : 0.f;
  }
  __syncthreads();
  float acc[MR][NR];
#pragma unroll
  for (int a = 0; a < MR; ++a)
#pragma unroll
    for (int b = 0; b < NR; ++b) acc[a][b] = 0.f;
#pragma unroll 4
  for (int k = 0; k < r; ++k) {
    float b[MR], w[NR];
#pragma unroll
    for (int h = 0; h < MR / 4; ++h)
      *reinterpret_cast<float4*>(b + 4 * h) = *reinterpret_cast<const float4*>(sB + k * TM + 64 * h + 4 * tx);
#pragma unroll
    for (int h = 0; h < NR / 4; ++h)
      *reinterpret_cast<float4*>(w + 4 * h) = *reinterpret_cast<const float4*>(sW + k * PW + 64 * h + 4 * ty);
#pragma unroll
    for (int a = 0; a < MR; ++a)
#pragma unroll
      for (int u = 0; u < NR; ++u) acc[a][u] = fmaf(b[a], w[u], acc[a][u]);
  }
#pragma unroll
  for (int u = 0; u < NR; ++u) {
    const int col = j0 + 64 * (u >> 2) + 4 * ty + (u & 3);
    if (col >= ncols) continue;
#pragma unroll
    for (int h = 0; h < MR / 4; ++h) {
      const int i = 64 * h + 4 * tx;
      TR* p = R + (int64_t)col * ldr + row0 + i;
      if (vecr && i + 4 <= rt) {
        float v[4];
        load4(p, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] += acc[4 * h + q][u];
        store4(p, v);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (i + q < rt) p[q] = conv<TR>(conv<float>(p[q]) + acc[4 * h + q][u]);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Coupling application of the low-precision factors, FP32 products:
// [W'_alpha; W'_beta] = K~^{-1} [W_beta; W_alpha] for the columns [0, nrhs) of every
// parent, over the children's first chunk slots (FP64, ld r). CTA = one parent x TN
// columns, thread = 8 rows x 4 columns; K~^{-1} and the right-hand side are rounded
// into shared memory once, so every read precedes the writes. (As a split-operand
// product, which keeps FP64, it took twice the time: 5.1 against 2.4 ms for the 4 x 4
// tiles before, N = 2^18, rank 64.)
template <int TN>
__global__ void __launch_bounds__(256) coupling_apply_f32_kernel(int64_t cpn, int r, double* P, size_t slot, int nrhs,
                                                                 const double* __restrict__ Kinv, int64_t cpn_read) {
  constexpr int PR = TN + 4;
  extern __shared__ __align__(16) float sm[];
  const int n = 2 * r;
  const int PK = (n + 7) / 8 * 8;
  float* sK = sm;            // [k][PK]: K~^{-1}(i, k)
  float* sR = sm + n * PK;   // [k][PR]
  const int tid = threadIdx.x;
  const int64_t j = blockIdx.x;
  const int j0 = blockIdx.y * TN;
  const double* Kj = Kinv + (size_t)j * n * n;
  double* Pa = P + (size_t)(2 * j) * cpn * slot;
  double* Pb = Pa + (size_t)cpn * slot;
#pragma unroll 8
  for (int e = tid; e < n * PK; e += 256) {
    const int i = e % PK, k = e / PK;
    sK[e] = i < n ? (float)Kj[(size_t)k * n + i] : 0.f;
  }
#pragma unroll 8
  for (int e = tid; e < n * TN; e += 256) {
    const int k = e % n, col = e / n;
    double v = 0.0;
    if (j0 + col < nrhs) {
      const double* p = (k < r ? Pb : Pa) + (size_t)(j0 + col) * r + (k < r ? k : k - r);
      for (int64_t q = 0; q < cpn_read; ++q) v += p[q * slot];
    }
    sR[k * PR + col] = (float)v;
  }
  __syncthreads();
  const int tx = tid & 15, ty = tid >> 4;
  const int i0 = (TN == 64 ? ty : ty & 7) * 8, c0 = 4 * tx + (TN == 64 ? 0 : (ty >> 3) * 64);
  if (i0 >= n) return;
  float acc[8][4];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[a][q] = 0.f;
#pragma unroll 4
  for (int k = 0; k < n; ++k) {
    float kv[8], xv[4];
    *reinterpret_cast<float4*>(kv) = *reinterpret_cast<const float4*>(sK + k * PK + i0);
    *reinterpret_cast<float4*>(kv + 4) = *reinterpret_cast<const float4*>(sK + k * PK + i0 + 4);
    *reinterpret_cast<float4*>(xv) = *reinterpret_cast<const float4*>(sR + k * PR + c0);
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[a][q] = fmaf(kv[a], xv[q], acc[a][q]);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (j0 + c0 + q >= nrhs) break;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const int i = i0 + a;
      if (i < n) (i < r ? Pa : Pb)[(size_t)(j0 + c0 + q) * r + (i < r ? i : i - r)] = (double)acc[a][q];
    }
  }
}

cudaError_t launch_coupling_apply_f32(int64_t cpn, int r, int c, double* P, int64_t sw, int nrhs, const double* Kinv,
                                      int64_t cpn_read, cudaStream_t s) {
  const int n = 2 * r, tn = r <= 32 ? 128 : 64;
  const size_t sm = (size_t)n * ((n + 7) / 8 * 8 + tn + 4) * sizeof(float);
  auto kern = r <= 32 ? coupling_apply_f32_kernel<128> : coupling_apply_f32_kernel<64>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  kern<<<dim3(1u << (c - 1), (unsigned)((nrhs + tn - 1) / tn)), 256, sm, s>>>(cpn, r, P, (size_t)r * sw, nrhs, Kinv, cpn_read);
  note_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
template <typename TB, typename TR, int WR, int WC, int WK>
static cudaError_t project_f32_go(int64_t N, int r, int c, const TB* Bas, int64_t ldb, int bas_block, const TR* R,
                                  int64_t ldr, int ncols, double* P, cudaStream_t s) {
  const int64_t ch = chunk_rows(N, c);
  const size_t stages = 2 * WK * (WK > 2 ? 8 : 16) * ((32 * WR + 4) + (64 * WC + 4)) * sizeof(float);
  const size_t sums = (size_t)WR * WC * 2048 * sizeof(float);
  const size_t sm = stages > sums ? stages : sums;
  cudaError_t e = cudaFuncSetAttribute(project_f32_kernel<TB, TR, WR, WC, WK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sm);
  if (e != cudaSuccess) return e;
  dim3 grid((unsigned)num_chunks(N, c), (unsigned)((ncols + 64 * WC - 1) / (64 * WC)));
  project_f32_kernel<TB, TR, WR, WC, WK><<<grid, 256, sm, s>>>(N, r, c, Bas, ldb, bas_block, vec4_ok(Bas, ldb, ch), R, ldr,
                                                           vec4_ok(R, ldr, ch), ncols, P);
  note_launches(1);
  return cudaGetLastError();
}

template <typename TB, typename TR>
cudaError_t launch_project_f32(int64_t N, int r, int c, const TB* Bas, int64_t ldb, int bas_block, const TR* R,
                               int64_t ldr, int ncols, double* P, cudaStream_t s) {
  if (r <= 32) {
    if (ncols <= 64) return project_f32_go<TB, TR, 1, 1, 8>(N, r, c, Bas, ldb, bas_block, R, ldr, ncols, P, s);
    if (ncols <= 128) return project_f32_go<TB, TR, 1, 2, 4>(N, r, c, Bas, ldb, bas_block, R, ldr, ncols, P, s);
    return project_f32_go<TB, TR, 1, 4, 2>(N, r, c, Bas, ldb, bas_block, R, ldr, ncols, P, s);
  }
  if (ncols <= 64) return project_f32_go<TB, TR, 2, 1, 4>(N, r, c, Bas, ldb, bas_block, R, ldr, ncols, P, s);
  if (ncols <= 128) return project_f32_go<TB, TR, 2, 2, 2>(N, r, c, Bas, ldb, bas_block, R, ldr, ncols, P, s);
  return project_f32_go<TB, TR, 2, 4, 1>(N, r, c, Bas, ldb, bas_block, R, ldr, ncols, P, s);
}

template <typename TB, typename TR, int MR, int NR>
static cudaError_t update_f32_go(int64_t N, int r, int c, const TB* Bas, int64_t ldb, int bas_block, TR* R,
                                 int64_t ldr, int ncols, const double* Wbase, int64_t wstride, int swap_sibling,
                                 double alpha, cudaStream_t s) {
  const int64_t n = N >> c;
  const size_t sm = (size_t)r * (16 * MR + 16 * NR + 4) * sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(update_f32_kernel<TB, TR, MR, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sm);
  if (e != cudaSuccess) return e;
  const int64_t tiles = ((int64_t)1 << c) * ((n + 16 * MR - 1) / (16 * MR));
  dim3 grid((unsigned)tiles, (unsigned)((ncols + 16 * NR - 1) / (16 * NR)));
  update_f32_kernel<TB, TR, MR, NR><<<grid, 256, sm, s>>>(N, r, c, Bas, ldb, bas_block, vec4_ok(Bas, ldb, n), R, ldr,
                                                      vec4_ok(R, ldr, n), ncols, Wbase, wstride, swap_sibling, alpha);
  note_launches(1);
  return cudaGetLastError();
}

// Rows: 128 at a time unless the nodes have at most 64. Columns: 64 at a time for
// up to 64 of them (and for 129 to 192, where a third tile of 128 would be half
// empty), else 128.
template <typename TB, typename TR>
cudaError_t launch_update_f32(int64_t N, int r, int c, const TB* Bas, int64_t ldb, int bas_block, TR* R,
                              int64_t ldr, int ncols, const double* Wbase, int64_t wstride, int swap_sibling,
                              double alpha, cudaStream_t s) {
  const bool narrow = ncols <= 64 || (ncols > 128 && ncols <= 192);
  if ((N >> c) <= 64) {
    if (narrow)
      return update_f32_go<TB, TR, 4, 4>(N, r, c, Bas, ldb, bas_block, R, ldr, ncols, Wbase, wstride, swap_sibling, alpha, s);
    return update_f32_go<TB, TR, 4, 8>(N, r, c, Bas, ldb, bas_block, R, ldr, ncols, Wbase, wstride, swap_sibling, alpha, s);
  }
  if (narrow)
    return update_f32_go<TB, TR, 8, 4>(N, r, c, Bas, ldb, bas_block, R, ldr, ncols, Wbase, wstride, swap_sibling, alpha, s);
  return update_f32_go<TB, TR, 8, 8>(N, r, c, Bas, ldb, bas_block, R, ldr, ncols, Wbase, wstride, swap_sibling, alpha, s);
}

#define HODLR_INST(TB, TR)                                                                                          \
  template cudaError_t launch_project_f32<TB, TR>(int64_t, int, int, const TB*, int64_t, int, const TR*, int64_t,  \
                                                  int, double*, cudaStream_t);                                     \
  template cudaError_t launch_update_f32<TB, TR>(int64_t, int, int, const TB*, int64_t, int, TR*, int64_t, int,    \
                                                 const double*, int64_t, int, double, cudaStream_t);
HODLR_INST(float, float)
HODLR_INST(__nv_bfloat16, float)
HODLR_INST(__nv_bfloat16, __nv_bfloat16)
#undef HODLR_INST

}  // namespace hodlr
