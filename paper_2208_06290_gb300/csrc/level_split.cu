// FP64 projections and rank-r updates of the level stage on the FP16 tensor
// cores (fp64_split.cuh): projections from two columns on, updates from three (from two on
// small trees of high rank).
#include "fp64_split.cuh"

namespace hodlr {
using namespace split;

// ---------------------------------------------------------------------------
// Projection partials P[q] = Bas(rows_q, block)^T R(rows_q, 0:ncols), q a row
// chunk. CTA = (chunk, 8 WN columns of R, 32 basis columns); warp (wn, wk)
// takes eight columns and every WK-th block of 16 NK rows. Per block: the CTA
// splits the basis rows into shared memory in fragment order (A operand, shared
// by the WN warps); every warp splits its own R entries in registers (B
// operand) straight from their loads, so R passes once through the SM; 36
// digit products per k16 step; the exact sums are added to FP64 accumulators.
template <typename TB, int MT, int WN, int WK, int NK>
__global__ void __launch_bounds__(256, 2) project_split_kernel(int64_t N, int r, int c, const TB* __restrict__ Bas,
                                                               int64_t ldb, int bas_block, bool vecb,
                                                               const double* __restrict__ R, int64_t ldr, bool vecr,
                                                               int ncols, double* __restrict__ P) {
  constexpr int BK = 16 * NK;            // rows of one warp's block
  constexpr int kFrag = MT * NK * kPlanes * 512;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* sA = smem_raw;                                       // [WK][MT][NK][plane][lane] 16 B
  int* sE = reinterpret_cast<int*>(smem_raw + WK * kFrag);            // [WK][32] exponents of the basis columns
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int wn = warp % WN, wk = warp / WN;
  const int64_t ch = chunk_rows(N, c);
  const int64_t q = blockIdx.x, row0 = q * ch;
  const int b0 = blockIdx.z * 32;                 // first basis column
  const int j0 = (blockIdx.y * WN + wn) * 8;      // first column of R of this warp
  const int rb = min(r - b0, MT * 16);
  const TB* B0 = Bas + ((int64_t)bas_block * r + b0) * ldb + row0;
  const bool mine = j0 + g < ncols;
  const double* R0 = R + (int64_t)(mine ? j0 + g : 0) * ldr + row0;
  const bool active = j0 < ncols;
  double acc[MT][4];
#pragma unroll
  for (int a = 0; a < MT; ++a)
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[a][u] = 0.0;

  for (int64_t k0 = 0; k0 < ch; k0 += BK * WK) {
    const int64_t kw = k0 + (int64_t)wk * BK;
    // this warp's R entries: lane (g, t) holds rows 16 s + 4 t .. + 3 of column g
    double x[NK][4];
#pragma unroll
    for (int s = 0; s < NK; ++s) {
      const int64_t k = kw + 16 * s + 4 * t;
      load_run4(R0 + k, mine ? ch - k : 0, vecr, x[s]);
    }
    // basis rows to shared memory: thread (column j, t, kh) splits rows
    // 16 (kh NK/2 + s) + 4 t .. + 3
    __syncthreads();
#pragma unroll
    for (int w = 0; w < WK; ++w) {
      const int j = tid >> 3;
      if (MT == 2 || j < 16) {
        const int tt = tid & 3, kh = (tid >> 2) & 1;
        double y[NK / 2][4];
#pragma unroll
        for (int s = 0; s < NK / 2; ++s) {
          const int64_t k = k0 + (int64_t)w * BK + 16 * (kh * (NK / 2) + s) + 4 * tt;
          load_run4(B0 + (int64_t)(j < rb ? j : 0) * ldb + k, j < rb ? ch - k : 0, vecb, y[s]);
        }
        const int e = shared_exp<NK / 2, 7>(y);
        if ((tid & 7) == 0) sE[w * 32 + j] = e;
        unsigned char* dst = sA + w * kFrag + (j >> 4) * NK * kPlanes * 512 + ((j & 7) * 4 + tt) * 16 +
                             ((j >> 3) & 1) * 8;
#pragma unroll
        for (int s = 0; s < NK / 2; ++s) {
          uint2 d[kDigits];
          split4(y[s], e, d);
          store_planes(dst + (kh * (NK / 2) + s) * kPlanes * 512, d);
        }
      }
    }
    const int er = shared_exp<NK, 3>(x);
    __syncthreads();
    if (active) {
      uint2 bf[NK][kDigits];
#pragma unroll
      for (int s = 0; s < NK; ++s) split4(x[s], er, bf[s]);
      const int eb0 = __shfl_sync(0xffffffffu, er, 8 * t), eb1 = __shfl_sync(0xffffffffu, er, 8 * t + 4);
#pragma unroll
      for (int a = 0; a < MT; ++a) {
        const uint4* fa = reinterpret_cast<const uint4*>(sA + wk * kFrag + a * NK * kPlanes * 512) + lane;
        const int ea0 = sE[wk * 32 + a * 16 + g], ea1 = sE[wk * 32 + a * 16 + g + 8];
        double v[4];
        tile<NK == 2>(StagedA<NK>{fa, bf}, ea0, ea1, eb0, eb1, v, [&](int u) {
          const int j = a * 16 + g + (u >> 1) * 8, col = j0 + 2 * t + (u & 1);
          double d = 0.0;
          if (j < rb && col < ncols)
#pragma unroll 8
            for (int64_t k = kw; k < ch && k < kw + BK; ++k)
              d = fma(to_d(B0[(int64_t)j * ldb + k]), R[(int64_t)col * ldr + row0 + k], d);
          return d;
        });
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[a][u] += v[u];
      }
    }
  }
  if (WK > 1) {  // sum the row groups in order through shared memory
    __syncthreads();
    double* sP = reinterpret_cast<double*>(smem_raw);
    if (wk > 0) {
#pragma unroll
      for (int a = 0; a < MT; ++a)
#pragma unroll
        for (int u = 0; u < 4; ++u) sP[(((wk - 1) * WN + wn) * MT * 4 + a * 4 + u) * 32 + lane] = acc[a][u];
    }
    __syncthreads();
    if (wk > 0) return;
#pragma unroll
    for (int w = 0; w < WK - 1; ++w)
#pragma unroll
      for (int a = 0; a < MT; ++a)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[a][u] += sP[((w * WN + wn) * MT * 4 + a * 4 + u) * 32 + lane];
  }
  double* Pq = P + (size_t)q * r * ncols;
#pragma unroll
  for (int a = 0; a < MT; ++a)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = a * 16 + g + (u >> 1) * 8, col = j0 + 2 * t + (u & 1);
      if (j < rb && col < ncols) Pq[(size_t)col * r + b0 + j] = acc[a][u];
    }
}

// At most eight columns: the basis is the large operand, so every warp takes
// its own rows (32 at a time, the CTA's eight warps every 256) and splits the
// basis entries in registers as well; no shared memory until the warps' sums
// are added in order at the end.
template <typename TB, int MT>
__global__ void __launch_bounds__(256, 2) project_split_skinny_kernel(int64_t N, int r, int c,
                                                                      const TB* __restrict__ Bas, int64_t ldb,
                                                                      int bas_block, bool vecb,
                                                                      const double* __restrict__ R, int64_t ldr,
                                                                      bool vecr, int ncols, double* __restrict__ P) {
  __shared__ double sP[8][MT * 4][32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int64_t ch = chunk_rows(N, c);
  const int64_t q = blockIdx.x, row0 = q * ch;
  const int b0 = blockIdx.z * 32;
  const int rb = min(r - b0, MT * 16);
  const TB* B0 = Bas + ((int64_t)bas_block * r + b0) * ldb + row0;
  const bool mine = g < ncols;
  const double* R0 = R + (int64_t)(mine ? g : 0) * ldr + row0;
  double acc[MT][4];
#pragma unroll
  for (int a = 0; a < MT; ++a)
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[a][u] = 0.0;
  for (int64_t kw = warp * 32; kw < ch; kw += 256) {
    double x[2][4];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int64_t k = kw + 16 * s + 4 * t;
      load_run4(R0 + k, mine ? ch - k : 0, vecr, x[s]);
    }
    const int er = shared_exp<2, 3>(x);
    uint2 bf[2][kDigits];
#pragma unroll
    for (int s = 0; s < 2; ++s) split4(x[s], er, bf[s]);
    const int eb0 = __shfl_sync(0xffffffffu, er, 8 * t), eb1 = __shfl_sync(0xffffffffu, er, 8 * t + 4);
#pragma unroll
    for (int a = 0; a < MT; ++a) {
      double y0[2][4], y1[2][4];  // basis columns a * 16 + g and + 8
      const int ja = a * 16 + g, jb = ja + 8;
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const int64_t k = kw + 16 * s + 4 * t;
        load_run4(B0 + (int64_t)(ja < rb ? ja : 0) * ldb + k, ja < rb ? ch - k : 0, vecb, y0[s]);
        load_run4(B0 + (int64_t)(jb < rb ? jb : 0) * ldb + k, jb < rb ? ch - k : 0, vecb, y1[s]);
      }
      const int ea0 = shared_exp<2, 3>(y0), ea1 = shared_exp<2, 3>(y1);
      float cd[kDigits][4];
      uint4 am[2];  // magnitudes
      clear_sums<true>(cd);
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        uint2 f0[kDigits], f1[kDigits];
        split4(y0[s], ea0, f0);
        split4(y1[s], ea1, f1);
#pragma unroll
        for (int i = 0; i < kDigits; ++i)
#pragma unroll
          for (int jd = 0; jd + i < kDigits; ++jd)
            mma_f16(cd[i + jd], f0[i].x, f1[i].x, f0[i].y, f1[i].y, bf[s][jd].x, bf[s][jd].y);
        am[s] = make_uint4(magnitude(f0[0].x, f0[1].x), magnitude(f1[0].x, f1[1].x), magnitude(f0[0].y, f0[1].y),
                           magnitude(f1[0].y, f1[1].y));
      }
      double v[4];
      finish_tile<true>(cd, ea0, ea1, eb0, eb1, v, [&](float (&mg)[4]) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const uint2 mb = magnitudes(bf[s]);
          mma_f16(mg, am[s].x, am[s].y, am[s].z, am[s].w, mb.x, mb.y);
        }
      }, [&](float (&c)[4]) {
        const TB* Br = again(B0);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const int64_t k = kw + 16 * s + 4 * t;
          double z[4];
          uint2 f0[kDigits], f1[kDigits];
          load_run4(Br + (int64_t)(ja < rb ? ja : 0) * ldb + k, ja < rb ? ch - k : 0, vecb, z);
          split4(z, ea0, f0);
          load_run4(Br + (int64_t)(jb < rb ? jb : 0) * ldb + k, jb < rb ? ch - k : 0, vecb, z);
          split4(z, ea1, f1);
#pragma unroll
          for (int i = 1; i < kDigits; ++i)
            mma_f16(c, f0[i].x, f1[i].x, f0[i].y, f1[i].y, bf[s][kDigits - i].x, bf[s][kDigits - i].y);
        }
      }, [&](int u) {
        const int j = a * 16 + g + (u >> 1) * 8, col = 2 * t + (u & 1);
        double d = 0.0;
        if (j < rb && col < ncols)
#pragma unroll 8
          for (int64_t k = kw; k < ch && k < kw + 32; ++k)
            d = fma(to_d(B0[(int64_t)j * ldb + k]), R[(int64_t)col * ldr + row0 + k], d);
        return d;
      });
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[a][u] += v[u];
    }
  }
#pragma unroll
  for (int a = 0; a < MT; ++a)
#pragma unroll
    for (int u = 0; u < 4; ++u) sP[warp][a * 4 + u][lane] = acc[a][u];
  __syncthreads();
  double* Pq = P + (size_t)q * r * ncols;
  for (int e = tid; e < MT * 4 * 32; e += 256) {
    const int au = e >> 5, ln = e & 31;
    const int j = (au >> 2) * 16 + (ln >> 2) + ((au >> 1) & 1) * 8, col = 2 * (ln & 3) + (au & 1);
    if (j < rb && col < ncols) {
      double v = sP[0][au][ln];
#pragma unroll
      for (int w = 1; w < 8; ++w) v += sP[w][au][ln];
      Pq[(size_t)col * r + b0 + j] = v;
    }
  }
}

// ---------------------------------------------------------------------------
// Rank-r update R(rows, 0:ncols) += alpha Bas(rows, block) W(node'). CTA = 128
// rows of one node; warp = 16 rows, whose basis entries are split once into
// registers (A operand) and used for every column; 64 columns of W at a time
// are split by the CTA into shared memory (B operand). KB = 32-term blocks
// (r <= 32 KB); grid.y shares the column tiles when there are few row tiles.
template <typename TB, int KB>
__global__ void __launch_bounds__(256, KB == 1 ? 2 : 1) update_split_kernel(
    int64_t N, int r, int c, const TB* __restrict__ Bas, int64_t ldb, int bas_block, double* __restrict__ R,
    int64_t ldr, int ncols, const double* __restrict__ Wbase, int64_t wstride, int swap_sibling, double alpha,
    bool vecr) {
  constexpr int NK = 2 * KB;  // k16 steps
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* sB = smem_raw;  // [col tile of 8][KB][plane][lane] 16 B
  int* sE = reinterpret_cast<int*>(smem_raw + 8 * KB * kPlanes * 512);
  const int64_t n = N >> c;
  const int64_t tpn = (n + 127) / 128;
  const int64_t node = blockIdx.x / tpn;
  const int64_t t0 = (blockIdx.x % tpn) * 128;
  const int64_t row0 = node * n + t0;
  const double* W = Wbase + (node ^ swap_sibling) * wstride;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int rt = (int)(n - t0 < 128 ? n - t0 : 128);
  const int i0 = warp * 16 + 2 * g;  // this lane's rows i0, i0 + 1 (fragment rows g, g + 8)
  const TB* B0 = Bas + (int64_t)bas_block * r * ldb + row0;
  uint2 af[NK][2][kDigits];  // [k16][row][digit]: (a0, a2) of row g, (a1, a3) of row g + 8
  int ea[2];
  {
    double x[2][NK][4];
#pragma unroll
    for (int s = 0; s < NK; ++s)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int k = 16 * s + 4 * t + q;
        const TB* p = B0 + (int64_t)(k < r ? k : 0) * ldb + i0;
        x[0][s][q] = (k < r && i0 < rt) ? to_d(p[0]) : 0.0;
        x[1][s][q] = (k < r && i0 + 1 < rt) ? to_d(p[1]) : 0.0;
      }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      ea[h] = shared_exp<NK, 3>(x[h]);
#pragma unroll
      for (int s = 0; s < NK; ++s) split4(x[h][s], ea[h], af[s][h]);
    }
  }
  for (int ct = blockIdx.y; ct * 64 < ncols; ct += gridDim.y) {
    const int j0 = ct * 64;
    __syncthreads();
    // W columns to shared memory: thread (column, 4 terms)
#pragma unroll
    for (int v = 0; v < 2 * KB; ++v) {
      const int task = v * 256 + tid;
      const int j = task / (8 * KB), grp = task % (8 * KB);
      double y[1][4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int k = 4 * grp + q;
        y[0][q] = (k < r && j0 + j < ncols) ? W[(size_t)(j0 + j) * r + k] : 0.0;
      }
      const int e = shared_exp<1, 8 * KB - 1>(y);
      if (grp == 0) sE[j] = e;
      uint2 d[kDigits];
      split4(y[0], e, d);
      unsigned char* dst = sB + ((j >> 3) * KB + (grp >> 3)) * kPlanes * 512 + ((j & 7) * 4 + (grp & 3)) * 16 +
                           ((grp >> 2) & 1) * 8;
      store_planes(dst, d);
    }
    __syncthreads();
    for (int nt = 0; nt < 8 && j0 + nt * 8 < ncols; ++nt) {
      const int col = j0 + nt * 8 + 2 * t;
      double* p0 = R + (int64_t)col * ldr + row0 + i0;
      double* p1 = p0 + ldr;
      const bool c0ok = col < ncols, c1ok = col + 1 < ncols;
      double o[4] = {0.0, 0.0, 0.0, 0.0};  // (row, col): (0,0) (1,0) (0,1) (1,1)
      if (vecr && i0 + 1 < rt) {
        if (c0ok) {
          const double2 u = *reinterpret_cast<const double2*>(p0);
          o[0] = u.x;
          o[1] = u.y;
        }
        if (c1ok) {
          const double2 u = *reinterpret_cast<const double2*>(p1);
          o[2] = u.x;
          o[3] = u.y;
        }
      } else {
        if (c0ok && i0 < rt) o[0] = p0[0];
        if (c0ok && i0 + 1 < rt) o[1] = p0[1];
        if (c1ok && i0 < rt) o[2] = p1[0];
        if (c1ok && i0 + 1 < rt) o[3] = p1[1];
      }
      const int eb0 = sE[nt * 8 + 2 * t], eb1 = sE[nt * 8 + 2 * t + 1];
      const uint4* fb = reinterpret_cast<const uint4*>(sB + nt * KB * kPlanes * 512) + lane;
      double v[4];
      tile<KB == 1>(StagedB<KB>{af, fb}, ea[0], ea[1], eb0, eb1, v, [&](int u) {
        const int i = i0 + (u >> 1), cc = col + (u & 1);
        double d = 0.0;
        if (i < rt && cc < ncols)
#pragma unroll 8
          for (int k = 0; k < r; ++k) d = fma(to_d(B0[(int64_t)k * ldb + i]), W[(size_t)cc * r + k], d);
        return d;
      });
      o[0] = fma(alpha, v[0], o[0]);
      o[1] = fma(alpha, v[2], o[1]);
      o[2] = fma(alpha, v[1], o[2]);
      o[3] = fma(alpha, v[3], o[3]);
      if (vecr && i0 + 1 < rt) {
        if (c0ok) *reinterpret_cast<double2*>(p0) = make_double2(o[0], o[1]);
        if (c1ok) *reinterpret_cast<double2*>(p1) = make_double2(o[2], o[3]);
      } else {
        if (c0ok && i0 < rt) p0[0] = o[0];
        if (c0ok && i0 + 1 < rt) p0[1] = o[1];
        if (c1ok && i0 < rt) p1[0] = o[2];
        if (c1ok && i0 + 1 < rt) p1[1] = o[3];
      }
    }
  }
}

// ---------------------------------------------------------------------------
template <typename TB, int MT, int WN, int WK, int NK>
static cudaError_t project_split_go(int64_t N, int r, int c, const TB* Bas, int64_t ldb, int bas_block, bool vecb,
                                    const double* R, int64_t ldr, bool vecr, int ncols, double* P, cudaStream_t s) {
  const size_t frag = (size_t)WK * MT * NK * kPlanes * 512;
  const size_t sums = (size_t)(WK - 1) * WN * MT * 4 * 32 * sizeof(double);
  const size_t sm = (frag > sums ? frag : sums) + WK * 32 * sizeof(int);
  cudaError_t e = cudaFuncSetAttribute(project_split_kernel<TB, MT, WN, WK, NK>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  dim3 grid((unsigned)num_chunks(N, c), (unsigned)((ncols + 8 * WN - 1) / (8 * WN)), (unsigned)((r + 31) / 32));
  project_split_kernel<TB, MT, WN, WK, NK><<<grid, 256, sm, s>>>(N, r, c, Bas, ldb, bas_block, vecb, R, ldr, vecr,
                                                                 ncols, P);
  note_launches(1);
  return cudaGetLastError();
}

template <typename TB, int MT>
static cudaError_t project_split_mt(int64_t N, int r, int c, const TB* Bas, int64_t ldb, int bas_block, bool vecb,
                                    const double* R, int64_t ldr, bool vecr, int ncols, double* P, cudaStream_t s) {
  if (ncols <= 8) {
    dim3 grid((unsigned)num_chunks(N, c), 1, (unsigned)((r + 31) / 32));
    project_split_skinny_kernel<TB, MT><<<grid, 256, 0, s>>>(N, r, c, Bas, ldb, bas_block, vecb, R, ldr, vecr, ncols,
                                                             P);
    note_launches(1);
    return cudaGetLastError();
  }
  if (ncols <= 16)
    return project_split_go<TB, MT, 2, 4, 2>(N, r, c, Bas, ldb, bas_block, vecb, R, ldr, vecr, ncols, P, s);
  if (ncols <= 32)
    return project_split_go<TB, MT, 4, 2, 4>(N, r, c, Bas, ldb, bas_block, vecb, R, ldr, vecr, ncols, P, s);
  return project_split_go<TB, MT, 8, 1, 4>(N, r, c, Bas, ldb, bas_block, vecb, R, ldr, vecr, ncols, P, s);
}

// Vector loads of four rows: every run starts at a multiple of four rows of a
// chunk, so the chunk starts, the leading dimension and the base decide.
template <typename T>
static bool vec4_ok(const T* p, int64_t ld, int64_t first, int64_t step) {
  return reinterpret_cast<uintptr_t>(p) % 16 == 0 && ld % 4 == 0 && first % 4 == 0 && step % 4 == 0;
}

template <typename TB>
cudaError_t launch_project_split(int64_t N, int r, int c, const TB* Bas, int64_t ldb, int bas_block, const double* R,
                                 int64_t ldr, int ncols, double* P, cudaStream_t s) {
  const int64_t ch = chunk_rows(N, c);
  const bool vecb = vec4_ok(Bas, ldb, 0, ch), vecr = vec4_ok(R, ldr, 0, ch);
  if (r <= 16) return project_split_mt<TB, 1>(N, r, c, Bas, ldb, bas_block, vecb, R, ldr, vecr, ncols, P, s);
  return project_split_mt<TB, 2>(N, r, c, Bas, ldb, bas_block, vecb, R, ldr, vecr, ncols, P, s);
}

template <typename TB, int KB>
static cudaError_t update_split_go(int64_t N, int r, int c, const TB* Bas, int64_t ldb, int bas_block, double* R,
                                   int64_t ldr, int ncols, const double* Wbase, int64_t wstride, int swap_sibling,
                                   double alpha, cudaStream_t s) {
  const size_t sm = (size_t)8 * KB * kPlanes * 512 + 64 * sizeof(int);
  cudaError_t e = cudaFuncSetAttribute(update_split_kernel<TB, KB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sm);
  if (e != cudaSuccess) return e;
  const int64_t n = N >> c;
  const int64_t tiles = ((int64_t)1 << c) * ((n + 127) / 128);
  const int ct = (ncols + 63) / 64;
  // few row tiles: split the column tiles over CTAs until every SM has two
  int gy = 1;
  while (gy < ct && tiles * gy < 2 * 152) ++gy;
  const bool vecr = reinterpret_cast<uintptr_t>(R) % 16 == 0 && ldr % 2 == 0 && n % 2 == 0;
  update_split_kernel<TB, KB><<<dim3((unsigned)tiles, gy), 256, sm, s>>>(N, r, c, Bas, ldb, bas_block, R, ldr, ncols,
                                                                        Wbase, wstride, swap_sibling, alpha, vecr);
  note_launches(1);
  return cudaGetLastError();
}

template <typename TB>
cudaError_t launch_update_split(int64_t N, int r, int c, const TB* Bas, int64_t ldb, int bas_block, double* R,
                                int64_t ldr, int ncols, const double* Wbase, int64_t wstride, int swap_sibling,
                                double alpha, cudaStream_t s) {
  if (r <= 32)
    return update_split_go<TB, 1>(N, r, c, Bas, ldb, bas_block, R, ldr, ncols, Wbase, wstride, swap_sibling, alpha,
                                  s);
  return update_split_go<TB, 2>(N, r, c, Bas, ldb, bas_block, R, ldr, ncols, Wbase, wstride, swap_sibling, alpha, s);
}

#define HODLR_INST(TB)                                                                                         \
  template cudaError_t launch_project_split<TB>(int64_t, int, int, const TB*, int64_t, int, const double*,     \
                                                int64_t, int, double*, cudaStream_t);                          \
  template cudaError_t launch_update_split<TB>(int64_t, int, int, const TB*, int64_t, int, double*, int64_t,   \
                                               int, const double*, int64_t, int, double, cudaStream_t);
HODLR_INST(double)
HODLR_INST(float)
#undef HODLR_INST

}  // namespace hodlr
