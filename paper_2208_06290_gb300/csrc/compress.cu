// GPU construction of the HODLR approximation of a kernel or boundary-integral
// matrix (Sec. 2.2): leaf blocks evaluated exactly (FP64), every off-diagonal
// sibling block A(I_alpha, I_beta) compressed to the fixed rank r by a
// partial-pivoted cross approximation (the approximate partial-pivoted LU the
// paper's kernel experiments used for this step on the CPU):
//
//   i_0 = first row of the block;  for k = 0 .. r-1:
//     rho(j)  = M(i_k, j) - sum_{l<k} u_l(i_k) v_l(j)          (residual row)
//     j_k     = argmax over unused j of |rho(j)|  (first maximum)
//     v_k     = rho / rho(j_k)
//     u_k(i)  = M(i, j_k) - sum_{l<k} u_l(i) v_l(j_k)         (residual column)
//     i_{k+1} = argmax over rows other than i_0 .. i_k of |u_k(i)|
//   A(I_alpha, I_beta) ~= sum_k u_k v_k^T = U_alpha V_beta^T.
//
// A residual that vanishes (rank exhausted) ends the block: its remaining u, v
// are zero. Kernel matrices are symmetric: one cross per sibling pair gives
// A(I_beta, I_alpha) = V_beta U_alpha^T, so U_big = V_big. The BIE matrix is
// not: both blocks of a pair are compressed.
//
// GPU form: blocks of up to 8192 rows take one cluster of CTAs each, one launch per
// level (aca_cluster_kernel). Above that all blocks of a level advance together, two
// launches per rank step: (1) one thread per column position forms the residual row of its
// block and the blocks' pivot columns are chosen by 64-bit atomic maxima of
// (|rho| bits, -j) keys (order-independent, so the choice is deterministic:
// largest |rho|, then the lowest column); (2) one thread per position forms
// v_k from the stored row and u_k of its block and chooses the next pivot
// rows the same way. Entries are rounded to FP32 (evaluated from FP64
// geometry), the residual updates are FP32 (from FP32 working copies of U and
// V); U and V are stored in FP64.
#include <cooperative_groups.h>

#include <cmath>
#include <vector>

#include "hodlr_internal.cuh"

namespace hodlr {
namespace {

struct Kern {
  int kind;        // hodlr_kernel
  int dim;
  const double* pts;  // N x dim, row-major
  double scale, nugget;
  int64_t N;
  float tol;       // stop a block once |pivot_k| <= tol |pivot_0| (0: fixed rank)
  double rate;     // Gaussian: 1 / (2 scale^2); Matern: sqrt(3) / scale
};

// A step is live when its residual row had a nonzero entry and (after the
// first step) its pivot is above the block's tolerance.
__device__ __forceinline__ bool step_live(unsigned long long ck, int k, float tol, const float* delta0,
                                          int64_t blk) {
  if ((ck >> 32) <= 1ull) return false;  // empty key or a vanishing residual
  if (k == 0 || tol <= 0.f) return true;
  const float piv = __uint_as_float((uint32_t)(ck >> 32) - 1u);
  return piv > tol * delta0[blk];
}

constexpr double kTwoPi = 6.283185307179586476925286766559;
constexpr int kGeo = 6;  // BIE geometry per point: x, y, normal (2), weight, curvature
constexpr size_t kWsAlign = 256;  // every workspace piece starts 256-byte aligned
inline size_t ws_align(size_t x) { return (x + kWsAlign - 1) / kWsAlign * kWsAlign; }

// Star curve rho(t) = 1 + 0.3 cos(5 t), t_i = 2 pi i / N (trapezoid rule):
// point, outward unit normal, weight w_i = |gamma'(t_i)| 2 pi / N and
// curvature, in FP64.
__device__ __forceinline__ void star_point(int64_t i, int64_t N, double& x, double& y, double& nx, double& ny,
                                           double& w, double& kappa) {
  const double t = (double)i * (kTwoPi / (double)N);
  const double rho = 1.0 + 0.3 * cos(5.0 * t), drho = -1.5 * sin(5.0 * t), ddrho = -7.5 * cos(5.0 * t);
  const double c = cos(t), s = sin(t);
  x = rho * c;
  y = rho * s;
  const double tx = drho * c - rho * s, ty = drho * s + rho * c;
  const double sp = sqrt(tx * tx + ty * ty);
  nx = ty / sp;
  ny = -tx / sp;
  w = sp * (kTwoPi / (double)N);
  kappa = (rho * rho + 2.0 * drho * drho - rho * ddrho) / pow(rho * rho + drho * drho, 1.5);
}

// Whether every FP64 value within `ulps` of q rounds to the same FP32 value as q:
// q is normal in FP32 and its low 29 bits are that far from the rounding boundary.
__device__ __forceinline__ bool rounds_alike(double q, int ulps) {
  const int e = (int)((uint32_t)__double2hiint(q) >> 20 & 0x7ffu);
  const int low = (int)((uint32_t)__double2loint(q) & 0x1fffffffu) - 0x10000000;
  return e > 1023 - 120 && e < 1023 + 120 && (low > ulps || low < -ulps);
}
__device__ __forceinline__ bool float_range(double q) {  // positive and well inside FP32's normal range
  const int hi = __double2hiint(q);
  return hi > (1023 - 120) << 20 && hi < (1023 + 120) << 20;
}

// Entry A(i, j), i != j (off-diagonal blocks), returned in FP32. The BIE
// entry is evaluated in FP64 from the FP64 geometry (x, y, normal, weight
// per point): for neighbouring points n(y).(x - y) is second order in the
// spacing while x - y is first order, so FP32 coordinates would lose most of
// its digits. The kernels take the squared distance in FP64 and the
// exponential in FP32.
// An FP64 division or square root is a sequence of 10 to 20 operations on a pipe
// that does two of them per clock and SM; with them these kernels were bound by
// that pipe. What is rounded to FP32 next needs fewer digits: one Newton step in
// FP64 from the FP32 reciprocal or reciprocal square root has a relative error
// below 2^-41, and unless the result lies that close to a rounding boundary (one
// entry in 10^4) it rounds to what the division or root would have given.
__device__ __forceinline__ float kernel_entry(const Kern& K, const double* __restrict__ g, int64_t i, int64_t j) {
  if (K.kind == HODLR_KERNEL_BIE_STAR) {
    // double layer: n(y).(x - y) / (2 pi |x - y|^2) w_y   (x = point i, y = point j)
    const double* gi = g + kGeo * i;
    const double* gj = g + kGeo * j;
    const double dx = gi[0] - gj[0], dy = gi[1] - gj[1];
    const double num = gj[2] * dx + gj[3] * dy, den = kTwoPi * (dx * dx + dy * dy), w = gj[4];
    if (float_range(den)) {
      double y = (double)__frcp_rn((float)den);
      y = fma(y, fma(-den, y, 1.0), y);
      const double q = num * y * w;
      if (rounds_alike(q, 8192)) return (float)q;
    }
    return (float)(num / den * w);
  }
  double pi[3], pj[3], d2 = 0.0;  // at most three coordinates, all loads in flight
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    pi[a] = a < K.dim ? g[(size_t)K.dim * i + a] : 0.0;
    pj[a] = a < K.dim ? g[(size_t)K.dim * j + a] : 0.0;
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double d = pi[a] - pj[a];
    if (a < K.dim) d2 = fma(d, d, d2);
  }
  if (K.kind == HODLR_KERNEL_GAUSSIAN) {
    double q = -d2 * K.rate;
    if (!rounds_alike(q, 16)) q = -d2 / (2.0 * K.scale * K.scale);
    return expf((float)q);
  }
  float a;  // Matern-3/2
  double q = 0.0;
  if (float_range(d2)) {
    const double y = (double)rsqrtf((float)d2);
    q = d2 * y;
    q = fma(fma(-q, q, d2), 0.5 * y, q) * K.rate;
  }
  if (rounds_alike(q, 8192)) a = (float)q;
  else a = (float)(1.7320508075688772 * sqrt(d2) / K.scale);
  return (1.f + a) * expf(-a);
}

// x - sum_{l < k} u[l step_u] v[l step_v], one rounding per term, in order; the
// loads of eight terms are in flight together.
__device__ __forceinline__ float residual(float x, const float* __restrict__ u, const float* __restrict__ v,
                                          int64_t step, int k) {
  int l = 0;
  for (; l + 8 <= k; l += 8) {
    float a[8], b[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      a[q] = u[(size_t)(l + q) * step];
      b[q] = v[(size_t)(l + q) * step];
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) x = fmaf(-a[q], b[q], x);
  }
  for (; l < k; ++l) x = fmaf(-u[(size_t)l * step], v[(size_t)l * step], x);
  return x;
}

__global__ void geometry_kernel(Kern K, double* __restrict__ g) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < K.N; i += (int64_t)gridDim.x * blockDim.x) {
    if (K.kind == HODLR_KERNEL_BIE_STAR) {
      double x, y, nx, ny, w, kap;
      star_point(i, K.N, x, y, nx, ny, w, kap);
      double* gi = g + kGeo * i;
      gi[0] = x;
      gi[1] = y;
      gi[2] = nx;
      gi[3] = ny;
      gi[4] = w;
      gi[5] = kap;
    } else {
      for (int a = 0; a < K.dim; ++a) g[(size_t)K.dim * i + a] = K.pts[(size_t)K.dim * i + a];
    }
  }
}

// Leaf blocks D_b (column-major m x m), FP64, from the FP64 geometry: BIE:
// the kernel off the diagonal and the smooth-quadrature diagonal
// -1/2 - w_i kappa_i / (4 pi); kernel matrices: k(|x_i - x_j|) + nugget on
// the diagonal.
// The blocks of symmetric kernels: one CTA per leaf and pair of 32 x 32 tiles on or
// above the diagonal; each entry is evaluated once (the FP64 pipe bounds this
// kernel) and its mirror image written through shared memory.
__global__ void __launch_bounds__(256) leaf_eval_sym_kernel(Kern K, const double* __restrict__ g, int m,
                                                            double* __restrict__ D) {
  __shared__ double sT[32][33];
  const int nt = (m + 31) / 32;
  int ti = blockIdx.y, tj = 0;  // pair number -> tiles ti <= tj
  while (ti >= nt - tj) ti -= nt - tj++;
  tj += ti;
  ti = tj - ti;
  const int64_t b = blockIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double* Db = D + (size_t)b * m * m;
  const int ii = ti * 32 + lane;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int jj = tj * 32 + w + 8 * q;
    if (ii < m && jj < m) {
      const int64_t i = b * m + ii, j = b * m + jj;
      double d2 = 0.0, v;
      for (int a = 0; a < K.dim; ++a) {
        const double d = g[(size_t)K.dim * i + a] - g[(size_t)K.dim * j + a];
        d2 += d * d;
      }
      if (K.kind == HODLR_KERNEL_GAUSSIAN) {
        v = exp(-d2 / (2.0 * K.scale * K.scale));
      } else {
        const double a = sqrt(3.0) * sqrt(d2) / K.scale;
        v = (1.0 + a) * exp(-a);
      }
      if (i == j) v += K.nugget;
      Db[(size_t)jj * m + ii] = v;
      sT[w + 8 * q][lane] = v;
    }
  }
  if (ti == tj) return;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int jj = ti * 32 + w + 8 * q, i2 = tj * 32 + lane;  // column jj of tile ti, row i2 of tile tj
    if (i2 < m && jj < m) Db[(size_t)jj * m + i2] = sT[lane][w + 8 * q];
  }
}

// The blocks of the BIE, which is not symmetric.
__global__ void leaf_eval_kernel(Kern K, const double* __restrict__ g, int m, double* __restrict__ D) {
  const int64_t total = K.N * (int64_t)m;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = e / ((int64_t)m * m);
    const int rem = (int)(e % ((int64_t)m * m));
    const int jj = rem / m, ii = rem % m;
    const int64_t i = b * m + ii, j = b * m + jj;
    double v;
    const double* gi = g + kGeo * i;
    const double* gj = g + kGeo * j;
    if (i == j) {
      v = -0.5 - gi[4] * gi[5] / (2.0 * kTwoPi);
    } else {
      const double dx = gi[0] - gj[0], dy = gi[1] - gj[1];
      v = (gj[2] * dx + gj[3] * dy) / (kTwoPi * (dx * dx + dy * dy)) * gj[4];
    }
    D[e] = v;
  }
}

// key = (|x| bits << 32) | (0xffffffff - local index): the atomic maximum is
// the largest |x|, then the lowest index. NaN ranks above every number.
__device__ __forceinline__ unsigned long long abs_key(float x, int64_t local) {
  uint32_t ab = __float_as_uint(x) & 0x7fffffffu;
  if (ab > 0x7f800000u) ab = 0x7f800000u;
  return ((unsigned long long)(ab + 1u) << 32) | (unsigned long long)(0xffffffffu - (uint32_t)local);
}
__device__ __forceinline__ int64_t key_index(unsigned long long key) {
  return (int64_t)(0xffffffffu - (uint32_t)(key & 0xffffffffull));
}

// Warp-aggregated atomic max of per-lane keys into keys[blk] (lanes of the
// warp may belong to different blocks).
__device__ __forceinline__ void key_max(unsigned long long* keys, int64_t blk, unsigned long long key, bool valid) {
  const unsigned mask = __ballot_sync(0xffffffffu, valid);
  if (!valid) return;
  const int64_t b0 = __shfl_sync(mask, blk, __ffs(mask) - 1);
  const bool same = __all_sync(mask, blk == b0);
  if (same && mask == 0xffffffffu) {
    unsigned long long k = key;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long t = __shfl_xor_sync(0xffffffffu, k, o);
      k = t > k ? t : k;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(keys + blk, k);
  } else {
    atomicMax(keys + blk, key);
  }
}

// Step (1): residual rows rho of every block's current pivot row, and the
// pivot columns. Thread per column position g (node beta = g / n is the
// column set of block beta ^ 1). The pivot row is read from the last step's row
// keys (no key: the residual vanished or fell below the tolerance, the block is
// done, marked -1, and its remaining u, v are zero) and recorded in prow.
__global__ void aca_row_kernel(Kern K, const double* __restrict__ geo, int64_t n, int c, int r, int k, int sym,
                               const float* __restrict__ U32, const float* __restrict__ V32, float* __restrict__ rho,
                               int* __restrict__ prow, const int* __restrict__ pcol,
                               const unsigned long long* __restrict__ lastkey,
                               unsigned long long* __restrict__ colkey) {
  const int64_t N = K.N;
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g - threadIdx.x < N;
       g += (int64_t)gridDim.x * blockDim.x) {
    const bool in = g < N;
    const int64_t gg = in ? g : N - 1;
    const int64_t beta = gg / n, blk = beta ^ 1;
    const bool active = in && (!sym || (blk & 1) == 0);
    float x = 0.f;
    unsigned long long key = 0;
    const int64_t jl = gg - beta * n;
    int ik = 0;  // local pivot row of this step; -1: block exhausted
    if (k > 0) {
      const unsigned long long lk = lastkey[blk];
      ik = lk ? (int)key_index(lk) : -1;
      if (in && jl == 0) prow[(size_t)blk * r + k] = ik;
    }
    if (active) {
      if (ik >= 0) {
        const int64_t gi = blk * n + ik;
        x = kernel_entry(K, geo, gi, gg);
        x = residual(x, U32 + gi, V32 + gg, N, k);
        bool used = false;
#pragma unroll 8
        for (int l = 0; l < k; ++l) used |= pcol[(size_t)blk * r + l] == (int)jl;
        key = used ? 0ull : abs_key(x, jl);
      }
      rho[gg] = x;
    }
    key_max(colkey, blk, key, active);
  }
}

// Step (2): v_k of every block from its residual row and pivot, u_k (residual
// column at the pivot column) and the next pivot rows. Thread per position g:
// as a row of node alpha = g / n (block alpha) it forms u_k(g); as a column
// of node beta = g / n (block beta ^ 1) it forms v_k(g).
__global__ void aca_col_kernel(Kern K, const double* __restrict__ geo, int64_t n, int c, int r, int k, int sym,
                               float* __restrict__ U32, float* __restrict__ V32, const float* __restrict__ rho,
                               const int* __restrict__ prow, int* __restrict__ pcol,
                               const unsigned long long* __restrict__ colkey, unsigned long long* __restrict__ rowkey,
                               double* __restrict__ Ub, double* __restrict__ Vb, int64_t ldu, int64_t ldv,
                               float* __restrict__ delta0) {
  const int64_t N = K.N;
  const int colblk = (c - 1) * r + k;  // column of U_big / V_big
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g - threadIdx.x < N;
       g += (int64_t)gridDim.x * blockDim.x) {
    const bool in = g < N;
    const int64_t gg = in ? g : N - 1;
    const int64_t node = gg / n;
    // v_k at column gg (block node ^ 1)
    {
      const int64_t blk = node ^ 1;
      if (in && (!sym || (blk & 1) == 0)) {
        const unsigned long long ck = colkey[blk];
        const bool live = step_live(ck, k, K.tol, delta0, blk);  // ck is 0 for a finished block
        // rho of block blk lives on node = blk ^ 1's positions
        const float piv = live ? rho[node * n + key_index(ck)] : 0.f;
        const float v = piv != 0.f ? rho[gg] / piv : 0.f;
        V32[(size_t)k * N + gg] = v;
        if (sym) {
          Ub[(size_t)colblk * ldu + gg] = (double)v;  // U(I_beta) = V(I_beta) for a symmetric kernel
          Vb[(size_t)colblk * ldv + gg] = (double)v;
        } else {
          Vb[(size_t)colblk * ldv + gg] = (double)v;
        }
      }
    }
    // u_k at row gg (block node)
    const int64_t blk = node;
    const bool active = in && (!sym || (blk & 1) == 0);
    unsigned long long key = 0;
    if (active) {
      const unsigned long long ck = colkey[blk];
      const bool live = step_live(ck, k, K.tol, delta0, blk);
      const int64_t jk = key_index(ck);
      const int64_t gj = (blk ^ 1) * n + jk;
      const int64_t il = gg - blk * n;
      float u = 0.f;
      if (live) {  // rows and columns of an off-diagonal block are disjoint
        u = kernel_entry(K, geo, gg, gj);
        u = residual(u, U32 + gg, V32 + gj, N, k);
      }
      U32[(size_t)k * N + gg] = u;
      Ub[(size_t)colblk * ldu + gg] = (double)u;
      if (sym) Vb[(size_t)colblk * ldv + gg] = (double)u;
      bool used = false;
#pragma unroll 8
      for (int l = 0; l <= k; ++l) used |= prow[(size_t)blk * r + l] == (int)il;
      key = (used || !live) ? 0ull : abs_key(u, il);
      if (il == 0) {
        pcol[(size_t)blk * r + k] = live ? (int)jk : -1;
        if (k == 0) delta0[blk] = live ? __uint_as_float((uint32_t)(ck >> 32) - 1u) : 0.f;
      }
    }
    key_max(rowkey, blk, key, active);
  }
}

// Levels of small nodes: all r steps of a block in one launch, by a cluster of CTAs
// that holds the block's keys in distributed shared memory and meets at a hardware
// barrier twice a step: about 10 us a step, a chain of loads from L2, against 25 us of
// the two launches above (Matern, N = 2^17, rank 64: 14.4 -> 10.7 ms). Thread
// positions, keys, pivots and roundings are those of the kernels above.
// At 8192 rows a cluster's eight SMs take 26 us a step, as long as the whole GPU's two
// launches; twice the rows would take longer.
constexpr int64_t kClusterRows = 8192;
constexpr int kClusterMax = 8, kClusterThreads = 256;

// Largest key over the cluster.
__device__ __forceinline__ unsigned long long cluster_max(unsigned long long key, unsigned long long* sWarp,
                                                          unsigned long long* sKey) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long t = __shfl_xor_sync(0xffffffffu, key, o);
    key = t > key ? t : key;
  }
  if (lane == 0) sWarp[warp] = key;
  __syncthreads();
  const unsigned ranks = cl.num_blocks(), rank = cl.block_rank();
  if (threadIdx.x < ranks) {
    key = sWarp[0];
#pragma unroll
    for (int w = 1; w < kClusterThreads / 32; ++w) key = sWarp[w] > key ? sWarp[w] : key;
    *cl.map_shared_rank(sKey + rank, threadIdx.x) = key;
  }
  cl.sync();
  key = sKey[0];
  for (unsigned q = 1; q < ranks; ++q) key = sKey[q] > key ? sKey[q] : key;
  return key;
}

// x - sum_{l < k} b[l] w[l step], as residual().
__device__ __forceinline__ float residual_shared(float x, const float* b, const float* w, int64_t step, int k) {
  int l = 0;
  for (; l + 32 <= k; l += 32) {
    float a[32];
#pragma unroll
    for (int q = 0; q < 32; ++q) a[q] = w[(size_t)(l + q) * step];
#pragma unroll
    for (int q = 0; q < 32; ++q) x = fmaf(-b[l + q], a[q], x);
  }
  for (; l + 8 <= k; l += 8) {
    float a[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) a[q] = w[(size_t)(l + q) * step];
#pragma unroll
    for (int q = 0; q < 8; ++q) x = fmaf(-b[l + q], a[q], x);
  }
#pragma unroll 4
  for (; l < k; ++l) x = fmaf(-b[l], w[(size_t)l * step], x);
  return x;
}

__global__ void __launch_bounds__(kClusterThreads) aca_cluster_kernel(Kern K, const double* __restrict__ geo,
                                                                      int64_t n, int c, int r, int sym, float* U32,
                                                                      float* V32, float* rho, int* prow, int* pcol,
                                                                      double* Ub, double* Vb, int64_t ldu,
                                                                      int64_t ldv) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ unsigned long long sWarp[kClusterThreads / 32], sKey[2][kClusterMax];
  __shared__ float sRow[64], sCol[64];
  const int tid = threadIdx.x;
  const int ranks = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int64_t unit = blockIdx.x / ranks;
  const int64_t blk = sym ? 2 * unit : unit;
  const int64_t r0 = blk * n, c0 = (blk ^ 1) * n, N = K.N;
  const int64_t first = (int64_t)rank * kClusterThreads + tid, step = (int64_t)ranks * kClusterThreads;
  int ik = 0;
  float delta0 = 0.f;
  uint32_t used_row = 0, used_col = 0;  // bit q: this thread's q-th position has been a pivot
  // the first keys go straight to the other CTAs' shared memory: all of them must have
  // started (later steps are ordered by the barriers of cluster_max)
  cl.sync();
  for (int k = 0; k < r; ++k) {
    const size_t col = (size_t)((c - 1) * r + k);
    // residual row of the pivot row
    if (tid < k && ik >= 0) sRow[tid] = U32[(size_t)tid * N + r0 + ik];
    if (tid == 0 && rank == 0) {
      prow[(size_t)blk * r + k] = ik;
      if (sym && k > 0) prow[(size_t)(blk ^ 1) * r + k] = -1;  // the mirrored block has no cross of its own
    }
    __syncthreads();
    unsigned long long key = 0;
    int q = 0;
    for (int64_t p = first; p < n; p += step, ++q) {
      float x = 0.f;
      if (ik >= 0) {
        x = kernel_entry(K, geo, r0 + ik, c0 + p);
        x = residual_shared(x, sRow, V32 + c0 + p, N, k);
        const unsigned long long t = (used_col >> q & 1u) ? 0ull : abs_key(x, p);
        key = t > key ? t : key;
      }
      rho[c0 + p] = x;
    }
    const unsigned long long ck = cluster_max(key, sWarp, sKey[0]);
    const bool live = step_live(ck, k, K.tol, &delta0, 0);
    const int64_t jk = key_index(ck);
    const float piv = live ? rho[c0 + jk] : 0.f;
    if (k == 0) delta0 = live ? __uint_as_float((uint32_t)(ck >> 32) - 1u) : 0.f;
    // v_k, the residual column at the pivot column and the next pivot row
    if (tid < k && live) sCol[tid] = V32[(size_t)tid * N + c0 + jk];
    if (tid == 0 && rank == 0) pcol[(size_t)blk * r + k] = live ? (int)jk : -1;
    __syncthreads();
    key = 0;
    q = 0;
    for (int64_t p = first; p < n; p += step, ++q) {
      if (live && p == jk) used_col |= 1u << q;
      if (p == ik) used_row |= 1u << q;
      const float v = piv != 0.f ? rho[c0 + p] / piv : 0.f;
      V32[(size_t)k * N + c0 + p] = v;
      Vb[col * ldv + c0 + p] = (double)v;
      if (sym) Ub[col * ldu + c0 + p] = (double)v;  // U(I_beta) = V(I_beta) for a symmetric kernel
      float u = 0.f;
      if (live) {
        u = kernel_entry(K, geo, r0 + p, c0 + jk);
        u = residual_shared(u, sCol, U32 + r0 + p, N, k);
        const unsigned long long t = (used_row >> q & 1u) ? 0ull : abs_key(u, p);
        key = t > key ? t : key;
      }
      U32[(size_t)k * N + r0 + p] = u;
      Ub[col * ldu + r0 + p] = (double)u;
      if (sym) Vb[col * ldv + r0 + p] = (double)u;
    }
    const unsigned long long rk = cluster_max(key, sWarp, sKey[1]);
    ik = rk ? (int)key_index(rk) : -1;
  }
}

// Rank of every block of a level: its live steps (pivot column >= 0).
__global__ void aca_ranks_kernel(int64_t nblk, int r, const int* __restrict__ pcol, int32_t* __restrict__ ranks) {
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nblk; b += (int64_t)gridDim.x * blockDim.x) {
    int k = 0;
    while (k < r && pcol[(size_t)b * r + k] >= 0) ++k;
    ranks[b] = k;
  }
}

unsigned grid_n(int64_t N) {
  int64_t b = (N + 255) / 256;
  return (unsigned)(b < 152 * 16 ? b : 152 * 16);
}

}  // namespace

size_t compress_workspace_bytes(const hodlr_desc& d) {
  const size_t N = (size_t)d.N, r = (size_t)d.r;
  size_t off = 0;
  auto take = [&](size_t bytes) { off += ws_align(bytes); };
  take(N * kGeo * sizeof(double));      // FP64 geometry / points
  take(2 * N * r * sizeof(float));      // FP32 working copies of one level's U, V columns
  take(N * sizeof(float));              // residual rows
  take(2 * r * ((size_t)1 << d.L) * sizeof(unsigned long long));  // column / row keys of every step
  take(2 * r * ((size_t)1 << d.L) * sizeof(int));                 // pivot rows / columns
  take(((size_t)1 << d.L) * sizeof(float));                       // first pivots of one level's blocks
  return off;
}

}  // namespace hodlr

using namespace hodlr;

extern "C" hodlr_status hodlr_compress_workspace_size(const hodlr_desc* desc, size_t* bytes) {
  hodlr_status st = check_desc_ext(desc);
  if (st != HODLR_OK) return st;
  if (!bytes) return HODLR_ERR_ARG;
  *bytes = compress_workspace_bytes(*desc);
  return HODLR_OK;
}

extern "C" hodlr_status hodlr_compress(const hodlr_desc* desc, const hodlr_kernel_desc* kern, double* D, double* U,
                                       double* V, int32_t* pivots, int32_t* ranks, void* workspace,
                                       size_t workspace_bytes, hodlr_stream_t stream) {
  hodlr_status st = check_desc_ext(desc);
  if (st != HODLR_OK) return st;
  if (!kern || !D || !U || !V) return HODLR_ERR_ARG;
  if (kern->kind != HODLR_KERNEL_BIE_STAR && kern->kind != HODLR_KERNEL_GAUSSIAN &&
      kern->kind != HODLR_KERNEL_MATERN32)
    return HODLR_ERR_ARG;
  if (kern->kind != HODLR_KERNEL_BIE_STAR && (!kern->points || kern->dim < 1 || kern->dim > 3 || !(kern->scale > 0.0)))
    return HODLR_ERR_ARG;
  if (!(kern->tol >= 0.0 && kern->tol < 1.0)) return HODLR_ERR_ARG;
  if (desc->N >= ((int64_t)1 << 31)) return HODLR_ERR_ARG;  // local indices are 32-bit
  const hodlr_desc& d = *desc;
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) % kWsAlign) || workspace_bytes < compress_workspace_bytes(d))
    return HODLR_ERR_WORKSPACE;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int64_t N = d.N;
  const int r = d.r, L = d.L;
  char* w = static_cast<char*>(workspace);
  size_t off = 0;
  auto take = [&](size_t bytes) { char* p = w + off; off += ws_align(bytes); return p; };
  double* geo = reinterpret_cast<double*>(take((size_t)N * kGeo * sizeof(double)));
  float* U32 = reinterpret_cast<float*>(take((size_t)N * r * sizeof(float)));
  float* V32 = reinterpret_cast<float*>(take((size_t)N * r * sizeof(float)));
  float* rho = reinterpret_cast<float*>(take((size_t)N * sizeof(float)));
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(
      take(2 * (size_t)r * ((size_t)1 << L) * sizeof(unsigned long long)));
  int* piv = reinterpret_cast<int*>(take(2 * (size_t)r * ((size_t)1 << L) * sizeof(int)));
  float* delta0 = reinterpret_cast<float*>(take(((size_t)1 << L) * sizeof(float)));
  Kern K{kern->kind, kern->kind == HODLR_KERNEL_BIE_STAR ? 2 : kern->dim, kern->points, kern->scale,
         kern->nugget, N, (float)kern->tol,
         kern->kind == HODLR_KERNEL_GAUSSIAN ? 1.0 / (2.0 * kern->scale * kern->scale) : 1.7320508075688772 / kern->scale};
  const int sym = kern->kind == HODLR_KERNEL_BIE_STAR ? 0 : 1;
  ProfScope prof_(KC_COMPRESS, s);
  note_work(8.0 * (double)N * d.m + 16.0 * (double)N * r * L, 2.0 * (double)N * r * r * L);
  geometry_kernel<<<grid_n(N), 256, 0, s>>>(K, geo);
  note_launches(1);
  if (sym) {
    const int nt = (d.m + 31) / 32;
    leaf_eval_sym_kernel<<<dim3(1u << L, nt * (nt + 1) / 2), 256, 0, s>>>(K, geo, d.m, D);
  } else {
    const int64_t tot = N * (int64_t)d.m;
    int64_t gb = (tot + 255) / 256;
    if (gb > 152 * 32) gb = 152 * 32;
    leaf_eval_kernel<<<(unsigned)gb, 256, 0, s>>>(K, geo, d.m, D);
  }
  note_launches(1);
  if (cudaGetLastError() != cudaSuccess) return HODLR_ERR_CUDA;
  for (int c = 1; c <= L; ++c) {
    const int64_t n = N >> c;
    const int64_t nblk = (int64_t)1 << c;
    unsigned long long* colkey = keys;                        // [r][nblk]
    unsigned long long* rowkey = keys + (size_t)r * nblk;     // [r][nblk]
    int* prow = piv;                                          // [nblk][r]
    int* pcol = piv + (size_t)r * nblk;                       // [nblk][r]
    if (cudaMemsetAsync(keys, 0, 2 * (size_t)r * nblk * sizeof(unsigned long long), s) != cudaSuccess ||
        cudaMemsetAsync(piv, 0, 2 * (size_t)r * nblk * sizeof(int), s) != cudaSuccess)
      return HODLR_ERR_CUDA;
    if (n <= kClusterRows) {
      int ranks = 1;
      while (ranks < kClusterMax && (int64_t)ranks * kClusterThreads < n) ranks *= 2;
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = ranks;
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      cfg.gridDim = dim3((unsigned)((sym ? nblk / 2 : nblk) * ranks));
      cfg.blockDim = dim3(kClusterThreads);
      cfg.stream = s;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      if (cudaLaunchKernelEx(&cfg, aca_cluster_kernel, K, (const double*)geo, n, c, r, sym, U32, V32, rho, prow, pcol,
                             U, V, d.ldu, d.ldv) != cudaSuccess)
        return HODLR_ERR_CUDA;
      note_launches(1);
    }
    for (int k = 0; n > kClusterRows && k < r; ++k) {
      aca_row_kernel<<<grid_n(N), 256, 0, s>>>(K, geo, n, c, r, k, sym, U32, V32, rho, prow, pcol,
                                               rowkey + (size_t)(k > 0 ? k - 1 : 0) * nblk,
                                               colkey + (size_t)k * nblk);
      aca_col_kernel<<<grid_n(N), 256, 0, s>>>(K, geo, n, c, r, k, sym, U32, V32, rho, prow, pcol,
                                               colkey + (size_t)k * nblk, rowkey + (size_t)k * nblk, U, V, d.ldu,
                                               d.ldv, delta0);
      note_launches(2);
    }
    if (ranks) {  // ranks of level c's blocks at offset 2^c - 2
      aca_ranks_kernel<<<(unsigned)((nblk + 255) / 256), 256, 0, s>>>(nblk, r, pcol, ranks + (nblk - 2));
      note_launches(1);
    }
    if (pivots) {
      // pivots of level c: [block][k] rows, then [block][k] columns (local indices)
      int32_t* pl = pivots + (size_t)2 * r * (((int64_t)1 << c) - 2);
      if (cudaMemcpyAsync(pl, piv, 2 * (size_t)r * nblk * sizeof(int), cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return HODLR_ERR_CUDA;
    }
    if (cudaGetLastError() != cudaSuccess) return HODLR_ERR_CUDA;
  }
  return HODLR_OK;
}

// ---------------------------------------------------------------------------
// Variable ranks per level (Eq. e:u with per-level widths): the ragged U_big
// / V_big hold level c's bases in columns off_c .. off_c + r_c - 1, each
// node's basis left-aligned (a node of lower rank has zero columns at the
// right). The same matrix in the uniform layout of width r >= max r_c has the
// level blocks zero-padded on the right, which every other entry point takes.
namespace hodlr {
namespace {

__global__ void pack_level_ranks_kernel(int64_t N, int r, int L, const int* __restrict__ lr,
                                        const int* __restrict__ off, const double* __restrict__ Ur, int64_t ldur,
                                        const double* __restrict__ Vr, int64_t ldvr, double* __restrict__ U,
                                        int64_t ldu, double* __restrict__ V, int64_t ldv) {
  const int col = blockIdx.y;  // uniform column (c - 1) r + j
  const int c = col / r + 1, j = col % r;
  const bool live = j < lr[c - 1];
  const int64_t src = live ? (int64_t)(off[c - 1] + j) : 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
    U[(int64_t)col * ldu + i] = live ? Ur[src * ldur + i] : 0.0;
    V[(int64_t)col * ldv + i] = live ? Vr[src * ldvr + i] : 0.0;
  }
}

}  // namespace
}  // namespace hodlr

extern "C" hodlr_status hodlr_pack_level_ranks(const hodlr_desc* desc, const int32_t* level_ranks, const double* Ur,
                                               int64_t ldur, const double* Vr, int64_t ldvr, double* U, double* V,
                                               void* workspace, size_t workspace_bytes, hodlr_stream_t stream) {
  hodlr_status st = check_desc_ext(desc);
  if (st != HODLR_OK) return st;
  const hodlr_desc& d = *desc;
  if (!level_ranks || !Ur || !Vr || !U || !V || ldur < d.N || ldvr < d.N) return HODLR_ERR_ARG;
  std::vector<int> lr(d.L), off(d.L);
  int tot = 0;
  for (int c = 0; c < d.L; ++c) {
    if (level_ranks[c] < 0 || level_ranks[c] > d.r) return HODLR_ERR_ARG;
    lr[c] = level_ranks[c];
    off[c] = tot;
    tot += lr[c];
  }
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) % kWsAlign) ||
      workspace_bytes < 2 * (size_t)d.L * sizeof(int))
    return HODLR_ERR_WORKSPACE;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int* dlr = static_cast<int*>(workspace);
  int* doff = dlr + d.L;
  std::vector<int> h(2 * d.L);
  for (int c = 0; c < d.L; ++c) {
    h[c] = lr[c];
    h[d.L + c] = off[c];
  }
  if (cudaMemcpyAsync(dlr, h.data(), h.size() * sizeof(int), cudaMemcpyHostToDevice, s) != cudaSuccess)
    return HODLR_ERR_CUDA;
  {
    ProfScope prof_(KC_VECTOR, s);
    note_work(16.0 * (double)d.N * (tot + d.r * d.L), 0.0);
    pack_level_ranks_kernel<<<dim3(grid_n(d.N), d.r * d.L), 256, 0, s>>>(d.N, d.r, d.L, dlr, doff, Ur, ldur, Vr,
                                                                         ldvr, U, d.ldu, V, d.ldv);
    note_launches(1);
  }
  // the host vector must outlive the asynchronous copy
  if (cudaStreamSynchronize(s) != cudaSuccess) return HODLR_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? HODLR_OK : HODLR_ERR_CUDA;
}
