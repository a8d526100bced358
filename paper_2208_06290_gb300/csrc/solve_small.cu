// FP64 solves of one to four columns: one launch per level.
//
// With so few columns a solve is a chain of short steps: at N = 4096 the leaf solve
// took 34 us and each level three launches of 5 to 16 us, bound by the FP64 pipe of
// the few SMs that had work (two FMAs per clock each) and by the launches. Here
//   * a level is one launch: each CTA takes at most 256 rows of a node, forms that
//     node's w from the children's projections and its rows of K~^{-1}, updates its
//     rows and projects them, still in shared memory, onto the next level's basis.
//     Every CTA of a node forms the same w; from nine projection chunks per child on
//     that costs more than a launch, and w comes from small_parent_kernel instead;
//   * row chunks are short (128 rows up to N = 2^15, else 256), so that small
//     problems reach more SMs; sums over the lanes are transposed, which takes 1.5
//     FP64 additions per basis column and warp instead of five;
//   * the leaf solves use the inverted diagonal blocks (leaf_split.cu) with all of a
//     CTA's warps on each block's terms, instead of one dependent step per unknown.
#include "hodlr_internal.cuh"
#include "substitute.cuh"

namespace hodlr {

namespace {

// Rows of a projection chunk at child level c: the node's, halved until they are few
// enough, but never below a leaf's.
int64_t small_rows(const hodlr_desc& d, int c) {
  int64_t n = d.N >> c;
  const int64_t most = d.N <= 32768 ? 128 : 256;
  while (n > most && n > d.m) n >>= 1;
  return n;
}

// Sums v over the warp; lane l ends with the total of value `idx` where
// l % (32 / NV) == 0.
template <int NV>
__device__ __forceinline__ double warp_sums(double (&v)[NV], int lane, int& idx) {
  idx = 0;
#pragma unroll
  for (int h = NV / 2, s = 16; s >= 1; s >>= 1, h >>= 1) {
    if (h >= 1) {
      const bool upper = (lane & s) != 0;
#pragma unroll
      for (int i = 0; i < h; ++i) {
        const double send = upper ? v[i] : v[i + h];
        const double keep = upper ? v[i + h] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
      }
      idx += upper ? h : 0;
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], s);
    }
  }
  return v[0];
}

// part[g][o KC + cc], g < G: partial sums of row off + o of K~^{-1} (or its transpose)
// times rhs (2r x KC, rhs[i KC + cc]); returns G.
template <int KC, int NT>
__device__ __forceinline__ int coupling_rows(int r, int rows, int off, const double* __restrict__ Kj, int trans,
                                             const double* rhs, double* part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n2 = 2 * r;
  const int tiles = (rows + 31) / 32;
  const int G = NT / 32 / tiles;
  const int o = warp % tiles * 32 + lane, g = warp / tiles;
  if (g < G) {
    double acc[KC];
#pragma unroll
    for (int cc = 0; cc < KC; ++cc) acc[cc] = 0.0;
    if (o < rows) {
      const int i = off + o;
#pragma unroll 8
      for (int j = g; j < n2; j += G) {
        const double kv = trans ? Kj[(size_t)i * n2 + j] : Kj[(size_t)j * n2 + i];
#pragma unroll
        for (int cc = 0; cc < KC; ++cc) acc[cc] = fma(kv, rhs[j * KC + cc], acc[cc]);
      }
#pragma unroll
      for (int cc = 0; cc < KC; ++cc) part[(g * rows + o) * KC + cc] = acc[cc];
    }
  }
  return G;
}

}  // namespace

struct SmallLevel {
  int64_t N;
  int r, k, trans;
  // update of level cu (0: none): own basis, coupling inverses of the level and the
  // projections of its nodes (cpn chunks each), or the finished w (wstride per node)
  int cu;
  const double* Ub;
  int64_t ldu;
  const double* K;
  const double* parts;
  int64_t cpn;
  const double* W;
  double* x;
  int64_t ldx;
  // projection of the CTA's rows (one chunk) onto the next level's basis (null: none)
  const double* Pb;
  int64_t ldp;
  double* out;
  int rows;  // rows of a CTA
};

template <int KC, int NT>
__global__ void __launch_bounds__(NT) small_level_kernel(SmallLevel a) {
  __shared__ double sRhs[2 * 64 * KC], sW[64 * KC], sX[KC][256];
  __shared__ double sPart[NT / 32 * 32 * KC];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r = a.r, k = a.k;
  const int64_t row0 = (int64_t)blockIdx.x * a.rows;
  const int64_t row = row0 + tid;
  const bool mine = tid < a.rows;
  double x[KC];
#pragma unroll
  for (int cc = 0; cc < KC; ++cc) x[cc] = (mine && cc < k) ? a.x[(int64_t)cc * a.ldx + row] : 0.0;
  if (a.cu > 0) {
    double pre[16];  // the first basis columns, loaded under the coupling product
#pragma unroll
    for (int j = 0; j < 16; ++j) pre[j] = (mine && j < r) ? a.Ub[(int64_t)j * a.ldu + row] : 0.0;
    const int64_t node = row0 / (a.N >> a.cu);
    const int64_t from = a.trans ? node ^ 1 : node;  // whose w
    if (a.W) {
      for (int e = tid; e < r * KC; e += NT) {
        const int j = e / KC, cc = e % KC;
        sW[e] = cc < k ? a.W[(size_t)from * r * k + cc * r + j] : 0.0;
      }
    } else {
      // right-hand side: K~ [w_a; w_b] = [s_b; s_a], transposed: K~^T t = [s_a; s_b]
      for (int e = tid; e < 2 * r * KC; e += NT) {
        const int i = e / KC, cc = e % KC;
        const int64_t child = (node & ~(int64_t)1) + ((i < r) == (a.trans == 0) ? 1 : 0);
        double s = 0.0;
        if (cc < k) {
          const double* p = a.parts + (size_t)child * a.cpn * r * k + cc * r + (i < r ? i : i - r);
          for (int64_t q = 0; q < a.cpn; ++q) s += p[(size_t)q * r * k];
        }
        sRhs[e] = s;
      }
      __syncthreads();
      const int G = coupling_rows<KC, NT>(r, r, (int)(from & 1) * r, a.K + (size_t)(node >> 1) * 4 * r * r, a.trans,
                                          sRhs, sPart);
      __syncthreads();
      for (int e = tid; e < r * KC; e += NT) {
        double s = sPart[e];
        for (int g = 1; g < G; ++g) s += sPart[g * r * KC + e];
        sW[e] = s;
      }
    }
    __syncthreads();
    if (mine) {
      double acc[KC];
#pragma unroll
      for (int cc = 0; cc < KC; ++cc) acc[cc] = 0.0;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        if (j < r) {
#pragma unroll
          for (int cc = 0; cc < KC; ++cc) acc[cc] = fma(pre[j], sW[j * KC + cc], acc[cc]);
        }
      }
#pragma unroll 8
      for (int j = 16; j < r; ++j) {
        const double b = a.Ub[(int64_t)j * a.ldu + row];
#pragma unroll
        for (int cc = 0; cc < KC; ++cc) acc[cc] = fma(b, sW[j * KC + cc], acc[cc]);
      }
#pragma unroll
      for (int cc = 0; cc < KC; ++cc) {
        x[cc] -= acc[cc];
        if (cc < k) a.x[(int64_t)cc * a.ldx + row] = x[cc];
      }
    }
  }
  if (!a.Pb) return;
#pragma unroll
  for (int cc = 0; cc < KC; ++cc) sX[cc][tid] = x[cc];
  __syncthreads();
  // four basis columns per warp at a time, rows along the lanes
  for (int j0 = warp * 4; j0 < r; j0 += NT / 32 * 4) {
    double v[4 * KC];
#pragma unroll
    for (int u = 0; u < 4 * KC; ++u) v[u] = 0.0;
#pragma unroll
    for (int i = 0; i < NT; i += 32) {
      if (i + lane < a.rows) {
        double b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) b[q] = j0 + q < r ? a.Pb[(int64_t)(j0 + q) * a.ldp + row0 + i + lane] : 0.0;
#pragma unroll
        for (int cc = 0; cc < KC; ++cc) {
          const double xv = sX[cc][i + lane];
#pragma unroll
          for (int q = 0; q < 4; ++q) v[cc * 4 + q] = fma(b[q], xv, v[cc * 4 + q]);
        }
      }
    }
    int idx;
    const double t = warp_sums<4 * KC>(v, lane, idx);
    const int cc = idx >> 2, j = j0 + (idx & 3);
    if (lane % (8 / KC) == 0 && cc < k && j < r) a.out[(size_t)blockIdx.x * r * k + cc * r + j] = t;
  }
}

// w of both children of every parent, from many projection chunks per child: the
// chunks are added by groups of threads, then the groups in order.
template <int KC>
__global__ void __launch_bounds__(512) small_parent_kernel(int r, int k, int trans, int64_t cpn,
                                                           const double* __restrict__ parts,
                                                           const double* __restrict__ K, double* __restrict__ W) {
  __shared__ double sSum[512 * KC], sRhs[2 * 64 * KC];
  const int tid = threadIdx.x;
  const int64_t p = blockIdx.x;
  const int n = 2 * r * k, G = 512 * KC / n;  // k <= KC and r <= 64: G >= 4
  for (int e = tid; e < G * n; e += 512) {
    const int g = e / n, i = e % n;          // i = child r k + column r + row
    const double* q0 = parts + (size_t)(2 * p + i / (r * k)) * cpn * r * k + i % (r * k);
    double s = 0.0;
#pragma unroll 4
    for (int64_t q = g; q < cpn; q += G) s += q0[(size_t)q * r * k];
    sSum[e] = s;
  }
  __syncthreads();
  for (int e = tid; e < 2 * r * KC; e += 512) {
    const int i = e / KC, cc = e % KC;
    const int child = (i < r) == (trans == 0) ? 1 : 0;
    double s = 0.0;
    if (cc < k)
      for (int g = 0; g < G; ++g) s += sSum[g * n + (child * k + cc) * r + (i < r ? i : i - r)];
    sRhs[e] = s;
  }
  __syncthreads();
  const int GK = coupling_rows<KC, 512>(r, 2 * r, 0, K + (size_t)p * 4 * r * r, trans, sRhs, sSum);
  __syncthreads();
  for (int e = tid; e < 2 * r * KC; e += 512) {
    const int o = e / KC, cc = e % KC;
    double s = sSum[e];
    for (int g = 1; g < GK; ++g) s += sSum[g * 2 * r * KC + e];
    if (cc < k) W[(size_t)(2 * p + o / r) * r * k + cc * r + o % r] = s;
  }
}

// X_b <- D_b^{-1} X_b or D_b^{-T} X_b, one CTA per leaf: left-looking substitution in
// blocks of 32 unknowns. The terms of a block (those of the solved blocks, then those
// of the inverted diagonal block) are dealt out to the eight warps, lane = row. Marked
// diagonal blocks (leaf_tinv_kernel) are substituted, a warp per column.
template <int KC>
__global__ void __launch_bounds__(256) small_leaf_kernel(int m, const double* __restrict__ LU,
                                                         const double* __restrict__ tinv,
                                                         const uint8_t* __restrict__ tsub,
                                                         const int* __restrict__ perm, const double* in, int64_t ldin,
                                                         double* out, int64_t ldout, int k, int trans) {
  __shared__ double sX[KC][256], sP[8][KC][32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t b = blockIdx.x;
  const int nb = (m + 31) / 32;
  const double* A = LU + (size_t)b * m * m;
  const double* T = tinv + (size_t)b * tinv_elems(m);
  const unsigned marked = __ballot_sync(0xffffffffu, lane < 2 * nb && tsub[(size_t)b * 2 * nb + (lane < 2 * nb ? lane : 0)] != 0);
  const int* pb = perm + (size_t)b * m;
  const int64_t row0 = b * m;
#pragma unroll
  for (int cc = 0; cc < KC; ++cc)
    sX[cc][tid] = (tid < m && cc < k) ? in[(int64_t)cc * ldin + row0 + (trans ? tid : pb[tid])] : 0.0;
  for (int sweep = 0; sweep < 2; ++sweep) {
    const bool useL = (sweep == 0) == (trans == 0);  // op(A) = L U, or U^T L^T
    for (int kk = 0; kk < nb; ++kk) {
      const int kb = sweep == 0 ? kk : nb - 1 - kk;
      const int row = kb * 32 + lane, nk = min(32, m - kb * 32);
      // diagonal block: terms 4 warp .. + 3 of row `lane`
      double tv[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int c = 4 * warp + q;
        const int i = trans ? c : lane, j = trans ? lane : c;  // element (i, j) of L^{-1} or U^{-1}
        const bool in_tri = useL ? i >= j : i <= j;
        tv[q] = 0.0;
        if (in_tri && row < m && kb * 32 + c < m) tv[q] = useL && i == j ? 1.0 : T[kb * 1024 + j * nk + i];
      }
      double acc[KC];
#pragma unroll
      for (int cc = 0; cc < KC; ++cc) acc[cc] = 0.0;
      const int c0 = (sweep == 0 ? 0 : (kb + 1) * 32) + warp * 4 * kk;
      __syncthreads();  // the solved blocks are in shared memory
      if (row < m) {
#pragma unroll 4
        for (int c = c0; c < c0 + 4 * kk; ++c) {
          if (c < m) {
            const double v = trans ? A[(size_t)row * m + c] : A[(size_t)c * m + row];
#pragma unroll
            for (int cc = 0; cc < KC; ++cc) acc[cc] = fma(v, sX[cc][c], acc[cc]);
          }
        }
      }
#pragma unroll
      for (int cc = 0; cc < KC; ++cc) sP[warp][cc][lane] = acc[cc];
      __syncthreads();
      if (tid < 32 * KC) {
        const int cc = tid >> 5;
        double s = sP[0][cc][lane];
#pragma unroll
        for (int w = 1; w < 8; ++w) s += sP[w][cc][lane];
        sX[cc][row] -= s;
      }
      __syncthreads();
      if (marked >> (2 * kb + (useL ? 0 : 1)) & 1u) {
        if (warp < KC) {
          double x[1] = {sX[warp][row]};
          substitute<1>(A + (size_t)kb * 32 * (m + 1), m, nk, sweep, useL, trans, lane, x);
          sX[warp][row] = x[0];
        }
        continue;
      }
#pragma unroll
      for (int cc = 0; cc < KC; ++cc) {
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q) s = fma(tv[q], sX[cc][kb * 32 + 4 * warp + q], s);
        sP[warp][cc][lane] = s;
      }
      __syncthreads();
      if (tid < 32 * KC) {
        const int cc = tid >> 5;
        double s = sP[0][cc][lane];
#pragma unroll
        for (int w = 1; w < 8; ++w) s += sP[w][cc][lane];
        sX[cc][row] = s;
      }
    }
  }
  __syncthreads();
  if (tid < m) {
    const int dst = trans ? pb[tid] : tid;
#pragma unroll
    for (int cc = 0; cc < KC; ++cc)
      if (cc < k) out[(int64_t)cc * ldout + row0 + dst] = sX[cc][tid];
  }
}

// ---------------------------------------------------------------------------
cudaError_t launch_leaf_solve_small(const Factor& F, const double* in, int64_t ldin, double* out, int64_t ldout,
                                    int k, int trans, cudaStream_t s) {
  const int m = F.d.m;
  const double Nd = (double)F.d.N;
  note_work(16.0 * Nd * k + 8.0 * Nd * m + 4.0 * Nd, 2.0 * m * Nd * k);
  const unsigned g = 1u << F.d.L;
  const double* lu = static_cast<const double*>(F.lu);
  if (k == 1) small_leaf_kernel<1><<<g, 256, 0, s>>>(m, lu, F.tinv, F.tsub, F.perm, in, ldin, out, ldout, k, trans);
  else if (k == 2) small_leaf_kernel<2><<<g, 256, 0, s>>>(m, lu, F.tinv, F.tsub, F.perm, in, ldin, out, ldout, k, trans);
  else small_leaf_kernel<4><<<g, 256, 0, s>>>(m, lu, F.tinv, F.tsub, F.perm, in, ldin, out, ldout, k, trans);
  note_launches(1);
  return cudaGetLastError();
}

// Projection chunks of every level and their count: two buffers in turn and the w's.
static int64_t small_parts(const hodlr_desc& d) {
  int64_t most = 0;
  for (int c = 1; c <= d.L; ++c) {
    const int64_t q = d.N / small_rows(d, c);
    if (q > most) most = q;
  }
  return most;
}

size_t solve_small_elems(const hodlr_desc& d, int k) { return 3 * (size_t)small_parts(d) * d.r * k; }

template <int KC>
static cudaError_t small_level(const hodlr_desc& d, SmallLevel a, cudaStream_t s) {
  const unsigned grid = (unsigned)(d.N / a.rows);
  if (a.rows <= 128) small_level_kernel<KC, 128><<<grid, 128, 0, s>>>(a);
  else small_level_kernel<KC, 256><<<grid, 256, 0, s>>>(a);
  note_launches(1);
  return cudaGetLastError();
}

template <int KC>
static cudaError_t solve_small(const Factor& F, double* x, int64_t ldx, int k, double* work, int trans,
                               cudaStream_t s) {
  const hodlr_desc& d = F.d;
  const int r = d.r, L = d.L;
  const double* Y = static_cast<const double*>(F.Y);
  const double* V = static_cast<const double*>(F.Vp);
  const size_t buf = (size_t)small_parts(d) * r * k;
  double* parts[2] = {work, work + buf};
  double* W = work + 2 * buf;
  // forward: x <- D^{-1} x, then levels L .. 1 (project V_c, update Y_c); adjoint:
  // levels 1 .. L (project Y_c, update V_c), then D^{-T}
  const double* pro = trans ? Y : V;
  const double* upd = trans ? V : Y;
  const int64_t ldpro = trans ? d.N : F.ldvp, ldupd = trans ? F.ldvp : d.N;
  cudaError_t e;
  if (!trans) {
    ProfScope prof_(KC_LEAF_SOLVE, s);
    if ((e = launch_leaf_solve_small(F, x, ldx, x, ldx, k, 0, s)) != cudaSuccess) return e;
  }
  SmallLevel a{};
  a.N = d.N;
  a.r = r;
  a.k = k;
  a.trans = trans;
  a.x = x;
  a.ldx = ldx;
  a.ldu = ldupd;
  a.ldp = ldpro;
  int64_t chunk = 0;  // rows per projection chunk of the level to be updated
  for (int i = 0; i <= L; ++i) {
    const int cu = i == 0 ? 0 : (trans ? i : L + 1 - i);       // level updated
    const int cp = i == L ? 0 : (trans ? i + 1 : L - i);       // level projected
    // a CTA's rows lie in one node of both levels: the lower of them decides
    const int low = trans ? (cp ? cp : cu) : (cu ? cu : cp);
    a.cu = cu;
    a.rows = (int)small_rows(d, low);
    a.Ub = cu ? upd + (size_t)(cu - 1) * r * ldupd : nullptr;
    a.Pb = cp ? pro + (size_t)(cp - 1) * r * ldpro : nullptr;
    a.out = parts[i & 1];
    a.W = nullptr;
    if (cu) {
      const int64_t n = d.N >> cu;
      a.parts = parts[(i - 1) & 1];
      a.cpn = n / chunk;
      a.K = F.K + F.Koff[cu] * 4 * r * r;
      if (a.cpn > 8) {
        ProfScope prof_(KC_COUPLING_APPLY, s);
        const double pr = (double)(1ll << (cu - 1));
        note_work(8.0 * ((double)(d.N / chunk) * r * k + pr * 4.0 * r * r + 2.0 * pr * r * k), pr * 8.0 * r * r * k);
        small_parent_kernel<KC><<<1u << (cu - 1), 512, 0, s>>>(r, k, trans, a.cpn, a.parts, a.K, W);
        note_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        a.W = W;
      }
    }
    ProfScope prof_(cu ? KC_UPDATE : KC_PROJECT, s);
    const double Nd = (double)d.N, both = (cu ? 1.0 : 0.0) + (cp ? 1.0 : 0.0);
    note_work(8.0 * Nd * r * both + 8.0 * Nd * k * (cu ? 2.0 : 1.0), 2.0 * Nd * r * k * both);
    if ((e = small_level<KC>(d, a, s)) != cudaSuccess) return e;
    chunk = a.rows;
  }
  if (trans) {
    ProfScope prof_(KC_LEAF_SOLVE, s);
    if ((e = launch_leaf_solve_small(F, x, ldx, x, ldx, k, 1, s)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_solve_small(const Factor& F, double* x, int64_t ldx, int k, double* work, int trans,
                               cudaStream_t s) {
  if (k == 1) return solve_small<1>(F, x, ldx, k, work, trans, s);
  if (k == 2) return solve_small<2>(F, x, ldx, k, work, trans, s);
  return solve_small<4>(F, x, ldx, k, work, trans, s);
}

}  // namespace hodlr
