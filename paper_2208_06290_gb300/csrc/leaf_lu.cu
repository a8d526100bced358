// Leaf stage: batched LU with partial pivoting of the 2^L leaf blocks (Alg. 1
// leaf loop; Alg. 3 first step).
#include "fp64_split.cuh"

namespace hodlr {

namespace {

constexpr int kPanel = 32;

// |x| as an ordered integer, two words, 0 for NaN (never a pivot while another
// entry can be one).
__device__ __forceinline__ uint2 pivot_key(float x) {
  const uint32_t u = __float_as_uint(x) & 0x7fffffffu;
  return make_uint2(u > 0x7f800000u ? 0u : u + 1u, 0u);
}
__device__ __forceinline__ uint2 pivot_key(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x) & 0x7fffffffu, lo = (uint32_t)__double2loint(x);
  const bool nan = hi > 0x7ff00000u || (hi == 0x7ff00000u && lo != 0u);
  return nan ? make_uint2(0u, 0u) : make_uint2(hi + 1u, lo);
}

template <typename T> struct Vec;
template <> struct Vec<float> {
  static constexpr int n = 4;
  using type = float4;
};
template <> struct Vec<double> {
  static constexpr int n = 2;
  using type = double2;
};

// 16 bytes of shared memory to or from registers.
template <typename T>
__device__ __forceinline__ void lds16(const T* p, T* o) {
  const typename Vec<T>::type v = *reinterpret_cast<const typename Vec<T>::type*>(p);
  o[0] = v.x;
  o[1] = v.y;
  if constexpr (Vec<T>::n == 4) {
    o[2] = v.z;
    o[3] = v.w;
  }
}
template <typename T>
__device__ __forceinline__ void sts16(T* p, const T* o) {
  typename Vec<T>::type v;
  v.x = o[0];
  v.y = o[1];
  if constexpr (Vec<T>::n == 4) {
    v.z = o[2];
    v.w = o[3];
  }
  *reinterpret_cast<typename Vec<T>::type*>(p) = v;
}

template <typename T> constexpr int kPitch = kPanel + Vec<T>::n;  // 16-byte rows, staggered banks

constexpr int kRowTile = 2 * split::kPlanes * 512;  // digits of 16 rows of L_21

template <typename T>
size_t leaf_lu_smem(int m) {
  const int n2 = m > kPanel ? m - kPanel : 0;
  return sizeof(T) * ((size_t)n2 * kPitch<T> + (size_t)kPanel * kPitch<T> + 2 * 8 * kPanel) + 256 * sizeof(double) +
         (sizeof(T) == 8 ? (size_t)((n2 + 15) / 16) * kRowTile : 0);
}

}  // namespace

// K1: leaf LU with partial pivoting (getrf's pivots: the first largest entry
// in the current row order), one CTA per leaf, one thread per row, panels of 32
// columns.
// A panel lives in the threads' registers. Each of its columns takes one
// barrier: every warp offers its largest entry together with that row, and all
// threads read the winner's row from shared memory. Rows are not moved while the
// panel is factored (every thread tracks the position of its row); the panel
// and the trailing columns are written back in the new order, earlier panels at
// the end. The pivot rows' trailing part U_12 is solved for with one column per
// lane. FP32: every thread updates its own row from registers (L_21) and
// broadcast reads of U_12, sixteen columns at a time. FP64: the update is a
// product of split operands on the tensor cores (fp64_split.cuh), L_21 split by
// the rows' threads into shared memory, eight columns of U_12 by each warp.
// A row that moves takes the place of a pivot row, whose trailing part is in
// shared memory by then, so the rows are updated in place without a barrier;
// U_12 itself is written last.
// A rank-1 update of the whole trailing block per column, three barriers each
// (the form before), was bound by those barriers and by memory passes; this one
// passes over the block m / 32 times through L2 and is bound by the panels'
// column steps. FP32, m = 256: 27.9 -> 3.0 ms for 2048 leaves (0.24 ms of HBM traffic);
// FP64 with the diagonal blocks' inverses, m = 256, 64 leaves: 7.0 -> 1.1 ms; m = 128, 1024
// leaves: 3.9 -> 1.75 ms.
template <typename T, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) leaf_lu_kernel(int m, const double* D,  // may alias LU (in place)
                                                             T* LU, int* __restrict__ perm,
                                                             double* __restrict__ leaf_ld, DevStatus* st) {
  constexpr int V = Vec<T>::n, PT = kPitch<T>;
  constexpr int CB = 16;
  constexpr bool kSplit = sizeof(T) == 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* sPiv = reinterpret_cast<double*>(smem_raw);  // pivots (256)
  T* sCand = reinterpret_cast<T*>(sPiv + 256);         // [2][8][kPanel] the warps' candidate rows
  T* sL = sCand + 2 * 8 * kPanel;                      // [rank][PT] L_11
  T* sU = sL + kPanel * PT;                            // [trailing column][PT] U_12
  unsigned char* sA = reinterpret_cast<unsigned char*>(sU + (m > kPanel ? m - kPanel : 0) * PT);  // digits of L_21
  __shared__ uint4 sKey[2][8];
  __shared__ int sRow[kPanel];
  __shared__ uint8_t sPerm[8][256], sMap[256];
  __shared__ int sE[kSplit ? 256 : 1];         // exponents of the rows of L_21
  __shared__ uint8_t sOld[kSplit ? 256 : 1];   // their places before the panel
  const int b = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const double* Db = D + (size_t)b * m * m;
  T* Ab = LU + (size_t)b * m * m;
  const int np = (m + kPanel - 1) / kPanel;
  int swaps = 0, sing = -1, step = 0;
  bool bad = false;

  for (int p = 0; p < np; ++p) {
    const int k0 = p * kPanel;
    const int nb = min(kPanel, m - k0);
    const bool live = tid >= k0 && tid < m;
    int pos = live ? tid : 0x7fffffff;
    bool open = live;  // not yet a pivot row
    T x[kPanel];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kPanel; ++j) {
      x[j] = T(0);
      if (live && j < nb) {
        if (p == 0) {
          const double v = Db[(size_t)j * m + tid];
          bad |= !f64_finite_bits(v);
          x[j] = conv<T>(v);
        } else {
          x[j] = Ab[(size_t)(k0 + j) * m + tid];
        }
      }
    }
#pragma unroll
    for (int k = 0; k < kPanel; ++k) {
      if (k < nb) {
        const int buf = step & 1;
        ++step;
        const uint2 key = open ? pivot_key(x[k]) : make_uint2(0u, 0u);
        const uint32_t mh = __reduce_max_sync(0xffffffffu, key.x);
        bool cand = open && key.x == mh;
        uint32_t ml = 0;
        if constexpr (sizeof(T) == 8) {
          ml = __reduce_max_sync(0xffffffffu, cand ? key.y : 0u);
          cand &= key.y == ml;
        }
        const uint32_t mp = __reduce_min_sync(0xffffffffu, cand ? (uint32_t)pos : 0x7fffffffu);
        if (cand && (uint32_t)pos == mp) {
          T* q = sCand + (buf * 8 + warp) * kPanel;
#pragma unroll
          for (int j = k / V * V; j < kPanel; j += V) sts16(q + j, &x[j]);
        }
        if (lane == 0) sKey[buf][warp] = make_uint4(mh, ml, mp, 0u);
        __syncthreads();
        uint4 best = sKey[buf][0];
        int bw = 0;
        for (int w = 1; w < nw; ++w) {
          const uint4 o = sKey[buf][w];
          const bool gt = o.x > best.x || (o.x == best.x && (o.y > best.y || (o.y == best.y && o.z < best.z)));
          if (gt) {
            best = o;
            bw = w;
          }
        }
        const int bp = (int)best.z;  // position of the pivot row
        swaps ^= bp != k0 + k;
        if (open) {
          if (pos == bp) {
            pos = k0 + k;
            open = false;
          } else if (pos == k0 + k) {
            pos = bp;
          }
        }
        T pr[kPanel];
#pragma unroll
        for (int j = k / V * V; j < kPanel; j += V) lds16(sCand + (buf * 8 + bw) * kPanel + j, &pr[j]);
        const T piv = pr[k];
        if (tid == 0) sPiv[k0 + k] = (double)piv;
        if (piv != T(0)) {
          if (open) {
            const T l = x[k] / piv;
            x[k] = l;
#pragma unroll
            for (int j = k + 1; j < kPanel; ++j) x[j] -= l * pr[j];
          }
        } else if (sing < 0) {
          sing = k0 + k;
        }
      }
    }
    if (live) {
#pragma unroll
      for (int j = 0; j < kPanel; ++j)
        if (j < nb) Ab[(size_t)(k0 + j) * m + pos] = x[j];
    }
    if (tid < m) sPerm[p][tid] = (uint8_t)(live ? pos : tid);
    const int n2 = m - k0 - kPanel;
    if (n2 <= 0) break;
    const bool pivot_row = live && pos < k0 + kPanel;
    const int rank = pos - k0;
    if (pivot_row) {
      sRow[rank] = tid;
#pragma unroll
      for (int j = 0; j < kPanel; j += V) sts16(sL + rank * PT + j, &x[j]);
    }
    if constexpr (kSplit) {
      const int idx = live ? rank - kPanel : -1;  // row of L_21
      if (idx >= 0) {
        uint32_t mh = 0;
        bool tiny = false;
#pragma unroll
        for (int j = 0; j < kPanel; ++j) {
          mh = max(mh, split::abs_hi(x[j]));
          tiny |= x[j] != T(0);
        }
        const int e = split::vector_exp(mh, tiny);
        sE[idx] = e;
        sOld[idx] = (uint8_t)tid;
        unsigned char* dst = sA + (idx >> 4) * kRowTile + (idx & 7) * 64 + ((idx >> 3) & 1) * 8;
#pragma unroll
        for (int q = 0; q < kPanel / 4; ++q) {  // q = 4 s + t
          const double y[4] = {x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]};
          uint2 d[split::kDigits];
          split::split4(y, e, d);
          split::store_planes(dst + (q >> 2) * split::kPlanes * 512 + (q & 3) * 16, d);
        }
      }
      if (tid < 16 && n2 + tid < 256) sE[n2 + tid] = split::kZeroExp;  // padding of the last row tile
    }
    __syncthreads();
    // U_12: the pivot rows' trailing columns, then L_11^{-1} applied, column per lane
    const int j2 = k0 + kPanel;
    for (int j = warp; j < n2; j += nw) {
      const size_t at = (size_t)(j2 + j) * m + sRow[lane];
      T v;
      if (p == 0) {
        bad |= !f64_finite_bits(Db[at]);
        v = conv<T>(Db[at]);
      } else {
        v = Ab[at];
      }
      sU[j * PT + lane] = v;
    }
    __syncthreads();
    for (int j = tid; j < n2; j += blockDim.x) {
      T u[kPanel];
#pragma unroll
      for (int k = 0; k < kPanel; k += V) lds16(sU + j * PT + k, &u[k]);
#pragma unroll
      for (int k = 1; k < kPanel; ++k) {
#pragma unroll
        for (int l = 0; l < k; l += V) {
          T lv[V];
          lds16(sL + k * PT + l, lv);
#pragma unroll
          for (int q = 0; q < V; ++q)
            if (l + q < k) u[k] -= lv[q] * u[l + q];
        }
      }
#pragma unroll
      for (int k = 0; k < kPanel; k += V) sts16(sU + j * PT + k, &u[k]);
    }
    __syncthreads();
    if constexpr (kSplit) {
      using namespace split;
      const int g = lane >> 2, t = lane & 3;
      for (int ct = warp; ct * 8 < n2; ct += nw) {
        uint2 bf[2][kDigits];
        int eb0, eb1;
        {
          double y[2][4];
          const T* uc = sU + min(ct * 8 + g, n2 - 1) * PT + 4 * t;
#pragma unroll
          for (int s = 0; s < 2; ++s) {
            lds16(uc + 16 * s, y[s]);
            lds16(uc + 16 * s + 2, y[s] + 2);
          }
          const int e = shared_exp<2, 3>(y);
#pragma unroll
          for (int s = 0; s < 2; ++s) split4(y[s], e, bf[s]);
          eb0 = __shfl_sync(0xffffffffu, e, 8 * t);
          eb1 = __shfl_sync(0xffffffffu, e, 8 * t + 4);
        }
        const int col = ct * 8 + 2 * t;
        for (int rt = 0; rt * 16 < n2; ++rt) {
          const int i0 = rt * 16 + g;
          double a[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + (u >> 1) * 8, j = col + (u & 1);
            a[u] = 0.0;
            if (i < n2 && j < n2) {
              const size_t at = (size_t)(j2 + j) * m + sOld[i];
              a[u] = p == 0 ? Db[at] : (double)Ab[at];
              if (p == 0) bad |= !f64_finite_bits(a[u]);
            }
          }
          const uint4* fa = reinterpret_cast<const uint4*>(sA + rt * kRowTile) + lane;
          double v[4];
          tile<true>(StagedA<2>{fa, bf}, sE[i0], sE[i0 + 8], eb0, eb1, v, [&](int u) {
            const int i = i0 + (u >> 1) * 8, j = col + (u & 1);
            double d = 0.0;
            if (i < n2 && j < n2)
#pragma unroll 8
              for (int k = 0; k < kPanel; ++k) d = fma((double)Ab[(size_t)(k0 + k) * m + j2 + i], (double)sU[j * PT + k], d);
            return d;
          });
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + (u >> 1) * 8, j = col + (u & 1);
            if (i < n2 && j < n2) Ab[(size_t)(j2 + j) * m + j2 + i] = a[u] - v[u];
          }
        }
        __syncwarp();
        for (int j = ct * 8; j < min(ct * 8 + 8, n2); ++j) Ab[(size_t)(j2 + j) * m + k0 + lane] = sU[j * PT + lane];
      }
    } else {
      for (int c0 = 0; c0 < n2; c0 += CB) {
        if (live && !pivot_row) {
          T a[CB];
#pragma unroll
          for (int c = 0; c < CB; ++c) {
            a[c] = T(0);
            if (c0 + c < n2) {
              const size_t at = (size_t)(j2 + c0 + c) * m + tid;
              if (p == 0) {
                const double v = Db[at];
                bad |= !f64_finite_bits(v);
                a[c] = conv<T>(v);
              } else {
                a[c] = Ab[at];
              }
            }
          }
#pragma unroll
          for (int c = 0; c < CB; ++c) {
            const T* uc = sU + min(c0 + c, n2 - 1) * PT;
#pragma unroll
            for (int l = 0; l < kPanel; l += V) {
              T uv[V];
              lds16(uc + l, uv);
#pragma unroll
              for (int q = 0; q < V; ++q) a[c] -= x[l + q] * uv[q];
            }
          }
#pragma unroll
          for (int c = 0; c < CB; ++c)
            if (c0 + c < n2) Ab[(size_t)(j2 + c0 + c) * m + pos] = a[c];
        }
      }
      __syncthreads();
      for (int j = warp; j < n2; j += nw) Ab[(size_t)(j2 + j) * m + k0 + lane] = sU[j * PT + lane];
    }
    if (p == 0 && bad) set_status(st, HODLR_ERR_NONFINITE, b, 0);
  }
  if (m <= kPanel && bad) set_status(st, HODLR_ERR_NONFINITE, b, 0);

  // earlier panels' rows into the final order: map = where the row at this
  // position after panel p ends
  int map = tid;
  for (int p = np - 1; p >= 0; --p) {
    __syncthreads();
    sMap[tid & 255] = (uint8_t)map;
    __syncthreads();
    map = tid < m ? sMap[sPerm[p][tid]] : tid;
    if (p == 0) break;
    if (!__syncthreads_or(map != tid)) continue;
    for (int c0 = (p - 1) * kPanel; c0 < p * kPanel; c0 += CB) {
      T a[CB];
      if (tid < m) {
#pragma unroll
        for (int c = 0; c < CB; ++c) a[c] = Ab[(size_t)(c0 + c) * m + tid];
      }
      __syncthreads();
      if (tid < m) {
#pragma unroll
        for (int c = 0; c < CB; ++c) Ab[(size_t)(c0 + c) * m + map] = a[c];
      }
    }
  }
  if (tid < m) perm[(size_t)b * m + map] = tid;
  if (tid == 0 && sing >= 0) set_status(st, HODLR_ERR_SINGULAR_LEAF, b, sing);
  // log|det D_b| and its sign, FP64
  if (tid < 32) {
    double la = 0.0;
    int neg = 0;
    for (int i = tid; i < m; i += 32) {
      const double u = sPiv[i];
      la += log(fabs(u));
      neg ^= (u < 0.0);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      la += __shfl_down_sync(0xffffffffu, la, off);
      neg ^= __shfl_down_sync(0xffffffffu, neg, off);
    }
    if (tid == 0) {
      leaf_ld[2 * b] = la;
      leaf_ld[2 * b + 1] = (sing >= 0) ? 0.0 : ((neg ^ swaps) ? -1.0 : 1.0);
    }
  }
}

template <typename T, int MAXT, int MINB>
static cudaError_t leaf_lu_go(const Factor& F, const double* D, cudaStream_t s) {
  const int m = F.d.m;
  const size_t sm = leaf_lu_smem<T>(m);
  cudaError_t e = cudaFuncSetAttribute(leaf_lu_kernel<T, MAXT, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sm);
  if (e != cudaSuccess) return e;
  leaf_lu_kernel<T, MAXT, MINB><<<1u << F.d.L, (m + 31) / 32 * 32, sm, s>>>(m, D, static_cast<T*>(F.lu), F.perm,
                                                                            F.leaf_ld, F.status);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_leaf_lu(const Factor& F, const double* D, cudaStream_t s) {
  ProfScope prof_(KC_LEAF_LU, s);
  if (leaf_uses_inverse(F)) return launch_leaf_inv(F, D, s);
  const int m = F.d.m;
  const double nleaf = (double)((int64_t)1 << F.d.L);
  const double e = F.prec == HODLR_PREC_FP64 ? 8.0 : 4.0;
  note_work((8.0 + e) * nleaf * m * m + 4.0 * nleaf * m, 2.0 / 3.0 * m * m * (double)m * nleaf);
  if (F.prec == HODLR_PREC_FP64) {
    const cudaError_t err = m <= 128 ? leaf_lu_go<double, 128, 2>(F, D, s) : leaf_lu_go<double, 256, 1>(F, D, s);
    return err != cudaSuccess ? err : launch_leaf_tinv(F, s);
  }
  return m <= 128 ? leaf_lu_go<float, 128, 4>(F, D, s) : leaf_lu_go<float, 256, 2>(F, D, s);
}

}  // namespace hodlr
