// FP64 products on the FP16 tensor cores.
//
// This GPU's FP64 pipe does 2 FMA per clock and SM (1.26 TFLOP/s), so every
// FP64 contraction of the library (projections, rank-r updates, leaf products)
// was bound by it while the memory system idled. Here an FP64 dot product is
// evaluated exactly up to a fixed-point grid finer than FP64's own rounding of
// it (the splitting of Ozaki et al., "Error-free transformations of matrix
// multiplication", Numer. Algorithms 59, 2012, with integer digits):
//
//   * every vector of the contraction (a row of A, a column of B, over a block
//     of at most 64 terms) gets the exponent e of its largest entry; an entry
//     x becomes the integer v, |v| < 2^62, x = v 2^(e - 1084) (exact for entries
//     within 2^9 of the largest, truncated below 2^-61 of its binade), written
//     in eight balanced base-256 digits, v = sum_i d_i 256^(7 - i),
//     -128 <= d_i <= 127, |d_0| <= 64;
//   * the digits are FP16 integers, and mma.sync m16n8k16 accumulates
//     c_d = sum_{i + j = d} A_i B_j for d = 0 .. 7 in FP32. |c_d| <= 7 * 2^14 *
//     64 < 2^24, so every accumulator holds its integer exactly (and below 2^22
//     for 32 terms);
//   * the eight integers are combined into one 63-bit integer in units of 2^-54 of the
//     smallest product that two largest entries can have (2^0 2^0 of their binades),
//     and rounded to FP64 on the integer pipe. The digit pairs with i + j = 8 are left
//     out: at worst 7 2^14 256^6 a term, 3.5 units for 32 terms, typically 0.1. With the
//     unit's rounding and the entries' truncation (2^-6 units a term) a sum is off by at
//     most 5 units (9 for 64 terms), typically by 0.3.
//   * That is within FP64's own rounding of a sum unless the vectors' large entries
//     do not meet. So one more mma a step adds up the products of the entries' leading 16
//     bits, s ~ sum |a| |b|. Where s is below 2^52 units (a quarter of that smallest
//     product of two largest entries) the pairs with i + j = 8 and the bits below the unit
//     are added, which leaves the entries' truncation: half a unit for 32 terms, typically
//     2^-5. Where s is below 2^48 units too the element is formed with FP64 FMAs.
//   * So no element is off by more than (n + 1) 2^-53 of its own sum |a| |b| over n terms,
//     one rounding above the bound of FP64 FMAs; root mean squares are at or below theirs
//     (tests/test_gpu_split.py has both). The second look is taken by none of the tiles
//     of normally distributed operands, by most of those on the diagonal of a dominant
//     leaf.
//
// The magnitudes' sums and the second look cost 1 to 3% (64 columns on N = 2^18, leaf 256,
// rank 32, both ways: 12.23 -> 12.39 ms) against looking only at small results.
//
// 36 digit products at the measured 935 FP16 MAC/clk/SM of mma.sync are 26
// FP64 MAC/clk/SM against the FP64 pipe's 2. Splitting costs about 28 integer
// operations per entry (64 per clock and SM), close to the 8 bytes per entry
// of HBM traffic; the rebuilt sum costs one FP64 addition. (Seven digits and 28
// products are a fifth cheaper, but their 2^-54 truncation of the largest
// product shows where one term dominates a row, as in diagonally dominant
// leaves: 1.8 times the rounding error of FMAs for 64-row leaves.)
//
// A vector with a non-finite entry, or whose largest entry lies outside
// [2^-400, 2^400], is left to the callers' FP64 loops (same result as plain
// FMAs), so infinities, NaN and extreme scales behave as in FP64 arithmetic.
#pragma once

#include "hodlr_internal.cuh"

namespace hodlr {
namespace split {

constexpr int kDigits = 8;
constexpr int kPlanes = 9;  // staged operands: the digits, then the magnitudes
constexpr int kMinExp = 1023 - 400, kMaxExp = 1023 + 400;  // biased exponents the digits cover

// Largest |x| of a vector so far, as the high word of its bits (ordered like |x|).
__device__ __forceinline__ uint32_t abs_hi(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }

// Exponent of a vector from the high word of its largest entry: kBadExp when the
// digits cannot represent it; `any_tiny` tells whether a vector below the range
// has a nonzero entry (an all-zero vector is exact, every digit is 0: kZeroExp).
// Both stand in sums of two exponents so that an element with a bad vector is
// always looked at again (finish_tile), one with a zero vector and no bad one never.
constexpr int kBadExp = 100000, kZeroExp = -4000;
__device__ __forceinline__ int vector_exp(uint32_t maxhi, bool any_tiny) {
  const int e = (int)(maxhi >> 20);
  if (e > kMaxExp || (e < kMinExp && any_tiny)) return kBadExp;
  return e < kMinExp ? kZeroExp : e;
}

// The biased digits of x in a vector of exponent e: byte 7 - i of the result
// holds d_i + 128.
__device__ __forceinline__ uint2 digits(double x, int e) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int sh = min(e - (int)((hi >> 20) & 0x7ffu), 63);  // zeros, denormals and bad vectors shift out
  uint64_t m = (((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | lo) << 9;
  m >>= sh;
  const int32_t s = (int32_t)hi >> 31;
  m ^= (uint64_t)(int64_t)s;
  m += 0x8080808080808080ull + (uint32_t)(s & 1);
  return make_uint2((uint32_t)m, (uint32_t)(m >> 32));
}

// Digit I of two entries as a pair of FP16 integers (x in the low half): the
// biased digit b < 256 under the exponent of 1024 is 1024 + b, less 1152.
template <int I>
__device__ __forceinline__ uint32_t digit_pair(uint2 x, uint2 y) {
  constexpr uint32_t sel = (I & 3) == 0 ? 0x0703 : (I & 3) == 1 ? 0x0602 : (I & 3) == 2 ? 0x0501 : 0x0400;
  uint32_t p = I < 4 ? __byte_perm(x.y, y.y, sel) : __byte_perm(x.x, y.x, sel);
  p = (p & 0x00ff00ffu) | 0x64006400u;
  uint32_t r;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(p), "r"(0x64806480u));
  return r;
}

// The digits of four consecutive terms, in the order of an mma fragment's
// k = (2t, 2t + 1 | 2t + 8, 2t + 9): out[i] = digit i of terms (0, 1), (2, 3).
__device__ __forceinline__ void split4(const double (&x)[4], int e, uint2 (&out)[kDigits]) {
  uint2 w[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) w[q] = digits(x[q], max(e, kMinExp));
#define HODLR_SPLIT_DIGIT(I) out[I] = make_uint2(digit_pair<I>(w[0], w[1]), digit_pair<I>(w[2], w[3]));
  HODLR_SPLIT_DIGIT(0)
  HODLR_SPLIT_DIGIT(1)
  HODLR_SPLIT_DIGIT(2)
  HODLR_SPLIT_DIGIT(3)
  HODLR_SPLIT_DIGIT(4)
  HODLR_SPLIT_DIGIT(5)
  HODLR_SPLIT_DIGIT(6)
  HODLR_SPLIT_DIGIT(7)
#undef HODLR_SPLIT_DIGIT
}

__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                        uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The FP64 value of the accumulators i[0 .. 7] of a row of exponent ea and a
// column of exponent eb (one rounding, to nearest).
// rest: what it rounds off, c_6 and c_7's part below the unit, in units of 256^7.
__device__ __forceinline__ double combine(const int (&i)[kDigits], int ea, int eb, int& rest) {
  const int p0 = i[0] * 256 + i[1], p1 = i[2] * 256 + i[3], p2 = i[4] * 256 + i[5], p3 = i[6] * 256 + i[7];
  int64_t t = (int64_t)p2 * 16 + ((p3 + 2048) >> 12);
  rest = ((p3 + 2048) & 4095) - 2048;
  t += (int64_t)p1 * (1 << 20);
  t += (int64_t)((uint64_t)(uint32_t)(p0 * 16) << 32);
  // t 2^(ea + eb - 2100), |t| < 2^63: normalize on the integer pipe
  const int32_t s = (int32_t)(t >> 63);
  uint64_t a = (uint64_t)(t ^ (int64_t)s) - (int64_t)s;
  if (a == 0) return 0.0;
  const int n = __clzll((int64_t)a);
  a <<= n;
  uint64_t b = (a >> 11) + ((uint64_t)(uint32_t)(ea + eb - 1015 - n) << 52);  // the leading 1 adds to the exponent
  b += (a >> 10) & 1u;
  return __longlong_as_double((int64_t)(b | ((uint64_t)(uint32_t)s & 0x80000000u) << 32));
}

__device__ __forceinline__ double combine_f32(const float (&c)[kDigits][4], int q, int ea, int eb, int& rest) {
  int i[kDigits];
#pragma unroll
  for (int d = 0; d < kDigits; ++d) i[d] = __float2int_rn(c[d][q]);
  return combine(i, ea, eb, rest);
}

// Accumulators started at 1.5 * 2^23 hold integers of at most 2^22 in their
// low significand bits (32 terms): no conversion is needed to read them.
constexpr float kMagic = 12582912.f;
__device__ __forceinline__ double combine_magic(const float (&c)[kDigits][4], int q, int ea, int eb, int& rest) {
  int i[kDigits];
#pragma unroll
  for (int d = 0; d < kDigits; ++d) i[d] = __float_as_int(c[d][q]) - 0x4B400000;
  return combine(i, ea, eb, rest);
}

// |leading 16 bits| of a pair of entries from its two first digits, as FP16 (11 bits).
__device__ __forceinline__ uint32_t magnitude(uint32_t d0, uint32_t d1) {
  uint32_t r;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(d0), "r"(0x5c005c00u), "r"(d1));  // 256 d0 + d1
  return r & 0x7fff7fffu;
}

__device__ __forceinline__ uint2 magnitudes(const uint2 (&d)[kDigits]) {
  return make_uint2(magnitude(d[0].x, d[1].x), magnitude(d[0].y, d[1].y));
}

// Digits and magnitudes of four entries to their planes, 512 bytes apart.
__device__ __forceinline__ void store_planes(unsigned char* dst, const uint2 (&d)[kDigits]) {
#pragma unroll
  for (int i = 0; i < kDigits; ++i) *reinterpret_cast<uint2*>(dst + i * 512) = d[i];
  *reinterpret_cast<uint2*>(dst + kDigits * 512) = magnitudes(d);
}

template <bool MAGIC>
__device__ __forceinline__ void clear_sums(float (&cd)[kDigits][4]) {
#pragma unroll
  for (int d = 0; d < kDigits; ++d)
#pragma unroll
    for (int u = 0; u < 4; ++u) cd[d][u] = MAGIC ? kMagic : 0.f;
}

// The same value to the program, another one to the compiler: what is loaded or
// computed from it is not kept from an earlier use (kept fragments of a rare branch
// spilled the products' registers).
template <typename T>
__device__ __forceinline__ const T* again(const T* p) {
  asm volatile("" : "+l"(p));
  return p;
}

// A tile's operands: A staged in planes of (a0, a2 | a1, a3) per k16 step and lane, B
// split in registers.
template <int NK>
struct StagedA {
  const uint4* fa;
  const uint2 (&bf)[NK][kDigits];
  __device__ __forceinline__ void products(float (&cd)[kDigits][4]) const {
#pragma unroll
    for (int s = 0; s < NK; ++s) {
#pragma unroll
      for (int i = 0; i < kDigits; ++i) {
        const uint4 f = fa[(s * kPlanes + i) * 32];
#pragma unroll
        for (int j = 0; j + i < kDigits; ++j) mma_f16(cd[i + j], f.x, f.z, f.y, f.w, bf[s][j].x, bf[s][j].y);
      }
    }
  }
  __device__ __forceinline__ void sums(float (&mg)[4]) const {
#pragma unroll
    for (int s = 0; s < NK; ++s) {
      const uint4 f = fa[(s * kPlanes + kDigits) * 32];
      const uint2 b = magnitudes(bf[s]);
      mma_f16(mg, f.x, f.z, f.y, f.w, b.x, b.y);
    }
  }
  __device__ __forceinline__ void eighth(float (&c)[4]) const {
    const uint4* fr = again(fa);
#pragma unroll
    for (int s = 0; s < NK; ++s)
#pragma unroll
      for (int i = 1; i < kDigits; ++i) {
        const uint4 f = fr[(s * kPlanes + i) * 32];
        mma_f16(c, f.x, f.z, f.y, f.w, bf[s][kDigits - i].x, bf[s][kDigits - i].y);
      }
  }
};

// A split in registers ([k16 step][fragment row g, g + 8]), B staged in planes of
// (b0, b1) of two k16 steps per lane.
template <int KB>
struct StagedB {
  const uint2 (&af)[2 * KB][2][kDigits];
  const uint4* fb;
  __device__ __forceinline__ void products(float (&cd)[kDigits][4]) const {
#pragma unroll
    for (int kb = 0; kb < KB; ++kb) {
      const uint2(&p)[2][kDigits] = af[2 * kb];
      const uint2(&q)[2][kDigits] = af[2 * kb + 1];
#pragma unroll
      for (int j = 0; j < kDigits; ++j) {
        const uint4 f = fb[(kb * kPlanes + j) * 32];
#pragma unroll
        for (int i = 0; i + j < kDigits; ++i) mma_f16(cd[i + j], p[0][i].x, p[1][i].x, p[0][i].y, p[1][i].y, f.x, f.y);
#pragma unroll
        for (int i = 0; i + j < kDigits; ++i) mma_f16(cd[i + j], q[0][i].x, q[1][i].x, q[0][i].y, q[1][i].y, f.z, f.w);
      }
    }
  }
  __device__ __forceinline__ void sums(float (&mg)[4]) const {
#pragma unroll
    for (int kb = 0; kb < KB; ++kb) {
      const uint2(&p)[2][kDigits] = af[2 * kb];
      const uint2(&q)[2][kDigits] = af[2 * kb + 1];
      const uint4 f = fb[(kb * kPlanes + kDigits) * 32];
      const uint2 p0 = magnitudes(p[0]), p1 = magnitudes(p[1]), q0 = magnitudes(q[0]), q1 = magnitudes(q[1]);
      mma_f16(mg, p0.x, p1.x, p0.y, p1.y, f.x, f.y);
      mma_f16(mg, q0.x, q1.x, q0.y, q1.y, f.z, f.w);
    }
  }
  __device__ __forceinline__ void eighth(float (&c)[4]) const {
    const uint4* fr = again(fb);
#pragma unroll
    for (int kb = 0; kb < KB; ++kb) {
      const uint2(&p)[2][kDigits] = af[2 * kb];
      const uint2(&q)[2][kDigits] = af[2 * kb + 1];
#pragma unroll
      for (int i = 1; i < kDigits; ++i) {
        const uint4 f = fr[(kb * kPlanes + kDigits - i) * 32];
        mma_f16(c, p[0][i].x, p[1][i].x, p[0][i].y, p[1][i].y, f.x, f.y);
        mma_f16(c, q[0][i].x, q[1][i].x, q[0][i].y, q[1][i].y, f.z, f.w);
      }
    }
  }
};

// The four elements of an accumulator tile: rows of exponents ea0, ea1 (fragment
// rows g, g + 8), columns of exponents eb0, eb1 (2t, 2t + 1); element u is row
// u >> 1, column u & 1. sums(mg) adds up the magnitudes' products (after the digit
// sums are combined: their registers are free by then), eighth(c) the digit pairs with
// i + j = 8; dot(u) is an element in FP64. Called by whole warps.
// Sums below kDirect (2^52 units) get the missing digits, below kFine (2^48) FMAs.
constexpr float kDirect = 16777216.f, kFine = 1048576.f;
template <bool MAGIC, class Sums, class Eighth, class Dot>
__device__ __forceinline__ void finish_tile(const float (&cd)[kDigits][4], int ea0, int ea1, int eb0, int eb1,
                                            double (&v)[4], Sums sums, Eighth eighth, Dot dot) {
  int rest[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int ea = u < 2 ? ea0 : ea1, eb = (u & 1) ? eb1 : eb0;
    v[u] = MAGIC ? combine_magic(cd, u, ea, eb, rest[u]) : combine_f32(cd, u, ea, eb, rest[u]);
  }
  float mg[4] = {0.f, 0.f, 0.f, 0.f};
  sums(mg);
  bool low[4], any = false;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    low[u] = mg[u] < kDirect && (u < 2 ? ea0 : ea1) + ((u & 1) ? eb1 : eb0) > 0;  // a zero vector (kZeroExp) is exact
    any |= low[u];
  }
  if (__any_sync(0xffffffffu, any)) {
    float c8[4] = {0.f, 0.f, 0.f, 0.f};
    eighth(c8);
    any = false;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = (u < 2 ? ea0 : ea1) + ((u & 1) ? eb1 : eb0);
      // |v| < 2^53 units: no rounding so far; the rest in units of 256^6, below 2^25
      if (low[u]) v[u] = fma((double)(rest[u] * 256 + __float2int_rn(c8[u])), __hiloint2double((e - 1097) << 20, 0), v[u]);
      low[u] = low[u] && mg[u] < kFine;
      any |= low[u];
    }
    if (!__any_sync(0xffffffffu, any)) return;
#pragma unroll 1
    for (int u = 0; u < 4; ++u) {
      if (__any_sync(0xffffffffu, low[0])) {
        const double d = low[0] ? dot(u) : 0.0;
        if (low[0]) v[0] = d;
      }
      // the next element to the front (static register indices)
      const double vf = v[0];
      const bool lf = low[0];
#pragma unroll
      for (int w = 0; w < 3; ++w) {
        v[w] = v[w + 1];
        low[w] = low[w + 1];
      }
      v[3] = vf;
      low[3] = lf;
    }
  }
}

// Products and elements of one tile.
template <bool MAGIC, class Operands, class Dot>
__device__ __forceinline__ void tile(const Operands& op, int ea0, int ea1, int eb0, int eb1, double (&v)[4], Dot dot) {
  float cd[kDigits][4];
  clear_sums<MAGIC>(cd);
  op.products(cd);
  finish_tile<MAGIC>(cd, ea0, ea1, eb0, eb1, v, [&](float (&mg)[4]) { op.sums(mg); },
                     [&](float (&c)[4]) { op.eighth(c); }, dot);
}

template <typename TB>
__device__ __forceinline__ double to_d(TB v) { return (double)v; }

// Four consecutive entries p[0 .. 3], those at or beyond `left` zero.
template <typename TB>
__device__ __forceinline__ void load_run4(const TB* p, int64_t left, bool vec, double (&x)[4]) {
  if (vec && left >= 4) {
    load4(p, x);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) x[q] = q < left ? to_d(p[q]) : 0.0;
  }
}
template <int NR>
__device__ __forceinline__ bool any_nonzero(const double (&x)[NR][4]) {
  bool b = false;
#pragma unroll
  for (int s = 0; s < NR; ++s)
#pragma unroll
    for (int q = 0; q < 4; ++q) b |= x[s][q] != 0.0;
  return b;
}

// Exponent of the vector whose entries are spread over the lanes that differ
// in the bits of LANES (power of two minus one, contiguous low bits).
template <int NR, int LANES>
__device__ __forceinline__ int shared_exp(const double (&x)[NR][4]) {
  uint32_t mh = 0;
#pragma unroll
  for (int s = 0; s < NR; ++s)
#pragma unroll
    for (int q = 0; q < 4; ++q) mh = max(mh, abs_hi(x[s][q]));
#pragma unroll
  for (int o = 1; o <= LANES / 2 + 1; o <<= 1) mh = max(mh, __shfl_xor_sync(0xffffffffu, mh, o));
  bool tiny = false;
  if (__any_sync(0xffffffffu, (mh >> 20) < (uint32_t)kMinExp)) {  // rare: an all-zero vector or a tiny one
    tiny = any_nonzero(x);
#pragma unroll
    for (int o = 1; o <= LANES / 2 + 1; o <<= 1) tiny |= __shfl_xor_sync(0xffffffffu, (int)tiny, o) != 0;
  }
  return vector_exp(mh, tiny);
}

}  // namespace split
}  // namespace hodlr
