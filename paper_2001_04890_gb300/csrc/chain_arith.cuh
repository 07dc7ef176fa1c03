// Element types and inner products of the triple products on the CUDA cores (sm_103a).
//
// FP64 products in fixed point.  The FP64 pipe of this GPU issues 2 multiply-adds per
// SM and clock (measured; FP64 mma.sync 1.75), the integer pipe 32 32 x 32 + 64 bit
// ones (a multiply and an addition; measured, see mad()).  So a tile of doubles is read as a block-scaled
// integer matrix: x = v 2^(E - 1079) with E the largest biased exponent of the tile
// and v a rounded integer, |v| < 2^57, kept as two signed limbs v = hi 2^29 + lo, |hi|, |lo| <= 2^28.
// A dot product accumulates sum hi hi' and sum (hi lo' + lo hi') exactly in two 64-bit
// registers: three multiply-adds per element product, the lo lo' term (2^-58 of the largest
// product at most, of either sign) dropped.  For a depth of 32 |sum hi hi'| <= 2^61 and
// |sum cross| <= 2^62.  The intermediate T = X Y is normalised back to 57 bits under an
// exponent of its own.  The sum over tasks is FP64, as f may be any double.
//
// The error is relative to a tile's largest elements: n 2^-55 max|X| max|Y| for a sum of n products
// (tests/test_gpu_products.py has the terms), where FP64 has n 2^-53 times the sum of |x| |y|.  An
// element below 2^-5 of its tile's largest has fewer than 53 bits, one below 2^-58 is zero.
//
// A tile with a NaN, an infinity or a largest element outside 2^+-256 is multiplied in FP64
// instead (slow paths of the kernels), so those values propagate as in FP64 arithmetic.
//
// FP32 elements: one FP32 multiply-add per element product.
#pragma once

#include <climits>
#include <cstdint>
#include <cuda_runtime.h>

namespace dmrg {

constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------- element types

// FX: 57-bit block-scaled integers in two limbs (from FP64), 8 bytes.
// else: FP32, 4 bytes.
template <bool FX>
struct Arith;

template <>
struct Arith<true> {
  using Elem = int2;
  using Out = double;
  static constexpr int VK = 2;  // elements per 128-bit shared load
  static constexpr int PAD = 2;  // row pitch TS + PAD
};

template <>
struct Arith<false> {
  using Elem = float;
  using Out = float;
  static constexpr int VK = 4;
  static constexpr int PAD = 4;
};

// t in [0, 1024), d in [1, 32]: t / d
__device__ __forceinline__ int small_div(int t, float inv) { return (int)(((float)t + 0.5f) * inv); }

__device__ __forceinline__ int2 limbs(long long v) {
  return make_int2((int)((v + (1ll << 28)) >> 29), (int)((unsigned)v << 3) >> 3);
}
__device__ __forceinline__ long long join(int2 v) { return ((long long)v.x << 29) + v.y; }

// the integer of x, |v| < 2^57, under tile exponent E (E >= x's own exponent field)
__device__ __forceinline__ int2 to_limbs(double x, int E) {
  const int h = __double2hiint(x);
  const int ex = (h >> 20) & 0x7ff;
  const unsigned mh = ((unsigned)h & 0xfffffu) | (ex ? 0x100000u : 0u);
  const unsigned long long m = ((unsigned long long)mh << 32 | (unsigned)__double2loint(x)) << 9;
  const int sh = min(E - ex + 4, 63);
  const unsigned long long v = ((m >> sh) + 1ull) >> 1;  // rounded to nearest
  const unsigned long long w = v + (1ull << 28);
  const int s = h >> 31;
  const int hi = (int)(w >> 29), lo = (int)((unsigned)w & 0x1fffffffu) - (1 << 28);
  return make_int2((hi ^ s) - s, (lo ^ s) - s);
}

__device__ __forceinline__ double limbs_to_double(int2 v, int e) {
  return scalbn((double)join(v), e);
}

// What a tile's elements allow: the largest |high word|, or an escape to FP64.
struct TileMax {
  unsigned hi = 0, any = 0;
  __device__ __forceinline__ void add(double x) {
    const unsigned h = (unsigned)__double2hiint(x) & 0x7fffffffu;
    hi = max(hi, h);
    any |= h | (unsigned)__double2loint(x);
  }
};
// The exponent of a tile: that of its largest element, -1 if fixed point does not take it, 0 if
// every element is zero.  Scale factors are made of exponents by integer additions to the exponent
// field and stay normal numbers for any that lie within 2^+-256; zero_as_one() gives them one for
// a tile of zeros, whose integers are zero under any exponent.
__device__ __forceinline__ int tile_exponent(unsigned hi, unsigned any) {
  const int E = (int)(hi >> 20);
  return any == 0u ? 0 : E > 1023 + 256 || E < 1023 - 256 ? -1 : E;
}
__device__ __forceinline__ int zero_as_one(int E) { return E == 0 ? 1023 : E; }

template <int TS>
struct Shift {
  // sums of at most TS products of |hi| <= 2^28: the top bits that stay free
  static constexpr int value = TS == 32 ? 1 : 2;
};

// hh 2^58 + cr 2^29 as a 64-bit integer in units of 2^(58 - s)
template <int S>
__device__ __forceinline__ long long fold(long long hh, long long cr) {
  return (hh << S) + ((cr + (1ll << (28 - S))) >> (29 - S));
}
// d += a b.  A loop of nothing but mad.wide.s32 on the same operands measured 63 per SM and clock,
// this form 32; but with mad.wide.s32 here the general kernel was slower (14 orbitals, M 1200 and
// 300: 42.2 against 37.0 ms; M 1600 and 500: 85.9 against 73.7 ms).
__device__ __forceinline__ void mad(long long &d, int a, int b) {
  asm("{\n\t.reg .s64 q;\n\tmul.wide.s32 q, %1, %2;\n\tadd.s64 %0, %0, q;\n\t}" : "+l"(d) : "r"(a), "r"(b));
}

// ---------------------------------------------------------------- inner products

// acc[a][b] += sum_k A[4a][k] B[8b][k] over the rows a < na; A and B point at this
// lane's first row and column.
template <int P, int NB>
__device__ __forceinline__ void mm(const int2 *A, const int2 *B, int kc, int na, long long (&hh)[4][NB],
                                   long long (&cr)[4][NB]) {
  for (int k = 0; k < kc; k += 2) {
    int4 y[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) y[b] = *reinterpret_cast<const int4 *>(B + 8 * b * P + k);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      if (a < na) {
        const int4 x = *reinterpret_cast<const int4 *>(A + 4 * a * P + k);
#pragma unroll
        for (int b = 0; b < NB; ++b) mad(hh[a][b], x.x, y[b].x);
#pragma unroll
        for (int b = 0; b < NB; ++b) mad(cr[a][b], x.x, y[b].y);
#pragma unroll
        for (int b = 0; b < NB; ++b) mad(hh[a][b], x.z, y[b].z);
#pragma unroll
        for (int b = 0; b < NB; ++b) mad(cr[a][b], x.y, y[b].x);
#pragma unroll
        for (int b = 0; b < NB; ++b) mad(cr[a][b], x.z, y[b].w);
#pragma unroll
        for (int b = 0; b < NB; ++b) mad(cr[a][b], x.w, y[b].z);
      }
    }
  }
}

template <int P, int NB>
__device__ __forceinline__ void mm(const float *A, const float *B, int kc, int na, float (&s)[4][NB]) {
  for (int k = 0; k < kc; k += 4) {
    float4 y[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) y[b] = *reinterpret_cast<const float4 *>(B + 8 * b * P + k);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      if (a < na) {
        const float4 x = *reinterpret_cast<const float4 *>(A + 4 * a * P + k);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          s[a][b] = fmaf(x.x, y[b].x, s[a][b]);
          s[a][b] = fmaf(x.y, y[b].y, s[a][b]);
          s[a][b] = fmaf(x.z, y[b].z, s[a][b]);
          s[a][b] = fmaf(x.w, y[b].w, s[a][b]);
        }
      }
    }
  }
}

// acc[a][b] += sum_k A[4a][k] B[8b][k] for a < NA and b < NB; row pitches pa and pb
template <int NA, int NB, int NAT, int NBT>
__device__ __forceinline__ void mm_acc(const float *A, int pa, const float *B, int pb, int kc,
                                       float (&acc)[NAT][NBT]) {
  pa *= 4;
  pb *= 8;
#pragma unroll 1
  for (int k = 0; k < kc; k += 4, A += 4, B += 4) {
    float4 y[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) y[b] = *reinterpret_cast<const float4 *>(B + b * pb);
#pragma unroll
    for (int a = 0; a < NA; ++a) {
      const float4 x = *reinterpret_cast<const float4 *>(A + a * pa);
#pragma unroll
      for (int b = 0; b < NB; ++b) acc[a][b] = fmaf(x.x, y[b].x, acc[a][b]);
#pragma unroll
      for (int b = 0; b < NB; ++b) acc[a][b] = fmaf(x.y, y[b].y, acc[a][b]);
#pragma unroll
      for (int b = 0; b < NB; ++b) acc[a][b] = fmaf(x.z, y[b].z, acc[a][b]);
#pragma unroll
      for (int b = 0; b < NB; ++b) acc[a][b] = fmaf(x.w, y[b].w, acc[a][b]);
    }
  }
}

// for the na <= 4 row groups and nb <= NBT column groups that hold outputs
template <int NB, int NBT>
__device__ __forceinline__ void mm_rows(const float *A, int pa, const float *B, int pb, int kc, int na,
                                        float (&acc)[4][NBT]) {
  if (na == 1) mm_acc<1, NB>(A, pa, B, pb, kc, acc);
  else if (na == 2) mm_acc<2, NB>(A, pa, B, pb, kc, acc);
  else if (na == 3) mm_acc<3, NB>(A, pa, B, pb, kc, acc);
  else mm_acc<4, NB>(A, pa, B, pb, kc, acc);
}
template <int NBT>
__device__ __forceinline__ void mm_any(const float *A, int pa, const float *B, int pb, int kc, int na, int nb,
                                       float (&acc)[4][NBT]) {
  if constexpr (NBT == 2) {
    if (nb == 1) mm_rows<1>(A, pa, B, pb, kc, na, acc);
    else mm_rows<2>(A, pa, B, pb, kc, na, acc);
  } else {
    if (nb == 1) mm_rows<1>(A, pa, B, pb, kc, na, acc);
    else if (nb == 2) mm_rows<2>(A, pa, B, pb, kc, na, acc);
    else if (nb == 3) mm_rows<3>(A, pa, B, pb, kc, na, acc);
    else mm_rows<4>(A, pa, B, pb, kc, na, acc);
  }
}

__device__ __forceinline__ unsigned magnitude(long long t) { return (unsigned)((t ^ (t >> 63)) >> 32); }

// f 2^e for an f whose exponent is moderate (|e| stays below 1000, see tile_exponent)
__device__ __forceinline__ double scaled(double f, int e) {
  return __hiloint2double(__double2hiint(f) + (e << 20), __double2loint(f));
}

__device__ __forceinline__ double muladd(double s, int2 v, double d) {
  return fma(s, (double)join(v), d);
}

}  // namespace dmrg
