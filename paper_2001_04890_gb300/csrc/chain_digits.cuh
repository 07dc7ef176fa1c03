// Digit images of FP64 blocks for chain_mma.cu: what an element becomes and where it lies.
#pragma once

#include <cstdint>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace dmrg {

// An image of an R x K block is cut into 8 x 16 blocks, those of the same 16 columns below one
// another, zeros to their edges.  A block holds what the 32 lanes of a warp take into their
// registers: for each of the six digits the pairs r0 (columns 2 t, 2 t + 1, t = lane % 4) and r1
// (2 t + 8, 2 t + 9) of row lane / 4.  Digits 2 v and 2 v + 1 make up vector v of a lane.  In
// the images of operators, which are the multiply's 16-row operand, two blocks that make up 16
// rows lie together: vector d of a lane is (r0, r0 of row + 8, r1, r1 of row + 8) of digit d,
// the four registers that the instruction takes.  12 bytes an element.
constexpr int kDigBlock = 1536;  // bytes of a block

__host__ __device__ constexpr int64_t dig_image_size(int R, int K) {  // in units of 8 bytes
  return (int64_t)((R + 7) / 8) * ((K + 15) / 16) * (kDigBlock / 8);
}

// the integer of x under block exponent E (E >= x's own exponent field): |v| < 2^58
__device__ __forceinline__ long long to_fixed(double x, int E) {
  const int h = __double2hiint(x);
  const int ex = (h >> 20) & 0x7ff;
  const unsigned mh = ((unsigned)h & 0xfffffu) | (ex ? 0x100000u : 0u);
  const unsigned long long m = ((unsigned long long)mh << 32 | (unsigned)__double2loint(x)) << 9;
  const long long v = (long long)(((m >> min(E - ex + 3, 63)) + 1ull) >> 1);  // rounded to nearest
  return h < 0 ? -v : v;
}

// The balanced digits (base 2^10, most significant first) of two integers |v| <= 2^58 as pairs
// of FP16.  With 512 added to each digit they are fields of 10 bits; 0x6400 | field is 1024 +
// field in FP16.
constexpr unsigned long long kDigBias =
    512ull * (1ull + (1ull << 10) + (1ull << 20) + (1ull << 30) + (1ull << 40) + (1ull << 50));
__device__ __forceinline__ void digits2(long long v, long long w, uint32_t (&d)[6]) {
  const unsigned long long a = (unsigned long long)v + kDigBias, b = (unsigned long long)w + kDigBias;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const unsigned x = (unsigned)(a >> (10 * (5 - i))), y = (unsigned)(b >> (10 * (5 - i)));
    const uint32_t bits = (__byte_perm(x, y, 0x5410) & 0x03ff03ffu) | 0x64006400u;
    const __half2 r = __hsub2(*reinterpret_cast<const __half2 *>(&bits), __half2half2(__ushort_as_half(0x6600)));
    d[i] = *reinterpret_cast<const uint32_t *>(&r);
  }
}

// The image of an R x K block whose element (r, k) is the integer get(r, k), by nthr threads;
// OPERATOR: blocks that make up 16 rows lie together.
template <bool OPERATOR, class Get>
__device__ __forceinline__ void write_digits(void *dst, int R, int K, int tid, int nthr, Get get) {
  const int step = OPERATOR ? 16 : 8;
  const int nr = (R + step - 1) / step, nb = (R + 7) / 8, n = nr * ((K + 15) / 16) * 32;
  for (int i = tid; i < n; i += nthr) {
    const int lane = i & 31, grp = (i >> 5) % nr, kc = (i >> 5) / nr;
    const int r = grp * step + (lane >> 2), k = kc * 16 + 2 * (lane & 3);
    uint32_t d[2][2][6];  // [row + 8][columns + 8]
#pragma unroll
    for (int h = 0; h < (OPERATOR ? 2 : 1); ++h)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int rr = r + 8 * h, kk = k + 8 * c;
        digits2(rr < R && kk < K ? get(rr, kk) : 0ll, rr < R && kk + 1 < K ? get(rr, kk + 1) : 0ll, d[h][c]);
      }
    uint4 *p = reinterpret_cast<uint4 *>(static_cast<char *>(dst) + (int64_t)(kc * nb + grp * (step / 8)) * kDigBlock) + lane;
    if (OPERATOR && R - grp * 16 > 8) {
#pragma unroll
      for (int u = 0; u < 6; ++u) p[32 * u] = make_uint4(d[0][0][u], d[1][0][u], d[0][1][u], d[1][1][u]);
    } else {
#pragma unroll
      for (int u = 0; u < 3; ++u)
        p[32 * u] = make_uint4(d[0][0][2 * u], d[0][1][2 * u], d[0][0][2 * u + 1], d[0][1][2 * u + 1]);
    }
  }
}

}  // namespace dmrg
