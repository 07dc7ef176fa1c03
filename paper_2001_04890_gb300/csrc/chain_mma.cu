// FP64 triple products of H.psi on the FP16 tensor pipe (sm_103a): D = sum_e f_e X_e Y_e Z_e
// over prepared operands (Sec. 2.2.1, Eq. dgemm).
//
// The FP64 pipe issues 2 multiply-adds per SM and clock, the integer pipe 10 products of 57-bit
// integers in two limbs (32 multiply-adds of 32 x 32 + 64 bits), the FP16 tensor pipe 1011
// products (mma.sync, all measured): at 26 per product of 58 bits, 39.  tcgen05 has 64 rows at
// least and no FP64 or wide integer form; the blocks here have 1 to 120, most below 32, and the
// 16 x 8 tile of mma.sync wastes less of them than its rate loses.
//
// Arithmetic (splitting into digits whose products add up without error: Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59, 2012).  A block is read as x = v 2^(E - 1080) with E its largest
// biased exponent and v an integer, |v| < 2^58, and v as six balanced digits in base 2^10,
// v = sum_i d_i 2^(10 (5 - i)), |d_i| <= 512, |d_0| <= 256.  Digits are exact in FP16, their
// products are integers of at most 2^18, and FP32 sums of integers are exact up to 2^24.  So 26
// multiplications with FP32 accumulators give the sums G_o = sum_(i+j=o) D_i D'_j, o = 0..6, over a
// depth of 16 (|G_0| to |G_4| are at most 2^24; G_5 and G_6 reach 1.25 2^24, where an FP32 sum
// is off by 2 at most, 2^-9 of a unit of the sum below).  After each depth of 16 the G are added
// up in one 64-bit integer in units of 2^60, below 2^63 for inner dimensions up to kPipeMaxN: the
// FP32 sum of G_4 and below rounds by one unit, what is left out (o > 6) is 2^-6 of one.  T = X Y
// goes back to 58 bits under an exponent of its own per 8 rows and 16 columns, and the sum over
// tasks is FP64.
//
// So the error is relative to the blocks' largest elements (tests/test_gpu_products.py has the
// bound and, for the digit orders and the longest sums, the worst cases).  Against H psi in 80
// bits at 10 orbitals, M 120, relative 2-norm: 5.0e-16 for the ground state (FP64 products
// 5.7e-16), 1.14e-15 for a random psi (1.18e-15); element by element within a block, elements
// 1 to 12 decades below the largest, the median errors are FP64's too (1.0e-15 and 1.1e-15 one decade
// below, 8.9e-9 and 9.1e-9 eight decades below): the sums that make up a small element have terms
// as large as those of a large one.  A vector for which that does not hold loses what lies
// below 2^-58 of a block's largest element.
//
// Data path.  The operands' images (chain_digits.cuh) are stored in the order of the multiply's
// registers, so a lane's share of an 8 x 16 block is three 128-bit loads and digits need no shared
// memory, no transposition and no barrier; lines are asked for one task ahead.  T comes out of the
// first product in the layout that the second one takes as its B operand, so for up to 32
// columns it never leaves the registers: D^T = sum Z^T T^T.  It is made 16 columns at a time:
// the sums of 32 want registers that the second product needs (24 orbitals, M 512: 8.7 against
// 8.2 ms, 12, M 800: 18.0 against 15.9 ms at equal occupancy), though D is then added to twice as
// often.
//
// What bounds it: latency.  206 to 310 instructions a multiply of 26 (sums to integers, digits of T, D)
// keep the tensor pipe 24 to 33% busy at the 3 to 4 warps a scheduler that registers allow.  Blocks are padded
// to 16 x 8 x 8: a third of the products at 24 orbitals, M 512, are of the problem.
//
// Time per H psi, limbs on the integer pipe -> this: 8 orbitals, M 64: 196 -> 178 us; 11, M 150:
// 585 -> 353 us; 24, M 512: 11.2 -> 7.6 ms; 12, M 800: 23.1 -> 14.9 ms.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>

#include "chain_arith.cuh"
#include "chain_digits.cuh"
#include "kernels.cuh"

namespace dmrg {

namespace {

__device__ __forceinline__ void prefetch(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// c + a b for 16 rows, 8 columns and a depth of 16, or 8 (HALF)
template <bool HALF>
__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2],
                                    float c0, float c1, float c2, float c3) {
  if constexpr (HALF)
    asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%7,%8,%9,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(b[0]), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
  else
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}

// this lane's share of an 8 x 16 block: digits d, registers r (columns 2t.. and 2t + 8..)
__device__ __forceinline__ void load_block(const char *p, int lane, uint32_t (&b)[6][2]) {
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    const uint4 x = *reinterpret_cast<const uint4 *>(p + v * 512 + lane * 16);
    b[2 * v][0] = x.x;
    b[2 * v][1] = x.y;
    b[2 * v + 1][0] = x.z;
    b[2 * v + 1][1] = x.w;
  }
}
// 16 x 16 of an operator: blocks that lie together, or (full = false) one block of at most 8 rows
// and, if have, another one's
__device__ __forceinline__ void load_rows(const char *p, bool full, const char *hi, bool have, int lane,
                                          uint32_t (&a)[6][4]) {
  if (full) {
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      const uint4 x = *reinterpret_cast<const uint4 *>(p + d * 512 + lane * 16);
      a[d][0] = x.x;
      a[d][1] = x.y;
      a[d][2] = x.z;
      a[d][3] = x.w;
    }
  } else {
    uint32_t x[6][2], y[6][2] = {};
    load_block(p, lane, x);
    if (have) load_block(hi, lane, y);
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      a[d][0] = x[d][0];
      a[d][1] = y[d][0];
      a[d][2] = x[d][1];
      a[d][3] = y[d][1];
    }
  }
}

// 1.5 2^23: the low bits of its sum with an integer below 2^22 are that integer.  G_0 and G_1 start
// from it, which saves them a conversion; the sum begins with what it adds taken off.
constexpr float kMagic = 12582912.f;
constexpr unsigned long long kMagicBits = 0x4b400000ull;
constexpr unsigned long long kMagicSum = (kMagicBits << 40) + (kMagicBits << 30);

template <bool HALF>
__device__ __forceinline__ void sums(const uint32_t (&a)[6][4], const uint32_t (&b)[6][2], float (&g)[7][4]) {
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const int o = i + j;
      if (o > 6) continue;
      if (i == 0 || (i == 1 && j == 5)) {
        const float c = o < 2 ? kMagic : 0.f;
        mma<HALF>(g[o], a[i], b[j], c, c, c, c);
      } else {
        mma<HALF>(g[o], a[i], b[j], g[o][0], g[o][1], g[o][2], g[o][3]);
      }
    }
}

// s = a b (16 rows, 8 columns) over a depth of 16, or 8 (half)
__device__ __forceinline__ void multiply(const uint32_t (&a)[6][4], const uint32_t (&b)[6][2], bool half,
                                         long long (&s)[4]) {
  float g[7][4];
  if (half) sums<true>(a, b, g);
  else sums<false>(a, b, g);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    s[e] = (long long)(0ull - kMagicSum);
    // units of 2^60: G_0 2^40 + G_1 2^30 + G_2 2^20 + G_3 2^10 + (G_4 + G_5 2^-10 + G_6 2^-20)
    s[e] += __float2int_rn(fmaf(fmaf(g[6][e], 0x1p-10f, g[5][e]), 0x1p-10f, g[4][e]));
    s[e] += (long long)__float2int_rn(g[3][e]) << 10;
    s[e] += (long long)__float2int_rn(g[2][e]) << 20;
    s[e] += (long long)__float_as_int(g[1][e]) << 30;
    const unsigned hi = (unsigned)(s[e] >> 32) + (__float_as_uint(g[0][e]) << 8);
    s[e] = (long long)((unsigned long long)hi << 32 | (unsigned)s[e]);
  }
}

// Digits of 8 rows and 16 columns of T: t[j][OFF + i] = column 8 j + 2 (lane & 3) + i of row lane / 4;
// out = the block as load_block gives it.  Returns the shift that took T to 58 bits.
template <int OFF>
__device__ __forceinline__ int digits_of(const long long (&t)[2][4], uint32_t (&out)[6][2]) {
  unsigned mx = 0;
#pragma unroll
  for (int j = 0; j < 2; ++j) mx = max(mx, max(magnitude(t[j][OFF]), magnitude(t[j][OFF + 1])));
  mx = __reduce_max_sync(kFull, mx);
  const int up = __clz(mx | 1) - 6;
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    long long v = t[j][OFF], w = t[j][OFF + 1];
    if (up >= 0) {
      v <<= up;
      w <<= up;
    } else {
      const long long half = 1ll << (-up - 1);
      v = (v + half) >> -up;
      w = (w + half) >> -up;
    }
    uint32_t d[6];
    digits2(v, w, d);
#pragma unroll
    for (int i = 0; i < 6; ++i) out[i][j] = d[i];
  }
  return up;
}

// The stacks of an item that fixed point does not take, in FP64 from the operators; added to
// the item's output, which the kernel has written.
__device__ __noinline__ void slow_stacks(const PipeEntry *P, const PipeStack *S, int nst, const ChainEntry *E,
                                         const int *pexp, const double *psi, const ChainGroup *gp, int r0, int c0,
                                         int rows, int cols, uint64_t db, double *T) {
  const ChainGroup g = *gp;
  const int tid = threadIdx.x, nthr = blockDim.x;
  double *D = reinterpret_cast<double *>(db + g.d * 8ull);
  for (int st = 0; st < nst; ++st) {
    if (!S[st].flags && pexp[S[st].yb] >= 0) continue;
    for (int i = S[st].e; i < S[st].e + S[st].ns; ++i) {
      const ChainEntry e = E[P[i].src];
      const bool xi = e.x == ~0ull, zi = e.z == ~0ull;
      const double *X = reinterpret_cast<const double *>(e.x * 8ull), *Y = psi + e.y;
      const double *Z = reinterpret_cast<const double *>(e.z * 8ull);
      for (int p0 = 0; p0 < e.p; p0 += 16) {
        const int pc = min(16, e.p - p0);
        __syncthreads();
        for (int t = tid; t < rows * pc; t += nthr) {
          const int64_t r = r0 + t / pc, k = p0 + t % pc;
          double s = 0.0;
          if (xi) s = Y[r * e.yrs + k * e.ycs];
          else
            for (int64_t j = 0; j < e.n; ++j) s = fma(X[r * e.xrs + j * e.xcs], Y[j * e.yrs + k * e.ycs], s);
          T[(t / pc) * 16 + t % pc] = s;
        }
        __syncthreads();
        for (int t = tid; t < rows * cols; t += nthr) {
          const int64_t r = t / cols, c = c0 + t % cols;
          double s = 0.0;
          if (zi) {
            if (c < p0 || c >= p0 + pc) continue;
            s = T[r * 16 + c - p0];
          } else {
            for (int64_t k = 0; k < pc; ++k) s = fma(T[r * 16 + k], Z[(p0 + k) * e.zrs + c * e.zcs], s);
          }
          double *d = D + (r0 + r) * g.drs + c * g.dcs;
          *d = fma(e.f, s, *d);
        }
      }
    }
  }
}

// One 16-row slice of a work item per CTA: rows [r0, r0 + 16) (slice blockIdx.y) and columns
// [c0, c0 + 16 NQ WC) of one chunk's output block.  A warp has 16 NQ columns.  WC = 1: the
// warps of the CTA take the chunk's stacks in turn, each by itself; their sums are added in
// warp order.  WC > 1: the WC warps each compute 16 columns of T, share the digits through
// shared memory and multiply them with their own columns of Z.
//
// A task at a time, or, for a slice of at most 8 rows, two tasks of a stack at a time: they
// share Y, so their X make up the 16 rows of the first product.
template <int NQ, int WC, int SMW>
__global__ void __launch_bounds__(WC == 1 ? 128 : 32 * WC, SMW / (WC == 1 ? 4 : WC))
    chain_mma_kernel(const PipeEntry *__restrict__ E, const PipeStack *__restrict__ stacks,
                     const int *__restrict__ nstacks, const ChainEntry *__restrict__ tasks,
                     const ChainGroup *__restrict__ G, const ChainItem *__restrict__ items,
                     const char *__restrict__ psi, const int *__restrict__ pexp, const double *__restrict__ psi64,
                     uint64_t db) {
  extern __shared__ __align__(16) unsigned char mma_smem[];
  __shared__ int te[2][WC][2];  // WC > 1: shifts of the chunks of T
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wcol = WC == 1 ? 0 : warp;
  const int grp = WC == 1 ? warp : 0, ngrp = WC == 1 ? (int)(blockDim.x >> 5) : 1;
  const ChainItem it = items[blockIdx.x];
  const ChainGroup *gp = G + it.g;
  const int gm = gp->m, gq = gp->q;
  const int nst = nstacks[it.g];
  const PipeStack *stk = stacks + gp->first;
  const int r0 = it.r0 + 16 * blockIdx.y, c0 = it.c0 + 16 * NQ * wcol;  // of this warp
  const int m = min(16, gm - r0), q = max(0, min(16 * NQ, gq - c0));
  if (m <= 0) return;
  const int rbx = (gm + 7) >> 3, rbz = (gq + 7) >> 3;  // 8-row blocks of the images of X and Z
  const bool pair = m <= 8;                            // two tasks at a time
  double D[2][NQ][4];  // [8 rows][16 columns]: rows 2 (lane & 3).., columns lane / 4..
#pragma unroll
  for (int b = 0; b < 2; ++b)
#pragma unroll
    for (int j = 0; j < NQ; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) D[b][j][e] = 0.0;
  bool any_special = false;
  int buf = 0;  // WC > 1: buffer of T

  // The stack at hand and the exponent of its Y, and the next one as read: when its turn comes it is
  // here, and what it points to is asked for while the tasks before it are computed.
  int4 d, nd;
  int si = grp, mem = 0, ey = 0, ns = 0;
  auto read = [&]() {
    nd = si < nst ? *reinterpret_cast<const int4 *>(stk + si) : make_int4(0, 0, 0, 0);
    si += ngrp;
  };
  auto next = [&]() {  // ns = 0: no further stack
    d = nd;
    ns = (d.w >> 24) & 15;
    mem = 0;
    if (ns > 0) {
      ey = pexp[d.w & 0xffffff];
      prefetch(E + d.x);
    }
    read();
  };
  read();
  next();
#pragma unroll 1
  while (ns > 0) {
    if (mem == 0 && (ey < 0 || (unsigned)d.w >> 28 != 0)) {  // not in fixed point
      any_special = true;
      next();
      continue;
    }
    const int n = d.y & 0xffff, p = (int)((unsigned)d.y >> 16), rby = (p + 7) >> 3;
    const char *Y = psi + (uint64_t)(uint32_t)d.z * 8;
    const PipeEntry *e0 = E + d.x + mem;
    const bool two = pair && mem + 1 < ns, x1 = !pair || two;
    const char *X0 = reinterpret_cast<const char *>(e0->x) + (r0 >> 3) * kDigBlock;
    const char *X1 = two ? reinterpret_cast<const char *>(e0[1].x) + (r0 >> 3) * kDigBlock : X0;
    const char *Z0 = reinterpret_cast<const char *>(e0->z) + (c0 >> 3) * kDigBlock;
    const char *Z1 = two ? reinterpret_cast<const char *>(e0[1].z) + (c0 >> 3) * kDigBlock : Z0;
    const int ney = ey;
    mem += pair ? 2 : 1;
    if (mem >= ns) next();  // from here on d, mem, ey and ns are those of the next task
    for (int k = 0; k < p; k += 16) {
      const int64_t o = (int64_t)(k >> 4) * rbz * kDigBlock;
      const int lines = min(2 * NQ, rbz - (c0 >> 3)) * (kDigBlock / 128);
      for (int i = lane; i < lines; i += 32) {
        prefetch(Z0 + o + i * 128);
        if (two) prefetch(Z1 + o + i * 128);
      }
    }
#pragma unroll 1
    for (int pb = 0; pb < p; pb += 16 * WC) {
      uint32_t td[2][6][2];  // digits of T: [8 rows]
      int up0 = 0, up1 = 0;
      const int pm = pb + 16 * wcol;  // this warp's columns of T
      if (pm < p) {
        long long t[2][4] = {};
        const int nj = min(2, rby - (pm >> 3));
#pragma unroll 1
        for (int k = 0; k < n; k += 16) {
          uint32_t a[6][4];
          load_rows(X0 + (k >> 4) * rbx * kDigBlock, !pair, X1 + (k >> 4) * rbx * kDigBlock, x1, lane, a);
          const bool half = n - k <= 8;
          const char *Yk = Y + ((k >> 4) * rby + (pm >> 3)) * kDigBlock;
#pragma unroll 1
          for (int j = 0; j < nj; ++j) {
            uint32_t b[6][2];
            load_block(Yk + j * kDigBlock, lane, b);
            long long s[4];
            multiply(a, b, half, s);
#pragma unroll
            for (int u = 0; u < 2; ++u)
              if (u == j) {
#pragma unroll
                for (int e = 0; e < 4; ++e) t[u][e] += s[e];
              }
          }
        }
        up0 = digits_of<0>(t, td[0]);
        if (x1) up1 = digits_of<2>(t, td[1]);
      }
      if (pb == 0 && ns > 0) {  // X and Y of the next task
        const int nn = d.y & 0xffff, np = (int)((unsigned)d.y >> 16);
        const PipeEntry *e = E + d.x + mem;
        const char *x = reinterpret_cast<const char *>(e->x) + (r0 >> 3) * kDigBlock;
        const char *xx = !pair ? x + kDigBlock
                         : mem + 1 < ns ? reinterpret_cast<const char *>(e[1].x) + (r0 >> 3) * kDigBlock
                                        : x;
        const int l = lane < 12 ? lane : lane - 12;
        for (int k = 0; k < nn; k += 16)
          if (lane < 24) prefetch((lane < 12 ? x : xx) + (k >> 4) * rbx * kDigBlock + l * 128);
        if (mem == 0) {
          const char *y = psi + (uint64_t)(uint32_t)d.z * 8;
          const int lines = ((np + 7) >> 3) * ((nn + 15) >> 4) * (kDigBlock / 128);
          for (int i = lane; i < lines; i += 32) prefetch(y + i * 128);
        }
      }
      const int nc = WC == 1 ? 1 : min(WC, (p - pb + 15) / 16);
      if constexpr (WC > 1) {
        uint4 *Ts = reinterpret_cast<uint4 *>(mma_smem + (buf * WC + wcol) * (2 * kDigBlock));
        if (pm < p) {
#pragma unroll
          for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int v = 0; v < 3; ++v)
              Ts[(b * 3 + v) * 32 + lane] = make_uint4(td[b][2 * v][0], td[b][2 * v][1], td[b][2 * v + 1][0], td[b][2 * v + 1][1]);
          if (lane == 0) {
            te[buf][wcol][0] = up0;
            te[buf][wcol][1] = up1;
          }
        }
        __syncthreads();
      }
#pragma unroll 1
      for (int c = 0; c < nc; ++c) {
        const int pc = pb + 16 * c;
        if constexpr (WC > 1) {
          const char *Ts = reinterpret_cast<const char *>(mma_smem + (buf * WC + c) * (2 * kDigBlock));
#pragma unroll
          for (int b = 0; b < 2; ++b) load_block(Ts + b * kDigBlock, lane, td[b]);
          up0 = te[buf][c][0];
          up1 = te[buf][c][1];
        }
        // 2^60 T64 = 2^(60 - up) T, and the same units again; f's exponent is in the entry's w
        const double f0 = e0->f, f1 = two ? e0[1].f : f0;
        const int s0 = 120 - 3240 - 1023 + ney - up0 + e0->w, s1 = 120 - 3240 - 1023 + ney - up1 + (two ? e0[1].w : e0->w);
        const double q0 = __hiloint2double((__double2hiint(f0) & 0x800fffff) | ((s0 + 1023) << 20), __double2loint(f0));
        const double q1 = __hiloint2double((__double2hiint(f1) & 0x800fffff) | ((s1 + 1023) << 20), __double2loint(f1));
        const bool half = p - pc <= 8;
#pragma unroll 1
        for (int j = 0; 16 * j < q; ++j) {
          const bool have = (c0 >> 3) + 2 * j + 1 < rbz;
          const int64_t off = (int64_t)((pc >> 4) * rbz + 2 * j) * kDigBlock;
          uint32_t a[6][4];
          load_rows(Z0 + off, have, Z0, false, lane, a);
          long long s[2][4];
          multiply(a, td[0], half, s[0]);
          if (x1) {
            if (two) load_rows(Z1 + off, have, Z1, false, lane, a);
            multiply(a, td[1], half, s[1]);
          }
#pragma unroll
          for (int u = 0; u < NQ; ++u)
            if (u == j) {
#pragma unroll
              for (int e = 0; e < 4; ++e) D[0][u][e] = fma(q0, (double)s[0][e], D[0][u][e]);
              if (two) {
#pragma unroll
                for (int e = 0; e < 4; ++e) D[0][u][e] = fma(q1, (double)s[1][e], D[0][u][e]);
              } else if (x1) {
#pragma unroll
                for (int e = 0; e < 4; ++e) D[1][u][e] = fma(q1, (double)s[1][e], D[1][u][e]);
              }
            }
        }
      }
      buf ^= 1;
    }
  }
  if constexpr (WC == 1) {
    if (ngrp > 1) {  // the warps' sums, added in warp order
      double *x = reinterpret_cast<double *>(mma_smem) + lane;
      for (int h = 1; h < ngrp; ++h) {
        if (grp == h) {
#pragma unroll
          for (int i = 0; i < 8 * NQ; ++i) x[i * 32] = D[i / (4 * NQ)][i / 4 % NQ][i % 4];
        }
        __syncthreads();
        if (grp == 0) {
#pragma unroll
          for (int i = 0; i < 8 * NQ; ++i) D[i / (4 * NQ)][i / 4 % NQ][i % 4] += x[i * 32];
        }
        __syncthreads();
      }
    }
  }
  if (grp == 0) {
    const int drs = gp->drs, dcs = gp->dcs, ri = 2 * (lane & 3), ci = lane >> 2;
    double *Dout = reinterpret_cast<double *>(db + gp->d * 8ull) + (int64_t)r0 * drs + (int64_t)c0 * dcs;
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int j = 0; j < NQ; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int r = 8 * b + ri + (e & 1), c = 16 * j + ci + 8 * (e >> 1);
          if (r < m && c < q) Dout[(int64_t)r * drs + (int64_t)c * dcs] = D[b][j][e];
        }
  }
  if (__syncthreads_or(any_special))
    slow_stacks(E, stk, nst, tasks, pexp, psi64, gp, r0, it.c0, m, min(16 * NQ * WC, gq - it.c0), db,
                reinterpret_cast<double *>(mma_smem));
}

// Warps that share a slice's tasks: chunks of many tasks are shared, so that no CTA runs on
// when the others are done, and so are chunks that alone would not fill the GPU.
int warps_per_slice(int n, int64_t tasks, int resident) {
  int k = 1;
  while (k < 4 && ((long long)n * k < resident || tasks > 16ll * k * n)) k *= 2;
  return k;
}

// SMW: warps that an SM holds, registers against latency.  At 12 a warp has the 168 registers
// that its sums, fragments and addresses want; at 16 it spills some (340 to 380 bytes), which pays
// where there are warps enough.  12 / 16 for every class but 0: 12 orbitals, M 800: 15.7 / 14.9 ms;
// 24, M 512: 7.9 / 7.6 ms; with few chunks (11, M 150) it costs 340 / 353 us.
template <int NQ, int WC, int SMW>
cudaError_t launch_mma(const PipeArgs &a, const ChainItem *items, const PipeClass &c, int slices, bool share,
                       cudaStream_t s) {
  if (c.items <= 0) return cudaSuccess;
  const int warps = WC > 1 ? WC : share ? warps_per_slice(c.items * slices, c.tasks, SMW * 152) : 1;
  // T of WC > 1 (two buffers), the sums of a warp, or T of slow_stacks
  const int bytes = std::max({WC > 1 ? 2 * WC * 2 * kDigBlock : 0, 8 * NQ * 32 * 8, 16 * 16 * 8});
  auto kern = chain_mma_kernel<NQ, WC, SMW>;
  add_kernel_launches(1);
  kern<<<dim3(c.items, slices), 32 * warps, bytes, s>>>(a.e, a.stacks, a.nstacks, a.tasks, a.g, items,
                                                        static_cast<const char *>(a.psi), a.pexp, a.psi64, a.db);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_chain_mma(const PipeArgs &a, const ChainItem *items, const PipeClass *c, int wide, cudaStream_t s,
                             cudaStream_t s1, cudaStream_t s2) {
  cudaError_t err;
  auto next = [&](int cls) {
    const ChainItem *p = items;
    items += c[cls].items;
    return p;
  };
  const ChainItem *i5 = next(5), *i4 = next(4), *i3 = next(3), *i2 = next(2), *i1 = next(1), *i0 = next(0);
  if ((err = launch_mma<2, 4, 16>(a, i5, c[5], 2, false, s1)) != cudaSuccess) return err;
  if ((err = launch_mma<2, 3, 15>(a, i4, c[4], 2, false, s)) != cudaSuccess) return err;
  if ((err = launch_mma<2, 2, 16>(a, i3, c[3], 2, false, s1)) != cudaSuccess) return err;
  if ((err = launch_mma<2, 1, 16>(a, i2, c[2], 2, wide != 0, s)) != cudaSuccess) return err;
  if ((err = launch_mma<2, 1, 16>(a, i1, c[1], 1, wide != 0, s1)) != cudaSuccess) return err;
  // 12 / 16: 8 orbitals, M 64 (459 items): 178 / 191 us; 24, M 512 (1,103): 7.56 / 7.43 ms; the batch of 16
  // problems (14,368): 11.8 / 10.8 ms.  An item has four warps at most: the line is two waves of 16 an SM.
  if (c[0].items > 2 * 4 * 152) return launch_mma<1, 1, 16>(a, i0, c[0], 1, wide != 0, s2);
  return launch_mma<1, 1, 12>(a, i0, c[0], 1, wide != 0, s2);
}

}  // namespace dmrg
