// The batched triple product D = sum_e f_e X_e Y_e Z_e on the CUDA cores (sm_103a).
//
// Used for H.psi (Sec. 2.2.1, Eq. dgemm: X = A_l, Y = psi^s, Z = A_r^T), for the
// renormalization O^T (A (x) o) O of Sec. 2.2.2 / Eq. renorm_mat (X = O^T, Y = A,
// Z = O), for the density matrix psi psi^T of Sec. 2.1 and for the wave-function
// prediction.  A chunk of tasks that share an output block is one work item: its
// sum stays in registers and is written once, so the result needs no atomics and
// does not depend on scheduling.
//
// FP64 tiles are multiplied as block-scaled integers (chain_arith.cuh).
//
// FP32 operators (FP64 psi rounded to FP32 as it is read, FP32 accumulation): the
// same tiling with one FP32 multiply-add per element product.
//
// Tiling.  A warp owns up to TS x TS outputs (TS = 16 or 32): lane (i, j) of a 4 x 8
// lane grid holds rows i + 4a and columns j + 8b, so ragged blocks waste at most 3 rows
// and 7 columns.  Operand tiles sit in shared memory with the summed index contiguous
// (row pitch = 4 banks mod 32: the 128-bit loads of a warp are free of conflicts).
// Blocks wider than 32 columns take WC warps per item (32 columns each) which share the
// rows' X tile and hand each other their part of T, so T is computed once.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>

#include "chain_arith.cuh"
#include "kernels.cuh"

namespace dmrg {

namespace {

constexpr uint64_t IDN = ~0ull;

// ---------------------------------------------------------------- tiles

// Read the R x K view src(r, k) = src[r rs + k cs] by nthr threads into registers.
// Element n of this thread has flat index t = n nthr + tid; the faster index follows the
// view's unit stride.
template <int TS>
struct View {
  int R, K, tot;
  bool kfast;
  float inv;
  __device__ __forceinline__ View(int R_, int K_, int rs, int cs) : R(R_), K(K_), tot(R_ * K_) {
    kfast = cs == 1 || rs != 1;
    inv = 1.0f / (float)(kfast ? K : R);
  }
  __device__ __forceinline__ void at(int t, int &r, int &k) const {
    const int q = small_div(t, inv);
    if (kfast) {
      r = q;
      k = t - q * K;
    } else {
      k = q;
      r = t - q * R;
    }
  }
};

// Columns [K, K rounded up to VK) of the first R rows of a tile are zeroed: the inner
// loops read whole 128-bit vectors.
template <bool FX, int P>
__device__ __forceinline__ void pad_tile(typename Arith<FX>::Elem *tile, int R, int K, int tid, int nthr) {
  constexpr int VK = Arith<FX>::VK;
  const int Kp = (K + VK - 1) / VK * VK;
  if (Kp == K) return;
  for (int r = tid; r < R; r += nthr)
    for (int k = K; k < Kp; ++k) tile[r * P + k] = typename Arith<FX>::Elem();
}

// A tile of doubles, read by nthr threads: raw values to their slots and the largest
// exponent, then (after the caller's reduction) each thread turns its own slots into limbs.
template <int TS, int P, typename T>
__device__ __forceinline__ TileMax read_raw(int2 *tile, const T *src, const View<TS> &V, int rs, int cs, int tid,
                                            int nthr) {
  TileMax mx;
#pragma unroll 1
  for (int t0 = tid; t0 < V.tot; t0 += 4 * nthr) {
    double v[4];
    int o[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int t = min(t0 + u * nthr, V.tot - 1);  // past the end: the last element again
      int r, k;
      V.at(t, r, k);
      o[u] = r * P + k;
      v[u] = (double)src[(int64_t)r * rs + (int64_t)k * cs];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      mx.add(v[u]);
      if (t0 + u * nthr < V.tot) *reinterpret_cast<double *>(tile + o[u]) = v[u];
    }
  }
  return mx;
}

template <int TS, int P>
__device__ __forceinline__ void raw_to_limbs(int2 *tile, const View<TS> &V, int E, int tid, int nthr) {
#pragma unroll 2
  for (int t = tid; t < V.tot; t += nthr) {
    int r, k;
    V.at(t, r, k);
    int2 *slot = tile + r * P + k;
    *slot = to_limbs(*reinterpret_cast<const double *>(slot), E);
  }
  pad_tile<true, P>(tile, V.R, V.K, tid, nthr);
}

// By one warp.  Returns the tile's exponent (tile_exponent).
template <int TS, int P, typename T>
__device__ __forceinline__ int load_fx(int2 *tile, const T *src, int R, int K, int rs, int cs, int lane) {
  const View<TS> V(R, K, rs, cs);
  const TileMax mx = read_raw<TS, P>(tile, src, V, rs, cs, lane, 32);
  const unsigned hi = __reduce_max_sync(kFull, mx.hi), any = __reduce_or_sync(kFull, mx.any);
  const int E = tile_exponent(hi, any);
  if (E >= 0) raw_to_limbs<TS, P>(tile, V, E, lane, 32);
  return E;
}

// By all warps of a CTA (barriers inside; red: 2 words per warp).
template <int TS, int P, int WC, typename T>
__device__ __forceinline__ int load_fx_cta(int2 *tile, const T *src, int R, int K, int rs, int cs, int tid,
                                           unsigned *red) {
  const View<TS> V(R, K, rs, cs);
  __syncthreads();  // the last readers of the tile and of red are done
  const TileMax mx = read_raw<TS, P>(tile, src, V, rs, cs, tid, 32 * WC);
  unsigned hi = __reduce_max_sync(kFull, mx.hi), any = __reduce_or_sync(kFull, mx.any);
  if ((tid & 31) == 0) {
    red[2 * (tid >> 5)] = hi;
    red[2 * (tid >> 5) + 1] = any;
  }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < WC; ++w) {
    hi = max(hi, red[2 * w]);
    any |= red[2 * w + 1];
  }
  const int E = tile_exponent(hi, any);
  if (E >= 0) raw_to_limbs<TS, P>(tile, V, E, tid, 32 * WC);
  __syncthreads();
  return E;
}

template <int TS, int P, typename T>
__device__ __forceinline__ void load_f32(float *tile, const T *src, int R, int K, int rs, int cs, int tid, int nthr) {
  const View<TS> V(R, K, rs, cs);
  for (int t0 = 0; t0 < V.tot; t0 += 4 * nthr) {
    float v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int t = t0 + u * nthr + tid;
      int r, k;
      V.at(t, r, k);
      v[u] = t < V.tot ? (float)src[(int64_t)r * rs + (int64_t)k * cs] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int t = t0 + u * nthr + tid;
      int r, k;
      V.at(t, r, k);
      if (t < V.tot) tile[r * P + k] = v[u];
    }
  }
  pad_tile<false, P>(tile, R, K, tid, nthr);
}

// ---------------------------------------------------------------- T = X Y

// One 16-row pass of T (+)= X Y over a chunk of the inner dimension.  While further
// chunks follow, the sums are kept in the T tile as 64-bit integers in units of 2^eraw;
// the last chunk normalises them to limbs under the exponent it returns.  A chunk with a tile
// of zeros (exponent 0) has an e below that of any other chunk, so that it never moves the sums
// of the others; sums that are all zero get eraw = 0.
template <int TS, int P, int NB>
__device__ __forceinline__ void stage1_fx(const int2 *X, const int2 *Y, int2 *T, int pass, int m, int pc, int kc,
                                          int lane, bool first, bool last, int extra, int e, int &eraw) {
  constexpr int S = Shift<TS>::value;
  const int lr = lane >> 3, lc = lane & 7;
  const int na = min(4, (m - 16 * pass + 3) >> 2);
  long long hh[4][NB], cr[4][NB];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < NB; ++b) hh[a][b] = cr[a][b] = 0;
  const int row = 16 * pass + lr;
  mm<P, NB>(X + row * P, Y + lc * P, kc, na, hh, cr);
  int2 *Tl = T + row * P + lc;
  e += extra;
  int d_old = 0, d_new = 0;  // alignment of the kept sums and of this chunk
  if (!first) {
    if (e > eraw) d_old = min(e - eraw, 63);
    else d_new = min(eraw - e, 63);
    e = max(e, eraw);
  }
  unsigned mx = 0;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    if (a < na) {
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        long long t = fold<S>(hh[a][b], cr[a][b]) >> extra;
        if (!first) t = (t >> d_new) + (*reinterpret_cast<const long long *>(Tl + 4 * a * P + 8 * b) >> d_old);
        if (last && (lc + 8 * b >= pc || row + 4 * a >= m)) t = 0;
        hh[a][b] = t;
        mx = max(mx, (unsigned)((t ^ (t >> 63)) >> 32));
      }
    }
  }
  if (!last) {
    eraw = e;
#pragma unroll
    for (int a = 0; a < 4; ++a)
      if (a < na) {
#pragma unroll
        for (int b = 0; b < NB; ++b) *reinterpret_cast<long long *>(Tl + 4 * a * P + 8 * b) = hh[a][b];
      }
    return;
  }
  mx = __reduce_max_sync(kFull, mx);
  int bits = 64 - __clz(mx);  // |t| < 2^bits
  if (mx == 0) {              // rare: every sum is below 2^32
    unsigned lo = 0;
#pragma unroll
    for (int a = 0; a < 4; ++a)
      if (a < na) {
#pragma unroll
        for (int b = 0; b < NB; ++b) lo = max(lo, (unsigned)(hh[a][b] ^ (hh[a][b] >> 63)));
      }
    lo = __reduce_max_sync(kFull, lo);
    bits = 33 - __clz(lo);
    if (lo == 0) {
      bits = 57;
      e = 0;
    }
  }
  const int sh = bits - 57;
  eraw = e + sh;
  const int left = max(-sh, 0), right = max(sh, 0);
  const long long half = right ? 1ll << (right - 1) : 0;
#pragma unroll
  for (int a = 0; a < 4; ++a)
    if (a < na) {
#pragma unroll
      for (int b = 0; b < NB; ++b) Tl[4 * a * P + 8 * b] = limbs(((hh[a][b] << left) + half) >> right);
    }
}

template <int TS, int P, int NB>
__device__ __forceinline__ void stage1_f32(const float *X, const float *Y, float *T, int pass, int m, int pc, int kc,
                                           int lane, bool first, bool apart) {
  const int lr = lane >> 3, lc = lane & 7;
  const int na = min(4, (m - 16 * pass + 3) >> 2);
  const int row = 16 * pass + lr;
  float *Tl = T + row * P + lc;
  float s[4][NB];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < NB; ++b) s[a][b] = (!first && !apart && a < na) ? Tl[4 * a * P + 8 * b] : 0.f;
  mm<P, NB>(X + row * P, Y + lc * P, kc, na, s);
#pragma unroll
  for (int a = 0; a < 4; ++a)
    if (a < na) {
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        float *t = Tl + 4 * a * P + 8 * b;
        if (!first && apart) s[a][b] += *t;
        *t = lc + 8 * b < pc ? s[a][b] : 0.f;
      }
    }
}

// ---------------------------------------------------------------- D += f T Z

template <int TS, int P, int NB, int NBMAX, int PASS>
__device__ __forceinline__ void stage2_fx(const int2 *T, const int2 *Z, int m, int kc, int lane, double scale,
                                          double (&D)[TS / 4][NBMAX]) {
  constexpr int S = Shift<TS>::value;
  const int na = min(4, (m - 16 * PASS + 3) >> 2);
  long long hh[4][NB], cr[4][NB];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < NB; ++b) hh[a][b] = cr[a][b] = 0;
  mm<P, NB>(T + (16 * PASS + (lane >> 3)) * P, Z + (lane & 7) * P, kc, na, hh, cr);
#pragma unroll
  for (int a = 0; a < 4; ++a)
    if (a < na) {
#pragma unroll
      for (int b = 0; b < NB; ++b)
        D[4 * PASS + a][b] = fma(scale, (double)fold<S>(hh[a][b], cr[a][b]), D[4 * PASS + a][b]);
    }
}

template <int TS, int P, int NB, int NBMAX, int PASS>
__device__ __forceinline__ void stage2_f32(const float *T, const float *Z, int m, int kc, int lane, float f,
                                           float (&D)[TS / 4][NBMAX]) {
  const int na = min(4, (m - 16 * PASS + 3) >> 2);
  float s[4][NB];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < NB; ++b) s[a][b] = 0.f;
  mm<P, NB>(T + (16 * PASS + (lane >> 3)) * P, Z + (lane & 7) * P, kc, na, s);
#pragma unroll
  for (int a = 0; a < 4; ++a)
    if (a < na) {
#pragma unroll
      for (int b = 0; b < NB; ++b) D[4 * PASS + a][b] = fmaf(f, s[a][b], D[4 * PASS + a][b]);
    }
}

// ---------------------------------------------------------------- the kernel

// One work item: rows [r0, r0 + TS) and columns [c0, c0 + TS WC) of one chunk's output
// block.  WC = 1: nsplit = blockDim / 32 warps take every nsplit-th task of the chunk
// and their sums are added in warp order.  WC > 1: warp w holds columns c0 + TS w ...
template <typename TX, typename TY, typename TZ, bool FX, int TS, int WC>
__global__ void __launch_bounds__(WC == 1 ? 256 : 32 * WC, WC == 1 ? (TS == 32 ? 1 : 2) : WC == 2 ? 4 : 2)
    chain_item_kernel(const ChainEntry *__restrict__ E, const ChainGroup *__restrict__ G,
                      const ChainItem *__restrict__ items, uint64_t xb, uint64_t yb, uint64_t zb, uint64_t db) {
  using A = Arith<FX>;
  using Elem = typename A::Elem;
  using Out = typename A::Out;
  constexpr int P = (TS + A::PAD);
  constexpr int NBMAX = TS / 8, NP = TS / 16;
  constexpr int TILE = TS * P;
  extern __shared__ __align__(16) unsigned char chain_smem[];
  __shared__ unsigned red[2 * WC];
  __shared__ int te[WC][NP];  // exponents of the T chunks, INT_MIN: the chunk holds doubles
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int lr = lane >> 3, lc = lane & 7;
  // WC = 1: per warp X, YZ, T.  WC > 1: X, then YZ per warp, then T per warp.
  Elem *base = reinterpret_cast<Elem *>(chain_smem);
  Elem *Xs = WC == 1 ? base + warp * 3 * TILE : base;
  Elem *Bs = WC == 1 ? Xs + TILE : base + (1 + warp) * TILE;
  Elem *Ts = WC == 1 ? Xs + 2 * TILE : base + (1 + WC) * TILE;  // chunk j at Ts + j TILE
  const ChainItem it = items[blockIdx.x];
  const ChainGroup g = G[it.g];
  const int m = min(TS, g.m - it.r0);
  const int col = it.c0 + (WC == 1 ? 0 : TS * warp);  // first output column of this warp
  const int q = max(0, min(TS, g.q - col));
  const int nbq = (q + 7) >> 3;
  const int step = WC == 1 ? (int)(blockDim.x >> 5) : 1;
  Out D[TS / 4][NBMAX];
#pragma unroll
  for (int a = 0; a < TS / 4; ++a)
#pragma unroll
    for (int b = 0; b < NBMAX; ++b) D[a][b] = 0;

  for (int ei = g.first + (WC == 1 ? warp : 0); ei < g.first + g.count; ei += step) {
    const ChainEntry e = E[ei];
    const bool xid = e.x == IDN, yid = e.y == IDN, zid = e.z == IDN;
    const TX *X = reinterpret_cast<const TX *>(xb + e.x * sizeof(TX)) + (int64_t)it.r0 * e.xrs;
    const TY *Y = reinterpret_cast<const TY *>(yb + e.y * sizeof(TY));
    const TZ *Z = reinterpret_cast<const TZ *>(zb + e.z * sizeof(TZ));
    const int n = e.n, p = e.p;
    const int nch = (n + TS - 1) / TS;
    // FP32 sums keep one order whatever the block size class: over chunks of 32 of the inner
    // dimension, added up for blocks of at most 32 x 32, running on for larger ones
    const bool apart = TS > 16 && g.m <= 32 && g.q <= 32;  // TS = 16: n <= 32
    int extra = 0;  // further bits kept free when the sum has many chunks
    if (FX && nch > 1) extra = nch <= 2 ? 1 : 32 - __clz(nch - 1);
    for (int p0 = 0; p0 < p; p0 += TS * WC) {
      if (zid && p0 != it.c0) continue;  // an identity Z: only the item's own columns of T
      // ---- this warp's chunk of T: columns pt .. pt + pc
      const int pt = p0 + (WC == 1 ? 0 : TS * warp);
      const int pc = max(0, min(TS, p - pt));
      Elem *T = Ts + (WC == 1 ? 0 : warp * TILE);
      int eT[NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) eT[i] = 0;
      bool slow = false;
      if (WC > 1) __syncthreads();  // T and te of the previous chunk have been read
      else __syncwarp();
      if (xid || yid) {
        const bool both = xid && yid;
        if constexpr (FX) {
          int E1 = -1;
          if (!both && pc > 0)
            E1 = xid ? load_fx<TS, P>(T, Y + (int64_t)it.r0 * e.yrs + (int64_t)pt * e.ycs, m, pc, e.yrs, e.ycs, lane)
                     : load_fx<TS, P>(T, X + (int64_t)pt * e.xcs, m, pc, e.xrs, e.xcs, lane);
#pragma unroll
          for (int i = 0; i < NP; ++i) eT[i] = zero_as_one(E1) - 1079;
          slow = E1 < 0;
        } else if (pc > 0) {
          if (both) {
            for (int t = lane; t < TS * TS; t += 32)
              T[(t / TS) * P + t % TS] = it.r0 + t / TS == pt + t % TS ? 1.f : 0.f;
          } else if (xid) {
            load_f32<TS, P>(T, Y + (int64_t)it.r0 * e.yrs + (int64_t)pt * e.ycs, m, pc, e.yrs, e.ycs, lane, 32);
          } else {
            load_f32<TS, P>(T, X + (int64_t)pt * e.xcs, m, pc, e.xrs, e.xcs, lane, 32);
          }
        }
      } else {
        for (int c = 0; c < nch; ++c) {
          const int n0 = c * TS, nc = min(TS, n - n0);
          const bool first = c == 0, last = c == nch - 1;
          if constexpr (FX) {
            const TX *Xc = X + (int64_t)n0 * e.xcs;
            const int Ex = WC == 1 ? load_fx<TS, P>(Xs, Xc, m, nc, e.xrs, e.xcs, lane)
                                   : load_fx_cta<TS, P, WC>(Xs, Xc, m, nc, e.xrs, e.xcs, tid, red);
            if (pc > 0) {
              const int Ey = load_fx<TS, P>(Bs, Y + (int64_t)n0 * e.yrs + (int64_t)pt * e.ycs, pc, nc, e.ycs, e.yrs,
                                            lane);
              slow |= Ex < 0 || Ey < 0;
              __syncwarp();
              if (!slow) {
                const int ex = Ex + Ey - 2100 - Shift<TS>::value;
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                  if (16 * i < m) {
                    switch ((pc + 7) >> 3) {
                      case 1: stage1_fx<TS, P, 1>(Xs, Bs, T, i, m, pc, nc, lane, first, last, extra, ex, eT[i]); break;
                      case 2: stage1_fx<TS, P, 2>(Xs, Bs, T, i, m, pc, nc, lane, first, last, extra, ex, eT[i]); break;
                      case 3: if constexpr (TS > 16) stage1_fx<TS, P, NBMAX - 1>(Xs, Bs, T, i, m, pc, nc, lane, first, last, extra, ex, eT[i]); break;
                      default: if constexpr (TS > 16) stage1_fx<TS, P, NBMAX>(Xs, Bs, T, i, m, pc, nc, lane, first, last, extra, ex, eT[i]); break;
                    }
                  }
                }
              }
            }
          } else {
            if (WC > 1) __syncthreads();
            load_f32<TS, P>(Xs, X + (int64_t)n0 * e.xcs, m, nc, e.xrs, e.xcs, WC == 1 ? lane : tid, 32 * WC);
            if (pc > 0)
              load_f32<TS, P>(Bs, Y + (int64_t)n0 * e.yrs + (int64_t)pt * e.ycs, pc, nc, e.ycs, e.yrs, lane, 32);
            if (WC > 1) __syncthreads();
            else __syncwarp();
            if (pc > 0) {
#pragma unroll
              for (int i = 0; i < NP; ++i) {
                if (16 * i < m) {
                  switch ((pc + 7) >> 3) {
                    case 1: stage1_f32<TS, P, 1>(Xs, Bs, T, i, m, pc, nc, lane, first, apart); break;
                    case 2: stage1_f32<TS, P, 2>(Xs, Bs, T, i, m, pc, nc, lane, first, apart); break;
                    case 3: if constexpr (TS > 16) stage1_f32<TS, P, NBMAX - 1>(Xs, Bs, T, i, m, pc, nc, lane, first, apart); break;
                    default: if constexpr (TS > 16) stage1_f32<TS, P, NBMAX>(Xs, Bs, T, i, m, pc, nc, lane, first, apart); break;
                  }
                }
              }
            }
          }
          if (!last) __syncwarp();  // the tiles are reused
        }
      }
      if constexpr (FX) {
        if (slow && pc > 0) {  // this chunk of T in FP64, straight from memory
          __syncwarp();
          for (int t = lane; t < m * pc; t += 32) {
            const int r = t / pc, k = t % pc;
            double s = 0.0;
            if (xid && yid) s = it.r0 + r == pt + k ? 1.0 : 0.0;
            else if (xid) s = (double)Y[(int64_t)(it.r0 + r) * e.yrs + (int64_t)(pt + k) * e.ycs];
            else if (yid) s = (double)X[(int64_t)r * e.xrs + (int64_t)(pt + k) * e.xcs];
            else
              for (int i = 0; i < n; ++i)
                s = fma((double)X[(int64_t)r * e.xrs + (int64_t)i * e.xcs],
                        (double)Y[(int64_t)i * e.yrs + (int64_t)(pt + k) * e.ycs], s);
            *reinterpret_cast<double *>(T + r * P + k) = s;
          }
#pragma unroll
          for (int i = 0; i < NP; ++i) eT[i] = INT_MIN;
        }
      }
      if constexpr (WC > 1) {
        if (FX && lane < NP) te[warp][lane] = lane == 0 ? eT[0] : eT[NP - 1];
        __syncthreads();
      } else {
        __syncwarp();
      }
      // ---- D += f T Z over the chunks of T
      if (q > 0) {
        for (int j = 0; j < WC; ++j) {
          const int kt = p0 + j * TS, kc = min(TS, p - kt);
          if (kc <= 0) break;
          if (zid && j != (WC == 1 ? 0 : warp)) continue;
          const Elem *Tj = Ts + j * TILE;
          if constexpr (FX) {
            int eTj[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) eTj[i] = WC == 1 ? eT[i] : te[j][i];
            const bool slowT = eTj[0] == INT_MIN;
            int Ez = 0;
            if (!zid) {
              __syncwarp();  // the tile's previous readers
              Ez = load_fx<TS, P>(Bs, Z + (int64_t)kt * e.zrs + (int64_t)col * e.zcs, q, kc, e.zcs, e.zrs, lane);
              __syncwarp();
            }
            const int ef = (__double2hiint(e.f) >> 20) & 0x7ff;
            const bool fok = ef <= 1023 + 100 && ef >= 1023 - 100;
            if (zid && !slowT && fok) {  // own columns of T
#pragma unroll
              for (int a = 0; a < TS / 4; ++a) {
                if (lr + 4 * a < m) {
                  const double sc = scaled(e.f, eTj[a / 4]);
#pragma unroll
                  for (int b = 0; b < NBMAX; ++b) {
                    const int2 v = lc + 8 * b < q ? Tj[(lr + 4 * a) * P + lc + 8 * b] : make_int2(0, 0);
                    D[a][b] = muladd(sc, v, D[a][b]);
                  }
                }
              }
            } else if (slowT || zid || Ez < 0 || !fok) {
              // values that fixed point does not take: FP64
              for (int k = 0; k < kc; ++k) {
                double z[NBMAX];
#pragma unroll
                for (int b = 0; b < NBMAX; ++b) {
                  const int c = lc + 8 * b;
                  z[b] = zid ? (c == k ? 1.0 : 0.0)
                             : c < q ? (double)Z[(int64_t)(kt + k) * e.zrs + (int64_t)(col + c) * e.zcs] : 0.0;
                }
#pragma unroll
                for (int a = 0; a < TS / 4; ++a) {
                  const int r = lr + 4 * a;
                  if (r < m) {
                    const double t = e.f * (slowT ? *reinterpret_cast<const double *>(Tj + r * P + k)
                                                  : limbs_to_double(Tj[r * P + k], eTj[a / 4]));
#pragma unroll
                    for (int b = 0; b < NBMAX; ++b)
                      if (!zid || lc + 8 * b == k) D[a][b] = fma(t, z[b], D[a][b]);
                  }
                }
              }
            } else {
              const int e0 = 58 - Shift<TS>::value + zero_as_one(Ez) - 1079;
              switch (nbq) {
                case 1:
                  stage2_fx<TS, P, 1, NBMAX, 0>(Tj, Bs, m, kc, lane, scaled(e.f, e0 + eTj[0]), D);
                  if (NP > 1 && m > 16) stage2_fx<TS, P, 1, NBMAX, NP - 1>(Tj, Bs, m, kc, lane, scaled(e.f, e0 + eTj[NP - 1]), D);
                  break;
                case 2:
                  stage2_fx<TS, P, 2, NBMAX, 0>(Tj, Bs, m, kc, lane, scaled(e.f, e0 + eTj[0]), D);
                  if (NP > 1 && m > 16) stage2_fx<TS, P, 2, NBMAX, NP - 1>(Tj, Bs, m, kc, lane, scaled(e.f, e0 + eTj[NP - 1]), D);
                  break;
                case 3:
                  if constexpr (TS > 16) {
                    stage2_fx<TS, P, NBMAX - 1, NBMAX, 0>(Tj, Bs, m, kc, lane, scaled(e.f, e0 + eTj[0]), D);
                    if (m > 16) stage2_fx<TS, P, NBMAX - 1, NBMAX, NP - 1>(Tj, Bs, m, kc, lane, scaled(e.f, e0 + eTj[NP - 1]), D);
                  }
                  break;
                default:
                  if constexpr (TS > 16) {
                    stage2_fx<TS, P, NBMAX, NBMAX, 0>(Tj, Bs, m, kc, lane, scaled(e.f, e0 + eTj[0]), D);
                    if (m > 16) stage2_fx<TS, P, NBMAX, NBMAX, NP - 1>(Tj, Bs, m, kc, lane, scaled(e.f, e0 + eTj[NP - 1]), D);
                  }
                  break;
              }
            }
          } else {
            const float f = (float)e.f;
            if (zid) {
#pragma unroll
              for (int a = 0; a < TS / 4; ++a)
#pragma unroll
                for (int b = 0; b < NBMAX; ++b)
                  if (lr + 4 * a < m && lc + 8 * b < q) D[a][b] = fmaf(f, Tj[(lr + 4 * a) * P + lc + 8 * b], D[a][b]);
            } else {
              __syncwarp();
              load_f32<TS, P>(Bs, Z + (int64_t)kt * e.zrs + (int64_t)col * e.zcs, q, kc, e.zcs, e.zrs, lane, 32);
              __syncwarp();
              switch (nbq) {
                case 1:
                  stage2_f32<TS, P, 1, NBMAX, 0>(Tj, Bs, m, kc, lane, f, D);
                  if (NP > 1 && m > 16) stage2_f32<TS, P, 1, NBMAX, NP - 1>(Tj, Bs, m, kc, lane, f, D);
                  break;
                case 2:
                  stage2_f32<TS, P, 2, NBMAX, 0>(Tj, Bs, m, kc, lane, f, D);
                  if (NP > 1 && m > 16) stage2_f32<TS, P, 2, NBMAX, NP - 1>(Tj, Bs, m, kc, lane, f, D);
                  break;
                case 3:
                  if constexpr (TS > 16) {
                    stage2_f32<TS, P, NBMAX - 1, NBMAX, 0>(Tj, Bs, m, kc, lane, f, D);
                    if (m > 16) stage2_f32<TS, P, NBMAX - 1, NBMAX, NP - 1>(Tj, Bs, m, kc, lane, f, D);
                  }
                  break;
                default:
                  if constexpr (TS > 16) {
                    stage2_f32<TS, P, NBMAX, NBMAX, 0>(Tj, Bs, m, kc, lane, f, D);
                    if (m > 16) stage2_f32<TS, P, NBMAX, NBMAX, NP - 1>(Tj, Bs, m, kc, lane, f, D);
                  }
                  break;
              }
            }
          }
        }
      }
    }
  }
  if constexpr (WC == 1) {
    if (step > 1) {  // the warps' sums, added in warp order
      __syncwarp();
      Out *mine = reinterpret_cast<Out *>(Xs);
      if (warp > 0) {
#pragma unroll
        for (int a = 0; a < TS / 4; ++a)
#pragma unroll
          for (int b = 0; b < NBMAX; ++b) mine[(a * NBMAX + b) * 32 + lane] = D[a][b];
      }
      __syncthreads();
      if (warp > 0) return;
      for (int w = 1; w < step; ++w) {
        const Out *other = reinterpret_cast<const Out *>(base + w * 3 * TILE);
#pragma unroll
        for (int a = 0; a < TS / 4; ++a)
#pragma unroll
          for (int b = 0; b < NBMAX; ++b) D[a][b] += other[(a * NBMAX + b) * 32 + lane];
      }
    }
  }
  double *Dout = reinterpret_cast<double *>(db + g.d * 8ull) + (int64_t)it.r0 * g.drs + (int64_t)col * g.dcs;
#pragma unroll
  for (int a = 0; a < TS / 4; ++a)
#pragma unroll
    for (int b = 0; b < NBMAX; ++b)
      if (lr + 4 * a < m && lc + 8 * b < q)
        Dout[(int64_t)(lr + 4 * a) * g.drs + (int64_t)(lc + 8 * b) * g.dcs] = (double)D[a][b];
}

template <typename TX, typename TY, typename TZ, bool FX, int TS, int WC>
cudaError_t launch_items(const ChainEntry *e, const ChainGroup *g, const ChainItem *items, int n, int warps,
                         uint64_t xb, uint64_t yb, uint64_t zb, uint64_t db, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  using A = Arith<FX>;
  constexpr int tile = TS * (TS + A::PAD) * (int)sizeof(typename A::Elem);
  const int smem = WC == 1 ? warps * 3 * tile : (1 + 2 * WC) * tile;
  auto kern = chain_item_kernel<TX, TY, TZ, FX, TS, WC>;
  const cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               WC == 1 ? 8 * 3 * tile : smem);
  if (err != cudaSuccess) return err;
  add_kernel_launches(1);
  kern<<<n, WC == 1 ? 32 * warps : 32 * WC, smem, s>>>(e, g, items, xb, yb, zb, db);
  return cudaGetLastError();
}

// Warps that share a chunk's tasks: one while the chunks alone fill the GPU.
int warps_per_item(int n, int resident) {
  int w = 1;
  while (w < 8 && (long long)n * w < resident) w *= 2;
  return w;
}

template <typename TX, typename TY, typename TZ, bool FX>
cudaError_t launch_chain_t(const ChainEntry *e, const ChainGroup *g, const ChainItem *items, const int *count,
                           uint64_t xb, uint64_t yb, uint64_t zb, uint64_t db, cudaStream_t s, int wide) {
  const int sms = 152;
  cudaError_t err;
  auto next = [&](int cls) {
    const ChainItem *p = items;
    items += count[cls];
    return p;
  };
  const ChainItem *i5 = next(5), *i4 = next(4), *i3 = next(3), *i1 = next(2), *i0 = (next(1), next(0));
  if ((err = launch_items<TX, TY, TZ, FX, 32, 4>(e, g, i5, count[5], 1, xb, yb, zb, db, s)) != cudaSuccess) return err;
  if ((err = launch_items<TX, TY, TZ, FX, 32, 3>(e, g, i4, count[4], 1, xb, yb, zb, db, s)) != cudaSuccess) return err;
  if ((err = launch_items<TX, TY, TZ, FX, 32, 2>(e, g, i3, count[3], 1, xb, yb, zb, db, s)) != cudaSuccess) return err;
  const int n32 = count[2] + count[1];  // rows <= 16 or not: the same kernel here
  const int w32 = wide && FX ? warps_per_item(n32, 8 * sms) : 1;  // FP32: one order of the sum
  if ((err = launch_items<TX, TY, TZ, FX, 32, 1>(e, g, i1, n32, w32, xb, yb, zb, db, s)) != cudaSuccess) return err;
  const int w16 = wide && FX ? warps_per_item(count[0], 16 * sms) : 1;
  return launch_items<TX, TY, TZ, FX, 16, 1>(e, g, i0, count[0], w16, xb, yb, zb, db, s);
}

}  // namespace

cudaError_t launch_chain_fp64(const ChainEntry *e, const ChainGroup *g, const ChainItem *items, const int *count,
                              uint64_t xb, uint64_t yb, uint64_t zb, uint64_t db, cudaStream_t s, int wide) {
  return launch_chain_t<double, double, double, true>(e, g, items, count, xb, yb, zb, db, s, wide);
}

cudaError_t launch_chain_f32ops(const ChainEntry *e, const ChainGroup *g, const ChainItem *items, const int *count,
                                uint64_t xb, uint64_t yb, uint64_t zb, uint64_t db, cudaStream_t s, int wide) {
  return launch_chain_t<float, double, float, false>(e, g, items, count, xb, yb, zb, db, s, wide);
}

// The work items of a group: its kernel class (index into the counts) and columns.
int chain_item_class(int m, int q, int nmax, int pmax) {
  // class 0: what the FP32 kernel for small blocks (chain_pipe.cu) holds in its tiles, at its row pitch
  const int pitch = ((nmax + 3) >> 3 << 3) + 4;
  if (m <= 16 && q <= 16 && nmax <= 32 && pmax <= 16 && std::max(m, pmax) * pitch <= kPipeTile) return 0;
  if (q <= 32) return m <= 16 ? 1 : 2;
  return q <= 64 ? 3 : q <= 96 ? 4 : 5;
}
int chain_item_cols(int cls) { return cls == 0 ? 16 : cls <= 2 ? 32 : 32 * (cls - 1); }

}  // namespace dmrg
