// H.psi on the CUDA cores (sm_103a): D = sum_e f_e X_e Y_e Z_e over prepared operands
// (Sec. 2.2.1, Eq. dgemm: X = A_l, Y = psi^s, Z = A_r^T).
//
// The operators of a position are read by thousands of tasks each, the psi blocks by
// hundreds, so both are put into the form that the inner loops take before the tasks run:
// the operators once per position, psi once per call.  FP64 becomes 58-bit block-scaled
// integers in two limbs (chain_arith.cuh has the arithmetic and its error), 8 bytes an
// element like the double it stands for, with one exponent per block; the FP32 mode rounds
// psi to FP32.
//
// An image of a block is a ready-made run of shared-memory tiles: the summed index cut into
// chunks of 32, each chunk rows x pitch with the summed index contiguous, zeros to the pitch.
// The pitch is 4 banks mod 8, so that the 128-bit loads of a warp (8 rows) are free of
// conflicts; any range of rows of a chunk is one contiguous copy.  A block has two images, of
// itself and of its transpose, so a task's operand needs no transposition on its way in.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>

#include "chain_arith.cuh"
#include "kernels.cuh"

namespace dmrg {

namespace {

constexpr int KD = 32;  // depth of a chunk

// row pitch of a chunk of w columns (elements)
template <bool FX>
__host__ __device__ constexpr int pitch_of(int w) {
  return FX ? ((w + 1) >> 2 << 2) + 2 : ((w + 3) >> 3 << 3) + 4;
}
// elements of an image with R rows and K columns
template <bool FX>
__host__ __device__ constexpr int64_t image_size(int R, int K) {
  return (int64_t)R * ((K / KD) * pitch_of<FX>(KD) + (K % KD ? pitch_of<FX>(K % KD) : 0));
}

// ---------------------------------------------------------------- preparation of operands

template <bool FX, typename T>
__device__ __forceinline__ typename Arith<FX>::Elem convert(T x, int E) {
  if constexpr (FX) return to_limbs((double)x, E);
  else return (float)x;
}

// The image of the R x K view src(r, k) = src[r rs + k cs] by nthr threads.
template <bool FX, typename T>
__device__ __forceinline__ void write_image(typename Arith<FX>::Elem *dst, const T *src, int R, int K, int64_t rs,
                                            int64_t cs, int E, int tid, int nthr) {
  using Elem = typename Arith<FX>::Elem;
  for (int k0 = 0; k0 < K; k0 += KD) {
    const int w = min(KD, K - k0), P = pitch_of<FX>(w);
    for (int t = tid; t < R * P; t += nthr) {
      const int r = t / P, k = t - r * P;
      dst[t] = k < w ? convert<FX>(src[r * rs + (k0 + k) * cs], E) : Elem();
    }
    dst += (int64_t)R * P;
  }
}

template <bool FX, typename T>
__device__ __forceinline__ int block_exponent(const T *src, int64_t n, int lane) {
  if (!FX) return 0;
  TileMax mx;
  for (int64_t i = lane; i < n; i += 32) mx.add((double)src[i]);
  const unsigned hi = __reduce_max_sync(kFull, mx.hi), any = __reduce_or_sync(kFull, mx.any);
  return tile_special(hi, any) ? -1 : (int)(hi >> 20);
}

// Images of the operator blocks, one warp per block.
template <bool FX, typename T>
__global__ void __launch_bounds__(256) op_images_kernel(const OpSlab *__restrict__ S, int nslabs, int64_t nblocks,
                                                        int16_t *exps) {
  using Elem = typename Arith<FX>::Elem;
  const int lane = threadIdx.x & 31;
  for (int64_t b = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); b < nblocks; b += (int64_t)gridDim.x * 8) {
    int lo = 0, hi = nslabs - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (S[mid].first <= b) lo = mid; else hi = mid - 1;
    }
    const OpSlab s = S[lo];
    const int64_t i = b - s.first, size = (int64_t)s.rows * s.cols;
    Elem *img = reinterpret_cast<Elem *>(s.img) + i * (image_size<FX>(s.rows, s.cols) + image_size<FX>(s.cols, s.rows));
    if (s.src == ~0ull) {  // an identity: its own transpose
      for (int k0 = 0; k0 < s.cols; k0 += KD) {
        const int w = min(KD, s.cols - k0), P = pitch_of<FX>(w);
        for (int t = lane; t < s.rows * P; t += 32) img[t] = t / P == k0 + t % P ? Arith<FX>::one() : Elem();
        img += s.rows * P;
      }
      if (lane == 0) exps[b] = 1023;
      continue;
    }
    const T *src = reinterpret_cast<const T *>(s.src * sizeof(T)) + i * size;
    const int E = block_exponent<FX>(src, size, lane);
    if (E >= 0) {
      write_image<FX>(img, src, s.rows, s.cols, s.cols, 1, E, lane, 32);
      write_image<FX>(img + image_size<FX>(s.rows, s.cols), src, s.cols, s.rows, 1, s.cols, E, lane, 32);
    }
    if (lane == 0) exps[b] = (int16_t)E;
  }
}

// Images of the psi blocks, one CTA per block.
template <bool FX>
__global__ void __launch_bounds__(128) psi_images_kernel(const PsiSpan *__restrict__ B, const double *__restrict__ psi,
                                                         typename Arith<FX>::Elem *out, int *exps) {
  __shared__ unsigned red[8];
  const PsiSpan s = B[blockIdx.x];
  const double *src = psi + s.off;
  const int n = s.rows * s.cols, tid = threadIdx.x;
  int E = 0;
  if constexpr (FX) {
    TileMax mx;
    for (int i = tid; i < n; i += 128) mx.add(src[i]);
    unsigned hi = __reduce_max_sync(kFull, mx.hi), any = __reduce_or_sync(kFull, mx.any);
    if ((tid & 31) == 0) {
      red[tid >> 5] = hi;
      red[4 + (tid >> 5)] = any;
    }
    __syncthreads();
    for (int w = 0; w < 4; ++w) {
      hi = max(hi, red[w]);
      any |= red[4 + w];
    }
    E = tile_special(hi, any) ? -1 : (int)(hi >> 20);
    if (tid == 0) exps[blockIdx.x] = E;
    if (E < 0) return;
  }
  write_image<FX>(out + s.img, src, s.rows, s.cols, s.cols, 1, E, tid, 128);
  write_image<FX>(out + s.img + image_size<FX>(s.rows, s.cols), src, s.cols, s.rows, 1, s.cols, E, tid, 128);
}

// The tasks of one chunk in the kernel's order and cut into stacks of consecutive tasks that
// share a psi block.  Limbs: sorted by psi block (kSortSpan at a time), so that those are many;
// FP32 tasks stay in the list's order, in which their FP32 sum is formed.
constexpr int kSortSpan = 1024;

template <bool FX>
__global__ void __launch_bounds__(256) pipe_entries_kernel(const ChainEntry *__restrict__ E,
                                                           const ChainGroup *__restrict__ G, PipeEntry *out,
                                                           PipeStack *stacks, int *nstacks, int *bad, OpTable ops,
                                                           const PsiSpan *__restrict__ B, int nblocks) {
  __shared__ unsigned long long key[kSortSpan];
  __shared__ int run0[kSortSpan];
  __shared__ int run1[kSortSpan];
  __shared__ int warp_sum[9];
  const ChainGroup g = G[blockIdx.x];
  const int tid = threadIdx.x;
  int ns = 0;  // stacks so far
  for (int b0 = 0; b0 < g.count; b0 += kSortSpan) {
    const int cnt = min(kSortSpan, g.count - b0);
    int len = 32;
    while (len < cnt) len *= 2;
    for (int i = tid; i < len; i += 256) {
      unsigned long long k = ~0ull;
      if (i < cnt) {
        const int64_t y = (int64_t)E[g.first + b0 + i].y;
        int lo = 0, hi = nblocks - 1;
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (B[mid].off <= y) lo = mid; else hi = mid - 1;
        }
        // limbs: tasks with a coefficient other than +-2^k run alone
        const double f = E[g.first + b0 + i].f;
        const bool alone = FX && ((__double2hiint(f) & 0xfffff) != 0 || __double2loint(f) != 0);
        k = (unsigned long long)(2 * lo + (alone ? 1 : 0)) << 32 | (unsigned)i;
      }
      key[i] = k;
    }
    __syncthreads();
    for (int size = 2; FX && size <= len; size *= 2)  // bitonic sort
      for (int stride = size / 2; stride > 0; stride /= 2) {
        for (int i = tid; i < len; i += 256) {
          const int j = i ^ stride;
          if (j > i) {
            const unsigned long long a = key[i], b = key[j];
            if ((a > b) == ((i & size) == 0)) {
              key[i] = b;
              key[j] = a;
            }
          }
        }
        __syncthreads();
      }
    // first and last position of the run that each position belongs to
    for (int i = tid; i < cnt; i += 256) {
      run0[i] = i == 0 || (key[i] >> 32) != (key[i - 1] >> 32) ? i : 0;
      run1[i] = i == cnt - 1 || (key[i] >> 32) != (key[i + 1] >> 32) ? i : cnt;
    }
    __syncthreads();
    for (int d = 1; d < cnt; d *= 2) {
      int v[kSortSpan / 256], w[kSortSpan / 256];
      for (int i = tid, u = 0; i < cnt; i += 256, ++u) {
        v[u] = i >= d ? max(run0[i], run0[i - d]) : run0[i];
        w[u] = i + d < cnt ? min(run1[i], run1[i + d]) : run1[i];
      }
      __syncthreads();
      for (int i = tid, u = 0; i < cnt; i += 256, ++u) {
        run0[i] = v[u];
        run1[i] = w[u];
      }
      __syncthreads();
    }
    for (int i0 = 0; i0 < cnt; i0 += 256) {
      const int i = i0 + tid;
      bool head = false;
      PipeStack st{};
      if (i < cnt) {
        const int yb = (int)(key[i] >> 33);
        const bool alone = (key[i] >> 32) & 1;
        const ChainEntry e = E[g.first + b0 + (int)(unsigned)key[i]];
        const bool xt = e.xcs != 1 || (e.xrs == 1 && e.n > 1), yt = e.ycs != 1 || (e.yrs == 1 && e.p > 1),
                   zt = e.zcs != 1 || (e.zrs == 1 && g.q > 1);
        // views of whole blocks: X m x n, Y n x p, Z p x q, row-major or transposed
        const bool xi = e.x == ~0ull, zi = e.z == ~0ull;
        const bool ok = e.n <= kPipeMaxN && e.p <= 65535 && e.y != ~0ull &&
                        (xi ? e.n == g.m : xt ? e.xrs == 1 && (e.n == 1 || e.xcs == g.m)
                                              : e.xcs == 1 && (g.m == 1 || e.xrs == e.n)) &&
                        (yt ? e.yrs == 1 && (e.p == 1 || e.ycs == e.n) : e.ycs == 1 && (e.n == 1 || e.yrs == e.p)) &&
                        (zi ? e.p == g.q : zt ? e.zrs == 1 && (g.q == 1 || e.zcs == e.p)
                                              : e.zcs == 1 && (e.p == 1 || e.zrs == g.q));
        PipeEntry p{};
        p.f = e.f;
        auto find = [&](uint64_t addr, int dim, bool transposed, uint64_t &img) -> int {
          int lo = 0, hi = ops.n - 1;
          int64_t i = 0;
          if (addr == ~0ull) {
            if (dim > ops.max_id) return -2;
            lo = ops.id[dim];
            if (lo < 0) return -2;
          } else {
            while (lo < hi) {
              const int mid = (lo + hi + 1) >> 1;
              if (ops.s[mid].src <= addr) lo = mid; else hi = mid - 1;
            }
            const uint64_t d = addr - ops.s[lo].src;
            i = (int64_t)(d / ((uint64_t)ops.s[lo].rows * ops.s[lo].cols));
          }
          const OpSlab s = ops.s[lo];
          const int64_t one = image_size<FX>(s.rows, s.cols);
          img = s.img + (uint64_t)((i * (one + image_size<FX>(s.cols, s.rows)) +
                                    (transposed && addr != ~0ull ? one : 0)) * (int64_t)sizeof(typename Arith<FX>::Elem));
          return ops.exps[s.first + i];
        };
        int ex = 0, ez = 0;
        if (ok) {
          ex = find(e.x, e.n, xt, p.x);
          ez = find(e.z, e.p, !zt, p.z);
        }
        if (!ok || ex == -2 || ez == -2) *bad = 1;
        const int ef = (__double2hiint(e.f) >> 20) & 0x7ff;
        if (FX && (ef > 1023 + 100 || ef < 1023 - 100)) ex = -1;  // a coefficient that needs FP64
        p.w = FX ? (ex < 0 || ez < 0 ? INT_MIN : ex + ez + ef) : 0;
        p.src = g.first + b0 + (int)(unsigned)key[i];
        const int cap = alone ? 1 : pipe_stack_cap(FX, g.tile0, g.m, g.q, e.n, e.p);
        head = (i - run0[i]) % cap == 0;
        st.e = g.first + b0 + i;
        st.ns = min(cap, run1[i] - i + 1);
        st.n = (uint16_t)e.n;
        st.p = (uint16_t)e.p;
        const int64_t one = image_size<FX>(B[yb].rows, B[yb].cols);
        st.y = (uint32_t)(B[yb].img + (yt ? 0 : one));  // rows: the columns of Y
        st.yb = yb;
        out[g.first + b0 + i] = p;
      }
      // number of stack heads before this one
      const unsigned ball = __ballot_sync(kFull, head);
      if ((tid & 31) == 0) warp_sum[tid >> 5] = __popc(ball);
      __syncthreads();
      if (tid == 0) {
        int run = 0;
        for (int w = 0; w < 8; ++w) {
          const int x = warp_sum[w];
          warp_sum[w] = run;
          run += x;
        }
        warp_sum[8] = run;
      }
      __syncthreads();
      if (head) stacks[g.first + ns + warp_sum[tid >> 5] + __popc(ball & ((1u << (tid & 31)) - 1))] = st;
      ns += warp_sum[8];
      __syncthreads();
    }
  }
  if (tid == 0) nstacks[blockIdx.x] = ns;
  if (FX) {  // stacks with a member that fixed point does not take are marked
    __threadfence_block();
    __syncthreads();
    for (int i = tid; i < ns; i += 256) {
      PipeStack &st = stacks[g.first + i];
      bool special = false;
      for (int j = 0; j < st.ns; ++j) special |= out[st.e + j].w == INT_MIN;
      st.flags = special ? 1 : 0;
    }
  }
}

// ---------------------------------------------------------------- the kernel

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void prefetch(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }
// n bytes (a multiple of 16) by the threads tid of nthr
__device__ __forceinline__ void copy_run(void *dst, const void *src, int n, int tid, int nthr) {
#pragma unroll 1
  for (int o = tid * 16; o < n; o += nthr * 16)
    cp_async16(static_cast<char *>(dst) + o, static_cast<const char *>(src) + o);
}

// Barrier of the group of threads [id nthr, (id + 1) nthr) of the CTA (whole warps).
__device__ __forceinline__ void group_sync(int id, int nthr) {
  if (nthr == 32)
    __syncwarp();
  else
    asm volatile("bar.sync %0, %1;" ::"r"(id + 1), "r"(nthr) : "memory");
}

// Group shapes.  A warp has 16 rows.  SMALL: output blocks of at most 16 x 16 and tasks whose X,
// Y and Z fit kPipeTile, 16 columns a warp; else 32 columns.
//
// Threads an SM holds of the kernel for small blocks.  At 512 a lane's 128 registers do not hold
// the limb sums, two stacks' descriptions and the addresses; measured at 384 / 512: H psi, 8
// orbitals, M 64: 196 / 216 us; 16 vectors, 24 orbitals, M 512: 13.4 / 12.8 ms; Davidson, 10
// orbitals, M 128: 157 / 168 ms.
constexpr int kSmallThreads = 384;
template <bool FX, bool SMALL, int WC>
struct PipeShape {
  static constexpr int NA = 4;              // rows per lane
  static constexpr int NB = SMALL ? 2 : 4;  // columns per lane
  static constexpr int CW = 8 * NB;         // columns of a warp
  static constexpr int PI = pitch_of<FX>(KD);  // row pitch of a whole chunk
  static constexpr int MAXTHREADS = WC == 1 ? 128 : 64 * WC;
  static constexpr int MINB = (SMALL ? kSmallThreads : WC == 4 ? 256 : 384) / MAXTHREADS;
};

// Shared memory of a group (elements): the X tile, each of the two Y / Z buffers, and the T tiles
// with row pitch pt, sized for the largest dimensions of the launch's tasks.
struct PipeSmem {
  int x, b, pt, group;
};

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

// One work item per CTA: rows [r0, r0 + 16 wr) and columns [c0, c0 + CW WC) of one chunk's
// output block.  The CTA holds one group of wr x WC warps, or (WC = 1) several that take the
// chunk's stacks in turn and whose sums are added in group order.  Lane (i, j) of a warp's
// 4 x 8 lane grid has rows i + 4 a and columns j + 8 b of the warp's tile, so a ragged block
// wastes at most 3 rows and 7 columns.
//
// A group works through units: for every stack and every CW WC columns of T, the chunks of
// stage 1 (T = X Y) and then those of stage 2 (D += f T Z).  A unit's tiles are copied while
// the unit before it is computed: X to its own buffer, Y and Z to two buffers in turn.
//
// The X of a stack's tasks lie below one another in the X tile, so stage 1 is one product with
// the Y that they share; their parts of T lie beside one another, and stage 2 sums over them.
// For that the parts of T get one scale, coefficients +-2^k and all; a task with another
// coefficient (a one-site term) is a stack of its own.
template <bool FX, bool SMALL, int WC>
__global__ void __launch_bounds__(PipeShape<FX, SMALL, WC>::MAXTHREADS, PipeShape<FX, SMALL, WC>::MINB)
    chain_pipe_kernel(const PipeEntry *__restrict__ E, const PipeStack *__restrict__ stacks,
                      const int *__restrict__ nstacks, const ChainEntry *__restrict__ tasks,
                      const ChainGroup *__restrict__ G, const ChainItem *__restrict__ items, int wr, PipeSmem sm,
                      const typename Arith<FX>::Elem *__restrict__ psi, const int *__restrict__ pexp,
                      const double *__restrict__ psi64, uint64_t db) {
  using A = Arith<FX>;
  using Elem = typename A::Elem;
  using Out = typename A::Out;
  using Acc = typename A::Acc;
  using S = PipeShape<FX, SMALL, WC>;
  constexpr int NA = S::NA, NB = S::NB, CW = S::CW, PI = S::PI, VK = A::VK, ES = (int)sizeof(Elem);
  extern __shared__ __align__(16) unsigned char pipe_smem[];
  __shared__ int te[8][WC];   // exponents of the T tiles
  const int gthr = 32 * wr * WC;
  const int grp = WC == 1 ? (int)threadIdx.x / gthr : 0, ngrp = WC == 1 ? (int)blockDim.x / gthr : 1;
  const int tid = (int)threadIdx.x - grp * gthr, warp = tid >> 5, lane = tid & 31;
  const int wrow = warp / WC, wcol = warp % WC;
  const int lr = lane >> 3, lc = lane & 7;
  const int PT = sm.pt;
  Elem *Xs = reinterpret_cast<Elem *>(pipe_smem) + grp * sm.group;
  Elem *Bs = Xs + sm.x;
  Elem *Ts = Bs + 2 * sm.b + wrow * WC * 16 * PT;  // this warp row's tiles
  int *tex = WC > 1 ? te[wrow] : te[threadIdx.x >> 5];
  const ChainItem it = items[blockIdx.x];
  const ChainGroup *gp = G + it.g;
  const int gm = gp->m, gq = gp->q, gfirst = gp->first;
  const int nst = nstacks[it.g];
  const PipeStack *stk = stacks + gfirst;
  const int mi = min(16 * wr, gm - it.r0), qi = min(CW * WC, gq - it.c0);  // of the item
  const int rw = WC == 1 && wr == 1 ? 16 : (mi + 4 * wr - 1) / (4 * wr) * 4;  // rows of a warp
  const int m = min(rw, mi - rw * wrow);                                     // of this warp
  const int q = min(CW, qi - CW * wcol);
  Out D[4][NB];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < NB; ++b) D[a][b] = 0;
  bool any_special = false;
  // FP32 sums over the inner dimension keep one order: chunks of 32 added up for blocks of at
  // most 32 x 32, running on for larger ones
  const bool apart = !FX && gm <= 32 && gq <= 32;

  // A stack (PipeStack as read, and the exponent of its Y).  It is read one stack ahead, and
  // what it points to is asked for in time, so that no copy waits for a chain of loads.
  struct Stack {
    int4 d;
    int ey;
    __device__ __forceinline__ int e() const { return d.x; }
    __device__ __forceinline__ int n() const { return d.y & 0xffff; }
    __device__ __forceinline__ int p() const { return (int)((unsigned)d.y >> 16); }
    __device__ __forceinline__ uint32_t y() const { return (uint32_t)d.z; }
    __device__ __forceinline__ int yb() const { return d.w & 0xffffff; }
    __device__ __forceinline__ int ns() const { return (d.w >> 24) & 15; }
    __device__ __forceinline__ bool special() const { return (unsigned)d.w >> 28 || ey < 0; }
  };
  int si = grp;
  auto member = [&](int ns) { return ns <= 1 ? 0 : tid >> (5 - (32 - __clz(ns - 1))); };  // stacks: one warp
  auto take = [&](Stack &t) {  // ns() = 0: no further stack of this group
    t.d = si < nst ? *reinterpret_cast<const int4 *>(stk + si) : make_int4(0, 0, 0, 0);
    t.ey = 0;
    si += ngrp;
  };
  auto ask = [&](Stack &t) {  // for the exponent of Y and this thread's share of the entries
    if (t.ns() == 0) return;
    if (FX) t.ey = pexp[t.yb()];
    prefetch(E + t.e() + min(member(t.ns()), t.ns() - 1));
  };
  auto skip_special = [&](Stack &t) {
    while (FX && t.ns() > 0 && t.special()) {
      any_special = true;
      take(t);
      ask(t);
    }
  };
  // Copy the tiles of a unit of t: chunk c of stage 1 or (two) of stage 2, columns of T from p0.
  auto copy_unit = [&](const Stack &t, int p0, int c, bool two, Elem *B) {
    const int ns = t.ns(), lg = ns <= 1 ? 0 : 32 - __clz(ns - 1), mem = lg ? tid >> (5 - lg) : 0, sub = gthr >> lg,
              st = lg ? tid & (sub - 1) : tid;
    const int k0 = two ? p0 + c * CW : c * KD;  // summed index
    const int w = min(KD, (two ? t.p() : t.n()) - k0), P = pitch_of<FX>(w);
    const int R = two ? gq : gm, r0 = two ? it.c0 : it.r0, rows = two ? qi : mi;
    if (mem < ns) {
      const PipeEntry &e = E[t.e() + mem];
      copy_run((two ? B : Xs) + mem * rows * P,
               reinterpret_cast<const char *>(two ? e.z : e.x) + ((int64_t)(k0 / KD) * R * PI + r0 * P) * ES, rows * P * ES,
               st, sub);
    }
    if (!two)
      copy_run(B, psi + t.y() + (int64_t)(k0 / KD) * t.p() * PI + p0 * P, min(CW * WC, t.p() - p0) * P * ES, tid, gthr);
    cp_commit();
  };

  Stack u, nx;  // the stack at hand and the next one
  take(u);
  ask(u);
  skip_special(u);
  if (u.ns() > 0) {
    copy_unit(u, 0, 0, false, Bs);
    take(nx);
  }
  int p0 = 0, c = 0;
  bool two = false;
  int par_b = 0;  // buffer of the current unit
  Acc acc[NA][NB];
#pragma unroll 1
  while (u.ns() > 0) {
    const int nch = (u.n() + KD - 1) / KD;
    // the unit after this one
    int vp = p0, vc = c + 1;
    bool vtwo = two, over = false;
    if (!two) {
      if (vc >= nch) {
        vc = 0;
        vtwo = true;
      }
    } else if (WC == 1 || vc >= min(WC, (u.p() - p0 + CW - 1) / CW)) {
      vc = 0;
      vtwo = false;
      vp += CW * WC;
      if (vp >= u.p()) {
        vp = 0;
        over = true;
      }
    }
    cp_wait<0>();
    group_sync(grp, gthr);  // the tiles are here, the unit before this one has been computed
    const bool late = !over && !two && !vtwo;  // X is still in use: copied after this unit
    if (!two && c == 0 && p0 == 0) ask(nx);
    if (over) {
      skip_special(nx);
      if (nx.ns() > 0) copy_unit(nx, 0, 0, false, Bs + (par_b ^ 1) * sm.b);
    } else if (!late) {
      copy_unit(u, vp, vc, vtwo, Bs + (par_b ^ 1) * sm.b);
    }
    const Elem *B = Bs + par_b * sm.b;
    const int ns = u.ns();
    const int pc = min(CW, u.p() - p0 - CW * (two ? c : wcol));  // columns of the T tile at hand
    const int pt = (pc + VK - 1) / VK * VK;                          // a member's columns in the tile
    const bool busy = m > 0 && (two ? q : pc) > 0;
    const int rows = two ? m : ns * m, na = (rows + 3) >> 2, nb = ((two ? q : pc) + 7) >> 3;
    if (busy) {
      // ---- sums of the unit: X Y, or over the members of T Z
      const int kc = two ? pc : min(KD, u.n() - c * KD), P = pitch_of<FX>(kc);
      if (two || c == 0 || apart) {
#pragma unroll
        for (int a = 0; a < NA; ++a)
#pragma unroll
          for (int b = 0; b < NB; ++b) acc[a][b] = Acc{};
      } else {
#pragma unroll
        for (int a = 0; a < NA; ++a)
#pragma unroll
          for (int b = 0; b < NB; ++b) carry(acc[a][b]);
      }
      const Elem *Ar = two ? Ts + c * 16 * PT + lr * PT : Xs + (rw * wrow + lr) * P;
      const Elem *Br = B + (wcol * CW + lc) * P;
#pragma unroll 1
      for (int mem = 0; mem < (two ? ns : 1); ++mem, Ar += pt, Br += qi * P) {
        mm_any(Ar, two ? PT : P, Br, P, kc, na, nb, acc);
        if constexpr (!FX) {
          if (two) {  // D += f (T Z), task by task
            const float f = (float)E[u.e() + mem].f;
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
              for (int b = 0; b < NB; ++b) {
                D[a][b] = fmaf(f, acc[a][b], D[a][b]);
                acc[a][b] = 0.f;
              }
          }
        }
      }
    }
    if (busy && two) {
      if constexpr (FX) {  // D += 2^e (sums)
        // a single task's coefficient is applied here; those of a stack are +-2^k and are in T
        const double f1 = ns == 1 ? E[u.e()].f : 1.0;
        const int e2 = 58 - 1 + (WC > 1 ? tex[c] : tex[0]);
        const double sc = __hiloint2double((__double2hiint(f1) & 0x800fffff) | ((e2 + 1023) << 20), __double2loint(f1));
#pragma unroll
        for (int a = 0; a < 4; ++a)
          if (a < na) {
#pragma unroll
            for (int b = 0; b < NB; ++b)
              if (b < nb) D[a][b] = fma(sc, (double)fold(acc[a][b], 1), D[a][b]);
          }
      }
    } else if (busy) {
      if (apart || c == nch - 1) {
        Elem *T = Ts + wcol * 16 * PT + lc;
        const float invm = 1.0f / (float)m;
        if constexpr (FX) {
          // the members' weights below the largest one (bits 0-5) and signs (bit 8): their parts
          // of T get one scale
          const int w = lane < ns ? E[u.e() + lane].w : INT_MIN;
          const int wmax = __reduce_max_sync(kFull, w);
          int below = 0;
          if (ns > 1 && lane < ns) below = min(wmax - w, 62) | (__double2hiint(E[u.e() + lane].f) < 0 ? 256 : 0);
          unsigned mx = 0;
#pragma unroll
          for (int a = 0; a < NA; ++a)
            if (a < na) {
              const int row = lr + 4 * a, sh = ns > 1 ? __shfl_sync(kFull, below, small_div(row, invm)) & 63 : 0;
#pragma unroll
              for (int b = 0; b < NB; ++b) {
                const unsigned h = sh < 32 ? magnitude(acc[a][b].hh) >> sh : 0u;
                mx = max(mx, b < nb && lc + 8 * b < pc && row < rows ? h : 0u);
              }
            }
          mx = __reduce_max_sync(kFull, mx);
          const int up = __clz(mx | 1) - 7;  // T = hh 2^(up - sh) + cross, below 2^57
          if (lane == 0) tex[WC > 1 ? wcol : 0] = wmax + u.ey - 2158 - 1023 - 1079 + 58 - up;
          const bool down = ns > 1 || up < 0;
#pragma unroll
          for (int a = 0; a < NA; ++a) {
            if (a < na) {
              const int row = lr + 4 * a, mem = ns > 1 ? small_div(row, invm) : 0;
              const int v = ns > 1 ? __shfl_sync(kFull, below, mem) : 0;
              const int net = up - (v & 63), l = max(net, 0), r = max(-net, 0);
              const long long half = 1ll << (28 - l), rhalf = (1ll << r) >> 1, sg = -(long long)(v >> 8);
              Elem *Tr = T + (row - mem * m) * PT + mem * pt;
              if (row < rows) {
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                  if (lc + 8 * b < pt) {
                    long long t = (acc[a][b].hh << l) + ((acc[a][b].cr + half) >> (29 - l));
                    if (down) t = (((t + rhalf) >> r) ^ sg) - sg;
                    Tr[8 * b] = lc + 8 * b < pc ? limbs(t) : Elem();
                  }
                }
              }
            }
          }
        } else {
#pragma unroll
          for (int a = 0; a < NA; ++a) {
            if (a < na) {
              const int row = lr + 4 * a, mem = ns > 1 ? small_div(row, invm) : 0;
              if (row < rows) {
                Elem *Tr = T + (row - mem * m) * PT + mem * pt;
#pragma unroll
                for (int b = 0; b < NB; ++b)
                  if (lc + 8 * b < pt)
                    Tr[8 * b] = lc + 8 * b < pc ? (apart && c > 0 ? Tr[8 * b] + acc[a][b] : acc[a][b]) : 0.f;
              }
            }
          }
        }
      }
    }
    if (late) {
      group_sync(grp, gthr);
      copy_unit(u, vp, vc, vtwo, Bs + (par_b ^ 1) * sm.b);
    }
    par_b ^= 1;
    p0 = vp;
    c = vc;
    two = vtwo;
    if (over) {
      u = nx;
      if (u.ns() > 0) take(nx);
    }
  }
  if constexpr (WC == 1) {
    if (ngrp > 1) {  // the groups' sums, added in group order
      __syncthreads();
      Out *mine = reinterpret_cast<Out *>(pipe_smem) + (size_t)threadIdx.x * (4 * NB + 1);
      if (grp > 0) {
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < NB; ++b) mine[a * NB + b] = D[a][b];
      }
      __syncthreads();
      if (grp == 0) {
        for (int h = 1; h < ngrp; ++h) {
          const Out *other = reinterpret_cast<const Out *>(pipe_smem) + (size_t)(h * gthr + tid) * (4 * NB + 1);
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < NB; ++b) D[a][b] += other[a * NB + b];
        }
      }
    }
  }
  if (grp == 0) {
    const int drs = gp->drs, dcs = gp->dcs;
    double *Dout = reinterpret_cast<double *>(db + gp->d * 8ull) + (int64_t)(it.r0 + rw * wrow) * drs +
                   (int64_t)(it.c0 + CW * wcol) * dcs;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < NB; ++b)
        if (lr + 4 * a < m && lc + 8 * b < q)
          Dout[(int64_t)(lr + 4 * a) * drs + (int64_t)(lc + 8 * b) * dcs] = (double)D[a][b];
  }
  if constexpr (FX) {
    if (__syncthreads_or(any_special))
      slow_stacks(E, stk, nst, tasks, pexp, psi64, gp, it.r0, it.c0, mi, qi, db, reinterpret_cast<double *>(pipe_smem));
  }
}

// Groups that share a chunk's tasks: chunks of many tasks are shared, so that no CTA runs on
// when the others are done, and so are chunks that alone would not fill the GPU.
int groups_per_item(int n, int64_t tasks, int wr, int resident) {
  int k = 1;
  while (32 * wr * k < 128 && ((long long)n * wr * k < resident || tasks > 16ll * k * n)) k *= 2;
  return k;
}

template <bool FX, bool SMALL, int WC>
cudaError_t launch_pipe(const PipeArgs &a, const ChainItem *items, const PipeClass &c, int wr, bool share,
                        cudaStream_t s) {
  if (c.items <= 0) return cudaSuccess;
  using S = PipeShape<FX, SMALL, WC>;
  using Elem = typename Arith<FX>::Elem;
  auto pitch = [](int w) { return pitch_of<FX>(w < KD ? w : KD); };
  const int mx = SMALL ? 0 : std::min(c.m, 16 * wr), qx = std::min(c.q, S::CW * WC), px = std::min(c.p, S::CW * WC);
  PipeSmem sm;
  // stacks of the small classes fill tiles of fixed size (pipe_stack_cap)
  sm.x = SMALL ? kPipeTile : wr == 1 ? 16 * pitch(c.n) : mx * pitch(c.n);
  sm.b = SMALL ? kPipeTile : std::max(px * pitch(c.n), (wr == 1 ? 32 : qx) * pitch(c.p));
  sm.pt = WC == 1 && c.p > 16 ? pitch(c.p) : pitch(KD);
  if (wr == 1) sm.pt = pitch(SMALL ? 16 : KD);
  sm.group = sm.x + 2 * sm.b + wr * WC * 16 * sm.pt;
  sm.group = std::max(sm.group, 32 * wr * WC * (4 * S::NB + 1));  // the exchange of the groups' sums
  const int bytes = sm.group * (int)sizeof(Elem);
  const int groups = share && FX ? groups_per_item(c.items, c.tasks, wr, (SMALL ? kSmallThreads / 32 : 12) * 152) : 1;
  auto kern = chain_pipe_kernel<FX, SMALL, WC>;
  const cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
  if (err != cudaSuccess) return err;
  add_kernel_launches(1);
  kern<<<c.items, 32 * wr * WC * groups, groups * bytes, s>>>(a.e, a.stacks, a.nstacks, a.tasks, a.g, items, wr, sm,
                                                             static_cast<const Elem *>(a.psi), a.pexp, a.psi64, a.db);
  return cudaGetLastError();
}

template <bool FX>
cudaError_t launch_pipe_all(const PipeArgs &a, const ChainItem *items, const PipeClass *c, bool wide, cudaStream_t s,
                            cudaStream_t s1, cudaStream_t s2) {
  cudaError_t err;
  auto next = [&](int cls) {
    const ChainItem *p = items;
    items += c[cls].items;
    return p;
  };
  const ChainItem *i5 = next(5), *i4 = next(4), *i3 = next(3), *i2 = next(2), *i1 = next(1), *i0 = next(0);
  if ((err = launch_pipe<FX, false, 4>(a, i5, c[5], 2, false, s1)) != cudaSuccess) return err;
  if ((err = launch_pipe<FX, false, 3>(a, i4, c[4], 2, false, s)) != cudaSuccess) return err;
  if ((err = launch_pipe<FX, false, 2>(a, i3, c[3], 2, false, s1)) != cudaSuccess) return err;
  if ((err = launch_pipe<FX, false, 1>(a, i2, c[2], 2, wide, s)) != cudaSuccess) return err;
  if ((err = launch_pipe<FX, false, 1>(a, i1, c[1], 1, wide, s1)) != cudaSuccess) return err;
  return launch_pipe<FX, true, 1>(a, i0, c[0], 1, wide, s2);
}

}  // namespace

cudaError_t launch_chain_pipe(const PipeArgs &a, bool f32, const ChainItem *items, const PipeClass *classes, int wide,
                              cudaStream_t s, cudaStream_t s1, cudaStream_t s2) {
  return f32 ? launch_pipe_all<false>(a, items, classes, wide != 0, s, s1, s2)
             : launch_pipe_all<true>(a, items, classes, wide != 0, s, s1, s2);
}

int64_t pipe_image_size(bool f32, int rows, int cols) {
  return f32 ? image_size<false>(rows, cols) : image_size<true>(rows, cols);
}

cudaError_t launch_op_images(const OpSlab *s, int nslabs, int64_t nblocks, int16_t *exps, bool f32, cudaStream_t st) {
  if (nblocks <= 0) return cudaSuccess;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((nblocks + 7) / 8, 152 * 16));
  add_kernel_launches(1);
  if (f32)
    op_images_kernel<false, float><<<grid, 256, 0, st>>>(s, nslabs, nblocks, exps);
  else
    op_images_kernel<true, double><<<grid, 256, 0, st>>>(s, nslabs, nblocks, exps);
  return cudaGetLastError();
}

cudaError_t launch_psi_images(const PsiSpan *b, int nblocks, const double *psi, void *out, int *exps, bool f32,
                              cudaStream_t st) {
  if (nblocks <= 0) return cudaSuccess;
  add_kernel_launches(1);
  if (f32)
    psi_images_kernel<false><<<nblocks, 128, 0, st>>>(b, psi, static_cast<float *>(out), exps);
  else
    psi_images_kernel<true><<<nblocks, 128, 0, st>>>(b, psi, static_cast<int2 *>(out), exps);
  return cudaGetLastError();
}

cudaError_t launch_pipe_entries(const ChainEntry *e, const ChainGroup *g, int ngroups, PipeEntry *out,
                                PipeStack *stacks, int *nstacks, int *bad, const OpTable &ops, const PsiSpan *b,
                                int nblocks, bool f32, cudaStream_t st) {
  if (ngroups <= 0) return cudaSuccess;
  add_kernel_launches(1);
  if (f32)
    pipe_entries_kernel<false><<<ngroups, 256, 0, st>>>(e, g, out, stacks, nstacks, bad, ops, b, nblocks);
  else
    pipe_entries_kernel<true><<<ngroups, 256, 0, st>>>(e, g, out, stacks, nstacks, bad, ops, b, nblocks);
  return cudaGetLastError();
}

}  // namespace dmrg
