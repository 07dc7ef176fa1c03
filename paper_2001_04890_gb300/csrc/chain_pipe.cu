// Prepared operands of H.psi, D = sum_e f_e X_e Y_e Z_e (Sec. 2.2.1, Eq. dgemm: X = A_l,
// Y = psi^s, Z = A_r^T), and its FP32 products on the CUDA cores (sm_103a).
//
// The operators of a position are read by thousands of tasks each, the psi blocks by
// hundreds, so both are put into the form that the inner loops take before the tasks run:
// the operators once per position, psi once per call.  FP64 becomes digits under one exponent
// per block (chain_digits.cuh, chain_mma.cu); the FP32 mode rounds psi to FP32.
//
// An FP32 image of a block is a ready-made run of shared-memory tiles: the summed index cut into
// chunks of 32, each chunk rows x pitch with the summed index contiguous, zeros to the pitch.
// The pitch is 4 banks mod 8, so that the 128-bit loads of a warp (8 rows) are free of
// conflicts; any range of rows of a chunk is one contiguous copy.  A block has two images, of
// itself and of its transpose, so a task's operand needs no transposition on its way in.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>

#include "chain_arith.cuh"
#include "chain_digits.cuh"
#include "kernels.cuh"

namespace dmrg {

namespace {

constexpr int KD = 32;  // depth of a chunk

// row pitch of a chunk of w columns (elements)
__host__ __device__ constexpr int pitch_of(int w) { return ((w + 3) >> 3 << 3) + 4; }
// elements of an image with R rows and K columns (FX: of 8 bytes)
template <bool FX>
__host__ __device__ constexpr int64_t image_size(int R, int K) {
  return FX ? dig_image_size(R, K) : (int64_t)R * ((K / KD) * pitch_of(KD) + (K % KD ? pitch_of(K % KD) : 0));
}

// ---------------------------------------------------------------- preparation of operands

template <bool FX>
using ImageElem = typename Arith<FX>::Elem;  // 8 bytes, or a float

// The image of an R x K block whose element (r, k) is get(r, k), an integer or a float, by nthr threads.
template <bool FX, bool OPERATOR, class Get>
__device__ __forceinline__ void write_image(ImageElem<FX> *dst, int R, int K, int tid, int nthr, Get get) {
  if constexpr (FX) {
    write_digits<OPERATOR>(dst, R, K, tid, nthr, get);
  } else {
    for (int k0 = 0; k0 < K; k0 += KD) {
      const int w = min(KD, K - k0), P = pitch_of(w);
      for (int t = tid; t < R * P; t += nthr) {
        const int r = t / P, k = t - r * P;
        dst[t] = k < w ? get(r, k0 + k) : 0.f;
      }
      dst += (int64_t)R * P;
    }
  }
}
// and of the view src[r rs + k cs]
template <bool FX, bool OPERATOR, typename T>
__device__ __forceinline__ void write_view(ImageElem<FX> *dst, const T *src, int R, int K, int64_t rs, int64_t cs, int E,
                                           int tid, int nthr) {
  write_image<FX, OPERATOR>(dst, R, K, tid, nthr, [&](int r, int k) {
    if constexpr (FX) return to_fixed((double)src[r * rs + k * cs], E);
    else return (float)src[r * rs + k * cs];
  });
}

template <bool FX, typename T>
__device__ __forceinline__ int block_exponent(const T *src, int64_t n, int lane) {
  if (!FX) return 0;
  TileMax mx;
  for (int64_t i = lane; i < n; i += 32) mx.add((double)src[i]);
  const unsigned hi = __reduce_max_sync(kFull, mx.hi), any = __reduce_or_sync(kFull, mx.any);
  return zero_as_one(tile_exponent(hi, any));
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
      write_image<FX, true>(img, s.rows, s.cols, lane, 32, [](int r, int k) {
        if constexpr (FX) return r == k ? 1ll << 57 : 0ll;
        else return r == k ? 1.f : 0.f;
      });
      if (lane == 0) exps[b] = 1023;
      continue;
    }
    const T *src = reinterpret_cast<const T *>(s.src * sizeof(T)) + i * size;
    const int E = block_exponent<FX>(src, size, lane);
    if (E >= 0) {
      write_view<FX, true>(img, src, s.rows, s.cols, s.cols, 1, E, lane, 32);
      write_view<FX, true>(img + image_size<FX>(s.rows, s.cols), src, s.cols, s.rows, 1, s.cols, E, lane, 32);
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
    E = zero_as_one(tile_exponent(hi, any));
    if (tid == 0) exps[blockIdx.x] = E;
    if (E < 0) return;
  }
  write_view<FX, false>(out + s.img, src, s.rows, s.cols, s.cols, 1, E, tid, 128);
  write_view<FX, false>(out + s.img + image_size<FX>(s.rows, s.cols), src, s.cols, s.rows, 1, s.cols, E, tid, 128);
}

// The tasks of one chunk in the kernel's order and cut into stacks of consecutive tasks that
// share a psi block.  Digits: sorted by psi block (kSortSpan at a time), so that those are many;
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
        k = (unsigned long long)lo << 32 | (unsigned)i;
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
        const int yb = (int)(key[i] >> 32);
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
        const int cap = pipe_stack_cap(FX, g.cls, g.m, g.q, e.n, e.p);
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

// ---------------------------------------------------------------- the FP32 kernel

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

// CTA shapes.  A warp has 16 rows.  SMALL: output blocks of at most 16 x 16 and tasks whose X,
// Y and Z fit kPipeTile, 16 columns a warp; else 32 columns.
template <bool SMALL, int WC>
struct PipeShape {
  static constexpr int NA = 4;              // rows per lane
  static constexpr int NB = SMALL ? 2 : 4;  // columns per lane
  static constexpr int CW = 8 * NB;         // columns of a warp
  static constexpr int PI = pitch_of(KD);   // row pitch of a whole chunk
  static constexpr int MAXTHREADS = 64 * WC;
  static constexpr int MINB = (WC == 4 ? 256 : 384) / MAXTHREADS;
};

// Shared memory (elements): the X tile, each of the two Y / Z buffers, and the T tiles with row
// pitch pt, sized for the largest dimensions of the launch's tasks.
struct PipeSmem {
  int x, b, pt, total;
};

// One work item per CTA: rows [r0, r0 + 16 wr) and columns [c0, c0 + CW WC) of one chunk's
// output block, wr x WC warps.  Lane (i, j) of a warp's 4 x 8 lane grid has rows i + 4 a and
// columns j + 8 b of the warp's tile, so a ragged block wastes at most 3 rows and 7 columns.
//
// The CTA works through units: for every stack and every CW WC columns of T, the chunks of
// stage 1 (T = X Y) and then those of stage 2 (D += f T Z).  A unit's tiles are copied while
// the unit before it is computed: X to its own buffer, Y and Z to two buffers in turn.
//
// The X of a stack's tasks lie below one another in the X tile, so stage 1 is one product with
// the Y that they share; their parts of T lie beside one another, and stage 2 adds their
// products to D task by task: the FP32 sums are formed in the task list's order, whatever the
// shapes and stacks.
template <bool SMALL, int WC>
__global__ void __launch_bounds__(PipeShape<SMALL, WC>::MAXTHREADS, PipeShape<SMALL, WC>::MINB)
    chain_pipe_kernel(const PipeEntry *__restrict__ E, const PipeStack *__restrict__ stacks,
                      const int *__restrict__ nstacks, const ChainGroup *__restrict__ G,
                      const ChainItem *__restrict__ items, int wr, PipeSmem sm, const float *__restrict__ psi,
                      uint64_t db) {
  using S = PipeShape<SMALL, WC>;
  constexpr int NA = S::NA, NB = S::NB, CW = S::CW, PI = S::PI, VK = 4, ES = (int)sizeof(float);
  extern __shared__ __align__(16) unsigned char pipe_smem[];
  const int nthr = 32 * wr * WC, tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wrow = warp / WC, wcol = warp % WC;
  const int lr = lane >> 3, lc = lane & 7;
  const int PT = sm.pt;
  float *Xs = reinterpret_cast<float *>(pipe_smem);
  float *Bs = Xs + sm.x;
  float *Ts = Bs + 2 * sm.b + wrow * WC * 16 * PT;  // this warp row's tiles
  const ChainItem it = items[blockIdx.x];
  const ChainGroup *gp = G + it.g;
  const int gm = gp->m, gq = gp->q, gfirst = gp->first;
  const int nst = nstacks[it.g];
  const PipeStack *stk = stacks + gfirst;
  const int mi = min(16 * wr, gm - it.r0), qi = min(CW * WC, gq - it.c0);  // of the item
  const int rw = WC == 1 && wr == 1 ? 16 : (mi + 4 * wr - 1) / (4 * wr) * 4;  // rows of a warp
  const int m = min(rw, mi - rw * wrow);                                     // of this warp
  const int q = min(CW, qi - CW * wcol);
  float D[4][NB];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < NB; ++b) D[a][b] = 0.f;
  // sums over the inner dimension keep one order: chunks of 32 added up for blocks of at
  // most 32 x 32, running on for larger ones
  const bool apart = gm <= 32 && gq <= 32;

  auto sync = [&]() {
    if (nthr == 32) __syncwarp();
    else __syncthreads();
  };
  // A stack (PipeStack as read).  It is read one stack ahead, and what it points to is asked for in
  // time, so that no copy waits for a chain of loads.
  struct Stack {
    int4 d;
    __device__ __forceinline__ int e() const { return d.x; }
    __device__ __forceinline__ int n() const { return d.y & 0xffff; }
    __device__ __forceinline__ int p() const { return (int)((unsigned)d.y >> 16); }
    __device__ __forceinline__ uint32_t y() const { return (uint32_t)d.z; }
    __device__ __forceinline__ int ns() const { return (d.w >> 24) & 15; }
  };
  int si = 0;
  auto member = [&](int ns) { return ns <= 1 ? 0 : tid >> (5 - (32 - __clz(ns - 1))); };  // stacks: one warp
  auto take = [&](Stack &t) {  // ns() = 0: no further stack
    t.d = si < nst ? *reinterpret_cast<const int4 *>(stk + si) : make_int4(0, 0, 0, 0);
    ++si;
  };
  auto ask = [&](const Stack &t) {  // for this thread's share of the entries
    if (t.ns() > 0) prefetch(E + t.e() + min(member(t.ns()), t.ns() - 1));
  };
  // Copy the tiles of a unit of t: chunk c of stage 1 or (two) of stage 2, columns of T from p0.
  auto copy_unit = [&](const Stack &t, int p0, int c, bool two, float *B) {
    const int ns = t.ns(), lg = ns <= 1 ? 0 : 32 - __clz(ns - 1), mem = lg ? tid >> (5 - lg) : 0, sub = nthr >> lg,
              st = lg ? tid & (sub - 1) : tid;
    const int k0 = two ? p0 + c * CW : c * KD;  // summed index
    const int w = min(KD, (two ? t.p() : t.n()) - k0), P = pitch_of(w);
    const int R = two ? gq : gm, r0 = two ? it.c0 : it.r0, rows = two ? qi : mi;
    if (mem < ns) {
      const PipeEntry &e = E[t.e() + mem];
      copy_run((two ? B : Xs) + mem * rows * P,
               reinterpret_cast<const char *>(two ? e.z : e.x) + ((int64_t)(k0 / KD) * R * PI + r0 * P) * ES, rows * P * ES,
               st, sub);
    }
    if (!two)
      copy_run(B, psi + t.y() + (int64_t)(k0 / KD) * t.p() * PI + p0 * P, min(CW * WC, t.p() - p0) * P * ES, tid, nthr);
    cp_commit();
  };

  Stack u, nx;  // the stack at hand and the next one
  take(u);
  ask(u);
  if (u.ns() > 0) {
    copy_unit(u, 0, 0, false, Bs);
    take(nx);
  }
  int p0 = 0, c = 0;
  bool two = false;
  int par_b = 0;  // buffer of the current unit
  float acc[NA][NB];
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
    sync();  // the tiles are here, the unit before this one has been computed
    const bool late = !over && !two && !vtwo;  // X is still in use: copied after this unit
    if (!two && c == 0 && p0 == 0) ask(nx);
    if (over) {
      if (nx.ns() > 0) copy_unit(nx, 0, 0, false, Bs + (par_b ^ 1) * sm.b);
    } else if (!late) {
      copy_unit(u, vp, vc, vtwo, Bs + (par_b ^ 1) * sm.b);
    }
    const float *B = Bs + par_b * sm.b;
    const int ns = u.ns();
    const int pc = min(CW, u.p() - p0 - CW * (two ? c : wcol));  // columns of the T tile at hand
    const int pt = (pc + VK - 1) / VK * VK;                          // a member's columns in the tile
    const bool busy = m > 0 && (two ? q : pc) > 0;
    const int rows = two ? m : ns * m, na = (rows + 3) >> 2, nb = ((two ? q : pc) + 7) >> 3;
    if (busy) {
      // ---- sums of the unit: X Y, or member by member T Z
      const int kc = two ? pc : min(KD, u.n() - c * KD), P = pitch_of(kc);
      if (two || c == 0 || apart) {
#pragma unroll
        for (int a = 0; a < NA; ++a)
#pragma unroll
          for (int b = 0; b < NB; ++b) acc[a][b] = 0.f;
      }
      const float *Ar = two ? Ts + c * 16 * PT + lr * PT : Xs + (rw * wrow + lr) * P;
      const float *Br = B + (wcol * CW + lc) * P;
#pragma unroll 1
      for (int mem = 0; mem < (two ? ns : 1); ++mem, Ar += pt, Br += qi * P) {
        mm_any(Ar, two ? PT : P, Br, P, kc, na, nb, acc);
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
    if (busy && !two && (apart || c == nch - 1)) {
      float *T = Ts + wcol * 16 * PT + lc;
      const float invm = 1.0f / (float)m;
#pragma unroll
      for (int a = 0; a < NA; ++a) {
        if (a < na) {
          const int row = lr + 4 * a, mem = ns > 1 ? small_div(row, invm) : 0;
          if (row < rows) {
            float *Tr = T + (row - mem * m) * PT + mem * pt;
#pragma unroll
            for (int b = 0; b < NB; ++b)
              if (lc + 8 * b < pt)
                Tr[8 * b] = lc + 8 * b < pc ? (apart && c > 0 ? Tr[8 * b] + acc[a][b] : acc[a][b]) : 0.f;
          }
        }
      }
    }
    if (late) {
      sync();
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

template <bool SMALL, int WC>
cudaError_t launch_pipe(const PipeArgs &a, const ChainItem *items, const PipeClass &c, int wr, cudaStream_t s) {
  if (c.items <= 0) return cudaSuccess;
  using S = PipeShape<SMALL, WC>;
  auto pitch = [](int w) { return pitch_of(w < KD ? w : KD); };
  const int mx = SMALL ? 0 : std::min(c.m, 16 * wr), qx = std::min(c.q, S::CW * WC), px = std::min(c.p, S::CW * WC);
  PipeSmem sm;
  // stacks of the small classes fill tiles of fixed size (pipe_stack_cap)
  sm.x = SMALL ? kPipeTile : wr == 1 ? 16 * pitch(c.n) : mx * pitch(c.n);
  sm.b = SMALL ? kPipeTile : std::max(px * pitch(c.n), (wr == 1 ? 32 : qx) * pitch(c.p));
  sm.pt = WC == 1 && c.p > 16 ? pitch(c.p) : pitch(KD);
  if (wr == 1) sm.pt = pitch(SMALL ? 16 : KD);
  sm.total = sm.x + 2 * sm.b + wr * WC * 16 * sm.pt;
  auto kern = chain_pipe_kernel<SMALL, WC>;
  const cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
  if (err != cudaSuccess) return err;
  add_kernel_launches(1);
  kern<<<c.items, 32 * wr * WC, sm.total * sizeof(float), s>>>(a.e, a.stacks, a.nstacks, a.g, items, wr, sm,
                                                               static_cast<const float *>(a.psi), a.db);
  return cudaGetLastError();
}

cudaError_t launch_pipe_f32(const PipeArgs &a, const ChainItem *items, const PipeClass *c, cudaStream_t s,
                            cudaStream_t s1, cudaStream_t s2) {
  cudaError_t err;
  auto next = [&](int cls) {
    const ChainItem *p = items;
    items += c[cls].items;
    return p;
  };
  const ChainItem *i5 = next(5), *i4 = next(4), *i3 = next(3), *i2 = next(2), *i1 = next(1), *i0 = next(0);
  if ((err = launch_pipe<false, 4>(a, i5, c[5], 2, s1)) != cudaSuccess) return err;
  if ((err = launch_pipe<false, 3>(a, i4, c[4], 2, s)) != cudaSuccess) return err;
  if ((err = launch_pipe<false, 2>(a, i3, c[3], 2, s1)) != cudaSuccess) return err;
  if ((err = launch_pipe<false, 1>(a, i2, c[2], 2, s)) != cudaSuccess) return err;
  if ((err = launch_pipe<false, 1>(a, i1, c[1], 1, s1)) != cudaSuccess) return err;
  return launch_pipe<true, 1>(a, i0, c[0], 1, s2);
}

}  // namespace

cudaError_t launch_chain_pipe(const PipeArgs &a, bool f32, const ChainItem *items, const PipeClass *classes, int wide,
                              cudaStream_t s, cudaStream_t s1, cudaStream_t s2) {
  return f32 ? launch_pipe_f32(a, items, classes, s, s1, s2) : launch_chain_mma(a, items, classes, wide, s, s1, s2);
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
