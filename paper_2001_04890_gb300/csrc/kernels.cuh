// Device kernels of the two-site QC-DMRG hot path (sm_103a) -- launch wrappers.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "plan.hpp"

namespace dmrg {

// Pre-summation task (Sec. 2.2.3, Eq. presum): out[t] = sum_u coef[t,u] src[u]
// for the K_out temporaries of one family in one sector transition.
struct LincombTask {
  uint64_t out;        // element address of the output slab (K_out blocks)
  uint64_t src;        // element address of the source slab (K_src blocks)
  uint64_t coef;       // element address of the K_out x K_src coefficient matrix
  int kout, ksrc;
  int rows, cols;      // output block shape
  int tr;              // source blocks read transposed (source block is cols x rows)
  int tile0;           // first tile of this task in the launch grid
};

// Bounded-wait / error flag shared by the kernels of one context.
struct DevStatus {
  int error;
};

// Work item of the CUDA-core kernels: the rows from r0 and columns from c0 of one group's output
// block, as many as the item's class takes (chain_item_class: 16 x 16, 16 x 32, 32 x 32, 32 x 64,
// 32 x 96, 32 x 128).
struct ChainItem {
  int g, r0, c0, pad;
};
constexpr int kChainClasses = 6;
int chain_item_class(int m, int q, int nmax, int pmax);  // largest n, p of the group's tasks
int chain_item_cols(int cls);
// D = sum over each group's tasks (written, not added).  items: those of class 5, then 4, 3, 2, 1, 0,
// count[class] of each.  wide: chunks that do not fill the GPU are shared by several warps.
cudaError_t launch_chain_fp64(const ChainEntry *e, const ChainGroup *g, const ChainItem *items, const int *count,
                              uint64_t xb, uint64_t yb, uint64_t zb, uint64_t db, cudaStream_t s, int wide = 1);
// same task list with FP32 operators X, Z (FP64 psi in, FP64 sigma out, FP32 accumulation)
cudaError_t launch_chain_f32ops(const ChainEntry *e, const ChainGroup *g, const ChainItem *items, const int *count,
                                uint64_t xb, uint64_t yb, uint64_t zb, uint64_t db, cudaStream_t s, int wide = 1);

// Prepared operands of H.psi (chain_pipe.cu): images of the operator blocks (limbs of the FP64
// operators, or FP32) and of the psi blocks.
struct OpSlab {   // blocks of equal shape, one after the other (the operators of one sector transition)
  uint64_t src;   // element address of the first block (~0: an identity)
  uint64_t img;   // byte address of its images: of the block, then of its transpose
  int64_t first;  // number of the slab's first block
  int rows, cols;
};
struct OpTable {
  const OpSlab *s = nullptr;  // sorted by src
  const int16_t *exps = nullptr;
  const int *id = nullptr;    // slab of the identity of each dimension up to max_id, or -1
  int n = 0, max_id = -1;
};
struct PsiSpan {
  int64_t off, img;  // element offset of the block in psi, and of its images among the images
  int rows, cols;
};
struct PipeEntry {
  uint64_t x, z;  // byte addresses of the images of X (rows: its rows) and Z (rows: its columns)
  double f;
  int w;          // digits: sum of the exponents of X, Z and f (INT_MIN: the task needs FP64)
  int src;        // the task in the execution list
};
static_assert(sizeof(PipeEntry) == 32, "PipeEntry is 32 bytes");
struct PipeStack {
  int e;          // first entry
  uint16_t n, p;  // Y is n x p
  uint32_t y;     // element offset of its image (rows: its columns)
  unsigned yb : 24, ns : 4, flags : 4;  // psi block, tasks, whether one of them needs FP64
};
static_assert(sizeof(PipeStack) == 16, "the kernel reads a PipeStack as one vector");
constexpr int kPipeMaxN = 120;  // inner dimension that 64-bit sums of digit products take
constexpr int kPipeTile = 320;  // elements of the X, Y and Z tiles of the kernel for small blocks
// Tasks on one psi block that run as one stack.  Digits: two, whose X make up the 16 rows of a
// product.  FP32: what the tiles of the class's kernel hold (rows of X, depth of T).
#ifdef __CUDACC__
__host__ __device__
#endif
inline int pipe_stack_cap(bool digits, int cls, int m, int q, int n, int p) {
  if (digits) return 2;
  if (cls > 1 || n > 32 || p > 32) return 1;
  const bool small = cls == 0;
  const int pn = ((n + 3) >> 3 << 3) + 4, pp = ((p + 3) >> 3 << 3) + 4, pt = (p + 3) & ~3;
  int c = (small ? 16 : 32) / pt;
  const int rows = 16 / m;
  if (rows < c) c = rows;
  if (small) {
    if (kPipeTile / (m * pn) < c) c = kPipeTile / (m * pn);
    if (kPipeTile / (q * pp) < c) c = kPipeTile / (q * pp);
  } else if (32 / q < c) {
    c = 32 / q;
  }
  return c < 1 ? 1 : c < 8 ? c : 8;
}
int64_t pipe_image_size(bool f32, int rows, int cols);  // elements of one image
// images and exponents of every block; s in block order
cudaError_t launch_op_images(const OpSlab *s, int nslabs, int64_t nblocks, int16_t *exps, bool f32, cudaStream_t st);
cudaError_t launch_psi_images(const PsiSpan *b, int nblocks, const double *psi, void *out, int *exps, bool f32,
                              cudaStream_t st);
// The tasks of every group as PipeEntry and their stacks (from the
// group's first entry on; nstacks per group); digits: sorted by psi block within the group.  *bad is
// set if a task has a form that the kernels do not take.
cudaError_t launch_pipe_entries(const ChainEntry *e, const ChainGroup *g, int ngroups, PipeEntry *out,
                                PipeStack *stacks, int *nstacks, int *bad, const OpTable &ops, const PsiSpan *b,
                                int nblocks, bool f32, cudaStream_t st);
struct PipeArgs {
  const PipeEntry *e;
  const PipeStack *stacks;
  const int *nstacks;
  const ChainEntry *tasks;  // the execution list (FP64 operators: for tasks that fixed point does not take)
  const ChainGroup *g;
  const void *psi;          // images of the psi blocks
  const int *pexp;          // digits: their exponents
  const double *psi64;      // the call's psi
  uint64_t db;
};
struct PipeClass {  // the items of a kernel class
  int items = 0;
  int64_t tasks = 0;
  int m = 0, q = 0, n = 0, p = 0;  // largest dimensions
};
// as launch_chain_fp64 / launch_chain_f32ops (f32), on prepared operands; classes 2 and 4 run on s,
// 1, 3 and 5 on s1, 0 on s2 (the caller orders them; all may be s)
cudaError_t launch_chain_pipe(const PipeArgs &a, bool f32, const ChainItem *items, const PipeClass *classes, int wide,
                              cudaStream_t s, cudaStream_t s1, cudaStream_t s2);
// its FP64 part (chain_mma.cu)
cudaError_t launch_chain_mma(const PipeArgs &a, const ChainItem *items, const PipeClass *classes, int wide,
                             cudaStream_t s, cudaStream_t s1, cudaStream_t s2);

// Split task lists: every output block's entries are cut into chunks whose
// partial blocks go to a scratch buffer; this adds them in chunk order.
struct ReduceGroup {
  int64_t e0;    // first flattened element of this block among all reduced elements
  int64_t soff;  // scratch offset of chunk 0 (chunks are m*q apart)
  uint64_t d;    // element offset of the output block
  int drs, dcs, m, q, nsplit;
};
cudaError_t launch_reduce_partials(const ReduceGroup *r, int nred, int64_t total, const double *scratch,
                                   double *out, cudaStream_t s);
cudaError_t launch_to_f32(float *out, const double *in, int64_t n, cudaStream_t s);
cudaError_t launch_lincomb_fp64(const LincombTask *t, int ntasks, int ntiles, cudaStream_t s);
cudaError_t launch_diag_fp64(const ChainEntry *e, const ChainGroup *g, int ngroups,
                             uint64_t xb, uint64_t zb, double *diag, cudaStream_t s);

// Davidson helpers (all FP64, deterministic two-stage reductions)
cudaError_t launch_dots(const double *V, int k, int64_t n, const double *w, double *partial,
                        double *out, cudaStream_t s);
cudaError_t launch_combine(double *out, const double *V, const double *y, int k, int64_t n,
                           double beta, cudaStream_t s);
cudaError_t launch_axpy(double *y, const double *x, double a, int64_t n, cudaStream_t s);
cudaError_t launch_scale(double *x, const double *a_dev, int invert_sqrt, int64_t n, cudaStream_t s);
cudaError_t launch_precond(double *t, const double *r, const double *diag, const double *theta,
                           int64_t n, cudaStream_t s);
cudaError_t launch_residual(double *r, const double *hx, const double *x, const double *theta,
                            int64_t n, cudaStream_t s);
cudaError_t launch_sub_proj(double *w, const double *V, const double *c, int k, int64_t n,
                            cudaStream_t s);
cudaError_t launch_fill_guess(double *x, int64_t n, uint64_t seed, cudaStream_t s);
cudaError_t launch_jacobi_eigh(const double *A, int n, int lda, double *evals, double *evecs,
                               cudaStream_t s);
cudaError_t launch_gather_columns(double *O, const double *evecs, int n, const int *cols,
                                  int kept, cudaStream_t s);

int dots_partial_blocks(int64_t n);

// tcgen05 self-test: C (128 x N) = A (128 x K) B^T (N x K), bf16 inputs, FP32 accumulation in TMEM
cudaError_t launch_tc_selftest(const float *A, const float *B, float *C, int N, int K, int *status,
                               cudaStream_t s);

// number of kernels this library has launched in the process
long long kernel_launch_count();
void add_kernel_launches(long long n);  // kernels run by CUDA-graph replays

}  // namespace dmrg

namespace dmrg {

// Tensor-core tiles: an R x K operand pre-split into bf16 hi / lo parts in the
// K-major core-matrix layout (8-row x 16-byte core matrices, core matrix
// (rg, kg) at byte (rg * K16/8 + kg) * 128), rows padded to R8 = ceil8(R),
// K to K16 = ceil16(K) with zeros; the lo part follows the hi part.
struct TileSpec {
  uint64_t src;     // byte address of the source view (FP32 or FP64; element (r, k) at element r*rs + k*cs)
  uint64_t dst;     // byte offset of the tile in the tile arena
  int rs, cs, R, K;
};
struct PsiTileSpec {
  int64_t src;      // element offset of the psi block (n x p, row-major) in psi
  uint64_t dst;     // byte offset of its transposed tile (rows p, K n)
  int n, p;
};
// One task of the pipelined tensor-core chain: D += f X Y Z with X, Y^T, Z^T given as tiles.
// 32 bytes, so any run of entries is one aligned bulk copy.
struct TcEntry {
  uint64_t xt, zt;      // byte offsets of the X and Z^T tiles in the operator tile arena
  uint32_t yt;          // byte offset of the Y^T tile in the psi tile arena
  float f;
  uint8_t n, p;         // inner dims (<= 128)
  uint8_t stack;        // first task of a stack: the number of consecutive tasks (same Y, same
                        // output block) whose X run stacked along M in one stage 1; others 0
  uint8_t pad0;
  uint32_t pad1;
};
static_assert(sizeof(TcEntry) == 32, "TcEntry is 32 bytes");
// The tensor-core kernel reads task descriptors in chunks of kTcChunkCopy entries,
// kTcChunk apart: the entry array carries kTcChunkCopy zero entries after its end.
constexpr int kTcChunk = 56;
constexpr int kTcChunkCopy = 64;
struct TcGroup {
  uint64_t d;       // element offset of the output block (or scratch slot)
  int drs, dcs, m, q;
  int first, count;
};

// operator tiles from FP32 (src_f64 false) or FP64 sources (src == ~0: exact identity tile)
cudaError_t launch_build_tiles(const TileSpec *t, int ntiles, uint8_t *arena, bool src_f64, cudaStream_t s);
// Y^T tiles of FP64 psi blocks
cudaError_t launch_psi_tiles(const PsiTileSpec *t, int ntiles, const double *psi, uint8_t *arena,
                             cudaStream_t s);
// tensor-core H.psi chain (split-BF16 x3, FP32 accumulation, FP64 output blocks), persistent
// CTAs taking groups (m, q <= 128, every entry n, p <= 128) from *counter (zeroed here on s);
// shape 1: every group has m, q <= 64 and every entry p <= 64 (MMA M = 64, four CTAs per SM);
// shape 2: m <= 64, q and p <= 32 (five CTAs per SM); shape 0: the rest;
// *status (8 ints) is raised if an mbarrier wait ran out
// pipeline-wait limit of the tensor-core kernel (tries <= 0: the default)
void set_tc_wait_tries(long long tries);
cudaError_t launch_chain_tc2(const TcEntry *e, const TcGroup *g, int ngroups, const uint8_t *optiles,
                             const uint8_t *psitiles, uint64_t db, int *counter, int *status, int shape,
                             cudaStream_t s);

}  // namespace dmrg
