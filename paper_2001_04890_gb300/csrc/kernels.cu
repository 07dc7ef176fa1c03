// FP64 device kernels of the two-site QC-DMRG hot path (sm_103a); the batched triple
// products are in chain_kernels.cu and tc_kernels.cu.
//
// reduce_partials: adds the chunks of a split task list in chunk order.
// lincomb_fp64: pre-summed operators (Sec. 2.2.3, Eq. presum) as a GEMM
//               [K_out x K_src] x [K_src x block elements] per sector.
// Davidson helpers, a round-robin parallel Jacobi eigensolver for the small subspace
// matrix, and a column gather that builds O from eigenvectors.
#include <cuda_runtime.h>

#include <atomic>

#include "kernels.cuh"

namespace dmrg {

#define IDN (~0ull)

static std::atomic<long long> g_launches{0};
long long kernel_launch_count() { return g_launches.load(); }
void add_kernel_launches(long long n) { g_launches.fetch_add(n); }
#define COUNT(n) g_launches.fetch_add(n)

__device__ __forceinline__ const double *dptr(uint64_t base, uint64_t off) {
  return reinterpret_cast<const double *>(base + off * 8ull);
}

// out[ red.d + ...] += sum over the task chunks of their partial blocks, in chunk order
__global__ void reduce_partials_kernel(const ReduceGroup *__restrict__ R, int nred, int64_t total,
                                       const double *__restrict__ scratch, double *out) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    int lo = 0, hi = nred - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (R[mid].e0 <= t) lo = mid; else hi = mid - 1;
    }
    const ReduceGroup r = R[lo];
    const int64_t loc = t - r.e0;
    const int i = (int)(loc / r.q), c = (int)(loc % r.q);
    const int64_t mq = (int64_t)r.m * r.q;
    double s = 0.0;
    for (int k = 0; k < r.nsplit; ++k) s += scratch[r.soff + k * mq + loc];
    out[r.d + (int64_t)i * r.drs + (int64_t)c * r.dcs] += s;
  }
}

cudaError_t launch_reduce_partials(const ReduceGroup *r, int nred, int64_t total, const double *scratch,
                                   double *out, cudaStream_t s) {
  if (nred <= 0 || total <= 0) return cudaSuccess;
  int64_t blocks = (total + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  COUNT(1);
  reduce_partials_kernel<<<(int)blocks, 256, 0, s>>>(r, nred, total, scratch, out);
  return cudaGetLastError();
}

__global__ void to_f32_kernel(float *out, const double *in, int64_t n) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    out[e] = (float)in[e];
}

__global__ void __launch_bounds__(256) lincomb_fp64_kernel(const LincombTask *__restrict__ T,
                                                           int ntasks) {
  __shared__ double Cs[32][33];
  __shared__ double Ss[32][33];
  const int tile = blockIdx.x;
  int lo = 0, hi = ntasks - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (T[mid].tile0 <= tile) lo = mid; else hi = mid - 1;
  }
  const LincombTask t = T[lo];
  const int64_t E = (int64_t)t.rows * t.cols;
  const int ne = (int)((E + 31) / 32);
  const int tl = tile - t.tile0;
  const int t0 = (tl / ne) * 32;
  const int64_t e0 = (int64_t)(tl % ne) * 32;
  const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
  const double *coef = dptr(0, t.coef);
  const double *src = dptr(0, t.src);
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int u0 = 0; u0 < t.ksrc; u0 += 32) {
    for (int idx = tid; idx < 1024; idx += 256) {
      const int i = idx >> 5, j = idx & 31;
      Cs[i][j] = (t0 + i < t.kout && u0 + j < t.ksrc) ? coef[(int64_t)(t0 + i) * t.ksrc + u0 + j] : 0.0;
      const int64_t e = e0 + j;
      double v = 0.0;
      if (u0 + i < t.ksrc && e < E) {
        int64_t se = e;
        if (t.tr) {
          const int64_t r = e / t.cols, c = e % t.cols;
          se = c * t.rows + r;
        }
        v = src[(int64_t)(u0 + i) * E + se];
      }
      Ss[i][j] = v;
    }
    __syncthreads();
    const int uc = min(32, t.ksrc - u0);
    for (int uu = 0; uu < uc; ++uu) {
      const double sv = Ss[uu][tx];
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[i] = fma(Cs[ty + 8 * i][uu], sv, acc[i]);
    }
    __syncthreads();
  }
  double *out = const_cast<double *>(dptr(0, t.out));
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int tt = t0 + ty + 8 * i;
    const int64_t e = e0 + tx;
    if (tt < t.kout && e < E) out[(int64_t)tt * E + e] = acc[i];
  }
}

static int grid_for(int64_t n);

cudaError_t launch_to_f32(float *out, const double *in, int64_t n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  COUNT(1);
  to_f32_kernel<<<grid_for(n), 256, 0, s>>>(out, in, n);
  return cudaGetLastError();
}

cudaError_t launch_lincomb_fp64(const LincombTask *t, int ntasks, int ntiles, cudaStream_t s) {
  if (ntasks <= 0 || ntiles <= 0) return cudaSuccess;
  COUNT(1);
  lincomb_fp64_kernel<<<ntiles, 256, 0, s>>>(t, ntasks);
  return cudaGetLastError();
}

// diag(H_eff): entries whose input block is their output block contribute f X_ii Z_jj.
__global__ void diag_fp64_kernel(const ChainEntry *__restrict__ E, const ChainGroup *__restrict__ G,
                                 uint64_t xb, uint64_t zb, double *diag) {
  const ChainGroup g = G[blockIdx.x];
  for (int ei = g.first; ei < g.first + g.count; ++ei) {
    const ChainEntry e = E[ei];
    if (e.y != g.d) continue;
    const bool xid = e.x == IDN, zid = e.z == IDN;
    const double *X = xid ? nullptr : dptr(xb, e.x);
    const double *Z = zid ? nullptr : dptr(zb, e.z);
    for (int idx = threadIdx.x; idx < g.m * g.q; idx += blockDim.x) {
      const int i = idx / g.q, j = idx % g.q;
      const double x = xid ? 1.0 : X[(int64_t)i * e.xrs + (int64_t)i * e.xcs];
      const double z = zid ? 1.0 : Z[(int64_t)j * e.zrs + (int64_t)j * e.zcs];
      diag[g.d + (int64_t)i * g.drs + (int64_t)j * g.dcs] += e.f * x * z;
    }
    __syncthreads();
  }
}

cudaError_t launch_diag_fp64(const ChainEntry *e, const ChainGroup *g, int ngroups, uint64_t xb,
                             uint64_t zb, double *diag, cudaStream_t s) {
  if (ngroups <= 0) return cudaSuccess;
  COUNT(1);
  diag_fp64_kernel<<<ngroups, 256, 0, s>>>(e, g, xb, zb, diag);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- Davidson helpers

int dots_partial_blocks(int64_t n) {
  int64_t b = (n + 2047) / 2048;
  if (b < 1) b = 1;
  if (b > 608) b = 608;  // 4 per SM on 152 SMs
  return (int)b;
}

// Partial dot products of the columns [C blockIdx.y, C blockIdx.y + C) of V with w.  An FP64
// operation takes a warp 64 clocks of its scheduler, and a vector of 16,600 elements has nine
// blocks' worth of elements, so the columns go to blocks of their own: 25 columns in one block took
// 37 us, most of it the reduction over the warp.  That reduction adds lane i + 16 to lane i, then
// + 8, ... for every column; half of the lanes do one column's additions and half another's as long
// as there are two, so C columns take C + 1 additions and not 5 C.
template <int C>
__global__ void __launch_bounds__(256) dots_stage1(const double *__restrict__ V, int k, int64_t n,
                                                   const double *__restrict__ w, double *partial) {
  __shared__ double red[8][C];
  const int nb = gridDim.x, c0 = C * blockIdx.y, kc = min(C, k - c0);
  const double *Vc = V + (int64_t)c0 * n;
  double s[C];
#pragma unroll
  for (int j = 0; j < C; ++j) s[j] = 0.0;
#pragma unroll 2
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)nb * blockDim.x) {
    const double we = w[e];
#pragma unroll
    for (int j = 0; j < C; ++j)
      if (j < kc) s[j] = fma(Vc[(int64_t)j * n + e], we, s[j]);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int o = 16;
#pragma unroll
  for (int h = C / 2; h > 0; h /= 2, o /= 2) {
#pragma unroll
    for (int j = 0; j < h; ++j) {  // columns j (lower lanes) and j + h (upper lanes)
      const bool up = lane & o;
      const double give = up ? s[j] : s[j + h], keep = up ? s[j + h] : s[j];
      s[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  for (; o > 0; o /= 2) s[0] += __shfl_xor_sync(0xffffffffu, s[0], o);
  if (lane % (32 / C) == 0) red[warp][lane / (32 / C)] = s[0];  // lane's upper bits select its column
  __syncthreads();
  if ((int)threadIdx.x < kc) {
    double x = 0.0;
    for (int w2 = 0; w2 < (int)(blockDim.x >> 5); ++w2) x += red[w2][threadIdx.x];
    partial[(int64_t)blockIdx.x * k + c0 + threadIdx.x] = x;
  }
}

__global__ void dots_stage2(const double *partial, int nb, int k, double *out) {
  const int j = blockIdx.x;
  __shared__ double red[256];
  double x = 0.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) x += partial[(int64_t)b * k + j];
  red[threadIdx.x] = x;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[j] = red[0];
}

cudaError_t launch_dots(const double *V, int k, int64_t n, const double *w, double *partial,
                        double *out, cudaStream_t s) {
  if (k <= 0) return cudaSuccess;
  const int nb = dots_partial_blocks(n);
  COUNT(1);
  // vectors of few blocks: fewer columns a block; long ones: w is read less often
  if (nb < 152) dots_stage1<4><<<dim3(nb, (k + 3) / 4), 256, 0, s>>>(V, k, n, w, partial);
  else dots_stage1<8><<<dim3(nb, (k + 7) / 8), 256, 0, s>>>(V, k, n, w, partial);
  COUNT(1);
  dots_stage2<<<k, 256, 0, s>>>(partial, nb, k, out);
  return cudaGetLastError();
}

__global__ void combine_kernel(double *out, const double *__restrict__ V, const double *__restrict__ y,
                               int k, int64_t n, double beta) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    double s = beta == 0.0 ? 0.0 : beta * out[e];
    for (int j = 0; j < k; ++j) s = fma(y[j], V[(int64_t)j * n + e], s);
    out[e] = s;
  }
}

static int grid_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  if (b < 1) b = 1;
  return (int)b;
}

cudaError_t launch_combine(double *out, const double *V, const double *y, int k, int64_t n,
                           double beta, cudaStream_t s) {
  COUNT(1);
  combine_kernel<<<grid_for(n), 256, 0, s>>>(out, V, y, k, n, beta);
  return cudaGetLastError();
}

__global__ void sub_proj_kernel(double *w, const double *__restrict__ V, const double *__restrict__ c,
                                int k, int64_t n) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    double s = w[e];
    for (int j = 0; j < k; ++j) s = fma(-c[j], V[(int64_t)j * n + e], s);
    w[e] = s;
  }
}

cudaError_t launch_sub_proj(double *w, const double *V, const double *c, int k, int64_t n,
                            cudaStream_t s) {
  if (k <= 0) return cudaSuccess;
  COUNT(1);
  sub_proj_kernel<<<grid_for(n), 256, 0, s>>>(w, V, c, k, n);
  return cudaGetLastError();
}

__global__ void axpy_kernel(double *y, const double *x, double a, int64_t n) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    y[e] = fma(a, x[e], y[e]);
}

cudaError_t launch_axpy(double *y, const double *x, double a, int64_t n, cudaStream_t s) {
  COUNT(1);
  axpy_kernel<<<grid_for(n), 256, 0, s>>>(y, x, a, n);
  return cudaGetLastError();
}

__global__ void scale_kernel(double *x, const double *a_dev, int invert_sqrt, int64_t n) {
  const double a = invert_sqrt ? 1.0 / sqrt(*a_dev) : *a_dev;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    x[e] *= a;
}

cudaError_t launch_scale(double *x, const double *a_dev, int invert_sqrt, int64_t n, cudaStream_t s) {
  COUNT(1);
  scale_kernel<<<grid_for(n), 256, 0, s>>>(x, a_dev, invert_sqrt, n);
  return cudaGetLastError();
}

__global__ void precond_kernel(double *t, const double *r, const double *diag, const double *theta,
                               int64_t n) {
  const double th = *theta;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    double d = th - diag[e];
    if (fabs(d) < 1e-8) d = d < 0.0 ? -1e-8 : 1e-8;
    t[e] = r[e] / d;
  }
}

cudaError_t launch_precond(double *t, const double *r, const double *diag, const double *theta,
                           int64_t n, cudaStream_t s) {
  COUNT(1);
  precond_kernel<<<grid_for(n), 256, 0, s>>>(t, r, diag, theta, n);
  return cudaGetLastError();
}

__global__ void residual_kernel(double *r, const double *hx, const double *x, const double *theta,
                                int64_t n) {
  const double th = *theta;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    r[e] = fma(-th, x[e], hx[e]);
}

cudaError_t launch_residual(double *r, const double *hx, const double *x, const double *theta,
                            int64_t n, cudaStream_t s) {
  COUNT(1);
  residual_kernel<<<grid_for(n), 256, 0, s>>>(r, hx, x, theta, n);
  return cudaGetLastError();
}

// SplitMix64 (Steele, Lea, Flood 2014) as a counter-based generator
__device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void fill_guess_kernel(double *x, int64_t n, uint64_t seed) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t r = splitmix64(seed * 0x100000001B3ull + (uint64_t)e);
    x[e] = 2.0 * ((double)(r >> 11) * (1.0 / 9007199254740992.0)) - 1.0;
  }
}

cudaError_t launch_fill_guess(double *x, int64_t n, uint64_t seed, cudaStream_t s) {
  COUNT(1);
  fill_guess_kernel<<<grid_for(n), 256, 0, s>>>(x, n, seed);
  return cudaGetLastError();
}

// Symmetric eigensolver for the small Davidson subspace matrix (n <= 32):
// two-sided Jacobi with the round-robin (circle) ordering, so each round
// applies n/2 disjoint rotations at once (they commute).  Rotation
// angles as in the classical cyclic method (t = sgn(th)/(|th|+sqrt(th^2+1)),
// th = (a_qq - a_pp)/(2 a_pq)); sweeps until the off-diagonal norm is below
// 1e-16 of the diagonal norm.  Eigenvalues ascending; evecs row-major with
// eigenvector j in column j.
//
// One SM's FP64 pipes bound it (an operation takes a warp 64 clocks of its scheduler).  The angles
// are one warp's chain of divisions and roots, so the other schedulers turn V by the round
// before meanwhile, and A <- J^T A J is one pass in which a thread has the four elements of two
// pairs.
__global__ void __launch_bounds__(256) jacobi_eigh_kernel(const double *A, int n, int lda, double *evals,
                                                          double *evecs) {
  __shared__ double a[32][33];
  __shared__ double v[32][33];
  __shared__ double rc[2][16], rs[2][16];
  __shared__ int rp[2][16], rq[2][16];  // rq < 0: p has no partner (odd n)
  __shared__ int done;
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int idx = tid; idx < n * n; idx += nt) {
    const int i = idx / n, j = idx % n;
    a[i][j] = A[(int64_t)i * lda + j];
    v[i][j] = (i == j) ? 1.0 : 0.0;
  }
  const int N = (n + 1) & ~1;  // an odd n gets a dummy index n (its pairs are skipped)
  const int npair = N / 2;
  const int warp = tid >> 5, vt = (((warp & 3) - 1) + 3 * (warp >> 2)) * 32 + (tid & 31);  // warps off the first scheduler
  int cur = 0;
  bool pending = false;  // V has not seen the rotations of buffer cur ^ 1
  auto turn_v = [&](int b, int t, int step) {  // V <- V J
    for (int it = t; it < n * npair; it += step) {
      const int k = it % n, m = it / n, p = rp[b][m], q = rq[b][m];
      if (q < 0) continue;
      const double c = rc[b][m], sn = rs[b][m];
      const double vkp = v[k][p], vkq = v[k][q];
      v[k][p] = c * vkp - sn * vkq;
      v[k][q] = sn * vkp + c * vkq;
    }
  };
  __syncthreads();
  for (int sweep = 0; sweep < 60; ++sweep) {
    if (tid < 32) {
      double off = 0.0, dg = 0.0;
      if (tid < n) {
        dg = a[tid][tid] * a[tid][tid];
        for (int j = tid + 1; j < n; ++j) off += a[tid][j] * a[tid][j];
      }
      for (int o = 16; o > 0; o >>= 1) {
        off += __shfl_xor_sync(0xffffffffu, off, o);
        dg += __shfl_xor_sync(0xffffffffu, dg, o);
      }
      if (tid == 0) done = off <= 1e-32 * (dg + 1e-300);
    }
    __syncthreads();
    if (done) break;
    for (int r = 0; r < N - 1; ++r) {
      if (tid < npair) {
        const int i0 = tid, i1 = N - 1 - tid;
        int p = i0 == 0 ? 0 : ((i0 - 1 + r) % (N - 1)) + 1;
        int q = ((i1 - 1 + r) % (N - 1)) + 1;
        if (p > q) {
          const int x = p;
          p = q;
          q = x;
        }
        double c = 1.0, sn = 0.0;
        if (q < n) {
          const double apq = a[p][q];
          if (fabs(apq) >= 1e-300) {
            const double th = (a[q][q] - a[p][p]) / (2.0 * apq);
            const double t = (th >= 0.0 ? 1.0 : -1.0) / (fabs(th) + sqrt(th * th + 1.0));
            c = 1.0 / sqrt(t * t + 1.0);
            sn = t * c;
          }
        } else {
          q = -1;
        }
        rp[cur][tid] = p;
        rq[cur][tid] = q;
        rc[cur][tid] = c;
        rs[cur][tid] = sn;
      }
      if (pending && (warp & 3)) turn_v(cur ^ 1, vt, 192);
      __syncthreads();
      for (int it = tid; it < npair * npair; it += nt) {  // A <- J^T (A J), rows of pair i, columns of pair j
        const int i = it / npair, j = it % npair;
        const int p = rp[cur][i], q = rq[cur][i], y = rp[cur][j], z = rq[cur][j];
        const double c = rc[cur][i], sn = rs[cur][i], d = rc[cur][j], e = rs[cur][j];
        double py = a[p][y], pz = 0.0, qy = 0.0, qz = 0.0;
        if (z >= 0) pz = a[p][z];
        if (q >= 0) qy = a[q][y];
        if (q >= 0 && z >= 0) qz = a[q][z];
        if (z >= 0) {
          const double u = py, w = qy;
          py = d * u - e * pz;
          pz = e * u + d * pz;
          qy = d * w - e * qz;
          qz = e * w + d * qz;
        }
        if (q >= 0) {
          const double u = py, w = pz;
          py = c * u - sn * qy;
          qy = sn * u + c * qy;
          pz = c * w - sn * qz;
          qz = sn * w + c * qz;
        }
        a[p][y] = py;
        if (z >= 0) a[p][z] = pz;
        if (q >= 0) a[q][y] = qy;
        if (q >= 0 && z >= 0) a[q][z] = qz;
      }
      cur ^= 1;
      pending = true;
      __syncthreads();
    }
  }
  if (pending) turn_v(cur ^ 1, tid, nt);
  __syncthreads();
  if (tid == 0) {
    for (int i = 0; i < n; ++i) {
      int m = i;
      for (int j = i + 1; j < n; ++j)
        if (a[j][j] < a[m][m]) m = j;
      if (m != i) {
        const double t = a[i][i];
        a[i][i] = a[m][m];
        a[m][m] = t;
        for (int r = 0; r < n; ++r) {
          const double x = v[r][i];
          v[r][i] = v[r][m];
          v[r][m] = x;
        }
      }
    }
  }
  __syncthreads();
  for (int idx = tid; idx < n * n; idx += nt) evecs[idx] = v[idx / n][idx % n];
  if (tid < n) evals[tid] = a[tid][tid];
}

cudaError_t launch_jacobi_eigh(const double *A, int n, int lda, double *evals, double *evecs,
                               cudaStream_t s) {
  if (n > 32 || n < 1) return cudaErrorInvalidValue;
  COUNT(1);
  jacobi_eigh_kernel<<<1, 256, 0, s>>>(A, n, lda, evals, evecs);
  return cudaGetLastError();
}

// O[i][c] = evecs[:, cols[c]][i] for column-major evecs (n x n)
__global__ void gather_columns_kernel(double *O, const double *evecs, int n, const int *cols, int kept) {
  const int64_t tot = (int64_t)n * kept;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < tot; idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx / kept, c = idx % kept;
    O[idx] = evecs[(int64_t)cols[c] * n + i];
  }
}

cudaError_t launch_gather_columns(double *O, const double *evecs, int n, const int *cols, int kept,
                                  cudaStream_t s) {
  if (kept <= 0 || n <= 0) return cudaSuccess;
  COUNT(1);
  gather_columns_kernel<<<grid_for((int64_t)n * kept), 256, 0, s>>>(O, evecs, n, cols, kept);
  return cudaGetLastError();
}

}  // namespace dmrg
