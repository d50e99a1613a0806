// SR solve S~ x = g (Sec. 3.3.2) by mixed-precision iterative refinement:
// the Jacobi-scaled matrix A = D S~ D (D = diag(S~_kk)^-1/2, unit diagonal)
// is inverted once in FP32 by blocked Gauss-Jordan elimination, and that
// inverse corrects an FP64 solution against FP64 residuals:
//   x_0 = 0,  r_i = g - S~ x_i  (FP64),  x_{i+1} = x_i + D A32^-1 D r_i,
// until |r| <= eps |g| (Wilkinson / Moler iterative refinement).  The
// result carries the FP64 residual of the direct solve; the O(Np^3) work is
// FP32 (this part's FP64 rate is 1/64 of its FP32 rate).  The caller falls
// back to the FP64 Cholesky when the refinement does not converge.
#include "vmc_common.cuh"

#include <math.h>

namespace {

constexpr int GB = 32;    // Gauss-Jordan block
constexpr int GT = 64;    // update tile (GT x GT outputs per CTA)

// d_k = S~_kk^-1/2 (S~_kk > 0 for a shifted overlap matrix; a non-positive
// entry marks the matrix as unusable: flag[1] = 1)
__global__ void k_ir_diag(const double *S, int n, double *dsc, int *flag) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const double a = S[(size_t)k * n + k];
  if (!(a > 0.0) || !isfinite(a)) {
    flag[1] = 1;
    dsc[k] = 1.0;
  } else {
    dsc[k] = 1.0 / sqrt(a);
  }
}

// The scaled matrix, and its first GB rows and columns beside it (k_gj_step)
__global__ void k_ir_scale(const double *S, int n, const double *dsc, float *A, float *R, float *C) {
  const size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= (size_t)n * n) return;
  const int i = (int)(q / n), j = (int)(q % n);
  const float a = (float)(dsc[i] * S[q] * dsc[j]);
  A[q] = a;
  if (i < GB) R[(size_t)i * n + j] = a;
  if (j < GB) C[(size_t)i * GB + j] = a;
}

// In-place inverse of the GB x GB block D by Gauss-Jordan elimination without
// pivoting (the scaled matrix is symmetric positive definite), 256 threads:
// thread = row tid / 8, columns tid % 8 + 8 j, in registers; one barrier per
// step, at which the next pivot row and column are published.
__device__ __forceinline__ void block_invert(float (*D)[GB + 1], float (*rowk)[GB],
                                             float (*colk)[GB]) {
  const int tid = threadIdx.x, r = tid >> 3, q = tid & 7;
  float d[GB / 8];
#pragma unroll
  for (int j = 0; j < GB / 8; ++j) d[j] = D[r][q + 8 * j];
  if (r == 0)
#pragma unroll
    for (int j = 0; j < GB / 8; ++j) rowk[0][q + 8 * j] = d[j];
  if (q == 0) colk[0][r] = d[0];
  __syncthreads();
#pragma unroll
  for (int k = 0; k < GB; ++k) {
    const float *rk = rowk[k & 1], *ck = colk[k & 1];
    const float ip = 1.0f / rk[k];
    const float m = ck[r] * ip;
#pragma unroll
    for (int j = 0; j < GB / 8; ++j) {
      const int c = q + 8 * j;
      const float row = rk[c];
      if (r == k) d[j] = c == k ? ip : row * ip;
      else d[j] = c == k ? -m : d[j] - m * row;
    }
    if (k + 1 < GB) {
      if (r == k + 1)
#pragma unroll
        for (int j = 0; j < GB / 8; ++j) rowk[(k + 1) & 1][q + 8 * j] = d[j];
      if (q == ((k + 1) & 7)) colk[(k + 1) & 1][r] = d[(k + 1) >> 3];
    }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < GB / 8; ++j) D[r][q + 8 * j] = d[j];
  __syncthreads();
}

// Gauss-Jordan step on pivot block K = [k0, k0 + nb), one GT x GT tile of A per
// CTA, in place.  R (GB x n) and C (n x GB) hold the rows and columns of K as
// they were before the step, Rn and Cn receive those of the next block, so a
// step reads nothing of A but its own tile and needs one launch.  Every CTA
// inverts A_KK (P) and forms its columns of the new row block, B = P A_Kj, or P
// itself for the columns of K; then
//   i in K:      A_ij <- B
//   i not in K:  A_ij <- (j in K ? 0 : A_ij) - sum_l C_il B_lj.
// What bounds it: latency (a 32-step inversion, two small products, one tile);
// n = 1069: 39 us in two launches per step -> 16 us from cold caches; the whole SR
// step of that size 2.17 -> 1.26 ms.
__global__ void __launch_bounds__(256) k_gj_step(float *A, int n, int k0, int nb, const float *R,
                                                 const float *C, float *Rn, float *Cn) {
  __shared__ float D[GB][GB + 1];
  __shared__ float Bs[GB][GT + 1];
  __shared__ float Cs[GT][GB + 1];
  __shared__ float rowk[2][GB], colk[2][GB];
  const int nt = (n + GT - 1) / GT;
  const int i0 = (blockIdx.x / nt) * GT, j0 = (blockIdx.x % nt) * GT, tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  auto inK = [&](int x) { return x >= k0 && x < k0 + nb; };
  // the tile and the operands are fetched while A_KK is inverted
  float a[4][4], rv[8];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int i = i0 + ty + 16 * u, j = j0 + tx + 16 * v;
      a[u][v] = (i < n && j < n && !inK(j)) ? A[(size_t)i * n + j] : 0.0f;
    }
  const int bl = tid >> 3, bc = tid & 7;   // B: row bl, columns bc + 8 u
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int j = j0 + bc + 8 * u;
    rv[u] = (bl < nb && j < n) ? R[(size_t)bl * n + j] : 0.0f;
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int r = (tid >> 5) + 8 * u, l = tid & 31, i = i0 + r;
    Cs[r][l] = (i < n && l < nb && !inK(i)) ? C[(size_t)i * GB + l] : 0.0f;
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = (tid >> 5) + 8 * u, c = tid & 31;
    D[r][c] = (r < nb && c < nb) ? R[(size_t)r * n + k0 + c] : (r == c ? 1.0f : 0.0f);
  }
  __syncthreads();
  block_invert(D, rowk, colk);
#pragma unroll
  for (int u = 0; u < 8; ++u) Bs[bl][bc + 8 * u] = rv[u];
  __syncthreads();
  float b[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) b[u] = 0.0f;
#pragma unroll 8
  for (int m = 0; m < GB; ++m) {
    const float p = D[bl][m];
#pragma unroll
    for (int u = 0; u < 8; ++u) b[u] += p * Bs[m][bc + 8 * u];
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int j = j0 + bc + 8 * u;
    Bs[bl][bc + 8 * u] = inK(j) ? D[bl][j - k0] : b[u];
  }
  __syncthreads();
  float acc[4][4] = {};
#pragma unroll 8
  for (int l = 0; l < GB; ++l) {
    float c[4], w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      c[u] = Cs[ty + 16 * u][l];
      w[u] = Bs[l][tx + 16 * u];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[u][v] += c[u] * w[v];
  }
  const int k1 = k0 + GB;   // next block
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int i = i0 + ty + 16 * u, j = j0 + tx + 16 * v;
      if (i >= n || j >= n) continue;
      const float x = inK(i) ? Bs[i - k0][tx + 16 * v] : a[u][v] - acc[u][v];
      A[(size_t)i * n + j] = x;
      if (i >= k1 && i < k1 + GB) Rn[(size_t)(i - k1) * n + j] = x;
      if (j >= k1 && j < k1 + GB) Cn[(size_t)i * GB + (j - k1)] = x;
    }
}

// x = 0, r = g, rs = D g (FP32), scal[1] = |g|^2, flag[0] = 0, iters = 0
__global__ void k_ir_init(const double *g, int n, const double *dsc, double *x, double *r,
                          float *rs, double *scal, int *flag) {
  __shared__ double red[256];
  double s = 0.0;
  for (int k = threadIdx.x; k < n; k += 256) {
    const double v = g[k];
    x[k] = 0.0;
    r[k] = v;
    rs[k] = (float)(dsc[k] * v);
    s += v * v;
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    scal[0] = 0.0;
    scal[1] = red[0];
    scal[2] = red[0];
    flag[0] = 0;
    flag[2] = 0;
  }
}

// x += D A32^-1 rs (one warp per row, FP32 products, FP64 update)
__global__ void k_ir_correct(const float *Ainv, int n, const double *dsc, const float *rs,
                             double *x, const int *flag) {
  if (flag[0] | flag[1]) return;
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (row >= n) return;
  const float *a = Ainv + (size_t)row * n;
  float s0 = 0.0f, s1 = 0.0f;
  int j = lane;
  for (; j + 32 < n; j += 64) {
    s0 += a[j] * rs[j];
    s1 += a[j + 32] * rs[j + 32];
  }
  if (j < n) s0 += a[j] * rs[j];
  float s = s0 + s1;
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) x[row] += dsc[row] * (double)s;
}

// r = g - S~ x (FP64, one warp per row); rs = D r in FP32; scal[0] += |r|^2.
// The CTA that finishes last (flag[3] counts them) tests convergence,
// |r|^2 <= eps^2 |g|^2 -> flag[0] = 1; scal[2] keeps the last |r|^2.
__global__ void k_ir_residual(const double *S, int n, const double *g, const double *x,
                              const double *dsc, double *r, float *rs, double *scal, int *flag,
                              double eps2) {
  if (flag[0] | flag[1]) return;
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (row < n) {
    const double *a = S + (size_t)row * n;
    double s0 = 0.0, s1 = 0.0;
    int j = lane;
    for (; j + 32 < n; j += 64) {
      s0 += a[j] * x[j];
      s1 += a[j + 32] * x[j + 32];
    }
    if (j < n) s0 += a[j] * x[j];
    double s = s0 + s1;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      const double v = g[row] - s;
      r[row] = v;
      rs[row] = (float)(dsc[row] * v);
      atomicAdd(scal, v * v);
      __threadfence();
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(flag + 3, 1) == (int)gridDim.x - 1) {
      flag[3] = 0;
      const double rr = atomicAdd(scal, 0.0);
      scal[0] = 0.0;
      scal[2] = rr;
      flag[2] += 1;
      if (rr <= eps2 * scal[1]) flag[0] = 1;
    }
  }
}

void ir_sequence(const SrWork &w, int max_iter, double eps, cudaStream_t st) {
  const int n = w.Np;
  cudaMemsetAsync(w.irflag, 0, sizeof(int) * 4, st);
  k_ir_diag<<<(n + 255) / 256, 256, 0, st>>>(w.S, n, w.dsc, w.irflag);
  const size_t n2 = (size_t)n * n;
  // the pivot block's rows and columns, alternating between two buffers
  float *R[2] = {w.gjR, w.gjR + (size_t)GB * n}, *C[2] = {w.gjC, w.gjC + (size_t)GB * n};
  k_ir_scale<<<(unsigned)((n2 + 255) / 256), 256, 0, st>>>(w.S, n, w.dsc, w.S32, R[0], C[0]);
  const int nt = (n + GT - 1) / GT;
  for (int k0 = 0, q = 0; k0 < n; k0 += GB, q ^= 1) {
    const int nb = n - k0 < GB ? n - k0 : GB;
    k_gj_step<<<nt * nt, 256, 0, st>>>(w.S32, n, k0, nb, R[q], C[q], R[q ^ 1], C[q ^ 1]);
  }
  k_ir_init<<<1, 256, 0, st>>>(w.g, n, w.dsc, w.x, w.r, w.rs32, w.scal, w.irflag);
  const int wb = (int)(((size_t)n * 32 + 255) / 256);
  for (int it = 0; it < max_iter; ++it) {
    k_ir_correct<<<wb, 256, 0, st>>>(w.S32, n, w.dsc, w.rs32, w.x, w.irflag);
    k_ir_residual<<<wb, 256, 0, st>>>(w.S, n, w.g, w.x, w.dsc, w.r, w.rs32, w.scal, w.irflag,
                                      eps * eps);
  }
}

}  // namespace

long long vmc_sr_ir_launches(int n, int max_iter) {
  return 3 + (n + GB - 1) / GB + 2LL * max_iter;
}

// Launch the refinement (the captured graph, made on first use).  Returns 0
// or -3 on a CUDA error.
int vmc_sr_ir_launch(SrWork &w, int max_iter, double eps, cudaStream_t st, long long *nl) {
  if (!w.ir_graph || w.ir_iter != max_iter || w.ir_eps != eps) {
    if (w.ir_graph) cudaGraphExecDestroy((cudaGraphExec_t)w.ir_graph);
    w.ir_graph = nullptr;
    cudaStream_t cs = nullptr;
    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) return -3;
    cudaGraph_t g = nullptr;
    cudaGraphExec_t ge = nullptr;
    bool ok = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
    if (ok) {
      ir_sequence(w, max_iter, eps, cs);
      ok = cudaStreamEndCapture(cs, &g) == cudaSuccess && g;
    }
    if (ok) ok = cudaGraphInstantiate(&ge, g, 0) == cudaSuccess;
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cs);
    if (!ok) {
      cudaGetLastError();
      return -3;
    }
    w.ir_graph = (void *)ge;
    w.ir_iter = max_iter;
    w.ir_eps = eps;
  }
  if (cudaGraphLaunch((cudaGraphExec_t)w.ir_graph, st) != cudaSuccess) return -3;
  *nl += vmc_sr_ir_launches(w.Np, max_iter);
  return 0;
}

// Enqueue the copies of the refinement's flags (4 ints) and scalars (3
// doubles) to host memory; evaluate them after the stream has synchronised.
int vmc_sr_ir_fetch(const SrWork &w, int *flags4, double *scal3, cudaStream_t st) {
  if (cudaMemcpyAsync(flags4, w.irflag, sizeof(int) * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return -3;
  if (cudaMemcpyAsync(scal3, w.scal, sizeof(double) * 3, cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return -3;
  return 0;
}

// 0: converged (*iters refinement steps, *rel_res = |r| / |g|); 1: not
// converged or S~ unusable (the caller solves by FP64 Cholesky).
int vmc_sr_ir_eval(const int *fl, const double *sc, int *iters, double *rel_res) {
  *iters = fl[2];
  *rel_res = sc[1] > 0.0 ? sqrt(sc[2] / sc[1]) : 0.0;
  return (fl[0] && !fl[1]) ? 0 : 1;
}

// Returns 0 (converged; *iters = refinement steps), 1 (not converged or S~
// unusable: the caller solves by FP64 Cholesky), or -3 on a CUDA error.
int vmc_sr_ir_solve(SrWork &w, int max_iter, double eps, int *iters, double *rel_res,
                    cudaStream_t st, long long *nl) {
  if (vmc_sr_ir_launch(w, max_iter, eps, st, nl)) return -3;
  int fl[4] = {0, 0, 0, 0};
  double sc[3] = {0, 0, 0};
  if (vmc_sr_ir_fetch(w, fl, sc, st)) return -3;
  if (cudaStreamSynchronize(st) != cudaSuccess) return -3;
  return vmc_sr_ir_eval(fl, sc, iters, rel_res);
}

void vmc_sr_ir_release(SrWork &w) {
  if (w.ir_graph) cudaGraphExecDestroy((cudaGraphExec_t)w.ir_graph);
  w.ir_graph = nullptr;
}
