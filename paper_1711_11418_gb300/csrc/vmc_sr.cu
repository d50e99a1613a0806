// Stochastic reconfiguration kernels (mVMC paper, Sec. 3.3.1-3.3.2):
//   o_k = <O_k>, E = <E_loc>,
//   S_km = <O_k O_m> - <O_k><O_m>  =  (1/N_MC) sum_mu (O_k,mu - o_k)(O_m,mu - o_m),
//   g_m  = <E O_m> - <E><O_m>      =  (1/N_MC) sum_mu (O_m,mu - o_m)(E_mu - E),
//   S~_kk = S_kk (1 + shift_rel) + shift_abs,
//   S~ x = g by Cholesky (S~ = L L^T) or by CG (Algorithm 1) with the SR-CG
//   product y = (1/N_MC) O^T (O v) - o (o . v) + shift terms,
//   alpha += -dtau x  (Eq. SR_equation_system).
// Sample rows are the rows of O (row-major, leading dimension ldO), in FP64
// (plain form) or FP32 (mixed form); every reduction accumulates in FP64.
#include "vmc_common.cuh"

#include <math.h>
#include <vector>

namespace {

constexpr int RB = 256;        // threads of the column-reduction kernels
constexpr int RMIN = 64;       // fewest rows per partial of a column reduction

}  // namespace

// Row chunks of a column reduction: enough CTAs to cover the SMs several
// times over, at least RMIN rows each.  Monotone in rows, so the partial
// buffer sized for the largest row count serves every smaller one.
int vmc_colreduce_parts(int rows, int Np) {
  const int ctiles = (Np + RB - 1) / RB;
  int target = (8 * 152 + ctiles - 1) / ctiles;
  const int most = (rows + RMIN - 1) / RMIN;
  if (target > most) target = most;
  return target < 1 ? 1 : target;
}

namespace {

template <typename TO>
__device__ __forceinline__ double ld(const TO *p) { return (double)*p; }

// FP64 value of a sample.  The FP64 pipe (two instructions a cycle and SM) also
// converts from FP32, so an FP32 word is widened by integer operations there:
// same bits for every normal number and zero; the rest is converted.
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) {
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  if (m - 0x00800000u >= 0x7f000000u && m != 0) return (double)x;   // subnormal, infinite, NaN
  const unsigned hi = m ? (b & 0x80000000u) | ((m >> 3) + 0x38000000u) : b;
  return __hiloint2double((int)hi, (int)(b << 29));
}

constexpr int CR_MEAN = 0;    // sum of O_rk
constexpr int CR_FORCE = 1;   // (O_rk - o_k) (E_r - ebar)                     (force g)
constexpr int CR_BOTH = 2;    // that, and (O_rk - o_k)^2 in a second partial  (g and diagonal of S)
constexpr int CR_DOT = 3;     // O_rk t_r                                      (CG: O^T t)

// Partial column reductions: part[c][k] = sum over the rows of chunk c; the
// second one follows the first at part2.  One thread per column, its rows in
// four accumulators by r mod 4, sixteen loads ahead.  The weights E_r - ebar
// are formed once per CTA.
//
// Bound by the FP64 pipe: 1 instruction per sample for the means, 3 for force
// and diagonal in one pass, where the separate passes with conversions took 2,
// 4 and 3.  FP32, 4096 x 32896 samples, all three results: a step of that model
// 54.4 -> 52.0 ms.
template <typename TO, int MODE>
__global__ void __launch_bounds__(RB) k_colreduce(const TO *O, int ldO, int rows, int Np,
                                                  const double *obar, const double *wvec,
                                                  const double *wshift, int chunk, double *part,
                                                  double *part2, const int *done) {
  constexpr bool WEIGHTS = MODE != CR_MEAN;
  constexpr int AHEAD = 16;
  __shared__ double ws[WEIGHTS ? RB : 1];
  if (done && *done) return;
  const int k = blockIdx.x * RB + threadIdx.x;
  const int c = blockIdx.y;
  const int r0 = c * chunk;
  const int r1 = min(rows, r0 + chunk);
  const bool on = k < Np;
  const double ok = (on && (MODE == CR_FORCE || MODE == CR_BOTH)) ? obar[k] : 0.0;
  const double shift = (MODE == CR_FORCE || MODE == CR_BOTH) ? *wshift : 0.0;
  const TO *col = O + (on ? k : 0);
  double s[4] = {0.0, 0.0, 0.0, 0.0}, d[4] = {0.0, 0.0, 0.0, 0.0};
  auto add = [&](int q, TO x, double wr) {
    const double o = widen(x);
    if constexpr (MODE == CR_MEAN) {
      s[q] += o;
    } else if constexpr (MODE == CR_DOT) {
      s[q] += o * wr;
    } else {
      const double z = o - ok;
      s[q] += z * wr;
      if constexpr (MODE == CR_BOTH) d[q] += z * z;
    }
  };
  for (int b0 = r0; b0 < r1; b0 += RB) {   // RB rows' weights at a time
    const int b1 = min(r1, b0 + RB);
    if constexpr (WEIGHTS) {
      __syncthreads();
      if (b0 + (int)threadIdx.x < b1)
        ws[threadIdx.x] = wvec[b0 + threadIdx.x] - shift;
      __syncthreads();
    }
    if (!on) continue;
    int r = b0;
    for (; r + AHEAD <= b1; r += AHEAD) {
      TO x[AHEAD];
#pragma unroll
      for (int u = 0; u < AHEAD; ++u) x[u] = col[(size_t)(r + u) * ldO];
#pragma unroll
      for (int u = 0; u < AHEAD; ++u) add(u & 3, x[u], WEIGHTS ? ws[r - b0 + u] : 0.0);
    }
    for (; r + 4 <= b1; r += 4) {
      TO x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = col[(size_t)(r + u) * ldO];
#pragma unroll
      for (int u = 0; u < 4; ++u) add(u, x[u], WEIGHTS ? ws[r - b0 + u] : 0.0);
    }
    for (; r < b1; ++r) add(0, col[(size_t)r * ldO], WEIGHTS ? ws[r - b0] : 0.0);
  }
  if (!on) return;
  part[(size_t)c * Np + k] = (s[0] + s[1]) + (s[2] + s[3]);
  if constexpr (MODE == CR_BOTH) part2[(size_t)c * Np + k] = (d[0] + d[1]) + (d[2] + d[3]);
}

__global__ void k_sum_parts(const double *part, int nparts, int Np, double scale, double *out,
                            const int *done) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= Np || (done && *done)) return;
  double s = 0.0;
  int c = 0;
  for (; c + 8 <= nparts; c += 8) {   // one chain of adds, eight loads ahead of it
    double x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = part[(size_t)(c + u) * Np + k];
#pragma unroll
    for (int u = 0; u < 8; ++u) s += x[u];
  }
  for (; c < nparts; ++c) s += part[(size_t)c * Np + k];
  out[k] = s * scale;
}

__global__ void k_mean_vec(const double *v, int n, double *out) {
  __shared__ double red[256];
  double s = 0.0;
  // one chain of adds per thread in order, sixteen loads ahead of it
  int i = threadIdx.x;
  for (; i + 15 * 256 < n; i += 16 * 256) {
    double x[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) x[u] = v[i + 256 * u];
#pragma unroll
    for (int u = 0; u < 16; ++u) s += x[u];
  }
  for (; i < n; i += 256) s += v[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = red[0] / n;
}

// Mirror the upper triangle and apply the diagonal shift.
__global__ void k_mirror_shift(double *S, int Np, double shift_rel, double shift_abs) {
  const size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (q >= (size_t)Np * Np) return;
  const int i = (int)(q / Np), j = (int)(q % Np);
  if (i > j) S[q] = S[(size_t)j * Np + i];
  else if (i == j) S[q] = S[q] * (1.0 + shift_rel) + shift_abs;
}

// Blocked right-looking Cholesky (lower triangle in place), panels of CB
// columns.  Per panel: k_chol_panel factors the diagonal block, L_jj L_jj^T,
// and forms the panel below (L_ij = A_ij L_jj^-T) and its part of the forward
// solution L z = g by substitution; k_syrk_trailing updates the trailing lower
// triangle (A -= L L^T) in 32x32 tiles and the rest of the right-hand side.
// What bounds it: the chain of n pivots (a reciprocal, a column, a barrier, up
// to eight multiply-adds on a pipe that takes 64 clocks for a warp's) and the
// FP64 pipe for n^3 / 3 multiply-adds.  n = 1069: panels 0.84 ms (one warp per
// block 2.37), trailing updates 0.65, backward solve 0.23 (both solves by
// themselves 1.32).  Products with the diagonal blocks'
// inverses are shorter chains, but their residual grows with the condition of
// the block: |S x - g| at neighbouring columns that are nearly alike, cond(S) =
// 1e10, was 2000 to 6000 times that of substitution, and past 1e13 the
// factorisation broke down.
constexpr int CB = 32;
constexpr int PT = 128;    // threads of k_chol_panel

// Panel step.  Every CTA factors the nb x nb diagonal block redundantly, lane =
// row, warp w the columns w, w + 4, ...: elimination without square roots
// (A = L1 D L1^T, L1 unit), L_jj = L1 D^1/2.  All CTAs but the last then solve
// X L_jj^T = A_i for CB rows below, four threads to a row, thread q the columns
// q, q + 4, ...: column c is finished and taken out of the later ones.  The last
// CTA records the first non-positive pivot in *info (1-based), stores 1 / L_kk
// (dinv) and the panel of the forward solution z, and the factored block: into A
// when it is the only CTA, else into dblk, from where the trailing update copies
// it (another CTA may still be reading the block).
__global__ void __launch_bounds__(PT) k_chol_panel(double *A, int n, int j0, int nb, int *info,
                                                   double *dblk, double *dinv, const double *y,
                                                   double *z) {
  __shared__ double Ls[CB][CB + 1];
  __shared__ double mcol[2][CB], acol[2][CB];   // multipliers, column before scaling
  __shared__ double dg[CB], sq[CB], rs[CB];
  __shared__ int bad_sh;
  const int tid = threadIdx.x, r = tid & 31, w = tid >> 5;
  const bool last = blockIdx.x == gridDim.x - 1;
  if (tid == 0) bad_sh = 0;
  double a[CB / 4];
#pragma unroll
  for (int j = 0; j < CB / 4; ++j) {
    const int c = w + 4 * j;
    a[j] = (r < nb && c <= r) ? A[(size_t)(j0 + r) * n + j0 + c] : (r == c ? 1.0 : 0.0);
  }
  // this thread's entries of the panel below, fetched while the block is factored
  const int q = tid & 3;
  const int i = j0 + nb + blockIdx.x * CB + (tid >> 2);
  const bool row_ok = !last && i < n;
  double x[CB / 4];
#pragma unroll
  for (int j = 0; j < CB / 4; ++j)
    x[j] = (row_ok && q + 4 * j < nb) ? A[(size_t)i * n + j0 + q + 4 * j] : 0.0;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < CB; ++k) {
    const int b = k & 1;
    if (w == (k & 3)) {
      double piv = __shfl_sync(0xffffffffu, a[k >> 2], k);
      if (!(piv > 0.0) || !isfinite(piv)) {
        if (r == 0 && !bad_sh) bad_sh = k + 1;
        piv = 1.0;
      }
      const double ip = vmc_recip(piv);
      const double m = r > k ? a[k >> 2] * ip : 0.0;
      acol[b][r] = a[k >> 2];
      mcol[b][r] = m;
      a[k >> 2] = r == k ? 1.0 : m;   // column k of L1
      if (r == 0) dg[k] = piv;
    }
    __syncthreads();
    const double m = mcol[b][r];
#pragma unroll
    for (int j = k >> 2; j < CB / 4; ++j) {
      const int c = w + 4 * j;
      if (c > k) a[j] = fma(-m, acol[b][c], a[j]);   // rows r >= c matter
    }
  }
  if (w == 0) {
    const double d = dg[r];
    const double s = sqrt(d);
    sq[r] = s;
    rs[r] = 1.0 / s;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < CB / 4; ++j) {
    const int c = w + 4 * j;
    Ls[r][c] = c <= r ? a[j] * sq[c] : 0.0;
  }
  __syncthreads();
  if (last) {
    const bool direct = gridDim.x == 1;
    for (int p = tid; p < CB * CB; p += PT) {
      const int rr = p / CB, c = p % CB;
      if (rr < nb && c <= rr) {
        if (direct) A[(size_t)(j0 + rr) * n + j0 + c] = Ls[rr][c];
        else dblk[rr * nb + c] = Ls[rr][c];
      }
    }
    if (tid == 0 && bad_sh && *info == 0) *info = j0 + bad_sh;
    if (w == 3) {
      double v = r < nb ? y[j0 + r] : 0.0;
#pragma unroll
      for (int k = 0; k < CB; ++k) {
        const double zk = __shfl_sync(0xffffffffu, v, k) * rs[k];
        if (r == k) v = zk;
        else if (r > k) v = fma(-Ls[r][k], zk, v);
      }
      if (r < nb) {
        z[j0 + r] = v;
        dinv[j0 + r] = rs[r];
      }
    }
    return;
  }
#pragma unroll
  for (int c = 0; c < CB; ++c) {
    const double xc = __shfl_sync(0xffffffffu, x[c >> 2], (tid & 28) | (c & 3)) * rs[c];
    if (q == (c & 3)) x[c >> 2] = xc;
#pragma unroll
    for (int j = c >> 2; j < CB / 4; ++j)
      if (q + 4 * j > c) x[j] = fma(-xc, Ls[q + 4 * j][c], x[j]);
  }
#pragma unroll
  for (int j = 0; j < CB / 4; ++j)
    if (row_ok && q + 4 * j < nb) A[(size_t)i * n + j0 + q + 4 * j] = x[j];
}

// Trailing update A[i][k] -= sum_l L[i][j0+l] L[k][j0+l] for j1 <= k <= i < n
// (j1 = j0 + nb): one 32x32 lower tile per CTA, tile (bi, bj) with bj <= bi
// decoded from the linear block index.  CTA 0 also stores the factored diagonal
// block from dblk (no CTA here reads that block).
// CTAs from n_tiles on take the panel out of the right-hand side instead:
// y_k -= sum_l L_{k,j0+l} z_{j0+l}, 256 rows k each.
__global__ void __launch_bounds__(256) k_syrk_trailing(double *A, int n, int j0, int nb,
                                                       const double *dblk, int n_tiles, double *y,
                                                       const double *z) {
  const int j1 = j0 + nb;
  if (blockIdx.x >= n_tiles) {
    __shared__ double zp[CB];
    if (threadIdx.x < CB) zp[threadIdx.x] = threadIdx.x < nb ? z[j0 + threadIdx.x] : 0.0;
    __syncthreads();
    const int k = j1 + (blockIdx.x - n_tiles) * 256 + threadIdx.x;
    if (k < n) {
      const double *row = A + (size_t)k * n + j0;
      double s0 = 0.0, s1 = 0.0;
#pragma unroll 8
      for (int l = 0; l < CB; l += 2) {
        if (l < nb) s0 = fma(row[l], zp[l], s0);
        if (l + 1 < nb) s1 = fma(row[l + 1], zp[l + 1], s1);
      }
      y[k] -= s0 + s1;
    }
    return;
  }
  if (blockIdx.x == 0)
    for (int q = threadIdx.x; q < nb * nb; q += 256) {
      const int r = q / nb, c = q % nb;
      if (c <= r) A[(size_t)(j0 + r) * n + j0 + c] = dblk[q];
    }
  int t = blockIdx.x, bi = 0;
  while (t >= bi + 1) {
    t -= bi + 1;
    ++bi;
  }
  const int bj = t;
  __shared__ double Pi[CB][33];
  __shared__ double Pk[CB][33];
  for (int q = threadIdx.x; q < CB * 32; q += 256) {
    const int r = q / CB, l = q % CB;
    const int ii = j1 + bi * 32 + r, kk = j1 + bj * 32 + r;
    Pi[l][r] = (l < nb && ii < n) ? A[(size_t)ii * n + j0 + l] : 0.0;
    Pk[l][r] = (l < nb && kk < n) ? A[(size_t)kk * n + j0 + l] : 0.0;
  }
  __syncthreads();
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  double a00 = 0, a01 = 0, a10 = 0, a11 = 0;
#pragma unroll 8
  for (int l = 0; l < CB; ++l) {
    const double x0 = Pi[l][ty], x1 = Pi[l][ty + 16];
    const double y0 = Pk[l][tx], y1 = Pk[l][tx + 16];
    a00 += x0 * y0; a01 += x0 * y1; a10 += x1 * y0; a11 += x1 * y1;
  }
  const double acc[2][2] = {{a00, a01}, {a10, a11}};
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int i = j1 + bi * 32 + ty + 16 * u, k = j1 + bj * 32 + tx + 16 * v;
      if (i < n && k < n && k <= i) A[(size_t)i * n + k] -= acc[u][v];
    }
}

// Backward solve L^T x = z, one launch per panel of CB unknowns, last first:
// every CTA solves L_pp^T x_p = z_p by substitution (a lane per unknown), then
// takes the panel out of its share of the entries above, z_i -= sum_l L_{p0+l,i}
// x_{p0+l} for i < p0 (thread per entry).  z is read and x written to another
// vector, so no CTA reads what another one writes.
constexpr int SV_COLS = 256;

__global__ void __launch_bounds__(SV_COLS) k_trsv_back(const double *L, int n, int p0,
                                                       const double *dinv, double *z, double *x) {
  __shared__ double Ls[CB][CB + 1], xp[CB];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nb = min(CB, n - p0);
#pragma unroll
  for (int u = 0; u < CB / 8; ++u) {
    const int r = warp + 8 * u;
    Ls[r][lane] = (r < nb && lane < r) ? L[(size_t)(p0 + r) * n + p0 + lane] : 0.0;
  }
  const int i = blockIdx.x * SV_COLS + tid;
  double col[CB];   // this thread's column of the panel, fetched while x_p is formed
#pragma unroll
  for (int l = 0; l < CB; ++l) col[l] = (i < p0 && l < nb) ? L[(size_t)(p0 + l) * n + i] : 0.0;
  __syncthreads();
  if (warp == 0) {
    double v = lane < nb ? z[p0 + lane] : 0.0;
    const double rd = lane < nb ? dinv[p0 + lane] : 0.0;
#pragma unroll
    for (int k = CB - 1; k >= 0; --k) {
      const double xk = __shfl_sync(0xffffffffu, v * rd, k);
      if (lane == k) v = xk;
      else if (lane < k) v = fma(-Ls[k][lane], xk, v);
    }
    xp[lane] = lane < nb ? v : 0.0;
    if (blockIdx.x == 0 && lane < nb) x[p0 + lane] = v;
  }
  __syncthreads();
  if (i < p0) {
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int l = 0; l < CB; l += 2) {
      s0 = fma(col[l], xp[l], s0);
      s1 = fma(col[l + 1], xp[l + 1], s1);
    }
    z[i] -= s0 + s1;
  }
}

// t = O v (one warp per row)
template <typename TO>
__global__ void k_gemv_rows(const TO *O, int ldO, int rows, int Np, const double *v, double *t,
                            const int *done) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= rows || *done) return;
  const TO *o = O + (size_t)warp * ldO;
  double s = 0.0;
  for (int k = lane; k < Np; k += 32) s += ld(o + k) * v[k];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) t[warp] = s;
}

__global__ void k_dot(const double *a, const double *b, int n, double *out) {
  __shared__ double red[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += a[i] * b[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = red[0];
}

// CG (Algorithm 1) on the device.  cg[0..1]: rho ping-pong, cg[2]: p.w,
// cg[3]: o.v, cg[4]: threshold eps^2 |b|^2; flags[0]: done, flags[1]:
// iterations, flags[2]: breakdown.
__global__ void k_cg_finish(const double *u, const double *obar, const double *odv,
                            const double *diagS, const double *v, double shift_rel,
                            double shift_abs, int n, double *w, const int *done) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n || *done) return;
  w[k] = u[k] - obar[k] * odv[0] + (shift_rel * diagS[k] + shift_abs) * v[k];
}

// x += alpha p, r -= alpha w with alpha = rho / (p.w)
__global__ void k_cg_update_xr(double *x, double *r, const double *p, const double *w,
                               const double *rho, const double *pw, int n, int *flags) {
  if (flags[0]) return;
  const double alpha = rho[0] / pw[0];
  if (!isfinite(alpha) || pw[0] == 0.0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      flags[2] = 1;
      flags[0] = 1;
    }
    return;
  }
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  x[k] += alpha * p[k];
  r[k] -= alpha * w[k];
}

// p = r + (rho'/rho) p
__global__ void k_cg_update_p(double *p, const double *r, const double *rho_new,
                              const double *rho, int n, const int *flags) {
  if (flags[0]) return;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  p[k] = r[k] + (rho_new[0] / rho[0]) * p[k];
}

__global__ void k_cg_init(double *cg, int *flags, double eps) {
  // cg[0] holds |b|^2 = rho_0 on entry
  cg[4] = eps * eps * cg[0];
  flags[0] = (cg[0] == 0.0) ? 1 : 0;
  flags[1] = 0;
  flags[2] = 0;
}

__global__ void k_update_params(double *p, const double *x, double dtau, int n) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) p[k] += -dtau * x[k];
}

template <typename TO, int MODE>
cudaError_t colreduce(const SrWork &w, const double *wvec, const double *wshift, double scale,
                      double *out, double *out2, cudaStream_t st, long long *nl,
                      const int *done = nullptr) {
  const int nparts = vmc_colreduce_parts(w.rows, w.Np);
  const int chunk = (w.rows + nparts - 1) / nparts;
  dim3 grid((w.Np + RB - 1) / RB, nparts);
  double *part2 = w.part + (size_t)nparts * w.Np;
  k_colreduce<TO, MODE><<<grid, RB, 0, st>>>((const TO *)w.O, w.ldO, w.rows, w.Np, w.obar, wvec,
                                             wshift, chunk, w.part, part2, done);
  const int g = (w.Np + 255) / 256;
  k_sum_parts<<<g, 256, 0, st>>>(w.part, nparts, w.Np, scale, out, done);
  *nl += 2;
  if (MODE == CR_BOTH) {
    k_sum_parts<<<g, 256, 0, st>>>(part2, nparts, w.Np, scale, out2, done);
    ++*nl;
  }
  return cudaGetLastError();
}

template <int MODE>
cudaError_t colreduce_any(const SrWork &w, const double *wvec, const double *wshift, double scale,
                          double *out, double *out2, cudaStream_t st, long long *nl) {
  return w.precision == 0
             ? colreduce<double, MODE>(w, wvec, wshift, scale, out, out2, st, nl)
             : colreduce<float, MODE>(w, wvec, wshift, scale, out, out2, st, nl);
}

}  // namespace

cudaError_t vmc_sr_means(const SrWork &w, cudaStream_t st, long long *nl) {
  k_mean_vec<<<1, 256, 0, st>>>(w.E, w.rows, w.ebar);
  ++*nl;
  return colreduce_any<CR_MEAN>(w, nullptr, nullptr, 1.0 / w.rows, w.obar, nullptr, st, nl);
}

// ebar is read by the kernel from device memory (no host round trip)
cudaError_t vmc_sr_build_g(const SrWork &w, bool diag, cudaStream_t st, long long *nl) {
  return diag ? colreduce_any<CR_BOTH>(w, w.E, w.ebar, 1.0 / w.rows, w.g, w.diagS, st, nl)
              : colreduce_any<CR_FORCE>(w, w.E, w.ebar, 1.0 / w.rows, w.g, nullptr, st, nl);
}

cudaError_t vmc_sr_build_S(const SrWork &w, double shift_rel, double shift_abs, cudaStream_t st,
                           long long *nl) {
  cudaError_t e = cudaMemsetAsync(w.S, 0, sizeof(double) * (size_t)w.Np * w.Np, st);
  if (e) return e;
  if ((e = vmc_sr_syrk_digits(w, st, nl))) return e;
  const size_t n2 = (size_t)w.Np * w.Np;
  k_mirror_shift<<<(unsigned)((n2 + 255) / 256), 256, 0, st>>>(w.S, w.Np, shift_rel, shift_abs);
  ++*nl;
  return cudaGetLastError();
}

// The launch sequence of the factorisation (with the forward solve) and the
// backward solve: three launches per panel.  Pointers are fixed for the life of
// the work area, so the sequence is captured once into a CUDA graph and
// replayed.
static void chol_sequence(const SrWork &w, cudaStream_t st) {
  const int n = w.Np;
  cudaMemsetAsync(w.info, 0, sizeof(int), st);
  // right-hand side y (= w.p, starts as g) -> z (= w.w), panel by panel
  cudaMemcpyAsync(w.p, w.g, sizeof(double) * n, cudaMemcpyDeviceToDevice, st);
  for (int j0 = 0; j0 < n; j0 += CB) {
    const int nb = n - j0 < CB ? n - j0 : CB;
    const int rem = n - j0 - nb;
    k_chol_panel<<<1 + (rem + CB - 1) / CB, PT, 0, st>>>(w.S, n, j0, nb, w.info, w.dblk, w.dinv, w.p,
                                                         w.w);
    if (rem > 0) {
      const int nt = (rem + 31) / 32, tiles = nt * (nt + 1) / 2;
      k_syrk_trailing<<<tiles + (rem + 255) / 256, 256, 0, st>>>(w.S, n, j0, nb, w.dblk, tiles, w.p, w.w);
    }
  }
  for (int p0 = ((n - 1) / CB) * CB; p0 >= 0; p0 -= CB) {
    const int grid = p0 > 0 ? (p0 + SV_COLS - 1) / SV_COLS : 1;
    k_trsv_back<<<grid, SV_COLS, 0, st>>>(w.S, n, p0, w.dinv, w.w, w.x);
  }
}

static long long chol_launches(int n) {
  long long c = 0;
  for (int j0 = 0; j0 < n; j0 += CB) c += (n - j0 > CB) ? 3 : 2;
  return c;
}

int vmc_sr_cholesky_launch(SrWork &w, cudaStream_t st, long long *nl) {
  if (!w.chol_graph) {
    // Capture on a private stream (the caller's may be the legacy stream,
    // which cannot be captured).
    cudaStream_t cs = nullptr;
    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) return -3;
    cudaGraph_t g = nullptr;
    cudaGraphExec_t ge = nullptr;
    bool ok = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
    if (ok) {
      chol_sequence(w, cs);
      ok = cudaStreamEndCapture(cs, &g) == cudaSuccess && g;
    }
    if (ok) ok = cudaGraphInstantiate(&ge, g, 0) == cudaSuccess;
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cs);
    if (!ok) {
      cudaGetLastError();
      return -3;
    }
    w.chol_graph = (void *)ge;
  }
  if (cudaGraphLaunch((cudaGraphExec_t)w.chol_graph, st) != cudaSuccess) return -3;
  *nl += chol_launches(w.Np);
  return 0;
}

// Factor and solve; returns 0, -4 (S~ not positive definite) or -3.
int vmc_sr_cholesky_solve(SrWork &w, cudaStream_t st, long long *nl) {
  if (vmc_sr_cholesky_launch(w, st, nl)) return -3;
  int info = 0;
  if (cudaMemcpyAsync(&info, w.info, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return -3;
  if (cudaStreamSynchronize(st) != cudaSuccess) return -3;
  return info ? -4 : 0;
}

void vmc_sr_release(SrWork &w) {
  if (w.chol_graph) cudaGraphExecDestroy((cudaGraphExec_t)w.chol_graph);
  w.chol_graph = nullptr;
}

// Mixed form (FP32 O): the two passes of the SR-CG product with FP32
// products summed in FP32 over 16 terms and the partial sums in FP64, so the
// FP64 pipe (1/64 of the FP32 rate on this part) does one add per 16
// products; relative error of each product sum about 1e-6 at most.  The
// operand vectors enter as FP32 copies.
constexpr int CH32 = 16;

__global__ void k_to_float(const double *v, int n, float *vf, const int *done) {
  if (done && *done) return;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) vf[k] = (float)v[k];
}

// t = O v, one warp per row; t in FP64 and as an FP32 copy
__global__ void k_gemv_rows_f32(const float *O, int ldO, int rows, int Np, const float *vf,
                                double *t, float *tf, const int *done) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= rows || *done) return;
  const float *o = O + (size_t)warp * ldO;
  double s = 0.0;
  for (int k0 = lane; k0 < Np; k0 += 32 * CH32) {
    float a = 0.0f;
#pragma unroll
    for (int u = 0; u < CH32; ++u) {
      const int k = k0 + 32 * u;
      if (k < Np) a = fmaf(o[k], vf[k], a);
    }
    s += (double)a;
  }
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) {
    t[warp] = s;
    tf[warp] = (float)s;
  }
}

// part[c][k] = sum over the rows of chunk c of O_rk t_r (thread per column)
__global__ void __launch_bounds__(RB) k_colreduce_t32(const float *O, int ldO, int rows, int Np,
                                                      const float *tf, int chunk, double *part,
                                                      const int *done) {
  const int k = blockIdx.x * RB + threadIdx.x;
  // the last rows first: they are what the row product left in L2
  const int c = gridDim.y - 1 - blockIdx.y;
  if (k >= Np || (done && *done)) return;
  const int r1 = min(rows, c * chunk + chunk);
  const float *col = O + k;
  double s = 0.0;
  for (int r = c * chunk; r < r1; r += CH32) {
    float a = 0.0f;
#pragma unroll
    for (int u = 0; u < CH32; ++u)
      if (r + u < r1) a = fmaf(col[(size_t)(r + u) * ldO], tf[r + u], a);
    s += (double)a;
  }
  part[(size_t)c * Np + k] = s;
}

// Dot products over many CTAs, summed in a fixed order (deterministic):
// dpart[b] = partial of CTA b; out = sum of the partials.
constexpr int DOT_MAXB = 512;

__global__ void k_dotp(const double *a, const double *b, int n, double *dpart, const int *done) {
  __shared__ double red[256];
  if (done && *done) return;
  double s = 0.0;
  for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) s += a[i] * b[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) dpart[blockIdx.x] = red[0];
}

__global__ void k_dotf(const double *dpart, int nb, double *out, const int *done) {
  __shared__ double red[256];
  if (done && *done) return;
  double s = 0.0;
  for (int i = threadIdx.x; i < nb; i += 256) s += dpart[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = red[0];
}

static int dot_blocks(int n) {
  const int nb = (n + 4095) / 4096;
  return nb < 1 ? 1 : (nb > DOT_MAXB ? DOT_MAXB : nb);
}

static void dot2(const double *a, const double *b, int n, double *out, double *dpart,
                 const int *done, cudaStream_t st, long long *nl) {
  const int nb = dot_blocks(n);
  k_dotp<<<nb, 256, 0, st>>>(a, b, n, dpart, done);
  k_dotf<<<1, 256, 0, st>>>(dpart, nb, out, done);
  *nl += 2;
}

// convergence test on rho' = r.r (computed by dot2): done if rho' < threshold
__global__ void k_cg_check2(const double *rho_new, const double *thr, int *flags) {
  if (flags[0]) return;
  const double v = rho_new[0];
  flags[1] += 1;
  if (!(v >= thr[0])) flags[0] = 1;   // converged (or NaN: flagged below)
  if (!isfinite(v)) flags[2] = 1;
}

// One SR-CG product out = S~ v (Sec. 3.3.2): t = O v, u = O^T t / rows,
// out = u - o (o . v) + shift terms.  2 (rows + 1) Np products for the S part.
static cudaError_t srcg_matvec(const SrWork &w, const double *v, double *out, double shift_rel,
                               double shift_abs, const int *done, cudaStream_t st, long long *nl) {
  const int threads = 256;
  const int blocks = (int)(((size_t)w.rows * 32 + threads - 1) / threads);
  if (w.precision == 0) {
    k_gemv_rows<double><<<blocks, threads, 0, st>>>((const double *)w.O, w.ldO, w.rows, w.Np, v, w.t, done);
    ++*nl;
    cudaError_t e = colreduce<double, CR_DOT>(w, w.t, nullptr, 1.0 / w.rows, w.r + w.Np, nullptr, st,
                                              nl, done);
    if (e) return e;
  } else {
    k_to_float<<<(w.Np + 255) / 256, 256, 0, st>>>(v, w.Np, w.vf, done);
    k_gemv_rows_f32<<<blocks, threads, 0, st>>>((const float *)w.O, w.ldO, w.rows, w.Np, w.vf,
                                                w.t, w.tf, done);
    const int nparts = vmc_colreduce_parts(w.rows, w.Np);
    const int chunk = (w.rows + nparts - 1) / nparts;
    dim3 grid((w.Np + RB - 1) / RB, nparts);
    k_colreduce_t32<<<grid, RB, 0, st>>>((const float *)w.O, w.ldO, w.rows, w.Np, w.tf, chunk,
                                         w.part, done);
    k_sum_parts<<<(w.Np + 255) / 256, 256, 0, st>>>(w.part, nparts, w.Np, 1.0 / w.rows,
                                                    w.r + w.Np, done);
    *nl += 4;
  }
  dot2(w.obar, v, w.Np, w.scal + 3, w.dpart, done, st, nl);
  k_cg_finish<<<(w.Np + 255) / 256, 256, 0, st>>>(w.r + w.Np, w.obar, w.scal + 3, w.diagS, v,
                                                   shift_rel, shift_abs, w.Np, out, done);
  *nl += 1;
  return cudaGetLastError();
}

// Dense product out = S~ v with S~ (shift included) stored row-major (one warp per row).
__global__ void k_gemv_dense(const double *S, int n, const double *v, double *out, const int *done) {
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (row >= n || *done) return;
  const double *r = S + (size_t)row * n;
  double s = 0.0;
  for (int k = lane; k < n; k += 32) s += r[k] * v[k];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) out[row] = s;
}

// Algorithm 1 with x0 = 0, run on the device in batches of iterations; the
// host reads the convergence flag once per batch.  w.r holds 2 Np doubles.
// dense = 0: SR-CG product from O (S never formed); dense = 1: product with
// the dense S~ in w.S.
int vmc_sr_cg_solve(const SrWork &w, double shift_rel, double shift_abs, double eps, int kmax,
                    int *iters, cudaStream_t st, long long *nl, int dense) {
  const int n = w.Np, g = (n + 255) / 256;
  int *flags = w.info;
  double *cg = w.scal;
  cudaMemsetAsync(w.x, 0, sizeof(double) * n, st);
  cudaMemcpyAsync(w.r, w.g, sizeof(double) * n, cudaMemcpyDeviceToDevice, st);
  cudaMemcpyAsync(w.p, w.g, sizeof(double) * n, cudaMemcpyDeviceToDevice, st);
  dot2(w.r, w.r, n, cg + 0, w.dpart, nullptr, st, nl);
  k_cg_init<<<1, 1, 0, st>>>(cg, flags, eps);
  *nl += 1;
  const int batch = 16;
  int h[3] = {0, 0, 0};
  for (int k = 1; k <= kmax; ++k) {
    double *rho = cg + ((k - 1) & 1), *rho_new = cg + (k & 1);
    if (dense) {
      k_gemv_dense<<<(int)(((size_t)n * 32 + 255) / 256), 256, 0, st>>>(w.S, n, w.p, w.w, flags);
      ++*nl;
    } else if (srcg_matvec(w, w.p, w.w, shift_rel, shift_abs, flags, st, nl) != cudaSuccess) {
      return -3;
    }
    dot2(w.p, w.w, n, cg + 2, w.dpart, flags, st, nl);
    k_cg_update_xr<<<g, 256, 0, st>>>(w.x, w.r, w.p, w.w, rho, cg + 2, n, flags);
    dot2(w.r, w.r, n, rho_new, w.dpart, flags, st, nl);
    k_cg_check2<<<1, 1, 0, st>>>(rho_new, cg + 4, flags);
    k_cg_update_p<<<g, 256, 0, st>>>(w.p, w.r, rho_new, rho, n, flags);
    *nl += 3;
    if (k % batch == 0 || k == kmax) {
      if (cudaMemcpyAsync(h, flags, sizeof(int) * 3, cudaMemcpyDeviceToHost, st) != cudaSuccess) return -3;
      if (cudaStreamSynchronize(st) != cudaSuccess) return -3;
      if (h[0]) break;
    }
  }
  if (cudaMemcpyAsync(h, flags, sizeof(int) * 3, cudaMemcpyDeviceToHost, st) != cudaSuccess) return -3;
  if (cudaStreamSynchronize(st) != cudaSuccess) return -3;
  *iters = h[1];
  if (h[2]) return -5;
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

cudaError_t vmc_sr_update_params(double *params, const double *x, double dtau, int Np,
                                 cudaStream_t st, long long *nl) {
  k_update_params<<<(Np + 255) / 256, 256, 0, st>>>(params, x, dtau, Np);
  ++*nl;
  return cudaGetLastError();
}

cudaError_t vmc_dot_dev(const double *a, const double *b, int n, double *out_dev, double *dpart,
                        cudaStream_t st, long long *nl) {
  dot2(a, b, n, out_dev, dpart, nullptr, st, nl);
  return cudaGetLastError();
}

cudaError_t vmc_dot_host(const double *a, const double *b, int n, double *out_host,
                         double *d_scratch, cudaStream_t st, long long *nl) {
  k_dot<<<1, 256, 0, st>>>(a, b, n, d_scratch);
  ++*nl;
  cudaError_t e = cudaMemcpyAsync(out_host, d_scratch, sizeof(double), cudaMemcpyDeviceToHost, st);
  if (e) return e;
  return cudaStreamSynchronize(st);
}
