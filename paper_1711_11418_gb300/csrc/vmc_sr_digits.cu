// Overlap matrix of the plain form, S = (1/N_MC) (O - o)^T (O - o) (mVMC paper,
// Sec. 3.3.1) from FP64 samples, to FP64 accuracy, on the tensor cores: every
// centred column becomes 56-bit fixed-point integers under one exponent, cut
// into 8-bit digits (vmc_digits.cuh), and S the sum of their exact products.
//
//   k_dig_max   largest exponent of every centred column
//   k_digits    a slab of samples as digits, in the order in which a lane
//               reads an operand of mma.sync m16n8k16: 16 bytes per lane for a
//               block of 16 parameters x 16 samples.  The same 16 bytes are a
//               row operand (16 x 16) and two column operands (16 x 8 each).
//   k_syrk_dig  64 x 64 tiles of S's upper triangle, split over sample ranges;
//               16 warps with a 16 x 16 tile each, 34 digit products of 16
//               samples at a time; every KC = 128 samples (7 x 128 x 2^14 <
//               2^24: the sums are exact up to there) the eight sums become one
//               FP64 number, added to the lane's entries in FP64.
//   k_syrk_nonfinite  the entries of columns with infinities or NaNs
//
// What is left out is below 2^-56 of a column's largest entry, at most the
// FP64 rounding of the entries themselves for all but the smallest ones.
// What bounds it: the tensor pipe behind mma.sync (34 BF16 products for one of
// FP64; 4 clocks per m16n8k16 and SM).  16384 x 1069: 2.2 ms, and 0.11 ms for
// the digits, against 21.2 ms on the FP64 pipe (15.6 ms at its full rate).
// Error against quad precision, relative to sqrt(S_kk S_mm): 2.0e-17 rms for
// normal columns (FP64 pipe 2.1e-17), largest
// 5.2e-16 with heavy tails (6.0e-16).  mma.sync and not tcgen05: the eight FP32
// accumulators of a 128 x 64 tile fill tensor memory, and every 128 samples they
// would all be read back; that kernel was not built.
#include "vmc_common.cuh"
#include "vmc_digits.cuh"

namespace {

using vmc_dig::NDIG;
using vmc_dig::NSUM;

constexpr int KC = 128;              // samples between flushes
constexpr int KS = 32;               // samples per stage (two blocks of 16)
constexpr int TS = 64;               // tile edge
constexpr int ST = 3;                // stages
constexpr int BLK = 512;             // bytes of one digit of a 16 x 16 block
constexpr int STAGE = 2 * (TS / 16) * NDIG * (KS / 16) * BLK;   // both operands
constexpr int THREADS = 512;
constexpr int NONFINITE = 0x7ff;     // exponent of a column with an infinity or a NaN

__global__ void k_dig_max(const double *O, int ldO, int rows, int Np, const double *obar, int chunk,
                          int *emax) {
  const int c = blockIdx.x * 32 + threadIdx.x;
  const int r0 = blockIdx.y * chunk, r1 = min(rows, r0 + chunk);
  __shared__ int sh[8][32];
  int e = 0;
  if (c < Np) {
    const double o = obar[c];
    for (int r = r0 + threadIdx.y; r < r1; r += 8)
      e = max(e, vmc_dig::expo(O[(size_t)r * ldO + c] - o));
  }
  sh[threadIdx.y][threadIdx.x] = e;
  __syncthreads();
  if (threadIdx.y == 0 && c < Np) {
    for (int q = 1; q < 8; ++q) e = max(e, sh[q][threadIdx.x]);
    atomicMax(emax + c, e);
    if (e == NONFINITE) emax[Np] = 1;   // the columns have one
  }
}

// Digits of samples row0 .. row0 + 16 kb_n of all parameters (zero beyond rows
// and Np): block (s, pb, kb) at D + ((s npb + pb) kb_n + kb) BLK.
__global__ void __launch_bounds__(256) k_digits(const double *O, int ldO, int rows, int Np,
                                                const double *obar, const int *emax, int row0,
                                                int kb_n, int npb, unsigned char *D) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const long long item = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (item >= (long long)kb_n * npb) return;
  const int pb = (int)(item % npb), kb = (int)(item / npb);   // neighbours share sample rows
  long long v[2][4];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int c = pb * 16 + g + 8 * h;
    const double o = c < Np ? obar[c] : 0.0;
    const int e = c < Np ? emax[c] : 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = row0 + kb * 16 + 2 * t + (u & 1) + 8 * (u >> 1);
      const double x = (c < Np && r < rows) ? O[(size_t)r * ldO + c] - o : 0.0;
      v[h][u] = vmc_dig::fixed(x, e);
    }
  }
#pragma unroll
  for (int s = 0; s < NDIG; ++s) {
    const uint4 w = make_uint4(vmc_dig::pair(v[0][0], v[0][1], s), vmc_dig::pair(v[1][0], v[1][1], s),
                               vmc_dig::pair(v[0][2], v[0][3], s), vmc_dig::pair(v[1][2], v[1][3], s));
    *reinterpret_cast<uint4 *>(D + (((size_t)s * npb + pb) * kb_n + kb) * BLK + lane * 16) = w;
  }
}

__device__ __forceinline__ void cp16(void *dst, const void *src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}

// Tile (bi, bj), bi <= bj, from blockIdx.x; samples of blocks kb0 .. from
// blockIdx.y.  Adds scale x the products into S (FP64 atomic adds, as S is
// summed over sample ranges and slabs).
__global__ void __launch_bounds__(THREADS, 1)
    k_syrk_dig(const unsigned char *D, int kb_n, int npb, int kb_split, int Np, const int *emax,
               double scale, double *S) {
  extern __shared__ __align__(128) unsigned char smem[];
  int tl = blockIdx.x, bi = 0;
  const int nt = npb / (TS / 16);
  while (tl >= nt - bi) {
    tl -= nt - bi;
    ++bi;
  }
  const int bj = bi + tl;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = warp >> 2, wn = warp & 3;
  const int k0 = blockIdx.y * kb_split, k1 = min(kb_n, k0 + kb_split);   // multiples of KC / 16
  const int nst = (k1 - k0) / (KS / 16);
  // one stage: for each operand, digit and 16-parameter block, KS / 16 blocks in a row
  constexpr int RUN = (KS / 16) * BLK;             // contiguous bytes
  constexpr int RUNS = 2 * NDIG * (TS / 16);
  auto load = [&](int st) {
    unsigned char *dst = smem + (size_t)(st % ST) * STAGE;
    for (int q = tid; q < RUNS * (RUN / 16); q += THREADS) {
      const int run = q / (RUN / 16), off = q % (RUN / 16) * 16;
      const int op = run / (NDIG * (TS / 16)), rem = run % (NDIG * (TS / 16));
      const int s = rem / (TS / 16), b = rem % (TS / 16);
      const int pb = (op ? bj : bi) * (TS / 16) + b;
      cp16(dst + (size_t)run * RUN + off,
           D + (((size_t)s * npb + pb) * kb_n + k0 + st * (KS / 16)) * BLK + off);
    }
  };
  double sum[2][4] = {};
  float acc[2][NSUM][4];
#pragma unroll
  for (int st = 0; st < ST - 1; ++st) {
    if (st < nst) load(st);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  // exponents of this lane's rows and columns
  const int r0 = bi * TS + wm * 16 + (lane >> 2), c0 = bj * TS + wn * 16 + 2 * (lane & 3);
  const int er[2] = {r0 < Np ? emax[r0] : 0, r0 + 8 < Np ? emax[r0 + 8] : 0};
  for (int st = 0; st < nst; ++st) {
    asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
    __syncthreads();   // stage st has landed for all; stage st - 1 is read by all
    if (st + ST - 1 < nst) load(st + ST - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (st % (KC / KS) == 0)
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int d = 0; d < NSUM; ++d)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[n][d][q] = 0.0f;
    const unsigned char *sa = smem + (size_t)(st % ST) * STAGE + (size_t)wm * RUN + lane * 16;
    const unsigned char *sb =
        smem + (size_t)(st % ST) * STAGE + (size_t)(NDIG * (TS / 16) + wn) * RUN + lane * 16;
#pragma unroll
    for (int ks = 0; ks < KS / 16; ++ks) {
      uint32_t a[NDIG][4];
#pragma unroll
      for (int s = 0; s < NDIG; ++s) {
        const uint4 w = *reinterpret_cast<const uint4 *>(sa + (size_t)s * (TS / 16) * RUN + ks * BLK);
        a[s][0] = w.x;
        a[s][1] = w.y;
        a[s][2] = w.z;
        a[s][3] = w.w;
      }
#pragma unroll
      for (int u = 0; u < NDIG; ++u) {
        const uint4 b = *reinterpret_cast<const uint4 *>(sb + (size_t)u * (TS / 16) * RUN + ks * BLK);
#pragma unroll
        for (int s = 0; s < NDIG; ++s)
          if (s + u < NSUM) {
            vmc_dig::mma(acc[0][s + u], a[s], b.x, b.z);
            vmc_dig::mma(acc[1][s + u], a[s], b.y, b.w);
          }
      }
    }
    if (st % (KC / KS) == KC / KS - 1) {
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          int v[NSUM];
#pragma unroll
          for (int d = 0; d < NSUM; ++d) v[d] = __float2int_rn(acc[n][d][q]);
          const int c = c0 + 8 * n + (q & 1);
          const int ec = c < Np ? emax[c] : 0;
          sum[n][q] += vmc_dig::scaled(vmc_dig::combine(v), vmc_dig::unit_expo(er[q >> 1], ec));
        }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
  for (int n = 0; n < 2; ++n)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = r0 + 8 * (q >> 1), j = c0 + 8 * n + (q & 1);
      if (i < Np && j < Np && i <= j) atomicAdd(S + (size_t)i * Np + j, sum[n][q] * scale);
    }
}

// Fixed point knows no infinities and NaNs: the entries of S of the columns that
// have one are summed in FP64 here, as IEEE arithmetic gives them (a row of S
// per CTA; returns at once where there is no such column).
__global__ void __launch_bounds__(256) k_syrk_nonfinite(const double *O, int ldO, int rows, int Np,
                                                        const double *obar, const int *emax,
                                                        double scale, double *S) {
  if (!emax[Np]) return;
  const int i = blockIdx.x;
  const bool all = emax[i] == NONFINITE;
  for (int j = i + threadIdx.x; j < Np; j += blockDim.x) {
    if (!all && emax[j] != NONFINITE) continue;
    double s = 0.0;
    for (int r = 0; r < rows; ++r)
      s += (O[(size_t)r * ldO + i] - obar[i]) * (O[(size_t)r * ldO + j] - obar[j]);
    S[(size_t)i * Np + j] = s * scale;
  }
}

// A slab of samples has at most 256 MiB of digits (17536 samples at 1069
// parameters), and at least KC samples.
constexpr size_t SLAB_BYTES = 256ull << 20;
int pad_blocks(int Np) { return (Np + TS - 1) / TS * (TS / 16); }
// bytes of KC samples' digits
size_t chunk_bytes(int Np) { return (size_t)NDIG * pad_blocks(Np) * BLK * (KC / 16); }

}  // namespace

size_t vmc_sr_digits_min_bytes(int Np) { return chunk_bytes(Np); }
size_t vmc_sr_digits_bytes(int rows, int Np) {
  const size_t all = (size_t)(rows + KC - 1) / KC, most = SLAB_BYTES / chunk_bytes(Np);
  return chunk_bytes(Np) * (all < most ? all : most > 1 ? most : 1);
}

// S (upper triangle; zeroed by the caller) += (1/rows) (O - o)^T (O - o) of the
// FP64 samples.  w.digits has w.digits_bytes, from vmc_sr_digits_min_bytes(Np)
// to vmc_sr_digits_bytes(rows, Np), which decide the samples of a slab; w.emax:
// Np + 1 ints.
cudaError_t vmc_sr_syrk_digits(const SrWork &w, cudaStream_t st, long long *nl) {
  const double *O = (const double *)w.O;
  unsigned char *digits = w.digits;
  int *emax = w.emax;
  cudaError_t e = cudaMemsetAsync(emax, 0, sizeof(int) * (w.Np + 1), st);
  if (e) return e;
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int ct = (w.Np + 31) / 32;
  int parts = (8 * nsm + ct - 1) / ct;
  const int most = (w.rows + 63) / 64;
  if (parts > most) parts = most;
  const int chunk = (w.rows + parts - 1) / parts;
  k_dig_max<<<dim3(ct, parts), dim3(32, 8), 0, st>>>(O, w.ldO, w.rows, w.Np, w.obar, chunk, emax);
  if ((e = cudaFuncSetAttribute(k_syrk_dig, cudaFuncAttributeMaxDynamicSharedMemorySize, ST * STAGE)))
    return e;
  const int npb = pad_blocks(w.Np), nt = npb / (TS / 16), ntiles = nt * (nt + 1) / 2;
  const size_t all = (size_t)(w.rows + KC - 1) / KC, have = w.digits_bytes / chunk_bytes(w.Np);
  const int slab = (int)(all < have ? all : have) * (KC / 16);
  if (slab < 1) return cudaErrorInvalidValue;
  for (int row0 = 0; row0 < w.rows; row0 += slab * 16) {
    const int left = (w.rows - row0 + KC - 1) / KC * (KC / 16);
    const int kb_n = left < slab ? left : slab;
    const long long items = (long long)kb_n * npb;
    k_digits<<<(unsigned)((items + 7) / 8), 256, 0, st>>>(O, w.ldO, w.rows, w.Np, w.obar, emax, row0,
                                                         kb_n, npb, digits);
    // sample ranges so that about eight waves of CTAs cover the SMs evenly
    const int chunks = kb_n / (KC / 16);
    int split = (8 * nsm + ntiles - 1) / ntiles;
    if (split > chunks) split = chunks;
    const int per = (chunks + split - 1) / split;
    split = (chunks + per - 1) / per;
    k_syrk_dig<<<dim3(ntiles, split), THREADS, ST * STAGE, st>>>(digits, kb_n, npb, per * (KC / 16),
                                                                 w.Np, emax, 1.0 / w.rows, w.S);
    *nl += 2;
  }
  k_syrk_nonfinite<<<w.Np, 256, 0, st>>>(O, w.ldO, w.rows, w.Np, w.obar, emax, 1.0 / w.rows, w.S);
  *nl += 2;
  return cudaGetLastError();
}
