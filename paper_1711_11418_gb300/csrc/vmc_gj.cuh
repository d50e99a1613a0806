// From-scratch inverse of one walker's M in FP64: blocked Gauss-Jordan
// elimination with partial pivoting in shared memory (mVMC paper, Sec. 3.2.1:
// the Pfaffian of the anti-parallel pair product is det M up to a sign,
// Pf^2 = det X), with log|det M| and its sign.  Shared by the translation
// units of the walker kernels (the plain walker and the projected one).
//
// In place on M padded to Npad rows and columns (a multiple of GB, identity
// in the padding), GB columns (a panel) at a time:
//   panel   one thread per row holds its GB entries in registers and takes
//           the GB elimination steps in FP64.  Rows are not moved: the row
//           that is the pivot of step k keeps its place (perm[k] = row).  The
//           panel then holds T (Npad x GB), the effect of its steps on every
//           other column;
//   update  A <- A_masked + T R for the columns outside the panel, R the GB
//           pivot rows before the panel and A_masked the rest (pivot rows 0).
// The update is a contraction over GB = 16 and nearly all of the
// multiply-adds, so it runs on the tensor cores, in fixed point: each row of
// T and each column of R becomes 56-bit integers (one exponent per row and
// column, after a power of two per pivot row that evens out R's rows), cut
// into seven signed 8-bit digits, which BF16 holds; the products of digits
// s + u = d are summed by mma.sync m16n8k16 in FP32 without rounding
// (integers below 2^23), d = 0..7; the eight sums make one integer, rounded
// once to FP64 and added to A.  (Splitting operands so that sums of products
// are free of error: Ozaki, Ogita, Oishi, Rump, Numer. Algorithms 59, 95,
// 2012.)  What is left out is about 2^-56 of (row maximum of T) x (column
// maximum of R), once per panel, where the elimination step by step rounds
// every entry once per step.
//
// What bounds it: the FP64 pipe (2 multiply-adds per clock and SM), which has
// the panels' N^2 GB multiply-adds and the update's N^3 / GB additions left
// of N^3, and the pivot chain of the panels.  4096 walkers, mixed form, with the
// walkers close to singular done again: N = 112 5.9 ms against 13.65 step by
// step; N = 128 9.5 against 26.7; N = 64 2.0 against 3.2.  mma.sync and not tcgen05: a tile's products are consumed at once
// by the warp that made them, eight 112 x 112 accumulators do not fit tensor
// memory, and two walkers share an SM so that one's panel chain runs under
// the other's update.
#pragma once

#include "vmc_common.cuh"
#include "vmc_digits.cuh"

namespace vmc_gj {

using vmc_dig::NDIG;
using vmc_dig::NOEXP;

constexpr int GB = 16;               // panel width: K of one mma.sync m16n8k16
constexpr int CT = 4;                // column tiles (of 8) whose digits are staged at a time
constexpr int MAX_THREADS = 2 * VMC_MAX_N;

__host__ __device__ inline int gj_pad(int N) { return (N + GB - 1) / GB * GB; }
// A warp per 16 rows for the update (a thread per row for the panel).
__host__ __device__ inline int gj_threads(int N) {
  const int t = (2 * gj_pad(N) + 31) / 32 * 32;
  return t < 64 ? 64 : t;
}
// Up to this N the step-by-step form below is taken: its kernels need 48
// registers a thread against 126, and the work per site around so small an
// elimination wants the CTAs (4096 walkers, Ns = 256: N = 8 1.03 ms against
// 1.20, N = 24 1.08 against 1.20; N = 32 1.20 against 1.16, N = 48 1.85
// against 1.47).
constexpr int GJ_STEPS_MAX_N = 24;
// Shared memory (bytes): the matrix, then the staged digits of R (free after
// the elimination).
__host__ __device__ inline size_t gj_matrix_bytes(int N) {
  return (size_t)gj_pad(N) * gj_pad(N) * sizeof(double);
}
constexpr size_t GJ_STAGE_BYTES = (size_t)NDIG * CT * 8 * 8 * sizeof(uint32_t);

// Entry (i, c) of the matrix: rows of Npad doubles, the 64-byte halves of
// each 128-byte group swapped in odd rows, so that the 16-byte accesses of an
// accumulator tile (two rows per eight lanes) touch every bank once.
__host__ __device__ inline int gj_at(int i, int c, int ld) { return i * ld + (c ^ ((i & 1) << 3)); }

struct GJShared {
  alignas(16) double cand[2][4][GB];   // candidate pivot row of each panel warp, by step parity
  unsigned long long ckey[2][4];
  double cinv[2][4];
  int crow[2][4];
  int perm[VMC_MAX_N];         // row that is the pivot of step k
  int step[VMC_MAX_N];         // step of which row i is the pivot
  int sig[GB];                 // power of two taken out of each pivot row
  int rexp[CT * 8];            // exponent of each staged column of R
  double val[4], pminw[4], amax[4];
  int neg[4];
  int bad, nonfinite;
  int sign;
  double logdet, pmin, pmax;   // log|det M|, smallest / largest |pivot|
};

// The accumulators start at 1.5 x 2^23, so that their bits hold the integers.
constexpr float GJ_MAGIC = 12582912.0f;
constexpr int GJ_MAGIC_BITS = 0x4B400000;

// The digit products' sum of entry q of a tile (vmc_dig::combine).  |n[d]| < 2^21.
__device__ __forceinline__ long long gj_combine(const float (&a)[8][4], int q) {
  int n[8];
#pragma unroll
  for (int d = 0; d < 8; ++d) n[d] = __float_as_int(a[d][q]) - GJ_MAGIC_BITS;
  const int p0 = n[0] * 256 + n[1], p1 = n[2] * 256 + n[3];
  const int p2 = n[4] * 256 + n[5] + ((n[6] * 256 + n[7] + 32768) >> 16);
  return (long long)p0 * 4294967296ll + (long long)p1 * 65536ll + (long long)p2;
}

// GB elimination steps on the panel of columns k0 .. k0 + GB - 1; threads
// tid < 32 ceil(Npad / 32), row tid each.  `mine` is the step of which this
// thread's row is the pivot (-1: none yet), `piv` that pivot.  Per step each
// warp's candidate (largest |a| among rows not yet used, ties to the lowest
// row) is published with its row and reciprocal, one barrier, and every
// thread takes the best of them.
__device__ __forceinline__ void gj_panel(double *A, int ld, int Npad, int k0, int &mine, double &piv,
                                         GJShared &g) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nw = (Npad + 31) >> 5;
  const bool row_ok = tid < Npad;
  double r[GB];
#pragma unroll
  for (int j = 0; j < GB; j += 2) {
    double2 v = make_double2(0.0, 0.0);
    if (row_ok) v = *reinterpret_cast<const double2 *>(A + gj_at(tid, k0 + j, ld));
    r[j] = v.x;
    r[j + 1] = v.y;
  }
#pragma unroll
  for (int k = 0; k < GB; ++k) {
    const int buf = k & 1;
    unsigned hi = (unsigned)__double2hiint(r[k]) & 0x7fffffffu, lo = (unsigned)__double2loint(r[k]);
    const bool use = row_ok && mine < 0 && !(hi > 0x7ff00000u || (hi == 0x7ff00000u && lo != 0u));
    if (!use) hi = lo = 0u;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    const unsigned bal = __ballot_sync(0xffffffffu, use && hi == mh && lo == ml);
    if (bal ? lane == __ffs(bal) - 1 : lane == 0) {
      g.ckey[buf][warp] = bal ? ((unsigned long long)mh << 32) | ml : 0ull;
      g.crow[buf][warp] = tid;
      g.cinv[buf][warp] = vmc_recip(r[k]);
#pragma unroll
      for (int j = 0; j < GB; j += 2)
        *reinterpret_cast<double2 *>(&g.cand[buf][warp][j]) = make_double2(r[j], r[j + 1]);
    }
    if (nw > 1)
      asm volatile("bar.sync 1, %0;" ::"r"(nw * 32) : "memory");
    else
      __syncwarp();
    int wb = 0;
    unsigned long long bk = g.ckey[buf][0];
    for (int q = 1; q < nw; ++q) {
      const unsigned long long kq = g.ckey[buf][q];
      if (kq > bk) {
        bk = kq;
        wb = q;
      }
    }
    if (bk == 0ull) {   // no finite non-zero entry left: singular (every thread agrees)
      if (tid == 0) g.bad = 1;
      return;
    }
    const int p = g.crow[buf][wb];
    const double ip = g.cinv[buf][wb];
    const bool is = tid == p;
    if (is) {
      mine = k0 + k;
      piv = r[k];
      g.perm[k0 + k] = p;
#pragma unroll
      for (int j = 0; j < GB; ++j) r[j] = 0.0;
    }
    const double m = is ? ip : -(r[k] * ip);
#pragma unroll
    for (int j = 0; j < GB; j += 2) {
      const double2 v = *reinterpret_cast<const double2 *>(&g.cand[buf][wb][j]);
      if (j != k) r[j] = fma(m, v.x, r[j]);
      if (j + 1 != k) r[j + 1] = fma(m, v.y, r[j + 1]);
    }
    r[k] = m;
  }
  if (row_ok) {
    g.step[tid] = mine;
#pragma unroll
    for (int j = 0; j < GB; j += 2)
      *reinterpret_cast<double2 *>(A + gj_at(tid, k0 + j, ld)) = make_double2(r[j], r[j + 1]);
  }
}

// In place on the padded matrix A (gj_at); blockDim.x >= gj_threads(N).  On
// return entry (k, c) of the inverse is A[perm[k]][step[c]] (gj_inverse_at).
__device__ __forceinline__ void gj_invert(double *A, uint32_t *stage, int N, GJShared &g) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int Npad = gj_pad(N), ld = Npad, nwarps = blockDim.x >> 5;
  const int np = (Npad + 31) >> 5;      // panel warps
  const int nrb = Npad / 16;            // row blocks of the update, one per warp
  const int gr = lane >> 2, gt = lane & 3;
  int mine = -1;
  double piv = 1.0;
  if (tid == 0) g.bad = g.nonfinite = 0;
  __syncthreads();
  for (int k0 = 0; k0 < Npad; k0 += GB) {
    if (warp < np) gj_panel(A, ld, Npad, k0, mine, piv, g);
    __syncthreads();
    if (g.bad) return;   // uniform
    const int ntile = Npad / 8 - 2;
    if (ntile == 0) break;
    // the power of two of each pivot row outside the panel
    for (int l = warp; l < GB; l += nwarps) {
      const int p = g.perm[k0 + l];
      int h = 0;
      for (int c = lane; c < Npad; c += 32)
        if (c < k0 || c >= k0 + GB) h = max(h, vmc_dig::expo(A[gj_at(p, c, ld)]));
      h = __reduce_max_sync(0xffffffffu, h);
      if (lane == 0) g.sig[l] = h ? h - 1023 : 0;
    }
    __syncthreads();
    // this warp's 16 rows of T as digits: the A operands of the update
    uint32_t a[NDIG][4];
    int ea = NOEXP, eb = NOEXP;
    const int ra = warp * 16 + gr, rb = ra + 8;
    bool pa = false, pb = false;
    if (warp < nrb) {
      double x[2][4];
      int sg[4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const double2 u = *reinterpret_cast<const double2 *>(A + gj_at(ra, k0 + 2 * gt + 8 * h, ld));
        const double2 v = *reinterpret_cast<const double2 *>(A + gj_at(rb, k0 + 2 * gt + 8 * h, ld));
        x[0][2 * h] = u.x;
        x[0][2 * h + 1] = u.y;
        x[1][2 * h] = v.x;
        x[1][2 * h + 1] = v.y;
        sg[2 * h] = g.sig[2 * gt + 8 * h];
        sg[2 * h + 1] = g.sig[2 * gt + 8 * h + 1];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int e0 = vmc_dig::expo(x[0][q]), e1 = vmc_dig::expo(x[1][q]);
        if (e0) ea = max(ea, e0 + sg[q]);
        if (e1) eb = max(eb, e1 + sg[q]);
        if (e0 == 0x7ff || e1 == 0x7ff) g.nonfinite = 1;
      }
      ea = max(ea, __shfl_xor_sync(0xffffffffu, ea, 1));
      eb = max(eb, __shfl_xor_sync(0xffffffffu, eb, 1));
      ea = max(ea, __shfl_xor_sync(0xffffffffu, ea, 2));
      eb = max(eb, __shfl_xor_sync(0xffffffffu, eb, 2));
      long long q0[4], q1[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        q0[q] = vmc_dig::fixed(x[0][q], ea - sg[q]);
        q1[q] = vmc_dig::fixed(x[1][q], eb - sg[q]);
      }
#pragma unroll
      for (int s = 0; s < NDIG; ++s) {
        a[s][0] = vmc_dig::pair(q0[0], q0[1], s);
        a[s][1] = vmc_dig::pair(q1[0], q1[1], s);
        a[s][2] = vmc_dig::pair(q0[2], q0[3], s);
        a[s][3] = vmc_dig::pair(q1[2], q1[3], s);
      }
      pa = g.step[ra] >= k0;
      pb = g.step[rb] >= k0;
    }
    for (int c0 = 0; c0 < ntile; c0 += CT) {
      const int nt = min(CT, ntile - c0);
      // digits of the pivot rows' entries in these columns, four threads to a
      // column: words (k pair t, k pair t + 4) of digit s of column j at
      // stage[(32 s + j) 8 + 2 t], as the B operands read them
      for (int q = tid; q < nt * 32; q += blockDim.x) {
        const int j = q >> 2, t = q & 3;
        const int tile = c0 + (j >> 3);
        const int c = (tile < k0 / 8 ? tile : tile + 2) * 8 + (j & 7);
        double x[4];
        int sg[4], e = NOEXP;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int l = 2 * t + (u & 1) + 8 * (u >> 1);
          x[u] = A[gj_at(g.perm[k0 + l], c, ld)];
          sg[u] = g.sig[l];
          const int ex = vmc_dig::expo(x[u]);
          if (ex) e = max(e, ex - sg[u]);
          if (ex == 0x7ff) g.nonfinite = 1;
        }
        e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
        e = max(e, __shfl_xor_sync(0xffffffffu, e, 2));
        long long v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = vmc_dig::fixed(x[u], e + sg[u]);
#pragma unroll
        for (int s = 0; s < NDIG; ++s)
          *reinterpret_cast<uint2 *>(stage + (size_t)(s * CT * 8 + j) * 8 + 2 * t) =
              make_uint2(vmc_dig::pair(v[0], v[1], s), vmc_dig::pair(v[2], v[3], s));
        if (t == 0) g.rexp[j] = e;
      }
      __syncthreads();
      if (warp < nrb) {
        for (int ti = 0; ti < nt; ++ti) {
          float acc[8][4];
#pragma unroll
          for (int d = 0; d < 8; ++d)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[d][q] = GJ_MAGIC;
#pragma unroll
          for (int u = 0; u < NDIG; ++u) {
            const uint2 b = *reinterpret_cast<const uint2 *>(
                stage + (size_t)(u * CT * 8 + ti * 8 + gr) * 8 + 2 * gt);
#pragma unroll
            for (int s = 0; s < NDIG; ++s)
              if (s + u < 8) vmc_dig::mma(acc[s + u], a[s], b.x, b.y);
          }
          const int tile = c0 + ti;
          const int c = (tile < k0 / 8 ? tile : tile + 2) * 8 + 2 * gt;
          const int f0 = g.rexp[ti * 8 + 2 * gt], f1 = g.rexp[ti * 8 + 2 * gt + 1];
          double2 *w0 = reinterpret_cast<double2 *>(A + gj_at(ra, c, ld));
          double2 *w1 = reinterpret_cast<double2 *>(A + gj_at(rb, c, ld));
          double2 v0 = *w0, v1 = *w1;
          v0.x = (pa ? 0.0 : v0.x) + vmc_dig::scaled(gj_combine(acc, 0), vmc_dig::unit_expo(ea, f0));
          v0.y = (pa ? 0.0 : v0.y) + vmc_dig::scaled(gj_combine(acc, 1), vmc_dig::unit_expo(ea, f1));
          v1.x = (pb ? 0.0 : v1.x) + vmc_dig::scaled(gj_combine(acc, 2), vmc_dig::unit_expo(eb, f0));
          v1.y = (pb ? 0.0 : v1.y) + vmc_dig::scaled(gj_combine(acc, 3), vmc_dig::unit_expo(eb, f1));
          *w0 = v0;
          *w1 = v1;
        }
      }
      __syncthreads();
    }
  }
  // log|det M|, the pivot range and the sign (pivots of rows below N)
  if (warp < np) {
    const bool in = tid < N;
    const double a = in ? fabs(piv) : 1.0;
    double ls = log(a), mn = in ? a : 1e300, mx = in ? a : 0.0;
    for (int o = 16; o > 0; o >>= 1) {
      ls += __shfl_xor_sync(0xffffffffu, ls, o);
      mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    const unsigned neg = __ballot_sync(0xffffffffu, in && piv < 0.0);
    // parity of the row order: pairs of steps taken out of order
    int inv = 0;
    if (in)
      for (int j = tid + 1; j < N; ++j) inv += g.perm[j] < g.perm[tid];
    const unsigned odd = __ballot_sync(0xffffffffu, inv & 1);
    if (lane == 0) {
      g.val[warp] = ls;
      g.pminw[warp] = mn;
      g.amax[warp] = mx;
      g.neg[warp] = __popc(neg) + __popc(odd);
    }
  }
  __syncthreads();
  if (tid == 0) {
    double a = 0.0, b = 1e300, c = 0.0;
    int n = 0;
    for (int q = 0; q < np; ++q) {
      a += g.val[q];
      b = fmin(b, g.pminw[q]);
      c = fmax(c, g.amax[q]);
      n += g.neg[q];
    }
    g.logdet = g.nonfinite ? nan("") : a;
    g.pmin = b;
    g.pmax = c;
    g.sign = (n & 1) ? -1 : 1;
  }
  __syncthreads();
}

__device__ __forceinline__ double gj_inverse_at(const double *A, int N, int k, int c,
                                                const GJShared &g) {
  return A[gj_at(g.perm[k], g.step[c], gj_pad(N))];
}

// ---------------------------------------------------------------------------
// The elimination step by step, every multiply-add in FP64.  The blocked form
// above differs from it in the last bits (about 1e-14 of the inverse, at no
// larger error).  It takes the matrices close to singular, of the plain and the
// projected state alike (gj_invert_guarded); and two users of the inverse turn
// last bits into visible differences of a trajectory and keep this form: the mixed form's projected
// state, whose FP32 inverses have no low words and whose ratios are sums over
// the operations that cancel, and the mixed form of models with exchange
// terms, whose SR-CG steps stop before convergence and follow the last bits
// of the samples (a relative change of 1e-9 in E moves the step by up to 5 %).
// Threads: 128, or 256 where one CTA fills an SM's shared memory (N > 112).
// The N^3 multiply-adds keep the FP64 pipe 67 % busy at N = 112, two CTAs per
// SM (608 x 256 inverses: 480 ms); a form with the matrix in registers (16 x 16
// threads, one CTA per SM) was slower there, 645 ms: nothing runs under its chain
// of pivots.
// In place on an N x N row-major matrix (row stride lda) in shared or global
// memory.  Two barriers per elimination step:
//   (P, B) two warps take the pivot of column k from the per-warp
//       candidates (largest |a|, ties: lowest row) and form 1/pivot; one
//       forms the multipliers m_i = a_ik / pivot (pivot row swapped in,
//       m_k = 0, kept negated so the update is one FMA), the other the raw
//       pivot row, swapping rows k and p and scaling row k;
//   (E) a_ic -= m_i r_c over all entries, spread flat over the threads in
//       whole warps; before it, each thread forms the updated value of its
//       row of column k+1 once more (one FMA, from a copy of the column taken
//       in (B)) for the next step's pivot candidates, reduced per warp by
//       integer compares of |a|'s bit patterns, so the next pivot search
//       needs no barrier of its own.
// Entries of the rank-1 update in flight per thread.
constexpr int GJ_ILP = 4;
constexpr int ST_WARPS = 8;          // most warps of the step-by-step form

struct GJSteps {
  double val[ST_WARPS];
  double amax[ST_WARPS];
  unsigned long long ckey[2][ST_WARPS];   // per-warp pivot candidates (|a| bits) ...
  int cidx[2][ST_WARPS];                  // ... and their signed_row()s, double-buffered by step
  int bad;
  int sign;
  double logdet;
  double pmin, pmax;   // smallest / largest |pivot|
  double ipiv;         // 1 / pivot of the current step
  double colk[VMC_MAX_N];   // negated multipliers -m_i of the current step (m_k = 0)
  double rowk[VMC_MAX_N];   // raw pivot row of the current step
  double coln[VMC_MAX_N];   // column k+1 before the current step's update
  double apiv[VMC_MAX_N];   // |pivot| of every step
  double pminw[ST_WARPS];
};

// A matrix the blocked form finds close to singular (max|M^-1| times the
// largest pivot above this, or no pivot at all) is eliminated again step by
// step.  The two forms' inverses differ by about 1e-16 of that product; the
// spin swap of the pair correlations, a difference of products of two entries
// that nearly cancel, multiplies it by the product's square, and one walker in
// thousands then decides the mean.  4096 placements at N = 112, mixed form: the
// correlations differ from those of the step-by-step inverses by up to 0.8 of
// their size with the blocked form alone, by 2e-5 with 3000 here (5e-7 with
// 1000); k_init takes 5.1, 5.9 and 6.2 ms.  About one random placement in 270
// is above.  (Set on placements at N = 112; the bound itself does not depend on
// N.)
constexpr double GJ_BLOCKED_COND = 3e3;
// Where the second elimination keeps GJSteps: in the staged digits' space,
// behind the part that its longer rows (odd stride) take.
constexpr size_t GJ_REDO_OFFSET = sizeof(double) * VMC_MAX_N;
static_assert(GJ_REDO_OFFSET + sizeof(GJSteps) <= GJ_STAGE_BYTES, "no room for the second elimination");

// |a| as an ordered integer key; NaN below every number (never a pivot)
__device__ __forceinline__ unsigned long long pivot_key(double a) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(a) & 0x7FFFFFFFFFFFFFFFull;
  return b > 0x7FF0000000000000ull ? 0ull : b + 1ull;
}

// a candidate's row with the sign of its entry in the lowest bit
__device__ __forceinline__ int signed_row(int i, double a) {
  return 2 * i + (__double2hiint(a) < 0 ? 1 : 0);
}

// warp-wide largest key (ties: lowest row); lane 0 records it in slot buf
__device__ __forceinline__ void pivot_candidates(unsigned long long key, int row, GJSteps &g,
                                                 int buf) {
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long ok = __shfl_xor_sync(0xffffffffu, key, o);
    const int orow = __shfl_xor_sync(0xffffffffu, row, o);
    if (ok > key || (ok == key && orow < row)) {
      key = ok;
      row = orow;
    }
  }
  if ((threadIdx.x & 31) == 0) {
    g.ckey[buf][threadIdx.x >> 5] = key;
    g.cidx[buf][threadIdx.x >> 5] = row;
  }
}

template <int NTH>   // threads of the CTA; 0: blockDim.x (at most 32 ST_WARPS)
__device__ __forceinline__ void gj_steps(double *A, int lda, int N, int *perm, GJSteps &g) {
  const int tid = threadIdx.x;
  const int nth = NTH ? NTH : (int)blockDim.x, nwarp = nth / 32;
  if (tid == 0) {
    g.logdet = 0.0;
    g.sign = 1;
    g.bad = 0;
    g.pmin = 1e300;
    g.pmax = 0.0;
  }
  // candidates of column 0
  {
    unsigned long long key = 0ull;
    int row = 2 * N;
    for (int i = tid; i < N; i += nth) {
      const double v = A[(size_t)i * lda];
      const unsigned long long kk = pivot_key(v);
      if (kk > key) {
        key = kk;
        row = signed_row(i, v);
      }
    }
    pivot_candidates(key, row, g, 0);
  }
  __syncthreads();
  const int qn = nth / N, rn = nth - (nth / N) * N;
  auto adv = [&](int &ii, int &cc) {
    ii += qn;
    cc += rn;
    if (cc >= N) {
      cc -= N;
      ++ii;
    }
  };
  for (int k = 0; k < N; ++k) {
    const int buf = k & 1;
    // (P) + (B) by warps 0 and 1 while the others wait: both take the pivot
    // from the per-warp candidates and form 1/pivot; warp 0 the negated
    // multipliers (pivot row swapped in) and the inverse's column k, warp 1
    // the raw pivot row, the swap of rows k and p with row k scaled, and the
    // copy of column k+1 (the two touch disjoint columns).
    if (tid < 64) {
      unsigned long long bk = g.ckey[buf][0];
      int row = g.cidx[buf][0];
      for (int q = 1; q < nwarp; ++q) {
        const unsigned long long kq = g.ckey[buf][q];
        const int iq = g.cidx[buf][q];
        if (kq > bk || (kq == bk && iq < row)) {
          bk = kq;
          row = iq;
        }
      }
      const int p = row >> 1;
      const int lane = tid & 31;
      const bool singular = bk <= 1ull || p >= N;   // zero (key 1) or no finite entry
      // the pivot from its candidate, not from A: warp 0 writes column k while
      // warp 1 may not have started
      const double piv = __longlong_as_double((long long)((bk - 1ull) | (unsigned long long)(row & 1) << 63));
      const double ipiv = __drcp_rn(piv);
      if (singular) {
        if (tid == 0) g.bad = 1;
      } else if (tid < 32) {
        if (tid == 0) {
          perm[k] = p;
          g.ipiv = ipiv;
          g.apiv[k] = fabs(piv);   // log|det| is summed after the elimination
          if ((piv < 0.0) != (p != k)) g.sign = -g.sign;
        }
        const double nipiv = -ipiv;   // negated multipliers: the update is one FMA
        for (int i = lane; i < N; i += 32) {
          const double a = (i == k) ? 0.0 : A[(size_t)(i == p ? k : i) * lda + k];
          g.colk[i] = a * nipiv;
        }
        __syncwarp();
        // the inverse's column k: -m_i, and 1/pivot at row k (rowk_k = 0
        // leaves it through the update)
        for (int i = lane; i < N; i += 32) A[(size_t)i * lda + k] = (i == k) ? ipiv : g.colk[i];
      } else {
        for (int c = lane; c < N; c += 32) {
          if (c == k) {
            g.rowk[c] = 0.0;
            continue;
          }
          const double r = A[(size_t)p * lda + c];
          g.rowk[c] = r;
          if (p != k) A[(size_t)p * lda + c] = A[(size_t)k * lda + c];
          A[(size_t)k * lda + c] = r * ipiv;
        }
        __syncwarp();
        // column k+1 as the update below finds it (rows swapped)
        if (k + 1 < N)
          for (int i = lane; i < N; i += 32) g.coln[i] = A[(size_t)i * lda + k + 1];
      }
    }
    __syncthreads();
    if (g.bad) return;   // uniform
    const int k1 = k + 1;
    // (E0) pivot candidates of column k+1 among rows >= k+1, from the values
    // the update below stores there (the same FMA), so the next pivot needs
    // no barrier of its own
    if (k1 < N) {
      unsigned long long key = 0ull;
      int row = 2 * N;
      for (int i = tid; i < N; i += nth) {
        const double v = fma(g.colk[i], g.rowk[k1], g.coln[i]);
        const unsigned long long kk = pivot_key(v);
        const bool t = (i >= k1) & (kk > key);
        key = t ? kk : key;
        row = t ? signed_row(i, v) : row;
      }
      pivot_candidates(key, row, g, buf ^ 1);
    }
    // (E) a_ic += (-m_i) r_c over all entries, spread flat over the threads
    // in whole warps, GJ_ILP entries in flight per thread (m_k = 0 leaves
    // row k, r_k = 0 leaves column k)
    {
      int i = tid / N, c = tid - (tid / N) * N;
      while (i < N) {
        int ii[GJ_ILP], cc[GJ_ILP];
        ii[0] = i;
        cc[0] = c;
#pragma unroll
        for (int u = 1; u < GJ_ILP; ++u) {
          ii[u] = ii[u - 1];
          cc[u] = cc[u - 1];
          adv(ii[u], cc[u]);
        }
        double *q[GJ_ILP];
        double a[GJ_ILP];
#pragma unroll
        for (int u = 0; u < GJ_ILP; ++u) {
          const bool ok = ii[u] < N;
          q[u] = A + (size_t)(ok ? ii[u] : i) * lda + (ok ? cc[u] : c);
          a[u] = *q[u];
        }
#pragma unroll
        for (int u = 0; u < GJ_ILP; ++u) {
          const int iu = ii[u] < N ? ii[u] : i, cu = ii[u] < N ? cc[u] : c;
          a[u] = fma(g.colk[iu], g.rowk[cu], a[u]);
        }
#pragma unroll
        for (int u = 0; u < GJ_ILP; ++u)
          if (u == 0 || ii[u] < N) *q[u] = a[u];
        i = ii[GJ_ILP - 1];
        c = cc[GJ_ILP - 1];
        adv(i, c);
      }
    }
    __syncthreads();
  }
  // log|det M| and the pivot range, off the elimination's serial path
  {
    double ls = 0.0, mn = 1e300, mx = 0.0;
    for (int i = tid; i < N; i += nth) {
      const double a = g.apiv[i];
      ls += log(a);
      mn = fmin(mn, a);
      mx = fmax(mx, a);
    }
    for (int o = 16; o > 0; o >>= 1) {
      ls += __shfl_xor_sync(0xffffffffu, ls, o);
      mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if ((tid & 31) == 0) {
      g.val[tid >> 5] = ls;
      g.pminw[tid >> 5] = mn;
      g.amax[tid >> 5] = mx;
    }
    __syncthreads();
    if (tid == 0) {
      double a = 0.0, b = 1e300, c = 0.0;
      for (int q = 0; q < nwarp; ++q) {
        a += g.val[q];
        b = fmin(b, g.pminw[q]);
        c = fmax(c, g.amax[q]);
      }
      g.logdet = a;
      g.pmin = b;
      g.pmax = c;
    }
  }
  for (int k = N - 1; k >= 0; --k) {
    const int p = perm[k];
    if (p == k) continue;   // uniform: perm is shared
    for (int r = tid; r < N; r += nth) {
      const double t0 = A[(size_t)r * lda + k];
      A[(size_t)r * lda + k] = A[(size_t)r * lda + p];
      A[(size_t)r * lda + p] = t0;
    }
    __syncthreads();
  }
  __syncthreads();
}

// The inverse by panels of the matrix entry(n, m), which A holds already (padded,
// gj_at); if it is close to singular, step by step after all, from entry() again,
// in rows of ld = N or N + 1 (odd).  stage: the staged digits' space (16-byte
// aligned), perm: N ints, red: a word per warp.  Every thread returns the same.
struct GJResult {
  int bad, sign;
  double logdet, pmin, pmax;
  bool steps;   // the inverse's entry (k, c) is A[k ld + c], else gj_inverse_at
};
template <typename Entry>
__device__ __forceinline__ GJResult gj_invert_guarded(double *A, uint32_t *stage, int N, int *perm,
                                                      GJShared &g, double *red, Entry entry) {
  const int tid = threadIdx.x, nwarps = blockDim.x >> 5, ld = (N % 2) ? N : N + 1;
  gj_invert(A, stage, N, g);
  GJResult r = {g.bad, g.sign, g.logdet, g.pmin, g.pmax, false};
  double amax = 0.0;
  if (!r.bad)   // the inverse's entries, in the order they are stored
    for (int i = tid >> 5; i < N; i += nwarps)
      for (int q = tid & 31; q < N; q += 32) amax = fmax(amax, fabs(A[gj_at(i, q, gj_pad(N))]));
  for (int o = 16; o > 0; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  if ((tid & 31) == 0) red[tid >> 5] = amax;
  __syncthreads();
  for (int q = 0; q < nwarps; ++q) amax = fmax(amax, red[q]);
  r.steps = r.bad || !(amax * r.pmax <= GJ_BLOCKED_COND);
  __syncthreads();
  if (r.steps) {
    GJSteps &g2 = *(GJSteps *)((unsigned char *)stage + GJ_REDO_OFFSET);
    for (int q = tid; q < N * N; q += blockDim.x) {
      const int n = q / N, m = q - n * N;
      A[n * ld + m] = entry(n, m);
    }
    __syncthreads();
    gj_steps<0>(A, ld, N, perm, g2);
    r.bad = g2.bad;
    r.sign = g2.sign;
    r.logdet = g2.logdet;
    r.pmin = g2.pmin;
    r.pmax = g2.pmax;
  }
  return r;
}

inline int gj_step_threads(int n_max) { return n_max > 112 ? 32 * ST_WARPS : 128; }

}  // namespace vmc_gj
