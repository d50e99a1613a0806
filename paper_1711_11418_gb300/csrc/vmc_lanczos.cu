// First-step power-Lanczos on the GPU (mVMC paper, Sec. 3.4): the local
// values F(x, H) = <x|H|psi>/<x|psi> (= E_loc) and F(x, H^2) of every walker's
// current configuration, and their walker means, the moments h1, h2(11),
// h2(20), h3(12) from which E_1(alpha) and alpha_1 follow.
//
// With D the diagonal part of H and h_t the matrix element of an off-diagonal
// term t (a hop: -t_ij, labels kept, so no fermion sign):
//
//   F(x, H)   = D(x) + sum_{t1} h_{t1} R(t1),
//   F(x, H^2) = D(x) F(x, H) + sum_{t1} h_{t1} [ D(x') R(t1) + sum_{t2} h_{t2} R(t1, t2) ],
//
// x' = t1 x, x'' = t2 x', R(t1) = psi(x')/psi(x), R(t1, t2) = psi(x'')/psi(x):
// every ratio is taken from x, so nothing divides by psi(x') (which may
// vanish).  The Pfaffian parts of the ratios come from three tables of the
// configuration, with B = M^-1:
//
//   Gu[b][k] = sum_l f(b, r_l,dn) B[l][k]   (up electron k to site b),
//   Gd[a][m] = sum_k f(r_k,up, a) B[m][k]   (down electron m to site a),
//   T[b][a]  = sum_k Gu[b][k] f(r_k,up, a),
//
// by the determinant lemma: two up electrons k1 -> b1, k2 -> b2 give
// Gu[b1][k1] Gu[b2][k2] - Gu[b1][k2] Gu[b2][k1] (two down electrons alike with
// Gd), and up k -> b with down m -> a give Gu[b][k] Gd[a][m] - B[m][k] (T[b][a] - f(b, a)).
// The correlation factors of x'' are those of two successive hops, the second
// on the occupations and Jastrow field of x'.
//
// One CTA of 256 threads per walker, the tables in a per-CTA slot of global
// memory (L2):
//  (1) M^-1 in shared memory; the tables as register-tiled products, 8 x 8
//      (FP32) or 8 x 4 (FP64) entries a thread, each entry one chain of
//      multiply-adds in the order of the sum;
//  (2) the hop terms that move x, listed per spin with what a pair needs of
//      them alone: sites, electron, Pfaffian ratio, log of the correlation
//      factor's ratio, matrix element.  A quarter of the terms, so a quarter
//      of the lanes' turns in (3);
//  (3) a warp per first term t1, lanes over the listed second terms.  A pair
//      needs five more numbers, each from a vector fixed by t1 (a row and a
//      column of Gu or Gd, a row or column of T, the change of the Jastrow
//      field), which the warp stages first.  The list holds the terms valid on
//      x; on x' a hop of the same spin into i1 or out of j1 drops out, and the
//      hops out of i1 (the same electron again) and into j1 come in, taken
//      from the terms by source and by target.
// What bounds it: (3) issue, about 40 instructions per pair and 2.5e5 pairs a
// walker at 16 x 16; (1) the loads that feed its multiply-adds.  Every pair
// reading four tables of the slot, and tables formed entry by entry from
// strided loads, took 35.9 ms for 1024 walkers of 16 x 16 (FP32); 4.9 ms so.
#include "vmc_common.cuh"
#include "vmc_dev.cuh"

#include <math.h>

namespace {

constexpr int LZ_NT = 256;           // threads per walker
constexpr int LZ_NW = LZ_NT / 32;

// A hop term that moves x: i2 | j2 << 12 | e2 << 24 | s2 << 31 (sites, label
// within the spin, spin; Ns <= 4096, N <= 128), its Pfaffian ratio, the log of
// its correlation-factor ratio, its matrix element -t.
template <typename T>
struct alignas(4 * sizeof(T)) LzTerm {
  unsigned pk;
  T r, c, h;
};

// A CTA's slot: Gu^T [N][Ns], Gd^T [N][Ns], T - f [Ns][Ns], the listed terms,
// their indices, and the warps' vectors where shared memory does not hold them.
struct LzSlot {
  size_t gd, tt, list, idx, vec, bytes;
};
template <typename T>
__host__ __device__ inline LzSlot lz_slot(int Ns, int N, int n_hop, bool vec_smem) {
  auto al = [](size_t x) { return (x + 63) / 64 * 64; };
  LzSlot s;
  s.gd = al(sizeof(T) * Ns * N);
  s.tt = s.gd + al(sizeof(T) * Ns * N);
  s.list = s.tt + al(sizeof(T) * Ns * Ns);
  s.idx = s.list + al(sizeof(LzTerm<T>) * 2 * (size_t)n_hop);
  s.vec = s.idx + al(sizeof(int) * 2 * (size_t)n_hop);
  s.bytes = s.vec + (vec_smem ? 0 : al(sizeof(T) * LZ_NW * (3 * (size_t)Ns + N)));
  return s;
}

// Shared memory: M^-1 (N x ldm), the Jastrow field, occupations, and the
// warps' vectors.
template <typename T>
__host__ __device__ inline size_t lz_smem(int Ns, int N, bool vec_smem) {
  const int ldm = (N % 2) ? N : N + 1;
  auto al = [](size_t x) { return (x + 15) / 16 * 16; };
  return al(sizeof(T) * (size_t)N * ldm) + al(sizeof(T) * Ns) + al(sizeof(int) * 2 * Ns) +
         (vec_smem ? sizeof(T) * LZ_NW * (3 * (size_t)Ns + N) : 0);
}

template <typename T>
__device__ __forceinline__ const T *minv_of(const SysDev &S, int w) {
  const size_t nb = ((size_t)S.N * S.ldm * sizeof(T) + 127) / 128 * 128;
  return (const T *)((const unsigned char *)S.minv + (size_t)w * nb);
}

// log P(y')/P(y) of a hop of a spin-s electron from site r to site t on a
// configuration y given by its occupations (occ, with the hop's own electron
// at r) and Jastrow field jf (Sec. 3.2.3), in the ratios' type (FP64, or FP32
// in the mixed form: GB300's FP64 pipe is 1/64 of the FP32 rate).
template <typename T>
__device__ __forceinline__ T corr_log(const SysDev &S, const int *occ, const T *jf, int s, int r,
                                      int t) {
  const int Ns = S.Ns, o = (1 - s) * Ns;
  const T *g = gtab<T>(S);
  T d = jf[t] - jf[r] - vtab<T>(S)[(size_t)r * Ns + t];
  d += (occ[o + t] >= 0 ? g[t] : (T)0) - (occ[o + r] >= 0 ? g[r] : (T)0);
  return d;
}

// Diagonal part of H (U n_up n_dn + V n n) of x moved by one hop of a spin-s
// electron r -> t (r = t = -1: x itself), by one warp.
__device__ double diag_energy(const SysDev &S, const int *occ, int s, int r, int t) {
  const int Ns = S.Ns, lane = threadIdx.x & 31;
  auto nsp = [&](int i, int sp) -> int {
    int v = occ[sp * Ns + i] >= 0;
    if (sp == s) v += (i == t) - (i == r);
    return v;
  };
  double d = 0.0;
  for (int i = lane; i < Ns; i += 32)
    if (nsp(i, 0) && nsp(i, 1)) d += S.U[i];
  for (int k = lane; k < S.n_V; k += 32) {
    const int a = S.V_i[k], b = S.V_j[k];
    d += S.V_val[k] * (double)((nsp(a, 0) + nsp(a, 1)) * (nsp(b, 0) + nsp(b, 1)));
  }
  return warp_sum(d);
}

// out[r][c] = sum_l a(l, r) y(l)[c], r < R, c < Ns, l < K ascending, by the
// CTA as 16 x 16 threads; store(r, c, value).
template <typename T, typename FA, typename FY, typename FS>
__device__ __forceinline__ void lz_product(int R, int Ns, int K, FA a, FY y, FS store) {
  constexpr int CW = sizeof(T) == 4 ? 8 : 4;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  for (int r0 = 0; r0 < R; r0 += 128)
    for (int c0 = 0; c0 < Ns; c0 += 16 * CW) {
      T acc[8][CW];
#pragma unroll
      for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int v = 0; v < CW; ++v) acc[u][v] = (T)0;
      int ri[8], ci[CW];
#pragma unroll
      for (int u = 0; u < 8; ++u) ri[u] = min(r0 + ty + 16 * u, R - 1);
#pragma unroll
      for (int v = 0; v < CW; ++v) ci[v] = min(c0 + tx + 16 * v, Ns - 1);
#pragma unroll 1
      for (int l = 0; l < K; ++l) {
        const T *yr = y(l);
        T av[8], yv[CW];
#pragma unroll
        for (int v = 0; v < CW; ++v) yv[v] = yr[ci[v]];
#pragma unroll
        for (int u = 0; u < 8; ++u) av[u] = a(l, ri[u]);
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
          for (int v = 0; v < CW; ++v) acc[u][v] += yv[v] * av[u];
      }
#pragma unroll
      for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int v = 0; v < CW; ++v)
          if (r0 + ty + 16 * u < R && c0 + tx + 16 * v < Ns)
            store(r0 + ty + 16 * u, c0 + tx + 16 * v, acc[u][v]);
    }
}

template <typename T, bool VS>   // VS: the warps' vectors are in shared memory
__global__ void __launch_bounds__(LZ_NT, sizeof(T) == 4 ? 2 : 1)
    k_lanczos(const SysDev *systems, int sys, unsigned char *slots, double *F1, double *F2) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ SysDev S;
  __shared__ int ele[2 * VMC_MAX_N];
  __shared__ double red[2 * LZ_NW];
  __shared__ int cnt[LZ_NW];
  load_sys(&S, systems + sys);
  const int N = S.N, Ns = S.Ns, Ne = S.Ne, ldm = S.ldm, tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  auto al = [](size_t x) { return (x + 15) / 16 * 16; };
  T *B = (T *)smem_raw;                                            // M^-1
  T *jf = (T *)((unsigned char *)B + al(sizeof(T) * (size_t)N * ldm));
  int *occ = (int *)((unsigned char *)jf + al(sizeof(T) * Ns));    // 2 Ns
  const LzSlot L = lz_slot<T>(Ns, N, S.n_hop, VS);
  unsigned char *slot = slots + (size_t)blockIdx.x * ((L.bytes + 255) / 256 * 256);
  T *Gu = (T *)slot, *Gd = (T *)(slot + L.gd), *Tt = (T *)(slot + L.tt);
  LzTerm<T> *list = (LzTerm<T> *)(slot + L.list);
  int *lidx = (int *)(slot + L.idx);
  T *vec = VS ? (T *)((unsigned char *)occ + al(sizeof(int) * 2 * Ns)) : (T *)(slot + L.vec);
  T *colv = vec + (size_t)warp * (3 * (size_t)Ns + N);             // Ns: column of Gu or Gd
  T *wv = colv + Ns, *tv = wv + Ns, *rowv = tv + Ns;               // Ns, Ns, N
  const T *F = ftab<T>(S);
  const T *FT = fTtab<T>(S);
  const T *V = vtab<T>(S);
  const T *G = gtab<T>(S);
  for (int w = blockIdx.x; w < S.W; w += gridDim.x) {
    __syncthreads();
    for (int k = tid; k < Ne; k += LZ_NT) ele[k] = S.ele[(size_t)w * Ne + k];
    for (int k = tid; k < 2 * Ns; k += LZ_NT) occ[k] = S.occ[(size_t)w * 2 * Ns + k];
    for (int k = tid; k < Ns; k += LZ_NT) jf[k] = ((const T *)S.jf)[(size_t)w * Ns + k];
    const T *Bg = minv_of<T>(S, w);
    for (int k = tid; k < N * ldm; k += LZ_NT) B[k] = Bg[k];
    __syncthreads();
    // (1) tables, by electron: Gu[k][b], Gd[m][a]; T[b][a] - f(b, a)
    lz_product<T>(
        N, Ns, N, [&](int l, int k) { return B[(size_t)l * ldm + k]; },
        [&](int l) { return FT + (size_t)ele[N + l] * Ns; },
        [&](int k, int b, T v) { Gu[(size_t)k * Ns + b] = v; });
    lz_product<T>(
        N, Ns, N, [&](int l, int m) { return B[(size_t)m * ldm + l]; },
        [&](int l) { return F + (size_t)ele[l] * Ns; },
        [&](int m, int a, T v) { Gd[(size_t)m * Ns + a] = v; });
    __syncthreads();
    lz_product<T>(
        Ns, Ns, N, [&](int k, int b) { return Gu[(size_t)k * Ns + b]; },
        [&](int k) { return F + (size_t)ele[k] * Ns; },
        [&](int b, int a, T v) { Tt[(size_t)b * Ns + a] = v - F[(size_t)b * Ns + a]; });
    // (2) the terms valid on x, per spin in order
    int n_up = 0, n_all = 0;
    for (int s = 0; s < 2; ++s) {
      for (int k0 = 0; k0 < S.n_hop; k0 += LZ_NT) {
        const int k = k0 + tid;
        int i = 0, j = 0, e = -1;
        if (k < S.n_hop) {
          i = S.hop_i[k];
          j = S.hop_j[k];
          e = occ[s * Ns + j];
          if (occ[s * Ns + i] >= 0 || (S.local_spin && occ[(1 - s) * Ns + i] >= 0) ||
              (S.lsite && (S.lsite[i] | S.lsite[j])))
            e = -1;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, e >= 0);
        __syncthreads();   // cnt of the round before is read
        if (lane == 0) cnt[warp] = __popc(bal);
        __syncthreads();
        int before = 0, total = 0;
        for (int q = 0; q < LZ_NW; ++q) {
          before += q < warp ? cnt[q] : 0;
          total += cnt[q];
        }
        if (e >= 0) {
          const int pos = n_all + before + __popc(bal & ((1u << lane) - 1u));
          const int el = s ? e - N : e;
          LzTerm<T> t;
          t.pk = (unsigned)i | ((unsigned)j << 12) | ((unsigned)el << 24) | ((unsigned)s << 31);
          t.r = (s ? Gd : Gu)[(size_t)el * Ns + i];
          t.c = corr_log<T>(S, occ, jf, s, j, i);
          t.h = (T)(-S.hop_t[k]);
          list[pos] = t;
          lidx[pos] = k;
        }
        n_all += total;
      }
      if (s == 0) n_up = n_all;
    }
    __syncthreads();
    // (3) pairs
    const double d0 = diag_energy(S, occ, 0, -1, -1);
    double f1 = 0.0, f2 = 0.0;   // f2: this lane's share
    for (int q1 = warp; q1 < n_all; q1 += LZ_NW) {
      const LzTerm<T> t1 = list[q1];
      const int i1 = t1.pk & 0xfffu, j1 = (t1.pk >> 12) & 0xfffu, e1 = (t1.pk >> 24) & 0x7fu;
      const int s1 = t1.pk >> 31;
      const T r1 = t1.r, c1 = t1.c;
      const double h1 = -S.hop_t[lidx[q1]];
      const T *G1 = (s1 ? Gd : Gu) + (size_t)e1 * Ns;
      __syncwarp();   // the vectors of the term before are read
      for (int x = lane; x < Ns; x += 32) {
        colv[x] = G1[x];
        wv[x] = V[(size_t)i1 * Ns + x] - V[(size_t)j1 * Ns + x];
        tv[x] = s1 ? Tt[(size_t)x * Ns + i1] : Tt[(size_t)i1 * Ns + x];
      }
      for (int x = lane; x < N; x += 32) rowv[x] = (s1 ? Gd : Gu)[(size_t)x * Ns + i1];
      __syncwarp();
      T acc = (T)0;
      // the other electrons of this spin
      const int a0 = s1 ? n_up : 0, a1 = s1 ? n_all : n_up;
      for (int q = a0 + lane; q < a1; q += 32) {
        const LzTerm<T> t = list[q];
        const int i2 = t.pk & 0xfffu, j2 = (t.pk >> 12) & 0xfffu, e2 = (t.pk >> 24) & 0x7fu;
        const T d = r1 * t.r - rowv[e2] * colv[i2];
        const T c2 = t.c + (wv[i2] - wv[j2]);
        const T R = d * corr_factor<T>(c1 + c2);
        if (i2 != i1 && j2 != j1) acc += t.h * R;
      }
      // the other spin: M changes in a row and a column
      const T gi = G[i1], gj = G[j1];
      const int b0 = s1 ? 0 : n_up, b1 = s1 ? n_up : n_all;
      for (int q = b0 + lane; q < b1; q += 32) {
        const LzTerm<T> t = list[q];
        const int i2 = t.pk & 0xfffu, j2 = (t.pk >> 12) & 0xfffu, e2 = (t.pk >> 24) & 0x7fu;
        const T d = r1 * t.r - B[s1 ? e1 * ldm + e2 : e2 * ldm + e1] * tv[i2];
        T c2 = t.c + (wv[i2] - wv[j2]);
        c2 += (i2 == i1 ? gi : i2 == j1 ? -gj : (T)0) - (j2 == i1 ? gi : j2 == j1 ? -gj : (T)0);
        acc += t.h * (d * corr_factor<T>(c1 + c2));
      }
      // the same electron again, out of i1 (back to x if to j1)
      for (int q = S.src_ptr[i1] + lane; q < S.src_ptr[i1 + 1]; q += 32) {
        const int i2 = S.src_i[q];
        if ((i2 != j1 && occ[s1 * Ns + i2] >= 0) || (S.lsite && (S.lsite[i2] | S.lsite[i1]))) continue;
        const T R = i2 == j1 ? (T)1
                             : colv[i2] * corr_factor<T>(corr_log<T>(S, occ, jf, s1, j1, i2));
        acc += (T)(-S.src_t[q]) * R;
      }
      // an electron of the same spin into j1
      for (int q = S.tgt_ptr[j1] + lane; q < S.tgt_ptr[j1 + 1]; q += 32) {
        const int j2 = S.tgt_j[q];
        const int e2 = occ[s1 * Ns + j2];
        if (j2 == i1 || e2 < 0 || (S.lsite && (S.lsite[j2] | S.lsite[j1]))) continue;
        const int el = s1 ? e2 - N : e2;
        const T d = r1 * (s1 ? Gd : Gu)[(size_t)el * Ns + j1] - rowv[el] * colv[j1];
        const T c2 = corr_log<T>(S, occ, jf, s1, j2, j1) + (wv[j1] - wv[j2]);
        acc += (T)(-S.tgt_t[q]) * (d * corr_factor<T>(c1 + c2));
      }
      f2 += h1 * (double)acc;
      // diagonal part of x'
      const int o = (1 - s1) * Ns;
      const double dx = S.n_V ? diag_energy(S, occ, s1, j1, i1)
                              : d0 + ((occ[o + i1] >= 0 ? S.U[i1] : 0.0) -
                                      (occ[o + j1] >= 0 ? S.U[j1] : 0.0));
      if (lane == 0) {
        const double hR = h1 * (double)(r1 * corr_factor<T>(c1));
        f1 += hR;
        f2 += hR * dx;
      }
    }
    f1 = warp_sum(f1);
    f2 = warp_sum(f2);
    if (lane == 0) {
      red[warp] = f1;
      red[LZ_NW + warp] = f2;
    }
    __syncthreads();
    if (tid == 0) {
      double a = 0.0, b = 0.0;
      for (int k = 0; k < LZ_NW; ++k) {
        a += red[k];
        b += red[LZ_NW + k];
      }
      const double e = d0 + a;
      F1[w] = e;
      F2[w] = d0 * e + b;
    }
  }
}

// h1 = <F1>, h2(11) = <F1^2>, h2(20) = <F2>, h3(12) = <F1 F2> over the walkers.
__global__ void k_lanczos_moments(const double *F1, const double *F2, int W, double *h) {
  __shared__ double red[4][NT];
  double a = 0.0, b = 0.0, c = 0.0, d = 0.0;
  for (int w = threadIdx.x; w < W; w += NT) {
    a += F1[w];
    b += F1[w] * F1[w];
    c += F2[w];
    d += F1[w] * F2[w];
  }
  red[0][threadIdx.x] = a;
  red[1][threadIdx.x] = b;
  red[2][threadIdx.x] = c;
  red[3][threadIdx.x] = d;
  __syncthreads();
  if (threadIdx.x < 4) {
    double s = 0.0;
    for (int k = 0; k < NT; ++k) s += red[threadIdx.x][k];
    h[threadIdx.x] = s / W;
  }
}

}  // namespace

namespace {

// Whether the warps' vectors fit shared memory beside the rest (always up to
// about 1000 sites); they go to the CTA's slot otherwise.
constexpr size_t LZ_SMEM_MAX = 224 * 1024;
template <typename T>
bool lz_vec_smem(int Ns, int N) {
  return lz_smem<T>(Ns, N, true) <= LZ_SMEM_MAX;
}

using LzKernel = void (*)(const SysDev *, int, unsigned char *, double *, double *);
LzKernel lz_kernel(int precision, bool vs) {
  if (precision == 0) return vs ? k_lanczos<double, true> : k_lanczos<double, false>;
  return vs ? k_lanczos<float, true> : k_lanczos<float, false>;
}

}  // namespace

size_t vmc_lanczos_slot_bytes(int precision, int Ns, int N, int n_hop) {
  return precision == 0 ? lz_slot<double>(Ns, N, n_hop, lz_vec_smem<double>(Ns, N)).bytes
                        : lz_slot<float>(Ns, N, n_hop, lz_vec_smem<float>(Ns, N)).bytes;
}

// The kernel for these sizes, its shared memory, and how many CTAs an SM holds.
static cudaError_t lz_config(int precision, int Ns, int N, LzKernel *k, size_t *smem, int *nb) {
  const bool vs = precision == 0 ? lz_vec_smem<double>(Ns, N) : lz_vec_smem<float>(Ns, N);
  *k = lz_kernel(precision, vs);
  *smem = precision == 0 ? lz_smem<double>(Ns, N, vs) : lz_smem<float>(Ns, N, vs);
  cudaError_t e = vmc_smem_limit((const void *)*k, *smem);
  if (e) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, *k, LZ_NT, *smem);
}

int vmc_lanczos_occupancy(int precision, int Ns, int N) {
  LzKernel k;
  size_t smem;
  int nb = 0;
  if (lz_config(precision, Ns, N, &k, &smem, &nb)) cudaGetLastError();
  return nb;
}

cudaError_t vmc_launch_lanczos(const SysDev *d_sys, int sys, int precision, int Ns, int N, int grid,
                               void *slots, double *F1, double *F2, int W, double *moments,
                               cudaStream_t st, long long *nl) {
  LzKernel k;
  size_t smem;
  int nb = 0;
  cudaError_t e = lz_config(precision, Ns, N, &k, &smem, &nb);
  if (e) return e;
  k<<<grid, LZ_NT, smem, st>>>(d_sys, sys, (unsigned char *)slots, F1, F2);
  k_lanczos_moments<<<1, NT, 0, st>>>(F1, F2, W, moments);
  *nl += 2;
  return cudaGetLastError();
}
