// Pair correlations of the current configurations (measurement mode of the
// mVMC paper, Sec. 2.2.3): ratio kernel, occupation counts, reduction.
#include "vmc_dev.cuh"

#include <type_traits>

namespace {

// ---------------------------------------------------------------------------
// Local estimators of Eq. MC, A acting on the ket |x>.  Off-diagonal kinds,
// per walker, from Green-function ratios of its M^-1 = B:
//   G_up[b, k] = sum_l f(b, r_l,dn) B_lk      (up electron k hops to b)
//   G_dn[a, m] = sum_k f(r_k,up, a) B_mk      (down electron m hops to a)
//   T[b, a]    = sum_k G_up[b, k] f(r_k,up, a)
// and, for the spin swap of up electron n on a with down electron m on b
// (both sites singly occupied; det of M with row n and column m replaced),
//   det M'/det M = G_up[b, n] G_dn[a, m] - B_mn (T[b, a] - f(b, a)).
//   kind 0 (c^dag_{b up} c_{j up}): up electron on j hops to b,
//          G_up[b, k] x P_G P_J ratio;
//   kind 1 (c^dag_{a dn} c_{b dn}): down electron on b hops to a,
//          G_dn[a, m] x P_G P_J ratio;
//   kind 4 (S^+_b S^-_a): the swap above, with the fermion sign -1 of
//          S^+S^- in the labelled basis (P_G, P_J unchanged).
// Only the entries an estimator uses are formed: G_up for sites b without an
// up electron, G_dn for sites a without a down electron, T for b singly
// occupied by a down electron and a by an up one.  At 16 x 16 and N = 112
// that is 4.1e6 multiply-adds a configuration (5.1e6 with the padding to 32
// electrons) where all sites took 9.6e6.
//
// Each of the three is a product of site rows of the f table, gathered at the
// electrons' sites, with a matrix in shared memory.  A warp takes BT sites at
// a time and all N electrons (U of 32 per lane): the gathered rows are staged
// in shared memory KC at a time and read as broadcast vectors, so BT U
// multiply-adds cost U + 2 shared loads (and T shares G_dn's rows, so both run
// in one pass).  The sum of every entry runs over the electrons in order from
// 0, one multiply-add each: the swap's difference cancels, so its factors keep
// the rounding that one order gives.  8 warps a CTA, two CTAs an SM where M^-1
// leaves room, so that one loads and gathers while the other multiplies.
// Bound by the shared-memory reads of the products and by instruction issue
// (by the FP64 pipe in the plain form).  4096 configurations of that system in
// the mixed form: 5.81 -> 2.24 ms (2.05 without the atomic adds; the
// multiply-adds alone are 0.55), against one thread per column and all sites.
//
// The estimators are added to one FP64 plane triple part[3][Ns][Ns] (diagonal
// entries stay 0; kind 4's plane holds [a][b], so that the lanes of a warp add
// to one row) by atomic adds without return, so the 24 Ns^2 bytes stay in L2
// and no thread waits on them; the order of the additions, and so the last
// bit of a sum, varies between runs.
// ---------------------------------------------------------------------------
constexpr int CNT = 256;          // threads of a CTA
constexpr int CW = CNT / 32;
constexpr int KC = 64;            // staged electrons of a warp's sites

// sites of a warp's tile: 32 bytes of staged words per electron
template <typename T> constexpr int corr_bt() { return 32 / (int)sizeof(T); }

// Shared memory of one walker; rows: rows of G_up kept for the spin swaps.
template <typename T>
struct CSmem {
  T *minv;        // N x ldm
  T *g;           // rows x ldm: G_up of down-occupied sites
  T *stage;       // CW x KC x BT
  T *jf;          // Ns
  int *ele;       // Ne
  short *occ;     // 2 Ns
  short *ul;      // Ns: sites without an up electron, those with a down one first
  short *al;      // Ns: sites without a down electron, those with an up one first
  short *pos;     // N: place of the down electron's site in ul, or -1
  int *cnt;       // n4 (head of ul), length of ul, head of al, length of al
};

template <typename T>
__host__ __device__ size_t corr_layout(int N, int Ns, int rows, unsigned char *base, CSmem<T> *sm) {
  const int ldm = (N % 2) ? N : N + 1;
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off = (off + bytes + 15) / 16 * 16; return o; };
  const size_t o_minv = take(((size_t)N * ldm * sizeof(T) + 127) / 128 * 128);
  const size_t o_stage = take((size_t)CW * KC * 32);
  const size_t o_jf = take(sizeof(T) * Ns);
  const size_t o_ele = take(sizeof(int) * 2 * N);
  const size_t o_occ = take(sizeof(short) * 2 * Ns);
  const size_t o_ul = take(sizeof(short) * Ns);
  const size_t o_al = take(sizeof(short) * Ns);
  const size_t o_pos = take(sizeof(short) * N);
  const size_t o_cnt = take(sizeof(int) * 4);
  const size_t o_g = take(sizeof(T) * (size_t)rows * ldm);
  if (sm) {
    sm->minv = (T *)(base + o_minv);
    sm->stage = (T *)(base + o_stage);
    sm->jf = (T *)(base + o_jf);
    sm->ele = (int *)(base + o_ele);
    sm->occ = (short *)(base + o_occ);
    sm->ul = (short *)(base + o_ul);
    sm->al = (short *)(base + o_al);
    sm->pos = (short *)(base + o_pos);
    sm->cnt = (int *)(base + o_cnt);
    sm->g = (T *)(base + o_g);
  }
  return off;
}

// One warp's tile: acc[j][u] = sum_l row_j[es[l]] A[col u][l] over l < N in
// order, and with TWO acc2 likewise with A2.  a[u], a2[u]: the lane's columns
// at l = 0, sl words apart from l to l + 1.  tab: table rows of Ns words;
// site[j]: the row of tile entry j.
template <typename T, int U, bool TWO>
__device__ __forceinline__ void corr_tile(const T *tab, int Ns, const int (&site)[corr_bt<T>()],
                                          const int *es, int N, T *stage, const T *const (&a)[U],
                                          const T *const (&a2)[U], int sl,
                                          T (&acc)[corr_bt<T>()][U], T (&acc2)[corr_bt<T>()][U]) {
  constexpr int BT = corr_bt<T>();
  using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
  constexpr int VN = 16 / (int)sizeof(T);
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int j = 0; j < BT; ++j)
#pragma unroll
    for (int u = 0; u < U; ++u) {
      acc[j][u] = (T)0;
      if constexpr (TWO) acc2[j][u] = (T)0;
    }
  for (int l0 = 0; l0 < N; l0 += KC) {
    const int len = (N - l0 < KC) ? N - l0 : KC;
    __syncwarp();
#pragma unroll
    for (int h = 0; h < KC / 32; ++h) {
      const int l = lane + 32 * h;
      if (l < len) {
        const int e = es[l0 + l];
        T v[BT];
#pragma unroll
        for (int j = 0; j < BT; ++j) v[j] = tab[(size_t)site[j] * Ns + e];
#pragma unroll
        for (int j = 0; j < BT; j += VN) {
          V x;
          if constexpr (sizeof(T) == 4) x = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
          else x = make_double2(v[j], v[j + 1]);
          *(V *)(stage + l * BT + j) = x;
        }
      }
    }
    __syncwarp();
#pragma unroll 2
    for (int l = 0; l < len; ++l) {
      T x[BT], m[U], m2[U];
#pragma unroll
      for (int j = 0; j < BT; j += VN) {
        const V y = *(const V *)(stage + l * BT + j);
        x[j] = y.x;
        x[j + 1] = y.y;
        if constexpr (sizeof(T) == 4) {
          x[j + 2] = y.z;
          x[j + 3] = y.w;
        }
      }
      const int o = (l0 + l) * sl;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        m[u] = a[u][o];
        if constexpr (TWO) m2[u] = a2[u][o];
      }
#pragma unroll
      for (int j = 0; j < BT; ++j)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          acc[j][u] += m[u] * x[j];
          if constexpr (TWO) acc2[j][u] += m2[u] * x[j];
        }
    }
  }
}

// log of the hop's correlation-factor ratio with v_tr for v_rt (v is
// symmetric), so that lanes with different r read one row of it.
template <typename T>
__device__ __forceinline__ T corr_hop_sym(const SysDev &S, const short *occ, const T *jf, int s,
                                          int r, int t) {
  return corr_hop_v<T>(occ, jf, gtab<T>(S), S.Ns, s, r, t, vtab<T>(S)[(size_t)t * S.Ns + r]);
}

// kind 1, and with SWAP kind 4, of the tile of sites al[i0 ..]
template <typename T, int U, bool SWAP>
__device__ __forceinline__ void corr_down(const SysDev &S, const CSmem<T> &sm, int i0, int n,
                                          int c0, int c1, T *stage, double *P1, double *P4) {
  constexpr int BT = corr_bt<T>();
  const int N = S.N, Ns = S.Ns, ldm = S.ldm, lane = threadIdx.x & 31;
  int site[BT];
#pragma unroll
  for (int j = 0; j < BT; ++j) site[j] = sm.al[i0 + j < n ? i0 + j : n - 1];
  const T *a[U], *a2[U];
  int place[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int m = lane + 32 * u;
    a[u] = sm.minv + (size_t)(m < N ? m : 0) * ldm;
    const int p = (SWAP && m < N) ? sm.pos[m] : -1;
    place[u] = (p >= c0 && p < c1) ? p - c0 : -1;
    a2[u] = SWAP ? sm.g + (size_t)(place[u] >= 0 ? place[u] : 0) * ldm : a[u];
  }
  T d[BT][U], t[BT][U];
  corr_tile<T, U, SWAP>(fTtab<T>(S), Ns, site, sm.ele, N, stage, a, a2, 1, d, t);
#pragma unroll
  for (int j = 0; j < BT; ++j) {
    if (i0 + j >= n) break;
    const int at = site[j];
    const int e = sm.occ[at];   // up electron on it, or -1
    const bool hop = c0 == 0 && !(S.local_spin && e >= 0);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int m = lane + 32 * u;
      if (m >= N) continue;
      const int bm = sm.ele[N + m];
      if (hop) {
        const T c = corr_factor<T>(corr_hop_sym<T>(S, sm.occ, sm.jf, 1, bm, at));
        atomicAdd(&P1[(size_t)at * Ns + bm], (double)(d[j][u] * c));
      }
      if constexpr (SWAP) {
        if (e >= 0 && place[u] >= 0) {
          // one rounding order, spelt out: the two products nearly cancel
          const T r = fma(a2[u][e], d[j][u],
                          -(a[u][e] * (t[j][u] - fTtab<T>(S)[(size_t)at * Ns + bm])));
          atomicAdd(&P4[(size_t)at * Ns + bm], -(double)r);
        }
      }
    }
  }
}

template <typename T, int U>
__global__ void __launch_bounds__(CNT, 2)
    k_corr(const SysDev *systems, int sys, int rows, double *part) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ SysDev S;
  load_sys(&S, systems + sys);
  constexpr int BT = corr_bt<T>();
  const int N = S.N, Ns = S.Ns, Ne = S.Ne, ldm = S.ldm, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  CSmem<T> sm;
  corr_layout<T>(N, Ns, rows, smem_raw, &sm);
  T *stage = sm.stage + (size_t)warp * KC * BT;
  const size_t ns2 = (size_t)Ns * Ns;
  double *P0 = part, *P1 = P0 + ns2, *P4 = P1 + ns2;
  const size_t nb = ((size_t)N * ldm * sizeof(T) + 127) / 128 * 128;
  for (int w = blockIdx.x; w < S.W; w += gridDim.x) {
    const uint4 *src = (const uint4 *)((const unsigned char *)S.minv + (size_t)w * nb);
    for (int k = tid; k < (int)(nb / 16); k += CNT) ((uint4 *)sm.minv)[k] = src[k];
    for (int k = tid; k < Ne; k += CNT) sm.ele[k] = S.ele[(size_t)w * Ne + k];
    for (int k = tid; k < 2 * Ns; k += CNT) sm.occ[k] = (short)S.occ[(size_t)w * 2 * Ns + k];
    for (int k = tid; k < Ns; k += CNT) sm.jf[k] = ((const T *)S.jf)[(size_t)w * Ns + k];
    for (int k = tid; k < N; k += CNT) sm.pos[k] = -1;
    __syncthreads();
    // warp 0 lists the sites b, warp 1 the sites a (in site order: first
    // those the swaps use, then those without any electron)
    if (warp < 2) {
      short *list = warp ? sm.al : sm.ul;
      const short *skip = sm.occ + (warp ? Ns : 0), *want = sm.occ + (warp ? 0 : Ns);
      int n = 0;
      for (int second = 0; second < 2; ++second) {
        for (int i0 = 0; i0 < Ns; i0 += 32) {
          const int i = i0 + lane;
          const bool in = i < Ns && skip[i] < 0 && ((want[i] < 0) == (second != 0));
          const unsigned mask = __ballot_sync(0xffffffffu, in);
          if (in) {
            const int p = n + __popc(mask & ((1u << lane) - 1));
            list[p] = (short)i;
            if (!warp && !second) sm.pos[want[i] - N] = (short)p;
          }
          n += __popc(mask);
        }
        if (lane == 0) sm.cnt[2 * warp + second] = n;
      }
    }
    __syncthreads();
    const int n4 = sm.cnt[0], nu = sm.cnt[1], na4 = sm.cnt[2], na = sm.cnt[3];
    // the swaps' sites b, `rows` at a time (all at once where they fit); the
    // first pass also takes the sites without an electron, and kind 1
    for (int c0 = 0; c0 == 0 || c0 < n4; c0 += rows) {
      const int c1 = (n4 - c0 < rows) ? n4 : c0 + rows;
      const int nc = c1 - c0, nb1 = nc + (c0 == 0 ? nu - n4 : 0);
      for (int i0 = warp * BT; i0 < nb1; i0 += CW * BT) {
        int site[BT];
#pragma unroll
        for (int j = 0; j < BT; ++j) {
          const int i = i0 + j < nb1 ? i0 + j : nb1 - 1;
          site[j] = sm.ul[i < nc ? c0 + i : n4 + i - nc];
        }
        const T *a[U];
#pragma unroll
        for (int u = 0; u < U; ++u) a[u] = sm.minv + (lane + 32 * u < N ? lane + 32 * u : 0);
        T g[BT][U], none[BT][U];
        corr_tile<T, U, false>(ftab<T>(S), Ns, site, sm.ele + N, N, stage, a, a, ldm, g, none);
#pragma unroll
        for (int j = 0; j < BT; ++j) {
          if (i0 + j >= nb1) break;
          const int b = site[j];
          const bool swap = i0 + j < nc;   // a down electron on b
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int k = lane + 32 * u;
            if (k >= N) continue;
            if (!(S.local_spin && swap)) {
              const int e = sm.ele[k];
              const T c = corr_factor<T>(corr_hop_sym<T>(S, sm.occ, sm.jf, 0, e, b));
              atomicAdd(&P0[(size_t)b * Ns + e], (double)(g[j][u] * c));
            }
            if (swap) sm.g[(size_t)(i0 + j) * ldm + k] = g[j][u];
          }
        }
      }
      __syncthreads();   // the swaps' rows of G_up are in place
      const int n1 = (c0 == 0) ? na : na4;
      for (int i0 = warp * BT; i0 < n1; i0 += CW * BT) {
        if (nc > 0 && i0 < na4) corr_down<T, U, true>(S, sm, i0, n1, c0, c1, stage, P1, P4);
        else corr_down<T, U, false>(S, sm, i0, n1, c0, c1, stage, P1, P4);
      }
      __syncthreads();
    }
  }
}

// Occupation products summed over the walkers of one system, exactly in
// integers: cnt[c][i][j] = sum_w x_i y_j with (x, y) = (n_up, n_up),
// (n_up, n_dn), (n_dn, n_up), (n_dn, n_dn) for c = 0..3.  These give every
// diagonal estimator (n_i n_j, S^z_i S^z_j and the i = j terms of kinds 0, 1,
// 4, 5).  A CTA takes a 32 x 32 tile of pairs and 256 walkers: each of its
// eight warps packs the occupations of 32 walkers at the tile's sites into one
// word a site (lane = site, so the loads are coalesced), and a pair's product
// is then eight ANDs and population counts.  cnt is zeroed by the launcher.
// Bound by the loads' issue; 4096 walkers of 256 sites: 0.84 ms with a thread
// per pair reading every walker's words, 0.05 with the reduction below.
__global__ void __launch_bounds__(256) k_corr_occ(const SysDev *systems, int sys, int *cnt) {
  __shared__ unsigned bits[4][8][32];   // n_up, n_dn at the rows' sites; at the columns'
  const SysDev &S = systems[sys];
  const int Ns = S.Ns, W = S.W, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int bi = blockIdx.y * 32, bj = blockIdx.x * 32;
  const int w0 = blockIdx.z * 256 + warp * 32;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int site = (q < 2 ? bi : bj) + lane;
    unsigned word = 0;
    if (site < Ns) {
      const int *o = S.occ + (size_t)w0 * 2 * Ns + (q & 1) * Ns + site;
#pragma unroll 8
      for (int k = 0; k < 32; ++k)
        if (w0 + k < W) word |= (o[(size_t)k * 2 * Ns] >= 0 ? 1u : 0u) << k;
    }
    bits[q][warp][lane] = word;
  }
  __syncthreads();
  const size_t ns2 = (size_t)Ns * Ns;
  const int j = bj + lane;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int y = warp + 8 * r, i = bi + y;
    int uu = 0, ud = 0, du = 0, dd = 0;
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const unsigned ui = bits[0][v][y], di = bits[1][v][y];
      const unsigned uj = bits[2][v][lane], dj = bits[3][v][lane];
      uu += __popc(ui & uj);
      ud += __popc(ui & dj);
      du += __popc(di & uj);
      dd += __popc(di & dj);
    }
    if (i < Ns && j < Ns) {
      const size_t q = (size_t)i * Ns + j;
      if (uu) atomicAdd(cnt + q, uu);
      if (ud) atomicAdd(cnt + ns2 + q, ud);
      if (du) atomicAdd(cnt + 2 * ns2 + q, du);
      if (dd) atomicAdd(cnt + 3 * ns2 + q, dd);
    }
  }
}

// out[kind][i][j] = walker mean of the local estimators (kinds 0..5 of the
// header): the ratio planes (n_part sets, summed in order) and the integer
// counts, scaled.  With a local_site mask (Kondo local spins: exactly one
// electron each) a hop c^dag_i c_j with i != j into or out of a marked site
// leaves the constrained space, where psi = 0: those entries of kinds 0 and 1
// are 0.  Spin swaps keep every site's occupation and are kept.
__global__ void k_corr_reduce(const double *part, int n_part, const int *cnt, int Ns, int W,
                              const signed char *lsite, double *out) {
  const size_t ns2 = (size_t)Ns * Ns;
  const double inv = 1.0 / (double)W;
  for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < ns2;
       q += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(q / Ns), j = (int)(q % Ns);
    const size_t qt = (size_t)j * Ns + i;
    double g0 = 0.0, g1 = 0.0, s4 = 0.0, s4t = 0.0;
    for (int b = 0; b < n_part; ++b) {
      const double *P = part + (size_t)b * 3 * ns2;
      g0 += P[q];
      g1 += P[ns2 + q];
      s4 += P[2 * ns2 + qt];   // kind 4's plane is transposed
      s4t += P[2 * ns2 + q];
    }
    const double uu = cnt[q], ud = cnt[ns2 + q], du = cnt[2 * ns2 + q], dd = cnt[3 * ns2 + q];
    const double szsz = 0.25 * (uu - ud - du + dd);
    double d0 = 0.0, d1 = 0.0, d4 = 0.0, d5 = 0.0;
    if (i == j) {   // n_up, n_dn, n_up (1 - n_dn), (n_up + n_dn - 2 n_up n_dn) / 2
      d0 = uu;
      d1 = dd;
      d4 = uu - ud;
      d5 = 0.5 * (uu - ud + dd - du);
    }
    if (lsite && i != j && (lsite[i] | lsite[j])) g0 = g1 = 0.0;
    out[q] = (g0 + d0) * inv;
    out[ns2 + q] = (g1 + d1) * inv;
    out[2 * ns2 + q] = (uu + ud + du + dd) * inv;
    out[3 * ns2 + q] = szsz * inv;
    out[4 * ns2 + q] = (s4 + d4) * inv;
    out[5 * ns2 + q] = (szsz + 0.5 * (s4 + s4t) + d5) * inv;
  }
}

using CorrKernel = void (*)(const SysDev *, int, int, double *);
template <typename T>
CorrKernel corr_kernel_of(int N) {
  switch ((N + 31) / 32) {
    case 1: return k_corr<T, 1>;
    case 2: return k_corr<T, 2>;
    case 3: return k_corr<T, 3>;
    default: return k_corr<T, 4>;
  }
}
CorrKernel corr_kernel(int precision, int N) {
  return precision == 0 ? corr_kernel_of<double>(N) : corr_kernel_of<float>(N);
}

}  // namespace

// Rows of G_up in shared memory: every singly occupied site's (at most
// min(N, Ns - N)) where two CTAs an SM still fit, or, where half the SM holds
// less than half of them, one CTA with as many as fit.
cudaError_t vmc_corr_shape(int precision, int N, int Ns, int W, CorrShape *out) {
  int dev = 0, nsm = 0, per_sm = 0, reserved = 0, optin = 0, per = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev))) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev))) return e;
  if ((e = cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev))) return e;
  if ((e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev))) return e;
  if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev))) return e;
  const CorrKernel kern = corr_kernel(precision, N);
  cudaFuncAttributes at;
  if ((e = cudaFuncGetAttributes(&at, (const void *)kern))) return e;
  const long long stat = (long long)at.sharedSizeBytes;
  const int ldm = (N % 2) ? N : N + 1;
  const long long row = (long long)ldm * (precision == 0 ? sizeof(double) : sizeof(float));
  const long long base = (long long)(precision == 0 ? corr_layout<double>(N, Ns, 0, nullptr, nullptr)
                                                    : corr_layout<float>(N, Ns, 0, nullptr, nullptr));
  const long long most = N < Ns - N ? N : Ns - N;
  const long long half = (per_sm / 2 - reserved - stat - base - 16) / row;
  const long long full = (optin - stat - base - 16) / row;
  long long rows = 2 * half >= most ? half : full;
  if (rows > most) rows = most;
  if (rows < 1) rows = 1;
  out->rows = (int)rows;
  out->smem = precision == 0 ? corr_layout<double>(N, Ns, (int)rows, nullptr, nullptr)
                             : corr_layout<float>(N, Ns, (int)rows, nullptr, nullptr);
  if ((e = vmc_smem_limit((const void *)kern, out->smem))) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, CNT, out->smem))) return e;
  if (per < 1) per = 1;
  const long long grid = (long long)nsm * per;
  out->grid = (int)(grid < W ? grid : (W > 0 ? W : 1));
  return cudaSuccess;
}

cudaError_t vmc_launch_corr(const SysDev *d_sys, int sys, int precision, int N,
                            const CorrShape &shape, double *part, cudaStream_t st, long long *nl) {
  corr_kernel(precision, N)<<<shape.grid, CNT, shape.smem, st>>>(d_sys, sys, shape.rows, part);
  ++*nl;
  return cudaGetLastError();
}

cudaError_t vmc_launch_corr_occ(const SysDev *d_sys, int sys, int Ns, int W, int *cnt,
                                cudaStream_t st, long long *nl) {
  const cudaError_t e = cudaMemsetAsync(cnt, 0, 4 * (size_t)Ns * Ns * sizeof(int), st);
  if (e) return e;
  const int t = (Ns + 31) / 32;
  const dim3 grid(t, t, (W + 255) / 256);
  k_corr_occ<<<grid, 256, 0, st>>>(d_sys, sys, cnt);
  ++*nl;
  return cudaGetLastError();
}

cudaError_t vmc_launch_corr_reduce(const double *part, int n_part, const int *cnt, int Ns, int W,
                                   const signed char *lsite, double *out, cudaStream_t st,
                                   long long *nl) {
  const size_t ns2 = (size_t)Ns * Ns;
  const size_t blocks = (ns2 + 255) / 256;
  const int grid = (int)(blocks < 4096 ? blocks : 4096);
  k_corr_reduce<<<grid, 256, 0, st>>>(part, n_part, cnt, Ns, W, lsite, out);
  ++*nl;
  return cudaGetLastError();
}
