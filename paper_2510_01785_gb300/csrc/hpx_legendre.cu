// Legendre stage of the HEALPix SHT (Sec. III-D Eq. 14-16, Eq. 24-27).
//
// lambda_lm(z) obeys the three-term recurrence of Eq. 16,
//   lambda_l = alpha_l (z lambda_{l-1} - lambda_{l-2} / alpha_{l-1}),
//   alpha_l = sqrt((4 l^2 - 1) / (l^2 - m^2)),
// started from lambda_mm = (-1)^m sqrt(prod_{k<=m} (2k+1)/(2k) / 4 pi) sin^m.
// It is run here in the rescaled variable mu_l = lambda_l / P_l with
// P_m = P_{m+1} = 1 and P_l = (alpha_l / alpha_{l-1}) P_{l-2}, which turns it
// into mu_l = c_l z mu_{l-1} - mu_{l-2} (c_l = alpha_l P_{l-1} / P_l): two
// FP64 operations per step.  P_l does not depend on the ring, so it is
// applied once per output coefficient (analysis) or once per input
// coefficient (synthesis) instead of once per step.
//
// Exponent rescaling: a plan-time pass runs every (m, ring) chain in a
// (mantissa, 2^(-512 k)) representation from lambda_mm until it first
// reaches 2^-200 (FP32 plans: the larger thresholds below which their values
// are zero anyway, see kSigExp64) and records l_c and (mu_{l_c-1}, mu_{l_c}).
// Values before l_c are dropped; after l_c they stay within the double range,
// so the per-transform kernels run the plain recurrence from the recorded
// state and skip the dropped part of every chain.
//
// Contraction with the rings (analysis) or coefficients (synthesis) uses the
// north/south symmetry lambda_lm(-z) = (-1)^(l+m) lambda_lm(z): each chain
// serves a mirrored ring pair, with S = G(y) + G(y') for even l - m and
// A = G(y) - G(y') for odd l - m.
#include <cooperative_groups.h>

#include <climits>
#include <vector>

#include <type_traits>

#include "hpx_internal.cuh"

namespace cg = cooperative_groups;

namespace hpx {

using T = double;  // the transform kernels of this file serve FP64 plans; hpx_legendre_f32.cu has the FP32 ones

constexpr int LB = 32;  // l values per block of the recurrence

// ---------------------------------------------------------------------------
// plan-time tables
// ---------------------------------------------------------------------------
// lambda_mm / sin^m theta = (-1)^m sqrt(prod_{k=1..m} (2k+1)/(2k) / (4 pi)),
// the product carried as an unevaluated double-double sum.
__global__ void k_lambda_mm_prefactor(int mmax, double* cmm) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m > mmax) return;
  double hi = 1.0, lo = 0.0;
  for (int k = 1; k <= m; ++k) {
    const double num = 2.0 * k + 1.0, den = 2.0 * k;
    const double qh = num / den;
    const double ql = fma(-qh, den, num) / den;  // num/den = qh + ql
    const double ph = hi * qh;
    double pe = fma(hi, qh, -ph);
    pe = fma(hi, ql, pe);
    pe = fma(lo, qh, pe);
    hi = ph + pe;
    lo = pe - (hi - ph);
  }
  const double inv4pi = 0.079577471545947667884;  // 1 / (4 pi)
  const double r = sqrt(hi * inv4pi) * (1.0 + 0.5 * lo / hi);
  cmm[m] = (m & 1) ? -r : r;
}

// c_l and P_l of the rescaled recurrence for every (l, m); packed like alm.
// coef_p (FP64 plans) or coef_pp (the others: hi + lo).
__global__ void k_recurrence_coefs(int lmax, int mmax, double* coef_c, double* coef_p, float2* coef_pp,
                                   float* coef_pf) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m > mmax) return;
  const long long base = (long long)m * (2 * lmax + 1 - m) / 2;
  auto put = [&](int l, double P) {
    const float hi = (float)P;
    if (coef_p) coef_p[base + l] = P;
    if (coef_pp) coef_pp[base + l] = make_float2(hi, (float)(P - (double)hi));
    coef_pf[base + l] = hi;
  };
  coef_c[base + m] = 0.0;
  put(m, 1.0);
  double p1 = 1.0, p2 = 1.0, a_prev = 0.0;  // P_{l-1}, P_{l-2}, alpha_{l-1}
  const double md = m;
  for (int l = m + 1; l <= lmax; ++l) {
    const double ld = l;
    const double a = sqrt((4.0 * ld * ld - 1.0) / (ld * ld - md * md));
    double P, c;
    if (l == m + 1) {
      P = 1.0;
      c = a;
    } else {
      P = (a / a_prev) * p2;
      c = a * p1 / P;
    }
    coef_c[base + l] = c;
    put(l, P);
    p2 = p1;
    p1 = P;
    a_prev = a;
  }
}

// Start of every chain (m, pair): the first l at which |mu_l| >= 2^-sig,
// with (mu_{l-1}, mu_l) there; l_c = lmax + 1 if the chain never gets there.
// FP32 plans (lgrid given, zeroed before): also, per group of 64 pairs, the
// largest over its chains of the first l past l_c at which |mu_l| >=
// 2^-kGridExp (lmax + 1 where a chain never gets there; a plain FP32
// recurrence finds it), and in gstart (large before) the earliest l_c.
// lc32 and start32, where given: the start from 2^-sig; lc_tab, start and the groups
// then are of the later one, 2^-sig2 (the same values on the way: scaling by powers
// of two is exact).
__global__ void k_chain_scan(const RingInfo* __restrict__ rings, const double* __restrict__ cmm,
                             const double* __restrict__ coef_c, const float2* __restrict__ coef_cf, int lmax,
                             int npair, int sig, int sig2, int* lc_tab, double* mu0_tab, double* mu1_tab,
                             float4* __restrict__ start, int* __restrict__ lgrid, int* __restrict__ gstart,
                             int ngrid, int* __restrict__ lc32, float4* __restrict__ start32) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  const int m = blockIdx.y;
  if (p >= npair) return;
  const double z = rings[p].z, s = rings[p].sinth;
  // sin^m by binary powering on (mantissa, exponent) pairs
  int es;
  const double fs = frexp(s, &es);
  double rm = 1.0, bm = fs;
  long long er = 0, eb = 0;
  for (int n = m; n > 0; n >>= 1) {
    int e;
    if (n & 1) {
      rm = frexp(rm * bm, &e);
      er += eb + e;
    }
    if (n > 1) {
      bm = frexp(bm * bm, &e);
      eb = 2 * eb + e;
    }
  }
  int e1;
  const double v0 = frexp(cmm[m] * rm, &e1);
  const long long E = er + (long long)m * es + e1;  // |lambda_mm| in [2^(E-1), 2^E)
  long long k = 0;
  if (E < -(sig - 1)) k = (-(sig - 1) - E + 511) / 512;
  const double up = ldexp(1.0, 512 - sig);
  double mu1 = ldexp(v0, (int)(E + 512 * k)), mu2 = 0.0;
  int l = m;
  const long long base = (long long)m * (2 * lmax + 1 - m) / 2;
  while (k > 0 && l < lmax) {
    ++l;
    const double mu = fma(coef_c[base + l] * z, mu1, -mu2);
    mu2 = mu1;
    mu1 = mu;
    if (fabs(mu1) >= up) {
      mu1 *= 0x1p-512;
      mu2 *= 0x1p-512;
      --k;
    }
  }
  const long long ci = (long long)m * npair + p;
  if (k > 0) mu1 = mu2 = 0.0;
  if (lc32) {
    lc32[ci] = k > 0 ? lmax + 1 : l;
    const Df d0 = df_of(mu2 * kDfUp), d1 = df_of(mu1 * kDfUp);
    start32[ci] = make_float4(d0.hi, d0.lo, d1.hi, d1.lo);
    const double up2 = ldexp(1.0, -sig2);
    while (k <= 0 && fabs(mu1) < up2) {
      if (l == lmax) {
        k = 1;  // never gets there
        mu1 = mu2 = 0.0;
        break;
      }
      ++l;
      const double mu = fma(coef_c[base + l] * z, mu1, -mu2);
      mu2 = mu1;
      mu1 = mu;
    }
  }
  lc_tab[ci] = k > 0 ? lmax + 1 : l;
  if (!start) {
    mu0_tab[ci] = mu2;
    mu1_tab[ci] = mu1;
    return;
  }
  const Df d0 = df_of(mu2 * kDfUp), d1 = df_of(mu1 * kDfUp);
  start[ci] = make_float4(d0.hi, d0.lo, d1.hi, d1.lo);
  int lg = lmax + 1;
  if (k <= 0 && !grid_never(p & ~63, npair, lmax)) {
    const float zf = (float)z;
    float x1 = (float)(mu1 * 0x1p100), x2 = (float)(mu2 * 0x1p100);
    lg = l;
    while (lg <= lmax && fabsf(x1) < 0x1p100f * (1.f / (1 << kGridExp))) {
      ++lg;
      if (lg > lmax) break;
      const float x = fmaf(coef_cf[base + lg].x * zf, x1, -x2);
      x2 = x1;
      x1 = x;
    }
    lg = max(lg, l + 1);
  }
  // one atomic per half group: the lanes of a warp with pairs share a 64-pair group
  const int left = npair - (p & ~31);
  const unsigned mask = left >= 32 ? 0xffffffffu : (1u << left) - 1u;
  lg = __reduce_max_sync(mask, lg);
  const int ls = __reduce_min_sync(mask, lc_tab[ci]);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(lgrid + (long long)m * ngrid + (p >> 6), lg);
    atomicMin(gstart + (long long)m * ngrid + (p >> 6), ls);
  }
}

// ---------------------------------------------------------------------------
// analysis
// ---------------------------------------------------------------------------
// Lane tiling of the (LB x 2CP) output block of one warp: each lane owns LPL
// consecutive l and CPL consecutive real components.
template <int C2N> struct LaneTile {  // LPL = C2N / CPL (LB = 32), both parities of l where CPL allows
  static constexpr int LPL = C2N <= 4 ? 1 : C2N == 16 ? 4 : 2, CPL = C2N / LPL;
};
static_assert(LB == 32, "lane tiles");

constexpr int kMuStride = LB + 16 / (int)sizeof(T);

// S/A coefficients, mu rows (each warp's partial sums of a block reuse its own
// 32 rows once it has read them), the double-buffered block partials, c_l
template <int CP>
size_t analysis_smem(int nthr) {
  constexpr int C2N = 2 * CP;
  static_assert(LB * C2N <= 32 * kMuStride, "partials fit a warp's mu rows");
  return sizeof(T) * ((size_t)nthr * 2 * C2N + (size_t)nthr * kMuStride + 2 * LB * C2N) +
         sizeof(double) * 2 * LB;
}

// One cluster per m, one recurrence chain per thread.  Warps take 32
// consecutive ring pairs (similar start l, so few idle lanes) and are dealt
// round-robin over the cluster's CTAs, so every CTA holds polar and
// equatorial chains alike and none idles at the cluster barrier.  Per block
// of LB l values: the chains write mu into shared memory (from the recurrence,
// or streamed from the lambda table when TAB), each warp contracts its 32
// chains with their S/A ring coefficients, the warps' partial sums are added
// in shared memory, and the cluster adds the CTAs' partials through
// distributed shared memory (double-buffered, one cluster barrier per block).
// Deterministic order.
template <int CP, bool TAB>
__global__ void __launch_bounds__(512)
k_legendre_analysis(const C2<T>* __restrict__ spec, T* __restrict__ alm, const RingInfo* __restrict__ rings,
                    const C2<T>* __restrict__ etab, const double* __restrict__ coef_c,
                    const double* __restrict__ coef_p, const int* __restrict__ lc_tab,
                    const double* __restrict__ mu0_tab, const double* __restrict__ mu1_tab, int lmax,
                    int npair, int nring, long long nspec, long long nalm, int b0, int nb, int use_w,
                    const LamTab<T> tb, double mfac) {
  using V = C2<T>;
  constexpr int C2N = 2 * CP;
  constexpr int CPL = LaneTile<C2N>::CPL, LPL = LaneTile<C2N>::LPL, NCQ = C2N / CPL;
  constexpr int MS = kMuStride;
  cg::cluster_group cluster = cg::this_cluster();
  const int crank = (int)cluster.block_rank(), csize = (int)cluster.num_blocks();
  const int nthr = blockDim.x, nwarp = nthr >> 5;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int m = blockIdx.y;
  const int p = (warp * csize + crank) * 32 + lane;
  const bool active = p < npair;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sG = reinterpret_cast<T*>(smem_raw);      // [nthr][2][C2N]  S, A
  T* sMu = sG + (size_t)nthr * 2 * C2N;        // [nthr][MS]; warp w's [LB][C2N] partials at row 32 w
  T* sC = sMu + (size_t)nthr * MS;             // [2][LB][C2N]
  double* sCz = reinterpret_cast<double*>(sC + 2 * LB * C2N);  // [2][LB] c_l of this and the next block

  double z = 0.0, s0 = 0.0, s1 = 0.0;
  int lc = INT_MAX;
  {
    T* g = sG + (size_t)t * 2 * C2N;
    if (active) {
      const int ys = (p == npair - 1) ? -1 : nring - 1 - p;
      const RingInfo Rn = rings[p];
      z = Rn.z;
      const long long ci = (long long)m * npair + p;
      lc = lc_tab[ci];
      s0 = mu0_tab[ci];
      s1 = mu1_tab[ci];
      if (lc > lmax) lc = INT_MAX;
      for (int c = 0; c < CP; ++c) {
        V gn = cmk<V>(0, 0), gs = cmk<V>(0, 0);
        if (c < nb && lc != INT_MAX) {
          gn = ring_coef<T>(spec, etab, Rn, m, b0 + c, nspec, use_w);
          if (ys >= 0) gs = ring_coef<T>(spec, etab, rings[ys], m, b0 + c, nspec, use_w);
        }
        const V S = cadd(gn, gs), A = csub(gn, gs);
        g[2 * c] = S.x;
        g[2 * c + 1] = S.y;
        g[C2N + 2 * c] = A.x;
        g[C2N + 2 * c + 1] = A.y;
      }
    } else {
      for (int c = 0; c < 2 * C2N; ++c) g[c] = (T)0;
    }
  }

  const long long base = alm_base(lmax, m);
  const int lq = lane / NCQ, cq = lane % NCQ;
  const int l0 = lq * LPL, c0 = cq * CPL;
  RecurD rc;
  rc.start(z, s0, s1);
  int buf = 0;
  if (t < LB) sCz[t] = (m + t <= lmax) ? coef_c[base + m + t] : 0.0;
  // TAB: this warp's group rows (32 coalesced 128-byte rows per block),
  // loaded one block ahead so the loads are in flight during the contraction
  // and the reductions of the block before
  int tls = INT_MAX;
  const T* ttg = nullptr;
  T nxt[TAB ? LB : 1];
  if constexpr (TAB) {
    const int g = warp * csize + crank;
    if (g < tb.ngroup) {
      tls = tb.lstart[(long long)m * tb.ngroup + g];
      ttg = tb.tab + tb.off[(long long)m * tb.ngroup + g] + lane;
    }
#pragma unroll
    for (int i = 0; i < LB; ++i) {
      const int l = m + i;
      nxt[i] = (l >= tls && l <= lmax) ? __ldcs(ttg + (long long)(l - tls) * 32) : (T)0;
    }
  }
  __syncthreads();
  for (int lb0 = m; lb0 <= lmax; lb0 += LB) {
    const double* cz = sCz + buf * LB;
    // --- recurrence: LB steps of mu_l = c_l z mu_{l-1} - mu_{l-2} ---
    T* myMu = sMu + (size_t)t * MS;
    if constexpr (TAB) {
#pragma unroll
      for (int i4 = 0; i4 < LB; i4 += 4) {
        *reinterpret_cast<double2*>(myMu + i4) = make_double2(nxt[i4], nxt[i4 + 1]);
        *reinterpret_cast<double2*>(myMu + i4 + 2) = make_double2(nxt[i4 + 2], nxt[i4 + 3]);
      }
#pragma unroll
      for (int i = 0; i < LB; ++i) {
        const int l = lb0 + LB + i;
        nxt[i] = (l >= tls && l <= lmax) ? __ldcs(ttg + (long long)(l - tls) * 32) : (T)0;
      }
    } else if (__any_sync(0xffffffffu, lc < lb0 + LB)) {
#pragma unroll
      for (int i4 = 0; i4 < LB; i4 += 4) {
        T v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = rc.step(cz[i4 + u], lb0 + i4 + u, lc);
        *reinterpret_cast<double2*>(myMu + i4) = make_double2(v[0], v[1]);
        *reinterpret_cast<double2*>(myMu + i4 + 2) = make_double2(v[2], v[3]);
      }
    } else {
#pragma unroll
      for (int i = 0; i < LB; ++i) myMu[i] = (T)0;
    }
    const int any_active = __syncthreads_or(lc < lb0 + LB);
    T* cpart = sC + buf * LB * C2N;
    if (any_active) {
      // --- contraction of this warp's 32 chains ---
      T acc[LPL][CPL];
#pragma unroll
      for (int a = 0; a < LPL; ++a)
#pragma unroll
        for (int c = 0; c < CPL; ++c) acc[a][c] = (T)0;
      const T* muw = sMu + (size_t)(warp * 32) * MS + l0;
      const T* gw = sG + (size_t)(warp * 32) * 2 * C2N + c0;
#pragma unroll 4
      for (int j = 0; j < 32; ++j) {
        T mv[LPL], gsv[CPL], gav[CPL];
#pragma unroll
        for (int a = 0; a < LPL; ++a) mv[a] = muw[(size_t)j * MS + a];
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
          gsv[c] = gw[(size_t)j * 2 * C2N + c];
          gav[c] = gw[(size_t)j * 2 * C2N + C2N + c];
        }
#pragma unroll
        for (int a = 0; a < LPL; ++a) {
          const bool odd = ((l0 + a) & 1) != 0;
#pragma unroll
          for (int c = 0; c < CPL; ++c) acc[a][c] = fma(mv[a], odd ? gav[c] : gsv[c], acc[a][c]);
        }
      }
      // this warp's partials over its own mu rows, which only it has read
      T* wp = sMu + (size_t)(warp * 32) * MS;
      __syncwarp();
#pragma unroll
      for (int a = 0; a < LPL; ++a)
#pragma unroll
        for (int c = 0; c < CPL; ++c) wp[(l0 + a) * C2N + c0 + c] = acc[a][c];
      __syncthreads();
      for (int o = t; o < LB * C2N; o += nthr) {
        T s = (T)0;
        for (int w = 0; w < nwarp; ++w) s += sMu[(size_t)(w * 32) * MS + o];
        cpart[o] = s;
      }
    } else {
      for (int o = t; o < LB * C2N; o += nthr) cpart[o] = (T)0;
    }
    // c_l of the next block, into the other half of the double buffer
    if (t < LB) {
      const int l = lb0 + LB + t;
      sCz[(buf ^ 1) * LB + t] = (l <= lmax) ? coef_c[base + l] : 0.0;
    }
    // --- cluster reduction; CTA r writes its share of the block ---
    cluster.sync();
    {
      const int nout = LB * C2N;
      const int per = (nout + csize - 1) / csize;
      const int q_end = min(nout, (crank + 1) * per);
      for (int q = crank * per + t; q < q_end; q += nthr) {
        const int part = q & 1, li = (q >> 1) % LB, bb = (q >> 1) / LB;
        const int l = lb0 + li;
        if (l > lmax || bb >= nb) continue;
        const int o = li * C2N + 2 * bb + part;
        T s = (T)0;
        for (int r = 0; r < csize; ++r) s += cluster.map_shared_rank(cpart, r)[o];
        alm[((long long)(b0 + bb) * nalm + base + l) * 2 + part] =
            (T)(coef_p[base + l] * (m > 0 ? mfac : 1.0) * (double)s);
      }
    }
    buf ^= 1;
  }
  cluster.sync();  // peers may still read this CTA's partials
}

// ---------------------------------------------------------------------------
// synthesis
// ---------------------------------------------------------------------------
// One thread per chain (m, pair): E_m = sum over even l - m of a_lm lambda_lm,
// O_m = sum over odd l - m; F_m(y) = E + O on the northern ring and
// F_m(y') = E - O on its mirror (Eq. 24 before the ring transform).  The
// block's coefficients (pre-multiplied by P_l) are broadcast from shared
// memory; mu comes from the recurrence, or from the lambda table when TAB.
template <int CP, bool TAB>
__global__ void __launch_bounds__(128)
k_legendre_synthesis(const T* __restrict__ alm, C2<T>* __restrict__ F, const RingInfo* __restrict__ rings,
                     const double* __restrict__ coef_c, const double* __restrict__ coef_p, const int* __restrict__ lc_tab,
                     const double* __restrict__ mu0_tab, const double* __restrict__ mu1_tab, int lmax,
                     int mmax, int npair, int nring, long long nalm, int b0, int nb, const LamTab<T> tb,
                     double mfac) {
  using V = C2<T>;
  constexpr int C2N = 2 * CP;
  __shared__ __align__(16) T sA[LB][C2N];
  __shared__ double sCz[LB];
  __shared__ int sMinLc;
  const int m = blockIdx.y, t = threadIdx.x, nthr = blockDim.x;
  const int p = blockIdx.x * nthr + t;
  const bool active = p < npair;
  double z = 0.0, s0 = 0.0, s1 = 0.0;
  int lc = INT_MAX;
  if (active) {
    z = rings[p].z;
    const long long ci = (long long)m * npair + p;
    lc = lc_tab[ci];
    s0 = mu0_tab[ci];
    s1 = mu1_tab[ci];
    if (lc > lmax) lc = INT_MAX;
  }
  if (t == 0) sMinLc = INT_MAX;
  __syncthreads();
  atomicMin(&sMinLc, lc);
  __syncthreads();
  const int lstart = sMinLc;
  T accE[C2N], accO[C2N];
#pragma unroll
  for (int c = 0; c < C2N; ++c) accE[c] = accO[c] = (T)0;
  const long long base = alm_base(lmax, m);
  RecurD rc;
  rc.start(z, s0, s1);
  if (lstart <= lmax) {
    for (int lb0 = m + ((lstart - m) / LB) * LB; lb0 <= lmax; lb0 += LB) {
      for (int q = t; q < LB * C2N; q += nthr) {
        const int li = q / C2N, c = q % C2N, bb = c >> 1, part = c & 1;
        const int l = lb0 + li;
        T v = (T)0;
        if (l <= lmax && bb < nb && !(m == 0 && part == 1)) {
          const T a = alm[((long long)(b0 + bb) * nalm + base + l) * 2 + part];
          v = coef_p[base + l] * (m > 0 ? mfac : 1.0) * a;
        }
        sA[li][c] = v;
      }
      if (t < LB) sCz[t] = (lb0 + t <= lmax) ? coef_c[base + lb0 + t] : 0.0;
      __syncthreads();
      // a warp whose chains all start after this block has nothing to add
      if (TAB && __any_sync(0xffffffffu, lc < lb0 + LB)) {
        const int g = p >> 5;
        const bool gok = g < tb.ngroup;
        const int ls = gok ? tb.lstart[(long long)m * tb.ngroup + g] : INT_MAX;
        const T* tg = tb.tab + (gok ? tb.off[(long long)m * tb.ngroup + g] : 0) + (p & 31);
#pragma unroll
        for (int h = 0; h < LB; h += 16) {
          T mv[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int l = lb0 + h + i;
            mv[i] = (l >= ls && l <= lmax) ? __ldcs(tg + (long long)(l - ls) * 32) : (T)0;
          }
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
#pragma unroll
            for (int c = 0; c < C2N; ++c) accE[c] = fma(mv[i], sA[h + i][c], accE[c]);
#pragma unroll
            for (int c = 0; c < C2N; ++c) accO[c] = fma(mv[i + 1], sA[h + i + 1][c], accO[c]);
          }
        }
      } else if (!TAB && __any_sync(0xffffffffu, lc < lb0 + LB)) {
#pragma unroll 4
        for (int i = 0; i < LB; i += 2) {
          {
            const T mf = rc.step(sCz[i], lb0 + i, lc);
#pragma unroll
            for (int c = 0; c < C2N; ++c) accE[c] = fma(mf, sA[i][c], accE[c]);
          }
          {
            const T mf = rc.step(sCz[i + 1], lb0 + i + 1, lc);
#pragma unroll
            for (int c = 0; c < C2N; ++c) accO[c] = fma(mf, sA[i + 1][c], accO[c]);
          }
        }
      }
      __syncthreads();
    }
  }
  if (active) {
    const int ys = (p == npair - 1) ? -1 : nring - 1 - p;
#pragma unroll
    for (int bb = 0; bb < CP; ++bb) {
      if (bb < nb) {
        const V e = cmk<V>(accE[2 * bb], accE[2 * bb + 1]);
        const V o = cmk<V>(accO[2 * bb], accO[2 * bb + 1]);
        F[((long long)(b0 + bb) * nring + p) * (mmax + 1) + m] = cadd(e, o);
        if (ys >= 0) F[((long long)(b0 + bb) * nring + ys) * (mmax + 1) + m] = csub(e, o);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static void analysis_shape(int npair, int* nthr, int* csize) {
  if (npair <= 256) {
    *nthr = ((npair + 31) / 32) * 32;
    *csize = 1;
  } else {
    *nthr = npair / 8 > 256 ? npair / 8 : 256;
    *csize = (npair + *nthr - 1) / *nthr;
  }
}

template <int CP, bool TAB>
static cudaError_t launch_analysis_cp(const hpx_plan_s* p, T* alm, bool use_w, double mfac, cudaStream_t s,
                                      int* nlaunch) {
  using V = C2<T>;
  int nthr, csize;
  analysis_shape(p->npair, &nthr, &csize);
  const size_t smem = analysis_smem<CP>(nthr);
  cudaError_t e = allow_max_smem(k_legendre_analysis<CP, TAB>);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(csize, p->mmax + 1, 1);
  cfg.blockDim = dim3(nthr, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = csize;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  for (int b0 = 0; b0 < p->nbatch; b0 += CP) {
    const int nb = (p->nbatch - b0) < CP ? (p->nbatch - b0) : CP;
    e = cudaLaunchKernelEx(&cfg, k_legendre_analysis<CP, TAB>, (const V*)p->d_spec, alm,
                           (const RingInfo*)p->d_ring, (const V*)p->d_etab, (const double*)p->d_coef_c,
                           (const double*)p->d_coef_p, (const int*)p->d_lc, (const double*)p->d_mu0,
                           (const double*)p->d_mu1, p->lmax, p->npair, p->nring, p->nspec, p->nalm, b0, nb,
                           use_w ? 1 : 0, lam_tab<T>(p), mfac);
    if (e != cudaSuccess) return e;
    ++*nlaunch;
  }
  return cudaGetLastError();
}

template <int CP>
static cudaError_t launch_analysis_sel(const hpx_plan_s* p, T* alm, bool use_w, double mfac, cudaStream_t s,
                                       int* nlaunch) {
  return p->d_tab ? launch_analysis_cp<CP, true>(p, alm, use_w, mfac, s, nlaunch)
                  : launch_analysis_cp<CP, false>(p, alm, use_w, mfac, s, nlaunch);
}

// f(integral_constant CP) for cp = 1 .. 8
template <typename F> static auto with_cp(int cp, F f) {
  switch (cp) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 3: return f(std::integral_constant<int, 3>{});
    case 4: return f(std::integral_constant<int, 4>{});
    case 5: return f(std::integral_constant<int, 5>{});
    case 6: return f(std::integral_constant<int, 6>{});
    case 7: return f(std::integral_constant<int, 7>{});
    default: return f(std::integral_constant<int, 8>{});
  }
}
// Channels a launch: as many launches as eight at most a launch need, of equal
// width.  The FP64 pipe bounds both stages, at two instructions for the
// recurrence and two a channel, so channels that are not there cost as much as
// those that are (Nside 128, three channels, widths 4 -> 3: analysis 0.438 -> 0.362
// ms, synthesis 0.481 -> 0.387; Nside 512, five, 8 -> 5: 8.88 -> 6.14 and 6.75 ->
// 4.54 ms).
static int channels_of(int nbatch, int launches) { return (nbatch + launches - 1) / launches; }
static int pick_cp(const hpx_plan_s* p) {
  int nthr, csize;
  analysis_shape(p->npair, &nthr, &csize);
  auto fits = [&](int c) { return with_cp(c, [&](auto k) { return analysis_smem<decltype(k)::value>(nthr); }) <= 200 * 1024; };
  int k = (p->nbatch + 7) / 8;
  while (channels_of(p->nbatch, k) > 1 && !fits(channels_of(p->nbatch, k))) ++k;
  return channels_of(p->nbatch, k);
}

template <>
cudaError_t launch_analysis<double>(const hpx_plan_s* p, double* alm, bool use_w, double mfac, cudaStream_t s,
                                    int* nlaunch) {
  return with_cp(pick_cp(p), [&](auto k) { return launch_analysis_sel<decltype(k)::value>(p, alm, use_w, mfac, s, nlaunch); });
}

template <int CP, bool TAB>
static cudaError_t launch_synthesis_cp(const hpx_plan_s* p, const T* alm, double mfac, cudaStream_t s,
                                       int* nlaunch) {
  using V = C2<T>;
  const int nthr = 128;
  dim3 grid((p->npair + nthr - 1) / nthr, p->mmax + 1);
  for (int b0 = 0; b0 < p->nbatch; b0 += CP) {
    const int nb = (p->nbatch - b0) < CP ? (p->nbatch - b0) : CP;
    k_legendre_synthesis<CP, TAB><<<grid, nthr, 0, s>>>(
        alm, (V*)p->d_F, p->d_ring, (const double*)p->d_coef_c, p->d_coef_p, p->d_lc, p->d_mu0, p->d_mu1,
        p->lmax, p->mmax, p->npair, p->nring, p->nalm, b0, nb, lam_tab<T>(p), mfac);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    ++*nlaunch;
  }
  return cudaSuccess;
}

template <int CP>
static cudaError_t launch_synthesis_sel(const hpx_plan_s* p, const T* alm, double mfac, cudaStream_t s,
                                        int* nlaunch) {
  return p->d_tab ? launch_synthesis_cp<CP, true>(p, alm, mfac, s, nlaunch)
                  : launch_synthesis_cp<CP, false>(p, alm, mfac, s, nlaunch);
}

template <>
cudaError_t launch_synthesis<double>(const hpx_plan_s* p, const double* alm, double mfac, cudaStream_t s,
                                     int* nlaunch) {
  return with_cp(channels_of(p->nbatch, (p->nbatch + 7) / 8),
                 [&](auto k) { return launch_synthesis_sel<decltype(k)::value>(p, alm, mfac, s, nlaunch); });
}

// c_l as the double-FP32 pairs of the FP32 plans' recurrence
__global__ void k_coef_pairs(const double* __restrict__ coef_c, float2* __restrict__ coef_cf, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const Df d = df_of(coef_c[i]);
    coef_cf[i] = make_float2(d.hi, d.lo);
  }
}

__global__ void k_z_pairs(const RingInfo* __restrict__ rings, float2* __restrict__ zf, int npair) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npair) return;
  const Df d = df_of(rings[p].z);
  zf[p] = make_float2(d.hi, d.lo);
}

cudaError_t build_recurrence_tables(hpx_plan_s* p, cudaStream_t s) {
  const int mb = (p->mmax + 1 + 127) / 128;
  k_lambda_mm_prefactor<<<mb, 128, 0, s>>>(p->mmax, p->d_cmm);
  k_recurrence_coefs<<<mb, 128, 0, s>>>(p->lmax, p->mmax, p->d_coef_c, p->d_coef_p, p->d_coef_pp, p->d_coef_pf);
  const long long nb = (p->nalm + 255) / 256;
  k_coef_pairs<<<(unsigned)(nb < 4096 ? nb : 4096), 256, 0, s>>>(p->d_coef_c, p->d_coef_cf, p->nalm);
  const int mode = tc_mode_of(p->dtype, p->flags);
  const bool half = mode > 0 && p->dtype != HPX_F32_BF16 && p->dtype != HPX_F32_BF16X3;
  const int sig = p->dtype == HPX_F64 ? kSigExp64 : half && !p->d_lc32 ? kSigExpHalf : kSigExp32;
  if (p->d_lgrid) {
    const size_t bytes = sizeof(int) * (size_t)(p->mmax + 1) * p->ngrid;
    cudaError_t e = cudaMemsetAsync(p->d_lgrid, 0, bytes, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(p->d_gstart, 0x7f, bytes, s);
    if (e != cudaSuccess) return e;
    k_z_pairs<<<(p->npair + 127) / 128, 128, 0, s>>>(p->d_ring, p->d_zf, p->npair);
  }
  k_chain_scan<<<dim3((p->npair + 127) / 128, p->mmax + 1), 128, 0, s>>>(
      p->d_ring, p->d_cmm, p->d_coef_c, p->d_coef_cf, p->lmax, p->npair, sig, half ? kSigExpHalf : sig, p->d_lc, p->d_mu0,
      p->d_mu1, p->d_start, p->d_lgrid, p->d_gstart, p->ngrid, p->d_lc32, p->d_start32);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// plan-resident lambda table
// ---------------------------------------------------------------------------
// Earliest chain start of each (m, 32-pair group) and its number of rows.
__global__ void k_table_groups(const int* __restrict__ lc_tab, int lmax, int npair, int ngroup, int align,
                               int* lstart, long long* rows) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  const int m = blockIdx.y;
  if (g >= ngroup) return;
  int ls = lmax + 1;
  for (int j = 0; j < 32; ++j) {
    const int p = g * 32 + j;
    if (p < npair) ls = min(ls, lc_tab[(long long)m * npair + p]);
  }
  // for the tensor-core analysis: aligned down to its tile grid m + align j,
  // so that a group covers a tile either entirely or not at all (the extra
  // rows hold zeros)
  if (ls <= lmax) ls = m + ((ls - m) / align) * align;
  lstart[(long long)m * ngroup + g] = ls;
  rows[(long long)m * ngroup + g] = lmax + 1 - ls;
}

// Rows of every group: the recurrence of the per-transform kernels (same
// operations), zero before a chain's start and for the padding lanes of a
// group.
template <typename E>
__global__ void k_table_fill(const RingInfo* __restrict__ rings, const double* __restrict__ coef_c,
                             const float2* __restrict__ coef_cf, const int* __restrict__ lc_tab,
                             const double* __restrict__ mu0_tab, const double* __restrict__ mu1_tab,
                             const float4* __restrict__ start, const int* __restrict__ lgrid, int ngrid,
                             const int* __restrict__ lstart,
                             const long long* __restrict__ off, int lmax, int npair, int ngroup, E* tab) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  const int m = blockIdx.y;
  const int g = p >> 5;
  if (g >= ngroup) return;
  const int ls = lstart[(long long)m * ngroup + g];
  E* out = tab + off[(long long)m * ngroup + g] + (p & 31);
  if (p >= npair) {
    for (int l = ls; l <= lmax; ++l) out[(long long)(l - ls) * 32] = (E)0;
    return;
  }
  if constexpr (sizeof(E) == 4) {
    Chain ch = chain_at<1>(rings, coef_cf, lc_tab, start, lgrid, ngrid, lmax, npair, m, p);
    for (int l = ls; l <= lmax; ++l) out[(long long)(l - ls) * 32] = ch.step(l);
  } else {
    const long long ci = (long long)m * npair + p;
    const int lc = lc_tab[ci];
    RecurD rc;
    rc.start(rings[p].z, mu0_tab[ci], mu1_tab[ci]);
    const long long base = alm_base(lmax, m);
    for (int l = ls; l <= lmax; ++l) out[(long long)(l - ls) * 32] = rc.step(coef_c[base + l], l, lc);
  }
}

template <typename E>
cudaError_t build_lambda_table(hpx_plan_s* p, cudaStream_t s) {
  const int ng = (p->npair + 31) / 32;
  p->ngroup = ng;
  const long long nent = (long long)(p->mmax + 1) * ng;
  cudaError_t e = cudaMalloc((void**)&p->d_tab_lstart, sizeof(int) * nent);
  if (e != cudaSuccess) return e;
  p->bytes += sizeof(int) * nent;
  e = cudaMalloc((void**)&p->d_tab_off, sizeof(long long) * nent);
  if (e != cudaSuccess) return e;
  p->bytes += sizeof(long long) * nent;
  k_table_groups<<<dim3((ng + 127) / 128, p->mmax + 1), 128, 0, s>>>(
      p->d_lc, p->lmax, p->npair, ng, (p->flags & HPX_PLAN_TENSOR_CORES) ? kTcTile : 1, p->d_tab_lstart, p->d_tab_off);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e;
  std::vector<long long> rows(nent);
  e = cudaMemcpy(rows.data(), p->d_tab_off, sizeof(long long) * nent, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return e;
  long long acc = 0;
  for (long long i = 0; i < nent; ++i) {
    const long long r = rows[i];
    rows[i] = acc;
    acc += 32 * r;
  }
  p->tab_elems = acc;
  e = cudaMemcpy(p->d_tab_off, rows.data(), sizeof(long long) * nent, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return e;
  e = cudaMalloc(&p->d_tab, sizeof(E) * (acc > 0 ? acc : 1));
  if (e != cudaSuccess) return e;
  p->bytes += sizeof(E) * (acc > 0 ? acc : 1);
  k_table_fill<E><<<dim3((ng * 32 + 127) / 128, p->mmax + 1), 128, 0, s>>>(
      p->d_ring, p->d_coef_c, p->d_coef_cf, p->d_lc, p->d_mu0, p->d_mu1, p->d_start, p->d_lgrid, p->ngrid, p->d_tab_lstart,
      p->d_tab_off, p->lmax, p->npair, ng, static_cast<E*>(p->d_tab));
  return cudaGetLastError();
}

template cudaError_t build_lambda_table<float>(hpx_plan_s*, cudaStream_t);
template cudaError_t build_lambda_table<double>(hpx_plan_s*, cudaStream_t);

}  // namespace hpx
