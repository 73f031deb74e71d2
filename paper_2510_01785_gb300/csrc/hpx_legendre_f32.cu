// Legendre stage of the FP32 plans on the CUDA cores (Sec. III-D Eq. 14-16,
// Eq. 24-27): lambda recomputed, or read from the plan's table, and contracted
// in FP32 FMAs.
//
// Both kernels give a lane two recurrence chains (ring pairs p and p + 32 of
// the warp's group of 64), stepped as hpx_internal.cuh describes.  They are bound by the FP32 pipe: per
// (l, m, ring pair) 12 operations of the recurrence and 2 a channel of the
// contraction, against 22 and 2 when every step was double-FP32.
// Where the old kernels lost the rest (analysis at 0.3 of the FP32 pipe's
// rate): one chain a lane leaves three shared-memory loads for every four
// FMAs of the analysis and one for every four of the synthesis; two chains
// and an 8 x 8 tile a lane make that one for sixteen and one for eight.
#include <cooperative_groups.h>

#include <climits>

#include "hpx_internal.cuh"

namespace cg = cooperative_groups;

namespace hpx {
namespace {

constexpr int LB = kGridBlock;  // l values per block

// This lane's columns of the lambda table: rows of the two 32-pair groups.
struct Rows2 {
  const float *ta = nullptr, *tb = nullptr;
  int lsa = INT_MAX, lsb = INT_MAX;
  __device__ __forceinline__ void init(const LamTab<float>& t, int m, int grp, int lane) {
    const long long e = (long long)m * t.ngroup + 2 * grp;
    if (2 * grp < t.ngroup) {
      lsa = t.lstart[e];
      ta = t.tab + t.off[e] + lane;
    }
    if (2 * grp + 1 < t.ngroup) {
      lsb = t.lstart[e + 1];
      tb = t.tab + t.off[e + 1] + lane;
    }
  }
  __device__ __forceinline__ float a(int l, int lmax) const {
    return (l >= lsa && l <= lmax) ? __ldcs(ta + (long long)(l - lsa) * 32) : 0.f;
  }
  __device__ __forceinline__ float b(int l, int lmax) const {
    return (l >= lsb && l <= lmax) ? __ldcs(tb + (long long)(l - lsb) * 32) : 0.f;
  }
};

__device__ __forceinline__ float4 dup(float2 c) { return make_float4(c.x, c.x, c.y, c.y); }
__device__ __forceinline__ float2 coef_at(const float2* __restrict__ c, int l, int lmax) {
  return l <= lmax ? c[l] : make_float2(0.f, 0.f);
}

// ---------------------------------------------------------------------------
// analysis
// ---------------------------------------------------------------------------
// One cluster per m; a warp takes 64 consecutive ring pairs, groups dealt
// round-robin over the cluster's CTAs (each holds polar and equatorial chains
// alike).  Per block of 32 l a warp writes its chains' mu into its tile --
// [chain][even l, odd l], rows of 36 floats: no bank conflicts either way --
// and contracts them with the chains' S (even l - m) and A (odd) ring
// coefficients: a lane sums 8 l of one parity x CT components over every KS-th
// chain, four 16-byte loads for 64 FMAs at 8 channels or more.  The lanes'
// sums are added over the warp's own mu rows.
//
// The sums over warps and CTAs are two more warps' work: nothing else waits for
// them.  With CTA-wide and cluster barriers at every block the warps spent 61%
// of their cycles at them: a warp in the general phase takes twice a grid
// block's time, there nearly always is one, and the sums' way through
// distributed shared memory and the stores was on every block's path.
//   compute -> sum warp: a block's sums in one of two slots; mbarriers
//     full[slot] (an arrival a warp) and empty[slot];
//   sum warp: adds the CTA's slots and sends the slice of l that CTA r owns to
//     r's inbox (st.async, which also completes r's in[place]), one of four
//     places; credit[place] (an arrival from every owner) frees it;
//   output warp: adds the cluster's slices of this CTA's l and writes alm.
// Every wait is bounded in time.  Deterministic order.  A sum or output warp whose
// wait has expired stops there: it sends nothing it has no credit for and gives no
// more credit, so that what can still be on its way to a CTA was sent before the
// final cluster barrier; a CTA that did not take it stays until it has landed.
//
// Four compute warps a CTA (256 chains; eight at Nside 2048, where clusters of
// more than eight CTAs would be needed).
template <int CP> struct ATile {
  static constexpr int C2N = 2 * CP;
  static constexpr int CT = C2N >= 16 ? 8 : C2N >= 4 ? 4 : 2;  // components a lane
  static constexpr int POS = 4 * (C2N / CT);                   // parities x 2 l halves x component groups
  static constexpr int KS = 32 / POS;                          // chains taken at a time
  static constexpr int MS = LB + 4;                            // floats of a mu row
  static constexpr int NOUT = LB * C2N;                        // sums of a block
  static constexpr int PS = NOUT + 4;                          // floats of one set of partial sums
  static constexpr int WARP = 64 * (2 * C2N + MS) + 2 * NOUT + 8 * LB;  // floats of a warp: G, mu, slots, c_l
  static_assert(KS * PS <= 64 * MS, "partial sums fit the warp's mu rows");
};

constexpr int kInbox = 4;  // places of the inbox

template <int CP> size_t analysis_smem(int warps) {
  using A = ATile<CP>;
  return 128 + sizeof(float) * ((size_t)warps * A::WARP + kInbox * A::NOUT);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t peer_addr(const void* p, int rank) {  // the same variable in another CTA
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_peer(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Waits for the phase of `bar` with this parity, at most 1 s, and not at all
// once a wait of this thread has expired (`late`).
__device__ __forceinline__ void mbar_wait(uint64_t* bar, uint32_t parity, bool& late) {
  if (late || mbar_test(bar, parity)) return;
  const unsigned long long t0 = global_ns();
  for (unsigned i = 1; i < (1u << 31); ++i) {
    if (mbar_test(bar, parity)) return;
    if ((i & 63u) == 0 && global_ns() - t0 > 1000000000ull) break;
  }
  late = true;
}

// The same by a whole warp, which gives up together.
__device__ __forceinline__ void mbar_wait_warp(uint64_t* bar, uint32_t parity, bool& late) {
  if (late || __all_sync(0xffffffffu, mbar_test(bar, parity))) return;
  const unsigned long long t0 = global_ns();
  for (unsigned i = 1; i < (1u << 31); ++i) {
    if (__all_sync(0xffffffffu, mbar_test(bar, parity))) return;
    if ((i & 63u) == 0 && __any_sync(0xffffffffu, global_ns() - t0 > 1000000000ull)) break;
  }
  late = true;
}

template <int CT> __device__ __forceinline__ void load_vec(float (&v)[CT], const float* src) {
  if constexpr (CT % 4 == 0) {
#pragma unroll
    for (int c = 0; c < CT; c += 4) {
      const float4 q = *reinterpret_cast<const float4*>(src + c);
      v[c] = q.x, v[c + 1] = q.y, v[c + 2] = q.z, v[c + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int c = 0; c < CT; c += 2) {
      const float2 q = *reinterpret_cast<const float2*>(src + c);
      v[c] = q.x, v[c + 1] = q.y;
    }
  }
}
template <int CT> __device__ __forceinline__ void store_vec(float* dst, const float (&v)[CT]) {
  if constexpr (CT >= 4) {
#pragma unroll
    for (int c = 0; c < CT; c += 4)
      *reinterpret_cast<float4*>(dst + c) = make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
  } else {
    *reinterpret_cast<float2*>(dst) = make_float2(v[0], v[1]);
  }
}

// (Two channels without a table: 96 registers are asked for, since 64, which the
// compiler may choose instead, spill: Nside 128 / lmax 383 60 -> 70 us, Nside 512 / lmax
// 1024 0.63 -> 0.65 ms.)
template <int CP, bool TAB>
__global__ void __launch_bounds__(320, (CP == 2 && !TAB ? 2 : 0))
k_legendre_analysis_f32(const float2* __restrict__ spec, float2* __restrict__ alm, const RingInfo* __restrict__ rings,
                        const float2* __restrict__ etab, const float2* __restrict__ coef_cf,
                        const float2* __restrict__ coef_pp, const int* __restrict__ lc_tab,
                        const float4* __restrict__ start, const float2* __restrict__ zf,
                        const int* __restrict__ lgrid, int ngrid, int lmax, int npair, int nring, long long nspec, long long nalm, int b0, int nb, int use_w,
                        const LamTab<float> tb, float mfac, int* __restrict__ status, int withhold) {
  using A = ATile<CP>;
  constexpr int C2N = A::C2N, CT = A::CT, KS = A::KS, MS = A::MS, PS = A::PS, NOUT = A::NOUT;
  cg::cluster_group cluster = cg::this_cluster();
  const int crank = (int)cluster.block_rank(), csize = (int)cluster.num_blocks();
  const int nwarp = (blockDim.x >> 5) - 2;  // compute warps, at most 8
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int m = blockIdx.y;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint64_t* full = reinterpret_cast<uint64_t*>(smem_raw);  // [2] a block's sums of all compute warps
  uint64_t* empty = full + 2;                              // [2] ... have been taken
  uint64_t* in = empty + 2;                                // [kInbox] the cluster's slices have arrived
  uint64_t* credit = in + kInbox;                          // [kInbox] every owner has taken its slice
  float* inbox = reinterpret_cast<float*>(smem_raw + 128); // [kInbox][csize][NOUT / csize]
  float* wbase = inbox + kInbox * NOUT;                    // per compute warp: G, mu rows, slots, c_l
  auto slot_of = [&](int w, int s) { return wbase + (size_t)w * A::WARP + 64 * (2 * C2N + MS) + s * NOUT; };

  if (t == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(full + s, nwarp);
      mbar_init(empty + s, 1);
    }
    for (int s = 0; s < kInbox; ++s) {
      mbar_init(in + s, csize > 1 ? 1 : 32);
      mbar_init(credit + s, csize);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  cluster.sync();

  const long long base = alm_base(lmax, m);
  const int nblk = (lmax - m) / LB + 1;
  bool late = false;
  if (warp < nwarp) {
    // ---- recurrence and contraction
    const int grp = warp * csize + crank;
    float* sG = wbase + (size_t)warp * A::WARP;  // [64][S, A: C2N]
    float* myMu = sG + 64 * 2 * C2N;             // [64][MS]
    float4* sCz = reinterpret_cast<float4*>(slot_of(warp, 2));  // [2][LB] c_l as (hi, hi, lo, lo)
    Chains2<1> ch;
    ch.init(zf, lc_tab, start, lgrid, ngrid, npair, lmax, m, grp, lane);
    Rows2 rows;
    if constexpr (TAB) rows.init(tb, m, grp, lane);
    // G of both chains: a ring's bin and phase (times its weight) once, then all
    // channels' loads in flight (channel by channel, with the bin's two integer
    // divisions each time, this took a third of the kernel at Nside 512)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int p = grp * 64 + 32 * h + lane;
      const bool on = p < npair && (h ? ch.lcb : ch.lca) != INT_MAX;
      const bool mirror = on && p < npair - 1;  // the equator ring has none
      const float2 *xn = spec, *xs = spec;
      float2 en = make_float2(0.f, 0.f), es = en;
      bool conj = false;
      if (on) {
        const RingInfo R = rings[p];
        const unsigned N = (unsigned)R.nphi, k = (unsigned)m % N, ip = ((unsigned)R.sigma * (unsigned)m) % (2u * N);
        conj = k > (N >> 1);
        const long long at = (long long)b0 * nspec + (conj ? N - k : k);
        xn += at + R.specoff;
        en = cscale(etab[R.etab + ip], use_w ? (float)R.w : 1.f);
        if (mirror) {  // the same length, shift and table
          const RingInfo& S = rings[nring - 1 - p];
          xs += at + S.specoff;
          es = cscale(etab[R.etab + ip], use_w ? (float)S.w : 1.f);
        }
      }
      float2 vn[CP], vs[CP];
#pragma unroll
      for (int c = 0; c < CP; ++c) {
        vn[c] = vs[c] = make_float2(0.f, 0.f);
        if (on && c < nb) vn[c] = xn[c * nspec];
        if (mirror && c < nb) vs[c] = xs[c * nspec];
      }
      float* g = sG + (size_t)(32 * h + lane) * 2 * C2N;
#pragma unroll
      for (int c = 0; c < CP; ++c) {
        const float2 gn = cmul(conj ? cconj(vn[c]) : vn[c], en), gs = cmul(conj ? cconj(vs[c]) : vs[c], es);
        *reinterpret_cast<float2*>(g + 2 * c) = cadd(gn, gs);
        *reinterpret_cast<float2*>(g + C2N + 2 * c) = csub(gn, gs);
      }
    }
    // until its first chain starts the warp's sums are zero
    for (int i = lane; i < 2 * NOUT; i += 32) slot_of(warp, 0)[i] = 0.f;
    const float2* cl = coef_cf + base;
    sCz[lane] = dup(coef_at(cl, m + lane, lmax));
    float nxa[TAB ? LB : 1], nxb[TAB ? LB : 1];  // TAB: the next block's rows, loaded a block ahead
    if constexpr (TAB) {
#pragma unroll
      for (int i = 0; i < LB; ++i) {
        nxa[i] = rows.a(m + i, lmax);
        nxb[i] = rows.b(m + i, lmax);
      }
    }
    __syncwarp();
    const int pos = lane % A::POS, ks = lane / A::POS;
    const int par = pos & 1, lh = (pos >> 1) & 1, c0 = (pos >> 2) * CT;
    for (int b = 0; b < nblk; ++b) {
      const int lb0 = m + b * LB, s = b & 1;
      const float4* cz = sCz + s * LB;
      const float2 cn = coef_at(cl, lb0 + LB + lane, lmax);
      const bool active = ch.lmin < lb0 + LB;
      if (active) {
        // --- this block's mu: even l at 0 .. 15 of a chain's row, odd l at 16 .. 31
        float *ra = myMu + lane * MS, *rb = ra + 32 * MS;
        auto put8 = [&](int i8, const float (&va)[8], const float (&vb)[8]) {
          const int h = i8 >> 1;
          *reinterpret_cast<float4*>(ra + h) = make_float4(va[0], va[2], va[4], va[6]);
          *reinterpret_cast<float4*>(ra + 16 + h) = make_float4(va[1], va[3], va[5], va[7]);
          *reinterpret_cast<float4*>(rb + h) = make_float4(vb[0], vb[2], vb[4], vb[6]);
          *reinterpret_cast<float4*>(rb + 16 + h) = make_float4(vb[1], vb[3], vb[5], vb[7]);
        };
        if constexpr (TAB) {
#pragma unroll
          for (int i8 = 0; i8 < LB; i8 += 8) {
            float va[8], vb[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              va[u] = nxa[i8 + u];
              vb[u] = nxb[i8 + u];
            }
            put8(i8, va, vb);
          }
        } else {
#pragma unroll 1
          for (int i8 = 0; i8 < LB; i8 += 8) {
            float va[8], vb[8];
            ch.steps8(cz + i8, lb0 + i8, va, vb);
            put8(i8, va, vb);
          }
        }
      }
      if constexpr (TAB) {
#pragma unroll
        for (int i = 0; i < LB; ++i) {
          nxa[i] = rows.a(lb0 + LB + i, lmax);
          nxb[i] = rows.b(lb0 + LB + i, lmax);
        }
      }
      if (active) {
        __syncwarp();
        // --- contraction over the warp's 64 chains
        float acc[8][CT];
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int c = 0; c < CT; ++c) acc[a][c] = 0.f;
        const float* mp = myMu + ks * MS + par * 16 + lh * 8;
        const float* gp = sG + ks * 2 * C2N + par * C2N + c0;
#pragma unroll 2
        for (int j = 0; j < 64; j += KS) {
          float mv[8], gv[CT];
          load_vec<8>(mv, mp);
          load_vec<CT>(gv, gp);
#pragma unroll
          for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int c = 0; c < CT; ++c) acc[a][c] = fmaf(mv[a], gv[c], acc[a][c]);
          mp += KS * MS;
          gp += KS * 2 * C2N;
        }
        __syncwarp();
        // the lanes' sums over the warp's mu rows: [ks][l][component], 4 floats
        // further on for the upper half of l (no bank conflicts)
        float* w = myMu + ks * PS + lh * 4 + c0;
#pragma unroll
        for (int a = 0; a < 8; ++a) store_vec<CT>(w + (2 * (lh * 8 + a) + par) * C2N, acc[a]);
      }
      sCz[(s ^ 1) * LB + lane] = dup(cn);
      __syncwarp();
      if (b >= 2) mbar_wait(empty + s, (uint32_t)((b - 2) >> 1) & 1u, late);
      if (active) {
        float* slot = slot_of(warp, s);
        for (int o = 4 * lane; o < NOUT; o += 128) {
          const float* src = myMu + o + (o / C2N >= LB / 2 ? 4 : 0);
          float4 v = *reinterpret_cast<const float4*>(src);
#pragma unroll
          for (int k = 1; k < KS; ++k) {
            const float4 u = *reinterpret_cast<const float4*>(src + k * PS);
            v.x += u.x, v.y += u.y, v.z += u.z, v.w += u.w;
          }
          *reinterpret_cast<float4*>(slot + o) = v;
        }
      }
      __syncwarp();
      if (lane == 0 && !withhold) mbar_arrive(full + s);
    }
  } else if (warp == nwarp) {
    // ---- sums over the warps, sent to their owners: CTA r owns l's r NOUT / csize floats of a block
    const int slice = NOUT / csize;
    for (int b = 0; b < nblk; ++b) {
      const int s = b & 1, q = b % kInbox;
      mbar_wait_warp(full + s, (uint32_t)(b >> 1) & 1u, late);
      if (b >= kInbox) mbar_wait_warp(credit + q, (uint32_t)(b / kInbox - 1) & 1u, late);
      if (late) break;
      for (int o = 4 * lane; o < NOUT; o += 128) {
        float4 u[8];
#pragma unroll
        for (int w = 0; w < 8; ++w) {
          u[w] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (w < nwarp) u[w] = *reinterpret_cast<const float4*>(slot_of(w, s) + o);
        }
        float4 v = u[0];
#pragma unroll
        for (int w = 1; w < 8; ++w) v.x += u[w].x, v.y += u[w].y, v.z += u[w].z, v.w += u[w].w;
        const int owner = o / slice;
        float* dst = inbox + q * NOUT + crank * slice + o % slice;
        if (csize > 1)
          asm volatile(
              "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                  peer_addr(dst, owner)),
              "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(peer_addr(in + q, owner))
              : "memory");
        else
          *reinterpret_cast<float4*>(dst) = v;
      }
      if (csize == 1) mbar_arrive(in + q);  // every lane
      __syncwarp();
      if (lane == 0) mbar_arrive(empty + s);
    }
  } else {
    // ---- sums over the cluster, and the output: this CTA's l of a block from crank nl on
    const int nl = LB / csize, slice = NOUT / csize, li = lane % nl;
    const float mf = m > 0 ? mfac : 1.f;  // a power of two
    for (int b = 0; b < nblk; ++b) {
      const int q = b % kInbox, l = m + b * LB + crank * nl + li;
      const float2 P = cscale(coef_at(coef_pp + base, l, lmax), mf);
      if (csize > 1 && lane == 0) mbar_expect(in + q, NOUT * sizeof(float));
      mbar_wait_warp(in + q, (uint32_t)(b / kInbox) & 1u, late);
      if (late) break;
      const float* src = inbox + q * NOUT + li * C2N;
      float2 v[CP];
#pragma unroll
      for (int i = 0; i < CP; ++i) {  // channels lane / nl + i csize (32 / nl = csize)
        const int bb = lane / nl + i * csize;
        v[i] = make_float2(0.f, 0.f);
        if (bb < CP)
          for (int r = 0; r < csize; ++r) v[i] = cadd(v[i], *reinterpret_cast<const float2*>(src + r * slice + 2 * bb));
      }
      __syncwarp();
      // before the stores, which its release would wait for
      if (lane < csize) mbar_arrive_peer(peer_addr(credit + q, lane));
#pragma unroll
      for (int i = 0; i < CP; ++i) {
        const int bb = lane / nl + i * csize;
        if (bb < nb && l <= lmax)
          alm[(long long)(b0 + bb) * nalm + base + l] =
              make_float2(fmaf(v[i].x, P.x, v[i].x * P.y), fmaf(v[i].y, P.x, v[i].y * P.y));
      }
    }
  }
  if (late) atomicExch(status, (int)HPX_ERR_TIMEOUT);
  cluster.sync();  // peers may still send to this CTA
  if (late && warp == nwarp + 1) {  // slices not taken: 20 us, a store's way to another SM takes one or two
    const unsigned long long t0 = global_ns();
    for (unsigned i = 0; i < (1u << 20) && global_ns() - t0 < 20000ull; ++i) {
    }
  }
}

// ---------------------------------------------------------------------------
// synthesis
// ---------------------------------------------------------------------------
// A lane sums E_m (even l - m) and O_m (odd) of its two chains in registers;
// F_m(y) = E + O on the northern ring and F_m(y') = E - O on its mirror
// (Eq. 24 before the ring transform).  The block's coefficients, times P_l, are
// broadcast from shared memory, one 16-byte load for 8 FMAs; the next block's
// are loaded into registers while a block is computed.  A CTA is one warp: its
// group's phase sets how long a block takes, and with several warps sharing
// the staged coefficients all of them waited for the slowest at each block's
// barrier (27% of the warps' cycles).
template <int CP, bool TAB>
__global__ void __launch_bounds__(32)
k_legendre_synthesis_f32(const float2* __restrict__ alm, float2* __restrict__ F, const float2* __restrict__ zf,
                         const float2* __restrict__ coef_cf, const float* __restrict__ coef_pf,
                         const int* __restrict__ lc_tab, const float4* __restrict__ start,
                         const int* __restrict__ lgrid, int ngrid, int lmax, int mmax, int npair, int nring,
                         long long nalm, int b0, int nb, const LamTab<float> tb, float mfac) {
  constexpr int C2N = 2 * CP;
  __shared__ __align__(16) float sA[2][LB][C2N];
  __shared__ __align__(16) float4 sCz[2][LB];
  const int m = blockIdx.y, lane = threadIdx.x, grp = blockIdx.x;
  Chains2<1> ch;
  ch.init(zf, lc_tab, start, lgrid, ngrid, npair, lmax, m, grp, lane);
  Rows2 rows;
  if constexpr (TAB) rows.init(tb, m, grp, lane);
  float e0[C2N], e1[C2N], o0[C2N], o1[C2N];  // E and O of chain p, of chain p + 32
#pragma unroll
  for (int c = 0; c < C2N; ++c) e0[c] = e1[c] = o0[c] = o1[c] = 0.f;
  const long long base = alm_base(lmax, m);
  const float mf = m > 0 ? mfac : 1.f;
  // this lane's l of a block, FQ channels at a time: fetched into registers,
  // put into shared memory once the 8 steps behind the loads are done
  constexpr int FQ = CP == 6 ? 2 : CP >= 4 ? CP / 4 : CP;
  static_assert(CP % FQ == 0 && CP / FQ <= LB / 8, "channels fetched a block ahead");
  float2 an[FQ], cn;
  auto fetch = [&](int lb, int q) {
    const int l = lb + lane;
    const bool in = l <= lmax;
    const float s = in ? coef_pf[base + l] * mf : 0.f;
#pragma unroll
    for (int i = 0; i < FQ; ++i) {
      const int bb = q * FQ + i;
      an[i] = make_float2(0.f, 0.f);
      if (in && bb < nb) {
        const float2 a = alm[(long long)(b0 + bb) * nalm + base + l];
        an[i] = make_float2(s * a.x, m == 0 ? 0.f : s * a.y);  // only Re a_l0 enters
      }
    }
    if (q == 0) cn = coef_at(coef_cf + base, l, lmax);
  };
  auto put = [&](int buf, int q) {
#pragma unroll
    for (int i = 0; i < FQ; ++i) *reinterpret_cast<float2*>(&sA[buf][lane][2 * (q * FQ + i)]) = an[i];
    if (q == 0) sCz[buf][lane] = dup(cn);
  };
  if (ch.lmin <= lmax) {
    int lb0 = m + ((ch.lmin - m) / LB) * LB, buf = 0;
    for (int q = 0; q < CP / FQ; ++q) {
      fetch(lb0, q);
      put(0, q);
    }
    __syncwarp();
    float nxa[TAB ? 8 : 1], nxb[TAB ? 8 : 1];
    if constexpr (TAB) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        nxa[u] = rows.a(lb0 + u, lmax);
        nxb[u] = rows.b(lb0 + u, lmax);
      }
    }
    for (; lb0 <= lmax; lb0 += LB, buf ^= 1) {
#pragma unroll 1
      for (int i8 = 0; i8 < LB; i8 += 8) {
        const bool next = lb0 + LB <= lmax && i8 / 8 < CP / FQ;
        if (next) fetch(lb0 + LB, i8 / 8);
        float va[8], vb[8];
        if constexpr (TAB) {
          // this group of 8 was loaded a group ago; the next one's loads go out
          // (16 channels leave no registers for that)
          constexpr bool AHEAD = CP < 16;
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            va[u] = AHEAD ? nxa[u] : rows.a(lb0 + i8 + u, lmax);
            vb[u] = AHEAD ? nxb[u] : rows.b(lb0 + i8 + u, lmax);
          }
          if constexpr (AHEAD) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              nxa[u] = rows.a(lb0 + i8 + 8 + u, lmax);
              nxb[u] = rows.b(lb0 + i8 + 8 + u, lmax);
            }
          }
        } else {
          ch.steps8(&sCz[buf][i8], lb0 + i8, va, vb);
        }
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
          float av[C2N];
          load_vec<C2N>(av, sA[buf][i8 + u]);
#pragma unroll
          for (int c = 0; c < C2N; ++c) {
            e0[c] = fmaf(va[u], av[c], e0[c]);
            e1[c] = fmaf(vb[u], av[c], e1[c]);
          }
          load_vec<C2N>(av, sA[buf][i8 + u + 1]);
#pragma unroll
          for (int c = 0; c < C2N; ++c) {
            o0[c] = fmaf(va[u + 1], av[c], o0[c]);
            o1[c] = fmaf(vb[u + 1], av[c], o1[c]);
          }
        }
        if (next) put(buf ^ 1, i8 / 8);
      }
      __syncwarp();
    }
  }
  auto write = [&](int p, const float (&e)[C2N], const float (&o)[C2N]) {
    if (p >= npair) return;
    const int ys = p == npair - 1 ? -1 : nring - 1 - p;
#pragma unroll
    for (int bb = 0; bb < CP; ++bb) {
      if (bb < nb) {
        const float2 ev = make_float2(e[2 * bb], e[2 * bb + 1]), ov = make_float2(o[2 * bb], o[2 * bb + 1]);
        F[((long long)(b0 + bb) * nring + p) * (mmax + 1) + m] = cadd(ev, ov);
        if (ys >= 0) F[((long long)(b0 + bb) * nring + ys) * (mmax + 1) + m] = csub(ev, ov);
      }
    }
  };
  write(grp * 64 + lane, e0, o0);
  write(grp * 64 + 32 + lane, e1, o1);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// Compute warps a CTA and CTAs a cluster of the analysis (npair is a power of two).
void analysis_shape(int npair, int* warps, int* csize) {
  const int groups = (npair + 63) / 64;
  *warps = groups <= 4 ? groups : groups <= 32 ? 4 : 8;
  *csize = (groups + *warps - 1) / *warps;
}

template <int CP, bool TAB>
cudaError_t launch_analysis_cp(const hpx_plan_s* p, float* alm, bool use_w, double mfac, cudaStream_t s, int* nlaunch) {
  int warps, csize;
  analysis_shape(p->npair, &warps, &csize);
  cudaError_t e = allow_max_smem(k_legendre_analysis_f32<CP, TAB>);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(csize, p->mmax + 1, 1);
  cfg.blockDim = dim3(32 * (warps + 2), 1, 1);
  cfg.dynamicSmemBytes = analysis_smem<CP>(warps);
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
    e = cudaLaunchKernelEx(&cfg, k_legendre_analysis_f32<CP, TAB>, (const float2*)p->d_spec, (float2*)alm,
                           (const RingInfo*)p->d_ring, (const float2*)p->d_etab, (const float2*)p->d_coef_cf,
                           (const float2*)p->d_coef_pp, (const int*)p->d_lc, (const float4*)p->d_start,
                           (const float2*)p->d_zf, (const int*)p->d_lgrid, p->ngrid, p->lmax, p->npair, p->nring,
                           p->nspec, p->nalm, b0, nb, use_w ? 1 : 0, lam_tab<float>(p), (float)mfac, p->d_status, p->test_withhold);
    if (e != cudaSuccess) return e;
    ++*nlaunch;
  }
  return cudaGetLastError();
}

template <int CP>
cudaError_t launch_analysis_sel(const hpx_plan_s* p, float* alm, bool use_w, double mfac, cudaStream_t s, int* nlaunch) {
  return p->d_tab ? launch_analysis_cp<CP, true>(p, alm, use_w, mfac, s, nlaunch)
                  : launch_analysis_cp<CP, false>(p, alm, use_w, mfac, s, nlaunch);
}

template <int CP, bool TAB>
cudaError_t launch_synthesis_cp(const hpx_plan_s* p, const float* alm, double mfac, cudaStream_t s, int* nlaunch) {
  const dim3 grid((p->npair + 63) / 64, p->mmax + 1);
  for (int b0 = 0; b0 < p->nbatch; b0 += CP) {
    const int nb = (p->nbatch - b0) < CP ? (p->nbatch - b0) : CP;
    k_legendre_synthesis_f32<CP, TAB><<<grid, 32, 0, s>>>(
        (const float2*)alm, (float2*)p->d_F, p->d_zf, p->d_coef_cf, p->d_coef_pf, p->d_lc, p->d_start, p->d_lgrid,
        p->ngrid, p->lmax, p->mmax, p->npair, p->nring, p->nalm, b0, nb, lam_tab<float>(p), (float)mfac);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    ++*nlaunch;
  }
  return cudaSuccess;
}

template <int CP>
cudaError_t launch_synthesis_sel(const hpx_plan_s* p, const float* alm, double mfac, cudaStream_t s, int* nlaunch) {
  return p->d_tab ? launch_synthesis_cp<CP, true>(p, alm, mfac, s, nlaunch)
                  : launch_synthesis_cp<CP, false>(p, alm, mfac, s, nlaunch);
}

// Channels a launch (each launch reruns the recurrence).
int channels(const hpx_plan_s* p, int most) {
  int cp = 1;
  while (cp < p->nbatch && cp < most) cp *= 2;
  return cp;
}

}  // namespace

template <>
cudaError_t launch_analysis<float>(const hpx_plan_s* p, float* alm, bool use_w, double mfac, cudaStream_t s,
                                   int* nlaunch) {
  switch (channels(p, 8)) {
    case 1: return launch_analysis_sel<1>(p, alm, use_w, mfac, s, nlaunch);
    case 2: return launch_analysis_sel<2>(p, alm, use_w, mfac, s, nlaunch);
    case 4: return launch_analysis_sel<4>(p, alm, use_w, mfac, s, nlaunch);
    default: return launch_analysis_sel<8>(p, alm, use_w, mfac, s, nlaunch);
  }
}

template <>
cudaError_t launch_synthesis<float>(const hpx_plan_s* p, const float* alm, double mfac, cudaStream_t s,
                                    int* nlaunch) {
  // as many launches as 16 channels at most need, of the narrowest width that
  // holds an equal share: the FP32 pipe works for channels that are not there too
  // (Nside 256, lmax 700: 3 channels 0.127 -> 0.109 ms, 6 0.186 -> 0.160, 12 from the
  // table 0.371 -> 0.213)
  const int k = (p->nbatch + 15) / 16, share = (p->nbatch + k - 1) / k;
  if (share <= 1) return launch_synthesis_sel<1>(p, alm, mfac, s, nlaunch);
  if (share <= 2) return launch_synthesis_sel<2>(p, alm, mfac, s, nlaunch);
  if (share <= 3) return launch_synthesis_sel<3>(p, alm, mfac, s, nlaunch);
  if (share <= 4) return launch_synthesis_sel<4>(p, alm, mfac, s, nlaunch);
  if (share <= 6) return launch_synthesis_sel<6>(p, alm, mfac, s, nlaunch);
  if (share <= 8) return launch_synthesis_sel<8>(p, alm, mfac, s, nlaunch);
  if (share <= 12) return launch_synthesis_sel<12>(p, alm, mfac, s, nlaunch);
  return launch_synthesis_sel<16>(p, alm, mfac, s, nlaunch);
}

}  // namespace hpx
