// Tensor-core Legendre stages whose lambda tiles are generated in shared
// memory (Sec. III-D Eq. 14-16, Eq. 24-27): the products of hpx_tc.cu without a
// table behind them.  Generator warps step the recurrence chains, split the
// values into 16-bit parts and write them straight into the swizzled operand
// tile that tcgen05.mma reads; nothing of lambda goes through global memory.
//
//   k_gen_analysis   D[l][n] = sum_p Lambda[l][p] Gt[n][p], a CTA all l of one m
//   k_gen_synthesis  D[p][n] = sum_l Lambda[l][p] At[n][l], a CTA 128 pairs of
//                    four m
//
// Used by the streamed-lambda plans of the split-product modes (all syntheses, and
// analyses of up to 96 or 160 channels, staged_analysis_pays; two 16-bit
// parts, three products: the same values, products and sums as the table
// tiles, so the same bits), and by the analysis of the FP32 plans without
// tensor-core tables, in three BF16 parts and six products: 3 x 8 significant
// bits hold a float exactly -- each channel's spectra are scaled by a power of two
// (chan_scale), so that the third part of a weak channel is no BF16 subnormal --
// and the products left out are below 2^-26 of a term.
//
// What bounds them is the FP32 pipe that steps the chains, 12 operations a
// value (the filled-table version moved 8 bytes a value through HBM and
// stepped 22): the products take a tenth to a third of the time behind it.
#include <cuda.h>

#include <climits>

#include "hpx_tcgen05.cuh"

namespace hpx {
namespace {

// Warps: the first 4 (analysis) or 8 (synthesis) drain, the next generate, the
// last two copy operands and issue products.
constexpr int kTileBytes = 128 * 128;  // one part of a lambda tile: 128 rows of 64 values

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
          taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
      "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Two floats as a pair of 16-bit values (a in the low half), and the pair's
// remainders.
template <typename E> struct Pair16;
template <> struct Pair16<__half> {
  static __device__ __forceinline__ uint32_t round(float& a, float& b) {
    const __half2 h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    a = __fsub_rn(a, f.x);
    b = __fsub_rn(b, f.y);
    return *reinterpret_cast<const uint32_t*>(&h);
  }
};
template <> struct Pair16<__nv_bfloat16> {
  static __device__ __forceinline__ uint32_t round(float& a, float& b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    const uint32_t u = *reinterpret_cast<const uint32_t*>(&h);
    a = __fsub_rn(a, __uint_as_float(u << 16));
    b = __fsub_rn(b, __uint_as_float(u & 0xFFFF0000u));
    return u;
  }
};

// Shared-memory matrix descriptor of an operand whose 128-byte rows run along
// M, in the 128-byte swizzle: 8-row (K) groups 1024 bytes apart, the second 64
// of M half a tile further on.
__device__ __forceinline__ uint64_t sdesc_mn128(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)(kTileBytes / 2 >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// Products of half h of a K block (64 values along K, four steps of 16; the
// halves become ready apart): A parts at aL + q kTileBytes, B parts at aB + q kB.
// The tensor cores add into the accumulator with truncation, so the fewer
// additions at the sum's own magnitude the better: small terms first, or in
// columns of their own.
// MN: A's rows run along M (a tile row is one K index), else along K as B's.
template <int NN, int PARTS, bool MN>
__device__ __forceinline__ void issue_half(uint32_t d, uint32_t aL, uint32_t aB, uint32_t fmt, int h) {
  constexpr uint32_t kB = NN * 128;
  auto idesc = [&](int n) {  // D f32, M = 128
    return (1u << 4) | (fmt << 7) | (fmt << 10) | (MN ? 1u << 15 : 0u) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
  };
  auto mma = [&](int n, int col, int pa, int pb, int j, bool acc) {
    const uint32_t ap = aL + pa * kTileBytes, kb = 64u * h + 32u * j;  // bytes along B's K
    umma_f16(d + col, MN ? sdesc_mn128(ap + 64u * kb) : sdesc_sw128(ap + kb), sdesc_sw128(aB + pb * kB + kb), idesc(n),
             acc ? 1u : 0u);
  };
  const bool more = h > 0;  // the accumulator holds the first half
  if constexpr (PARTS == 2) {
    // remainder of A first, then A against both parts of B (A read once)
    mma(NN, 0, 1, 0, 0, more);
    mma(NN, 0, 1, 0, 1, true);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint32_t kb = 64u * h + 32u * j;
      umma_f16_pair(d, MN ? sdesc_mn128(aL + 64u * kb) : sdesc_sw128(aL + kb), sdesc_sw128(aB + kB + kb),
                    sdesc_sw128(aB + kb), idesc(NN), 1u);
    }
  } else {
    // the B parts lie one after another, so one product takes A part q against
    // B parts 0 .. 2 - q; column regions 0 and 3 (the halves' terms of order
    // 1, two additions each), 1 and 2 (2^-8 and 2^-16)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (h == 0) {
        mma(3 * NN, 0, 0, 0, j, j > 0);
      } else {
        mma(NN, 3 * NN, 0, 0, j, j > 0);
        mma(2 * NN, NN, 0, 1, j, true);
      }
      mma(2 * NN, NN, 1, 0, j, true);
      mma(NN, 2 * NN, 2, 0, j, true);
    }
  }
}

// ---------------------------------------------------------------------------
// analysis
// ---------------------------------------------------------------------------
template <int NN, int PARTS> struct GenShape {
  static constexpr int kB = PARTS * NN * 128;      // operand tile bytes, all parts
  static constexpr int kStage = PARTS * kTileBytes;
  // a pair of generator warps each
  static constexpr int kNStage = PARTS == 3 ? (NN >= 64 ? 3 : 4) : NN == 32 ? 6 : NN == 64 ? 5 : 4;
  static constexpr int kThreads = 32 * (6 + 2 * kNStage);
  static constexpr int kCoef = 2 * kNStage * 1024;  // c_l of a tile, per generator warp
  static constexpr int kFree = 227 * 1024 - 3072 - kCoef - kNStage * kStage;
  static constexpr int kNB = kFree / kB < 4 ? kFree / kB : 4;  // operand tiles in flight
  static constexpr int kBuf = PARTS == 3 ? 4 * NN : NN;  // accumulator columns of a block
  static constexpr int kAlloc = 2 * kBuf <= 32 ? 32 : 2 * kBuf <= 64 ? 64 : 2 * kBuf <= 128 ? 128 : 2 * kBuf <= 256 ? 256 : 512;
  static constexpr size_t kSmem = 1024 + (size_t)kNStage * kStage + (size_t)kNB * kB + kCoef + 1024;
  static_assert(kNB >= 1 && 2 * kBuf <= 512 && kSmem <= 227 * 1024, "shape");
};

struct GenArgs {
  const float2* coef_cf;
  const int* lc;
  const float4* start;
  const float2* zf;
  const int* lgrid;
  const int* gstart;  // [m][group] earliest start of each 64-pair group
  int ngrid;
  LamTab<float> tab;  // FP32 table plans: lambda from here instead of the recurrence
  float4* state;      // [CTA][npair] chains between tiles
  const float* coef_pf;
  const float2* coef_pp;
  unsigned* bmax;     // the channels' largest spectrum components; three parts: left zero
  const float* binv;  // three parts: the inverse channel scales
  float sfac, lscale, mfac;
  float2* out;  // alm [b][nalm]
  int lmax, npair;
  long long nalm;
  int nb;
  uint32_t fmt;
  int* status;
  int nm, ncg;
  long long cg_rows;
  int withhold;
};

// One chain of a lane, 8 steps at a time; the state as in Chains2, scalar (an
// f32x2 FMA of three distinct register pairs takes three cycles, two scalar
// ones two and a half).  The products c z do not wait on the chain: two steps'
// are packed into one instruction each.
template <int S> struct Chain1 {
  static constexpr float kC = kGridC * S;
  GridState g;
  Df z;
  int lc, lg, m;
  int lmin, lmax_c;  // the warp's earliest and latest start
  // cz: per two steps (hi, hi, lo, lo) of c_l, c_{l+1}
  __device__ __forceinline__ void steps8(const float4* cz, int l, float (&v)[8]) {
    if (l + 8 <= lmin) {  // nothing has started
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = 0.f;
      return;
    }
    Df t[8];
    const F2 zh = pk2(z.hi, z.hi), zl = pk2(z.lo, z.lo);
#pragma unroll
    for (int u = 0; u < 8; u += 2) {  // df_mul(c, z) of both steps
      const float4 c = cz[u / 2];
      const F2 ch = pk2(c.x, c.y), cl = pk2(c.z, c.w), p = mul2(ch, zh);
      F2 e = fma2(ch, zh, neg2(p));
      e = fma2(ch, zl, e);
      e = fma2(cl, zh, e);
      unpk2(p, t[u].hi, t[u + 1].hi);
      unpk2(e, t[u].lo, t[u + 1].lo);
    }
    if (l >= lg) {
      if (l == lg) g = grid_enter(Df{g.s1, g.f1}, Df{g.s2, g.f2}, kC);
      else if (((l - m) & (kRegrid - 1)) == 0) regrid(g, kC);
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = grid_step(g, t[u], kC);
    } else if (lmax_c >= l) {
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = general_step<true>(g, t[u], l + u, lc);
    } else {
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = general_step<false>(g, t[u], l + u, lc);
    }
  }
};
// 8 consecutive l of a chain as 16-byte words of each part, kTileBytes apart
template <int PARTS, typename E>
__device__ __forceinline__ void put8(unsigned char* dst, float (&v)[8]) {
#pragma unroll
  for (int part = 0; part < PARTS; ++part) {
    uint32_t w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) w[u] = Pair16<E>::round(v[2 * u], v[2 * u + 1]);
    *reinterpret_cast<uint4*>(dst + part * kTileBytes) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}
// n coefficients c_l of a chain from l on, in Chain1's layout
__device__ __forceinline__ void stage_coefs(float4* cz, const float2* __restrict__ cl, int l, int n, int lmax, int lane) {
  for (int i = lane; i < n / 2; i += 32) {
    const float2 c0 = l + 2 * i <= lmax ? cl[l + 2 * i] : make_float2(0.f, 0.f);
    const float2 c1 = l + 2 * i + 1 <= lmax ? cl[l + 2 * i + 1] : make_float2(0.f, 0.f);
    cz[i] = make_float4(c0.x, c1.x, c0.y, c1.y);
  }
}

// A persistent CTA takes the (m, channel group) units blockIdx.x + i gridDim.x
// in turn (m ascending: the longest first).  Within one m it walks the tiles of
// 128 l, and in each the 64-pair groups that have started, in order: block =
// (tile, group).  Generator pair q = group mod kNStage owns stage q; its warps
// take the group's halves, a lane one chain, and keep the chains' states
// between tiles in global memory (16 bytes a chain every 128 steps, from L2).
// The tile is stored with l contiguous (a row a chain, M-major for the
// products), so that 8 steps of a chain leave as one 16-byte word; pair-major
// rows needed an exchange between lanes and four times the stores.
template <int NN, int PARTS, bool TAB, typename E>
__global__ void __launch_bounds__(GenShape<NN, PARTS>::kThreads, 1)
k_gen_analysis(const __grid_constant__ CUtensorMap tmB, const GenArgs a) {
  using SH = GenShape<NN, PARTS>;
  constexpr int NST = SH::kNStage, NB = SH::kNB, C2N = NN / 2, RB = PARTS * NN;
  constexpr int S = PARTS == 2 ? (int)kLamScale : 1;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* tiles = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* btile = tiles + NST * SH::kStage;
  float4* coefs = reinterpret_cast<float4*>(btile + NB * SH::kB);  // [warp][64]
  uint64_t* full = reinterpret_cast<uint64_t*>(reinterpret_cast<unsigned char*>(coefs) + SH::kCoef);
  uint64_t* empty = full + 2 * NST;  // a stage's halves apart
  uint64_t* bfull = empty + 2 * NST;
  uint64_t* bempty = bfull + NB;
  uint64_t* accf = bempty + NB;  // [2]
  uint64_t* acce = accf + 2;     // [2]
  uint64_t* done = acce + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* t0 = reinterpret_cast<int*>(tmem_slot + 2);  // [64] first tile of each group

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(SH::kAlloc));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (t == 32) {
    for (int s = 0; s < 2 * NST; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < NB; ++s) {
      mbar_init(&bfull[s], 1);
      mbar_init(&bempty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], 128);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  // three parts: the pack has read the maxima; the next ring transform finds zeros
  if (PARTS == 3 && blockIdx.x == 0)
    for (int b = t; b < a.nb; b += SH::kThreads) a.bmax[b] = 0u;
  unsigned kblk = 0;        // blocks so far (copies, products, drain)
  unsigned scount[NST] = {};  // products: blocks so far of each stage
  unsigned gcount = 0;      // generators: blocks so far of their stage
  bool alive = true;
  for (int unit = blockIdx.x; unit < a.nm * a.ncg; unit += gridDim.x) {
    const int m = unit / a.ncg, cgi = unit % a.ncg;
    const int b0 = cgi * (C2N / 2), nbl = min(C2N / 2, a.nb - b0);
    const int ntile = (a.lmax - m) / kTcTile + 1;
    if (t < a.ngrid) {
      const int gs = a.gstart[(long long)m * a.ngrid + t];
      t0[t] = gs <= a.lmax ? (gs - m) / kTcTile : INT_MAX;
    }
    __syncthreads();
    if (warp >= 4 && warp < 4 + 2 * NST) {
      // ---- generators
      const int gw = warp - 4, q = gw >> 1, h = gw & 1;
      float4* cz = coefs + gw * (kTcTile / 2);
      unsigned char* stage = tiles + q * SH::kStage;
      const float2* cl = a.coef_cf + alm_base(a.lmax, m);
      unsigned char* mine = stage + (32 * h + lane) * 128;  // this lane's row of both halves of M
      const uint32_t sw = (uint32_t)(lane & 7);
      for (int tile = 0; tile < ntile; ++tile) {
        const int l0 = m + kTcTile * tile;
        __syncwarp();
        if constexpr (!TAB) stage_coefs(cz, cl, l0, kTcTile, a.lmax, lane);
        __syncwarp();
        // a block's chain data (from L2) are loaded while the block before it
        // is generated
        auto first_from = [&](int g) {  // the next group of this pair that has started
          while (g < a.ngrid && tile < t0[g]) g += NST;
          return g;
        };
        struct Data {
          int lc, lg;
          float2 z;
          float4 st;
        };
        auto fetch = [&](int g) {
          Data d{INT_MAX, INT_MAX, make_float2(0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
          if (TAB || g >= a.ngrid) return d;
          const int p = 64 * g + 32 * h + lane;
          d.lg = a.lgrid[(long long)m * a.ngrid + g];
          if (p < a.npair) {
            d.lc = a.lc[(long long)m * a.npair + p];
            d.z = a.zf[p];
            d.st = tile > t0[g] ? a.state[(long long)blockIdx.x * a.npair + p] : a.start[(long long)m * a.npair + p];
          }
          return d;
        };
        int g = first_from(q);
        Data cur = fetch(g);
        while (g < a.ngrid) {
          const int gn = first_from(g + NST);
          const Data nxt = fetch(gn);
          const int p = 64 * g + 32 * h + lane;
          const bool on = p < a.npair;
          Chain1<S> ch;
          const float* row = nullptr;
          int ls = INT_MAX;
          if constexpr (TAB) {
            const int g2 = 2 * g + h;
            if (g2 < a.tab.ngroup) {
              const long long e = (long long)m * a.tab.ngroup + g2;
              ls = a.tab.lstart[e];
              row = a.tab.tab + a.tab.off[e] + lane;
            }
          } else {
            ch.m = m;
            ch.lc = cur.lc > a.lmax ? INT_MAX : cur.lc;
            ch.lg = grid_start(m, cur.lg);
            ch.z = Df{cur.z.x, cur.z.y};
            ch.lmin = __reduce_min_sync(0xffffffffu, ch.lc);
            ch.lmax_c = __reduce_max_sync(0xffffffffu, ch.lc);
            ch.g = tile > t0[g] ? GridState{cur.st.x, cur.st.y, cur.st.z, cur.st.w} : start_state(cur.st, (float)S);
          }
          if (alive && gcount > 0) alive = wait_phase(&empty[gw], (gcount - 1) & 1u, abort_flag, true);
          alive = __all_sync(0xffffffffu, alive);
          if (!alive) break;
          auto emit = [&](int i8, float (&v)[8]) {
            const uint32_t c = (uint32_t)i8 >> 3;  // 16-byte word of the 128 l
            put8<PARTS, E>(mine + (c >> 3) * (kTileBytes / 2) + (((c & 7) ^ sw) << 4), v);
          };
          if constexpr (TAB) {
            // 32 table rows in flight a lane
            float nx[4][8];
            auto rows8 = [&](int i8, float (&dst)[8]) {
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                const int l = l0 + i8 + u;
                dst[u] = l >= ls && l <= a.lmax ? __ldcs(row + (long long)(l - ls) * 32) : 0.f;
              }
            };
#pragma unroll
            for (int i = 0; i < 4; ++i) rows8(8 * i, nx[i]);
#pragma unroll 1
            for (int i32 = 0; i32 < kTcTile; i32 += 32)
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                emit(i32 + 8 * i, nx[i]);
                if (i32 + 32 < kTcTile) rows8(i32 + 32 + 8 * i, nx[i]);
              }
          } else {
#pragma unroll 1
            for (int i8 = 0; i8 < kTcTile; i8 += 8) {
              float v[8];
              ch.steps8(cz + i8 / 2, l0 + i8, v);
              emit(i8, v);
            }
          }
          if constexpr (!TAB) {
            if (on) a.state[(long long)blockIdx.x * a.npair + p] = make_float4(ch.g.s1, ch.g.f1, ch.g.s2, ch.g.f2);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(&full[gw]);
          ++gcount;
          g = gn;
          cur = nxt;
        }
        if (!alive) break;
      }
    } else if (warp == 4 + 2 * NST) {
      // ---- operand copies
      if (lane == 0 && !a.withhold) {
        const unsigned first = kblk;
        for (int tile = 0; tile < ntile && alive; ++tile)
          for (int g = 0; g < a.ngrid && alive; ++g) {
            if (tile < t0[g]) continue;
            const unsigned r = kblk % NB;
            if (kblk >= NB) alive = wait_phase(&bempty[r], (kblk / NB - 1) & 1u, abort_flag, true);
            if (!alive) break;
            mbar_expect_tx(&bfull[r], SH::kB);
            const int rb = (int)(((long long)m * a.ngrid + g) * RB + cgi * a.cg_rows);
#pragma unroll
            for (int part = 0; part < PARTS; ++part)
              tma_load_2d(btile + r * SH::kB + part * NN * 128, &tmB, 0, rb + part * NN, &bfull[r]);
            ++kblk;
          }
        // whatever was started completes before the CTA moves on
        for (unsigned k = kblk > NB ? kblk - NB : 0; k < kblk; ++k)
          if (k >= first) wait_phase(&bfull[k % NB], (k / NB) & 1u, abort_flag, false);
      }
    } else if (warp == 5 + 2 * NST) {
      // ---- products
      if (lane == 0) {
        bool started = false;
        for (int tile = 0; tile < ntile && alive; ++tile)
          for (int g = 0; g < a.ngrid; ++g) {
            if (tile < t0[g]) continue;
            const int q = g % NST, b = kblk & 1;
            const unsigned r = kblk % NB;
            unsigned sc = 0;
#pragma unroll
            for (int i = 0; i < NST; ++i)
              if (i == q) sc = scount[i]++;
            alive = wait_phase(&bfull[r], (kblk / NB) & 1u, abort_flag, true) &&
                    (kblk < 2 || wait_phase(&acce[b], ((kblk - 2) >> 1) & 1u, abort_flag, true));
            for (int h = 0; h < 2 && alive; ++h) {
              alive = wait_phase(&full[2 * q + h], sc & 1u, abort_flag, true);
              if (!alive) break;
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              issue_half<NN, PARTS, true>(tmem + (uint32_t)(b * SH::kBuf), smem_u32(tiles + q * SH::kStage),
                                          smem_u32(btile + r * SH::kB), a.fmt, h);
              umma_commit(&empty[2 * q + h]);
              started = true;
            }
            if (!alive) break;
            umma_commit(&bempty[r]);
            umma_commit(&accf[b]);
            ++kblk;
          }
        if (!alive && started) {  // what was started completes before the CTA ends
          umma_commit(done);
          wait_phase(done, 0, abort_flag, false);
        }
      }
    } else if (warp < 4) {
      // ---- drain: thread t owns row t of the tile
      const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
      const long long base = alm_base(a.lmax, m);
      float myinv = 1.f;  // two parts: the inverse scale of channel b0 + lane
      if (PARTS == 2 && lane < nbl) myinv = 1.f / chan_scale(a.bmax, b0 + lane, a.sfac);
      for (int tile = 0; tile < ntile; ++tile) {
        const int l = m + kTcTile * tile + t;
        const bool odd = (t & 1) != 0;
        float sum[C2N];
#pragma unroll
        for (int j = 0; j < C2N; ++j) sum[j] = 0.f;
        for (int g = 0; g < a.ngrid; ++g) {
          if (tile < t0[g]) continue;
          const int b = kblk & 1;
          if (alive) alive = wait_phase(&accf[b], (kblk >> 1) & 1u, abort_flag, true);
          alive = __all_sync(0xffffffffu, alive);
          if (!alive) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t c0 = trow + (uint32_t)(b * SH::kBuf);
          constexpr int NR = PARTS == 3 ? 4 : 1;  // column regions
          // a value from its regions: the smallest terms first, the two of
          // order 1 last
          auto total = [](const uint32_t (&v)[NR][16], int j) {
            if constexpr (PARTS == 3)
              return ((__uint_as_float(v[2][j]) + __uint_as_float(v[1][j])) + __uint_as_float(v[0][j])) +
                     __uint_as_float(v[3][j]);
            else
              return __uint_as_float(v[0][j]);
          };
          // the columns of this row's parity (S or A), 16 at a time; the load is
          // warp-wide, so both parities' are read
#pragma unroll
          for (int c = 0; c < C2N / 16; ++c) {
            uint32_t ve[NR][16], vo[NR][16];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
              tmem_ld16(c0 + (uint32_t)(r * NN + 16 * c), ve[r]);
              tmem_ld16(c0 + (uint32_t)(r * NN + C2N + 16 * c), vo[r]);
            }
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 16; ++j) sum[16 * c + j] += odd ? total(vo, j) : total(ve, j);
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          mbar_arrive(&acce[b]);
          ++kblk;
        }
        if (!alive) break;
        const bool row = l <= a.lmax;
        float2* out = a.out + (long long)b0 * a.nalm + base + l;
        const float mf = m > 0 ? a.mfac : 1.f;
        if constexpr (PARTS == 2) {
          // as the table tiles: P_l times powers of two, the channel scale last
          const float scale = row ? a.coef_pf[base + l] * mf * a.lscale : 0.f;
#pragma unroll
          for (int c = 0; c < C2N / 2; ++c) {
            const float inv = __shfl_sync(0xffffffffu, myinv, c);
            if (row && c < nbl)
              out[(long long)c * a.nalm] = make_float2(scale * sum[2 * c] * inv, scale * sum[2 * c + 1] * inv);
          }
        } else {
          if (row) {
            const float2 P = cscale(a.coef_pp[base + l], mf);
#pragma unroll
            for (int c = 0; c < C2N / 2; ++c)
              if (c < nbl) {
                const float inv = a.binv[b0 + c];  // a power of two
                const float re = sum[2 * c] * inv, im = sum[2 * c + 1] * inv;
                out[(long long)c * a.nalm] = make_float2(fmaf(re, P.x, re * P.y), fmaf(im, P.x, im * P.y));
              }
          }
        }
      }
    }
    __syncwarp();
    __syncthreads();  // every role is done with this m (and t0)
    if (*abort_flag) break;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (t == 0 && *abort_flag) atomicExch(a.status, (int)HPX_ERR_TIMEOUT);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(SH::kAlloc));
}

// ---------------------------------------------------------------------------
// synthesis
// ---------------------------------------------------------------------------
struct GenSynArgs {
  const float2* coef_cf;
  const int* lc;
  const float4* start;
  const float2* zf;
  const int* lgrid;
  int ngrid;
  const int* lstart;  // [m][pair tile] first l, aligned to m + 64 k
  int nptile;
  const long long* achunk;
  const unsigned* bmax;
  float sfac, lscale;
  float2* F;
  int lmax, mmax, npair, nring, nb;
  uint32_t fmt;
  int* status;
  int ncg;
  long long cg_rows;
  int withhold;
};

template <int NN> struct GenSynShape {
  static constexpr int kMq = NN == 128 ? 2 : 4;  // m of a CTA (the sums' tensor memory)
  static constexpr int kB = 2 * NN * 128, kStage = 2 * kTileBytes, kNB = NN == 128 ? 3 : 4;
  static constexpr int kThreads = 32 * (10 + 2 * kMq);
  static constexpr int kCoef = 2 * kMq * 64 * (int)sizeof(float4);  // c_l of a block, per generator warp
  static constexpr int kAlloc = (2 + kMq) * NN <= 256 ? 256 : 512;  // two block accumulators, the m's sums
  static_assert((2 + kMq) * NN <= 512 && kNB >= 2, "shape");
  static constexpr size_t kSmem = 1024 + kMq * (size_t)kStage + kNB * (size_t)kB + kCoef + 1024;
  static_assert(kSmem <= 227 * 1024, "shape");
};

// A CTA: 128 ring pairs of four (two at 32 channels) consecutive m, all l.  A
// pair of generator warps owns the j-th m's stage, 64 rows (ring pairs) each, a
// lane two chains, and writes 8 consecutive l of a row as one 16-byte word.  The m's blocks
// (64 l, in two halves of 32 so that one is generated while the other is
// contracted) are taken in turn, each accumulated alone and added to its m's
// sums in tensor memory; at the end every ring's values of the CTA's m leave
// as one piece of F (a 32-byte sector of four).
template <int NN, typename E>
__global__ void __launch_bounds__(GenSynShape<NN>::kThreads, 1)
k_gen_synthesis(const __grid_constant__ CUtensorMap tmB, const GenSynArgs a) {
  using SH = GenSynShape<NN>;
  constexpr int NB = SH::kNB, C2N = NN / 2, RB = 2 * NN, MQ = SH::kMq, KW = 64;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int ptile = (int)blockIdx.x / a.ncg, cgi = (int)blockIdx.x % a.ncg;
  const int m = blockIdx.y * MQ, nq = min(MQ, a.mmax + 1 - m);
  const int b0 = cgi * (C2N / 2), nbl = min(C2N / 2, a.nb - b0);
  extern __shared__ unsigned char smem_raw[];
  unsigned char* tiles = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* btile = tiles + MQ * SH::kStage;
  float4* coefs = reinterpret_cast<float4*>(btile + NB * SH::kB);  // [warp][64]
  uint64_t* full = reinterpret_cast<uint64_t*>(reinterpret_cast<unsigned char*>(coefs) + SH::kCoef);
  uint64_t* empty = full + 8;  // a stage's halves (32 l) apart
  uint64_t* bfull = empty + 8;
  uint64_t* bempty = bfull + NB;
  uint64_t* accf = bempty + NB;
  uint64_t* acce = accf + 2;
  uint64_t* done = acce + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* qna = reinterpret_cast<int*>(tmem_slot + 2);  // [MQ] blocks of each m
  int* qls = qna + 4;                                // [MQ] first l
  constexpr int kSum = 2 * NN;                       // first column of the sums

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(SH::kAlloc));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (warp == 1 && lane < MQ) {
    int n = 0, ls = 0;
    if (lane < nq) {
      ls = a.lstart[(long long)(m + lane) * a.nptile + ptile];
      if (ls <= a.lmax) n = (a.lmax - ls) / KW + 1;
    }
    qna[lane] = n;
    qls[lane] = ls;
  }
  if (t == 32) {
    for (int s = 0; s < 2 * MQ; ++s) {
      mbar_init(&full[s], 2);
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < NB; ++s) {
      mbar_init(&bfull[s], 1);
      mbar_init(&bempty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], 256);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  int rounds = 0;
  for (int j = 0; j < MQ; ++j) rounds = max(rounds, qna[j]);

  bool alive = true;
  if (warp >= 8 && warp < 8 + 2 * MQ) {
    // ---- generators
    const int gw = warp - 8, j = gw >> 1, h = gw & 1, mj = m + j, n = qna[j];
    if (n > 0) {
      float4* cz = coefs + gw * KW;
      Chains2<(int)kLamScale> ch;
      ch.init(a.zf, a.lc, a.start, a.lgrid, a.ngrid, a.npair, a.lmax, mj, ptile * 2 + h, lane);
      unsigned char* mine = tiles + j * SH::kStage + (64 * h + lane) * 128;  // rows of chains p, p + 32
      const uint32_t sw = (uint32_t)(lane & 7);                            // both rows' swizzle
      const float2* cl = a.coef_cf + alm_base(a.lmax, mj);
      auto coef = [&](int l) { return l <= a.lmax ? cl[l] : make_float2(0.f, 0.f); };
      float2 c0 = coef(qls[j] + lane), c1 = coef(qls[j] + 32 + lane);  // the next block's
      for (int k = 0; k < n; ++k) {
        const int lk = qls[j] + KW * k;
        __syncwarp();
        cz[lane] = make_float4(c0.x, c0.x, c0.y, c0.y);
        cz[32 + lane] = make_float4(c1.x, c1.x, c1.y, c1.y);
        __syncwarp();
        c0 = coef(lk + KW + lane);
        c1 = coef(lk + KW + 32 + lane);
        for (int hf = 0; hf < 2 && alive; ++hf) {
          if (k > 0) alive = wait_phase(&empty[2 * j + hf], (uint32_t)(k - 1) & 1u, abort_flag, true);
          alive = __all_sync(0xffffffffu, alive);
          if (!alive) break;
#pragma unroll 1
          for (int i8 = 32 * hf; i8 < 32 * hf + 32; i8 += 8) {
            float va[8], vb[8];
            if (lk + i8 + 8 <= ch.lmin) {
#pragma unroll
              for (int u = 0; u < 8; ++u) va[u] = vb[u] = 0.f;
            } else {
              ch.steps8(cz + i8, lk + i8, va, vb);
            }
            const uint32_t o = (((uint32_t)i8 >> 3) ^ sw) << 4;
            put8<2, E>(mine + o, va);
            put8<2, E>(mine + 32 * 128 + o, vb);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(&full[2 * j + hf]);
        }
        if (!alive) break;
      }
    }
  } else if (warp == 8 + 2 * MQ) {
    // ---- operand copies
    unsigned kblk = 0;
    if (lane == 0 && !a.withhold) {
      for (int it = 0; it < rounds && alive; ++it)
        for (int j = 0; j < MQ; ++j) {
          if (it >= qna[j]) continue;
          const unsigned r = kblk % NB;
          if (kblk >= NB) alive = wait_phase(&bempty[r], (kblk / NB - 1) & 1u, abort_flag, true);
          if (!alive) break;
          mbar_expect_tx(&bfull[r], SH::kB);
          const int rb = (int)((a.achunk[m + j] + (qls[j] - m - j) / KW + it) * RB + cgi * a.cg_rows);
          tma_load_2d(btile + r * SH::kB, &tmB, 0, rb, &bfull[r]);
          tma_load_2d(btile + r * SH::kB + NN * 128, &tmB, 0, rb + NN, &bfull[r]);
          ++kblk;
        }
      // whatever was started completes before the CTA moves on
      for (unsigned k = kblk > NB ? kblk - NB : 0; k < kblk; ++k)
        wait_phase(&bfull[k % NB], (k / NB) & 1u, abort_flag, false);
    }
  } else if (warp == 9 + 2 * MQ) {
    // ---- products, block by block (the first halves of all m before the
    // second ones, with an accumulator each, measured 9% slower)
    unsigned kblk = 0;
    if (lane == 0) {
      bool started = false;
      for (int it = 0; it < rounds && alive; ++it)
        for (int j = 0; j < MQ; ++j) {
          if (it >= qna[j]) continue;
          const int b = kblk & 1;
          const unsigned r = kblk % NB;
          alive = wait_phase(&bfull[r], (kblk / NB) & 1u, abort_flag, true) &&
                  (kblk < 2 || wait_phase(&acce[b], ((kblk - 2) >> 1) & 1u, abort_flag, true));
          for (int hf = 0; hf < 2 && alive; ++hf) {
            alive = wait_phase(&full[2 * j + hf], (uint32_t)it & 1u, abort_flag, true);
            if (!alive) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            issue_half<NN, 2, false>(tmem + (uint32_t)(b * NN), smem_u32(tiles + j * SH::kStage),
                                     smem_u32(btile + r * SH::kB), a.fmt, hf);
            umma_commit(&empty[2 * j + hf]);
            started = true;
          }
          if (!alive) break;
          umma_commit(&bempty[r]);
          umma_commit(&accf[b]);
          ++kblk;
        }
      if (started) {
        umma_commit(done);
        wait_phase(done, 0, abort_flag, false);
      }
    }
  } else if (warp < 8) {
    // ---- drain: warps 0-3 the first half of the columns, 4-7 the second;
    // a lane owns row 32 (warp mod 4) + lane (its ring pair)
    const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * C2N);
    unsigned kblk = 0;
    for (int it = 0; it < rounds && alive; ++it)
      for (int j = 0; j < MQ; ++j) {
        if (it >= qna[j]) continue;
        const int b = kblk & 1;
        if (alive) alive = wait_phase(&accf[b], (kblk >> 1) & 1u, abort_flag, true);
        alive = __all_sync(0xffffffffu, alive);
        if (!alive) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t cs = trow + (uint32_t)(kSum + j * NN), ca = trow + (uint32_t)(b * NN);
        constexpr int NC = C2N / 16, NW = NC < 2 ? NC : 2;  // NW loads of 16 columns of each in flight
#pragma unroll
        for (int c0 = 0; c0 < NC; c0 += NW) {
          uint32_t v[NW][16], w[NW][16];
#pragma unroll
          for (int c = 0; c < NW; ++c) {
            tmem_ld16(ca + 16 * (c0 + c), v[c]);
            if (it > 0) tmem_ld16(cs + 16 * (c0 + c), w[c]);
          }
          tmem_wait_ld();
          if (c0 + NW == NC) {  // the block's accumulator is read
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(&acce[b]);
          }
#pragma unroll
          for (int c = 0; c < NW; ++c) {
            if (it > 0) {
#pragma unroll
              for (int u = 0; u < 16; ++u) v[c][u] = __float_as_uint(__uint_as_float(w[c][u]) + __uint_as_float(v[c][u]));
            }
            tmem_st16(cs + 16 * (c0 + c), v[c]);
          }
        }
        tmem_wait_st();
        ++kblk;
      }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp < 4 && *abort_flag == 0) {
    // region j: E (columns 0 .. C2N-1) and O (C2N .. NN-1) of the j-th m (zero
    // without blocks); north ring p gets E + O, its mirror E - O
    const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)kSum;
    const int p = ptile * 128 + t;
    const int ys = p == a.npair - 1 ? -1 : a.nring - 1 - p;
    const long long mstride = a.mmax + 1;
#pragma unroll 1
    for (int cg = 0; cg < C2N / 8; ++cg) {  // 4 channels: 8 E and 8 O columns
      uint32_t e[MQ][8], o[MQ][8];
#pragma unroll
      for (int j = 0; j < MQ; ++j) {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(e[j][0]), "=r"(e[j][1]), "=r"(e[j][2]), "=r"(e[j][3]), "=r"(e[j][4]), "=r"(e[j][5]),
                       "=r"(e[j][6]), "=r"(e[j][7])
                     : "r"(trow + (uint32_t)(j * NN + 8 * cg)));
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(o[j][0]), "=r"(o[j][1]), "=r"(o[j][2]), "=r"(o[j][3]), "=r"(o[j][4]), "=r"(o[j][5]),
                       "=r"(o[j][6]), "=r"(o[j][7])
                     : "r"(trow + (uint32_t)(j * NN + C2N + 8 * cg)));
      }
      tmem_wait_ld();
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        const int c = 4 * cg + cc;
        if (p < a.npair && c < nbl) {
          const float inv = a.lscale / chan_scale(a.bmax, b0 + c, a.sfac);  // a power of two
#pragma unroll
          for (int side = 0; side < 2; ++side) {
            const int y = side ? ys : p;
            if (y < 0) continue;
            const long long at = ((long long)(b0 + c) * a.nring + y) * mstride + m;
            float2 w[MQ];
#pragma unroll
            for (int j = 0; j < MQ; ++j) {
              const bool has = qna[j] > 0;
              const float er = has ? __uint_as_float(e[j][2 * cc]) * inv : 0.f;
              const float ei = has ? __uint_as_float(e[j][2 * cc + 1]) * inv : 0.f;
              const float orr = has ? __uint_as_float(o[j][2 * cc]) * inv : 0.f;
              const float oi = has ? __uint_as_float(o[j][2 * cc + 1]) * inv : 0.f;
              w[j] = side ? make_float2(er - orr, ei - oi) : make_float2(er + orr, ei + oi);
            }
            if (nq == MQ && (at % MQ) == 0) {  // whole pieces: a sector of four m
              float4* dd = reinterpret_cast<float4*>(a.F + at);
#pragma unroll
              for (int h = 0; h < MQ / 2; ++h) dd[h] = make_float4(w[2 * h].x, w[2 * h].y, w[2 * h + 1].x, w[2 * h + 1].y);
            } else {
              for (int j = 0; j < MQ; ++j)
                if (j < nq) a.F[at + j] = w[j];
            }
          }
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  if (t == 0 && *abort_flag) atomicExch(a.status, (int)HPX_ERR_TIMEOUT);
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(SH::kAlloc));
}

template <int NN, int PARTS, bool TAB, typename E>
cudaError_t analysis_launch(const hpx_plan_s* p, const GenArgs& a, cudaStream_t s) {
  auto kern = k_gen_analysis<NN, PARTS, TAB, E>;
  cudaError_t e = allow_max_smem(kern);
  if (e != cudaSuccess) return e;
  const int units = a.nm * a.ncg, grid = units < p->gen_ctas ? units : p->gen_ctas;
  kern<<<grid, GenShape<NN, PARTS>::kThreads, GenShape<NN, PARTS>::kSmem, s>>>(*reinterpret_cast<const CUtensorMap*>(p->tm_gt), a);
  return cudaGetLastError();
}

template <int NN, typename E>
cudaError_t synthesis_launch(const hpx_plan_s* p, const GenSynArgs& a, cudaStream_t s) {
  auto kern = k_gen_synthesis<NN, E>;
  cudaError_t e = allow_max_smem(kern);
  if (e != cudaSuccess) return e;
  constexpr int MQ = GenSynShape<NN>::kMq;
  kern<<<dim3(p->nptile * a.ncg, (p->mmax + MQ) / MQ), GenSynShape<NN>::kThreads, GenSynShape<NN>::kSmem, s>>>(
      *reinterpret_cast<const CUtensorMap*>(p->tm_at), a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_gen_analysis(const hpx_plan_s* p, float* alm, double mfac, cudaStream_t s) {
  GenArgs a{};
  a.coef_cf = p->d_coef_cf;
  a.lc = p->d_lc;
  a.start = p->d_start;
  a.zf = p->d_zf;
  a.lgrid = p->d_lgrid;
  a.gstart = p->d_gstart;
  a.ngrid = p->ngrid;
  a.state = p->d_gen_state;
  a.coef_pf = p->d_coef_pf;
  a.coef_pp = p->d_coef_pp;
  a.mfac = (float)mfac;
  a.out = reinterpret_cast<float2*>(alm);
  a.lmax = p->lmax;
  a.npair = p->npair;
  a.nalm = p->nalm;
  a.nb = p->nbatch;
  a.status = p->d_status;
  a.nm = p->mmax + 1;
  a.cg_rows = p->gt_group_elems / 64;
  a.withhold = p->test_withhold;
  a.bmax = p->d_bmax;
  a.binv = reinterpret_cast<const float*>(p->d_bmax + p->bmax_stride);
  a.sfac = p->tc_sfac_a;
  const int nn = p->gen_parts == 3 ? p->gen_nn : p->tc_nn_a;
  a.ncg = (p->nbatch + nn / 4 - 1) / (nn / 4);
  if (p->gen_parts == 3) {
    a.fmt = 1;  // BF16
    a.tab = lam_tab<float>(p);
    const bool tab = p->d_tab != nullptr;
    switch (nn) {
      case 32: return tab ? analysis_launch<32, 3, true, __nv_bfloat16>(p, a, s) : analysis_launch<32, 3, false, __nv_bfloat16>(p, a, s);
      case 64: return tab ? analysis_launch<64, 3, true, __nv_bfloat16>(p, a, s) : analysis_launch<64, 3, false, __nv_bfloat16>(p, a, s);
    }
    return cudaErrorInvalidValue;
  }
  a.fmt = (uint32_t)p->tc_fmt;
  a.lscale = (float)(1.0 / kLamScale);
  switch (nn) {
    case 32: return a.fmt ? analysis_launch<32, 2, false, __nv_bfloat16>(p, a, s) : analysis_launch<32, 2, false, __half>(p, a, s);
    case 64: return a.fmt ? analysis_launch<64, 2, false, __nv_bfloat16>(p, a, s) : analysis_launch<64, 2, false, __half>(p, a, s);
    case 128: return a.fmt ? analysis_launch<128, 2, false, __nv_bfloat16>(p, a, s) : analysis_launch<128, 2, false, __half>(p, a, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_gen_synthesis(const hpx_plan_s* p, cudaStream_t s) {
  GenSynArgs a{};
  a.coef_cf = p->d_coef_cf;
  a.lc = p->d_lc;
  a.start = p->d_start;
  a.zf = p->d_zf;
  a.lgrid = p->d_lgrid;
  a.ngrid = p->ngrid;
  a.lstart = p->d_stab_lstart;
  a.nptile = p->nptile;
  a.achunk = p->d_achunk;
  a.bmax = p->d_bmax + p->bmax_stride;
  a.sfac = p->tc_sfac_s;
  a.lscale = (float)(1.0 / kLamScale);
  a.F = static_cast<float2*>(p->d_F);
  a.lmax = p->lmax;
  a.mmax = p->mmax;
  a.npair = p->npair;
  a.nring = p->nring;
  a.nb = p->nbatch;
  a.fmt = (uint32_t)p->tc_fmt;
  a.status = p->d_status;
  a.ncg = (p->nbatch + p->tc_nn_s / 4 - 1) / (p->tc_nn_s / 4);
  a.cg_rows = p->at_group_elems / 64;
  a.withhold = p->test_withhold;
  switch (p->tc_nn_s) {
    case 32: return a.fmt ? synthesis_launch<32, __nv_bfloat16>(p, a, s) : synthesis_launch<32, __half>(p, a, s);
    case 64: return a.fmt ? synthesis_launch<64, __nv_bfloat16>(p, a, s) : synthesis_launch<64, __half>(p, a, s);
    case 128: return a.fmt ? synthesis_launch<128, __nv_bfloat16>(p, a, s) : synthesis_launch<128, __half>(p, a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace hpx
