// Internal declarations shared by the libhpx translation units.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>
#include <string>

#include "hpx.h"

namespace hpx {

// ---------------------------------------------------------------------------
// complex helpers (float2 / double2)
// ---------------------------------------------------------------------------
template <typename T> struct Vec2;
template <> struct Vec2<float> { using type = float2; };
template <> struct Vec2<double> { using type = double2; };
template <typename T> using C2 = typename Vec2<T>::type;

template <typename V> __host__ __device__ __forceinline__ V cmk(decltype(V::x) a, decltype(V::x) b) {
  V r; r.x = a; r.y = b; return r;
}
template <typename V> __device__ __forceinline__ V cadd(V a, V b) { return cmk<V>(a.x + b.x, a.y + b.y); }
template <typename V> __device__ __forceinline__ V csub(V a, V b) { return cmk<V>(a.x - b.x, a.y - b.y); }
template <typename V> __device__ __forceinline__ V cconj(V a) { return cmk<V>(a.x, -a.y); }
template <typename V> __device__ __forceinline__ V cmul(V a, V b) {
  return cmk<V>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename V> __device__ __forceinline__ V cscale(V a, decltype(V::x) s) { return cmk<V>(a.x * s, a.y * s); }

// ---------------------------------------------------------------------------
// plan-resident tables
// ---------------------------------------------------------------------------
// One HEALPix ring (Sec. III-A).
struct RingInfo {
  long long start;    // first pixel in RING order
  long long specoff;  // offset of its half spectrum (N/2 + 1 bins) in the spectrum workspace
  long long etab;     // offset of its table E_N[r] = exp(-i pi r / N), r in [0, 2N)
  long long btab;     // offset of its Bluestein kernel spectrum, -1 if it needs none (N/2, FP32: N/4 a power of two)
  int nphi;           // N_y
  int sigma;          // phi_0 = sigma pi / N_y
  int logm;           // log2 of the FFT length used for the ring (FP32: fft32_shape)
  int pad;
  double z, sinth;    // cos(theta_y), sin(theta_y)
  double w;           // quadrature weight of every pixel on the ring (4 pi / Npix)
};

// FP32 ring transforms (hpx_fft_f32.cu): a ring of 4i pixels is two complex
// transforms of length i over M = A^2 R points; fft32_shape is 256 A + R.  i a
// power of two >= 16: M = i; else M >= 2i - 1 (Bluestein), i > 8.  A = 4 to M =
// 128, 8 to 512, then 16: smaller transforms spread over more threads, and R
// stays a small factor that M can be fitted with.
__host__ __device__ inline int fft32_shape(int i) {
  const int len = (i & (i - 1)) == 0 ? i : 2 * i - 1, A = len <= 128 ? 4 : len <= 512 ? 8 : 16;
  int r = (len + A * A - 1) / (A * A);
  if (r > 8) r += r & 1;  // radices 9, 11, 13 and 15 have no kernel
  return r + 256 * A;
}
__host__ __device__ inline int fft32_len(int i) { return (fft32_shape(i) >> 8) * (fft32_shape(i) >> 8) * (fft32_shape(i) & 255); }
__host__ __device__ inline bool fft32_bluestein(int i) { return i > 8 && (i & (i - 1)) != 0; }
// first-pass twiddles exp(-2 pi i j / M), j < M / A, of every M
__host__ __device__ inline int fft32_tw_offset(int A, int rad) { return 136 * (A - 4) + A * rad * (rad - 1) / 2; }
constexpr int kFft32Twiddles = 136 * (16 - 4) + 16 * 136;
__host__ __device__ inline long long fft32_chirp_offset(int i) { return (long long)i * (i - 1) / 2; }

}  // namespace hpx

struct hpx_plan_s {
  int nside, lmax, mmax, nbatch, dtype, device;
  unsigned flags;
  int nring, npair;
  long long npix, nalm, nspec;
  int logm_max;        // largest FFT length over the rings (log2)
  int logtw;           // log2 of the twiddle table's FFT length
  long long netab, nbtab;
  hpx::RingInfo* d_ring;
  void* d_etab;        // C2<T> per distinct ring length
  void* d_btab;        // C2<T> Bluestein kernel spectra, scaled 1/M (FP64: natural order; FP32: conjugated, hpx_fft_f32.cu)
  void* d_chirp;       // FP64: per cap ring i (offset i (i - 1)): exp(-pi i n^2 / H), n < H = 2i; FP32: fft32_chirp_offset,
                       // exp(-pi i n^2 / i), n < i
  void* d_tw;          // FP64: tw[j] = exp(-2 pi i j / 2^logtw), j < 2^(logtw-1); FP32: fft32_tw_offset
  // 16-bit single-product plans: rings and tables as an FP64 plan's (float2),
  // for their analysis
  hpx::RingInfo* d_ring16;
  void *d_btab16, *d_chirp16, *d_tw16;
  size_t nbtab16;
  int logm16;
  double* d_cmm;       // [mmax+1] lambda_mm / sin^m(theta) (sign included)
  double* d_coef_c;    // [nalm] recurrence coefficient c_l of mu_l = c_l z mu_{l-1} - mu_{l-2}
  float2* d_coef_cf;   // [nalm] c_l as a double-FP32 pair (hi, lo): the FP32 plans' recurrence
  double* d_coef_p;    // [nalm] P_l, lambda_l = P_l mu_l (FP64 plans)
  float2* d_coef_pp;   // [nalm] P_l as a sum of two floats (FP32 plans)
  float* d_coef_pf;    // [nalm] P_l rounded to float
  int* d_lc;           // [mmax+1][npair] first significant l of chain (m, pair)
  double* d_mu0;       // [mmax+1][npair] mu_{lc-1} (FP64 plans)
  double* d_mu1;       // [mmax+1][npair] mu_{lc}
  float4* d_start;     // [mmax+1][npair] both times 2^104 as double-FP32 pairs (FP32 plans)
  // FP16 hi/lo plans of a size that hpx_map2alm_noalloc takes: the same from
  // 2^-kSigExp32 on, for the FP32 recurrence of that call (d_lc's later starts are
  // exact for FP16 values only)
  int* d_lc32;
  float4* d_start32;
  int* d_lgrid;        // [mmax+1][ngrid] first l from which every chain of a 64-pair group has |mu| >= 2^-kGridExp
                       // and is past its start (lmax + 1 if some chain never is); FP32 plans
  int ngrid;           // 64-pair groups
  int* d_gstart;       // [mmax+1][ngrid] earliest start of a group's chains
  float2* d_zf;        // [npair] z as a sum of two floats
  // generated-lambda tensor-core stages (hpx_gen.cu)
  int gen_parts;       // 0: not used; 2: streamed split-product plans; 3: FP32 analysis in three BF16 parts,
                       // where it pays (gen_analysis)
  int gen_nn;          // 3: N columns of the analysis products
  int gen_wide;        // 2: N columns of the table tiles that wide analyses take instead, their lambda
                       // staged (0: no staging buffers); their operand in d_gt likewise
  long long gt_group_elems_wide;
  alignas(64) unsigned char tm_gt_wide[128];
  int gen_ctas;        // CTAs of the analysis (one per SM)
  float4* d_gen_state; // [gen_ctas][npair] chains between tiles
  void* d_spec;        // workspace [nbatch][nspec] C2<T>
  void* d_F;           // workspace [nbatch][nring][mmax+1] C2<T>
  void* d_io_map;      // device I/O buffers of the host-buffer entry points (lazy)
  void* d_io_alm;
  void* d_aio_map[2];  // pipelined host-buffer calls: two I/O slots (lazy)
  void* d_aio_alm[2];
  int aio_next;        // slot of the next pipelined call
  void* aio_streams;   // cudaStream_t[2]: host-to-device, device-to-host
  void* aio_events;    // cudaEvent_t[6]: uploaded[2], computed[2], slot free[2]
  void* d_it_map;      // iterative refinement: synthesis / residual map and correction (lazy)
  void* d_it_alm;
  void* timing;        // per-stage CUDA events while timing is enabled
  void* d_tab;         // plan-resident lambda table (HPX_PLAN_LAMBDA_TABLE), C2<T>'s real type
  long long* d_tab_off;  // [mmax+1][ngroup] first element of each (m, 32-pair group)
  int* d_tab_lstart;   // [mmax+1][ngroup] first l stored for the group
  int ngroup;
  long long tab_elems;
  // tensor-core Legendre stages (HPX_PLAN_TENSOR_CORES and the 16-bit dtypes)
  int tc_nn_a, tc_nn_s;  // N columns of the analysis / synthesis tiles (0: not used)
  int tc_mode;         // 0 FP32 table (3xTF32), 1 one 16-bit product, 2 16-bit x3 (hi, lo)
  int tc_fmt;          // 16-bit operand format: 0 FP16, 1 BF16
  float tc_sfac_a, tc_sfac_s;  // channel-scale bound factors of the current transform
  void* d_tab_lo;      // 16-bit x3: remainders of the row table
  void* d_gt;          // analysis operand Gt[cgroup][m][group][rows][row width] (per transform), one
                       // region per channel group of an analysis launch
  long long gt_group_elems;  // elements of one channel group's Gt region
  int gt_groups;       // channel groups Gt holds
  void* d_at;          // synthesis operand At[group][chunk][rows][row width] (per transform), one
                       // region per channel group of a synthesis launch
  long long at_group_elems;  // elements of one channel group's At region
  int at_groups;       // channel groups At holds (the plan's nbatch over channels per group)
  long long* d_achunk; // [mmax+2] first At chunk of each m
  unsigned* d_bmax;    // [2][bmax_stride] 16-bit modes: largest operand component per channel, of
                       // the analysis (spectra) and of the synthesis (alm), apart so that an
                       // analysis and a synthesis may run on the plan at the same time; FP32
                       // plans with gen_parts 3: [2][nbatch], the analysis' maxima (zero between
                       // analyses) and, from its pack on, the inverse channel scales (floats)
  int bmax_stride;     // the plan's own nbatch (views for fewer channels keep it)
  void* d_stab;        // column lambda table: blocks of 128 pairs x (32 or 64) l
  void* d_stab_lo;     // 16-bit x3: its remainders
  long long* d_stab_off;  // [mmax+1][nptile] first element of each (m, pair tile)
  int* d_stab_lstart;  // [mmax+1][nptile] first l stored
  int nptile;
  long long stab_elems;
  alignas(64) unsigned char tm_tab[128];   // TMA descriptors
  alignas(64) unsigned char tm_tablo[128];
  alignas(64) unsigned char tm_gt[128];
  alignas(64) unsigned char tm_stab[128];
  alignas(64) unsigned char tm_stablo[128];
  alignas(64) unsigned char tm_at[128];
  // out-of-core tables (HPX_PLAN_LAMBDA_HOST): pinned host copies, streamed
  // per block of m through two device staging buffers
  void* h_tab;
  void* h_tab_lo;
  void* h_stab;
  void* h_stab_lo;
  size_t host_bytes;   // pinned host memory of the tables
  void* d_stage[2];    // each: hi part, then (x3) lo part, stage_bytes apiece
  size_t stage_bytes;
  int stage_next;      // staging buffer of the next block
  int nblk_row, nblk_col;
  int* blk_row;        // host [nblk + 1]: m boundaries of the row-table blocks
  int* blk_col;
  long long* blk_row_base;  // host [nblk + 1]: first table element of each block
  long long* blk_col_base;
  alignas(64) unsigned char tm_stage[2][128];
  alignas(64) unsigned char tm_stagelo[2][128];
  void* copy_stream;   // cudaStream_t
  void* fft_streams;   // cudaStream_t[2]: the belt-ring launches of the analysis / synthesis ring
                       // transforms, beside the cap-ring launch on the caller's stream
  void* fft_events;    // cudaEvent_t[4]: fork / join of the analysis, then of the synthesis
  void* stage_events;  // cudaEvent_t[4]: copied[2], free[2]
  int* d_status;       // device-side wait status (HPX_OK or HPX_ERR_TIMEOUT)
  int test_withhold;   // test support: tile kernels issue no copies, FP32 analyses no sums (hpx_plan_test_withhold_copies)
  double w_max;        // largest ring weight (4 pi / Npix unless set)
  size_t bytes;
};

namespace hpx {

// Significance threshold of the recurrence chains: a chain contributes from
// the first l at which |mu_l| >= 2^-e; earlier values are dropped.  FP64 plans
// keep values down to 2^-200 (about 1.6e-60).  In the others e is where a
// value's stored or contracted form becomes exactly zero anyway (|mu| grows
// monotonically up to there), so nothing is lost: below 2^-136 for FP32 and
// BF16 (df_real flushes 2^9 mu below 2^-126), below 2^-34 for FP16 tables
// (2^9 |mu| < 2^-25 rounds to zero, the remainder too).  FP16 tables start
// 6.6% fewer rows that way at Nside 1024, lmax 3071.  hpx_map2alm_noalloc
// contracts FP32 values on plans with FP16 tables too, from starts of their own
// (d_lc32).
constexpr int kSigExp64 = 200, kSigExp32 = 136, kSigExpHalf = 34;

// Ring spectra that hpx_map2alm_noalloc has room for.
constexpr size_t kNoallocBytes = size_t(16) << 20;
// Whether a plan has the second set of chain starts (d_lc32).
inline bool has_starts32(int dtype, int tc_mode, int nbatch, size_t nspec) {
  return dtype == HPX_F32 && tc_mode > 0 && sizeof(float2) * (size_t)nbatch * nspec <= kNoallocBytes;
}

// Rows (l values) per tensor-core tile of the Legendre analysis; the lambda
// table's group starts are aligned to this grid relative to m.
constexpr int kTcTile = 128;

// error reporting (thread-local message)
void set_error(const char* fmt, ...);
hpx_status cuda_fail(cudaError_t e, const char* what);

// Let `func` launch with any dynamic shared memory size the current device
// allows.  The attribute is global per function, so plans of different sizes
// (and threads launching them) must not set it to their own sizes: one plan
// could lower it below what another, still live, launches with.  The launch
// size itself decides occupancy, not this limit.
template <typename F>
cudaError_t allow_max_smem(F* func) {
  int dev = 0, maxopt = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&maxopt, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, maxopt);
  return e;
}

// Double-FP32 numbers (Dekker's double-length arithmetic, 1971): a value is
// the unevaluated sum hi + lo of two floats, about 48 significant bits, and
// the arithmetic runs on the FP32 pipe, 64 times the FP64 pipe's rate on
// this part.  The FP32 plans run the recurrence in it: mu scaled by 2^104
// (chain starts are at least 2^-200 and |mu| stays below 2^8, so both
// parts stay normal floats; a power of two scales the linear recurrence
// exactly).  Explicitly rounded operations keep the compiler from fusing the
// error terms away.
struct Df {
  float hi, lo;
};
constexpr double kDfUp = 0x1p104;
__device__ __forceinline__ Df df_of(double x) {
  const float h = __double2float_rn(x);
  return Df{h, __double2float_rn(x - (double)h)};
}
// a b as an unnormalised pair: the rounded product, plus its rounding error
// (one FMA) and the cross terms (the lo lo term, below 2^-44 ab, dropped)
__device__ __forceinline__ Df df_mul(Df a, Df b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  return Df{p, __fmaf_rn(a.lo, b.hi, e)};
}
// t n1 - n2, renormalised: Knuth's TwoSum of the leading parts, the error
// terms added, then Dekker's FastTwoSum
__device__ __forceinline__ Df df_step(Df t, Df n1, Df n2) {
  const Df q = df_mul(t, n1);
  const float s = __fsub_rn(q.hi, n2.hi);
  const float v = __fsub_rn(s, q.hi);
  const float err = __fadd_rn(__fsub_rn(q.hi, __fsub_rn(s, v)), __fsub_rn(-n2.hi, v));
  const float f = __fadd_rn(err, __fsub_rn(q.lo, n2.lo));
  const float h = __fadd_rn(s, f);
  return Df{h, __fsub_rn(f, __fsub_rn(h, s))};
}
// the float value of a scaled pair: hi 2^-104, and 0 below 2^-126
__device__ __forceinline__ float df_real(Df x) { return fabsf(x.hi) < 0x1p-22f ? 0.f : __fmul_rn(x.hi, 0x1p-104f); }

// One recurrence chain mu_l = c_l z mu_{l-1} - mu_{l-2}, restarted at its first
// significant l (lc) with the stored (mu_{lc-1}, mu_lc) and zero before.  FP64
// plans (RecurD) step in FP64.  The others step in two phases:
//
// * General (RecurG): double-FP32, 19 FP32 operations a step, 3 more for the
//   value; good for any magnitude, so it carries a chain through its growth.
// * Grid (GridState), from the group's grid start on: the value is s + f with
//   s a multiple of a fixed quantum u (2^-18 in mu).  The product is split
//   into its multiple of u, q = (p s1 + C) - C with C = 1.5 2^23 u, and the
//   exact rest (one FMA), so s = q - s2 is exact and needs no TwoSum; f takes
//   the rest and the first-order terms in plain FP32.  |mu| is at most 17.9
//   for Nside <= 2048 (m = 0 on the first rings), so |s| < 2^23 u and q, of at
//   most twice that, stays a multiple of u / 2.  s absorbs f's whole quanta
//   every 16 steps (regrid), so f stays within tens of u and a step adds about
//   2^-39 absolute error.  11 operations a step and one for the value.
//
// A chain changes phase at the grid start of its 64-pair group: every chain of
// the group has started and has |mu| >= 2^-4 (it grows from there, and a step's
// error with it), aligned up to the 32-step blocks m + 32 k.  Near the pole a
// step's error grows linearly in l, up to 1 / sin(theta) times itself, so that
// a ring at theta ends with about 2^-42 lmax / theta; the groups next to the pole
// stay in the general phase (grid_never).  Simulated against extended precision
// (relative L2 over l of the worst chain, m = 0 .. 60): at lmax = 3 Nside - 1,
// 2^-24.2 or less for every Nside, and so at lmax 16384 (with all groups on the grid:
// Nside 64 2^-22, 256 2^-20.2, 2048 2^-18.8).  Rounding the values to FP32 alone
// gives 2^-25.  92% of the steps at Nside 2048 / lmax 6143 are grid steps, 78% at
// Nside 512 / lmax 1024.  Every FP32 kernel and table takes the same steps
// (operations rounded one by one, scalar or two chains packed), so their values
// agree bit for bit.
struct RecurD {
  double z = 0.0, s0 = 0.0, s1 = 0.0, n1 = 0.0, n2 = 0.0;
  __device__ __forceinline__ void start(double z_, double s0_, double s1_) {
    z = z_;
    s0 = s0_;
    s1 = s1_;
  }
  __device__ __forceinline__ double step(double c, int l, int lc) {
    double mu = fma(c * z, n1, -n2);
    if (l == lc) {
      mu = s1;
      n1 = s0;
    }
    n2 = n1;
    n1 = mu;
    return mu;
  }
};

constexpr int kGridExp = 4;     // see above
constexpr int kGridBlock = 32;  // the grid start's alignment relative to m
constexpr int kRegrid = 16;     // steps between regrids
constexpr float kGridC = 48.f;  // 1.5 2^23 u for u = 2^-18 (times the scale of scaled chains)
// Groups of 64 pairs (p0: the first) that stay in the general phase: from Nside
// 512 those below 1/32 of the pairs (lmax / theta = 120,000 at lmax = 3 Nside - 1,
// the most that the bound above allows; below Nside 512 no group reaches it); from
// lmax = 3 Nside on, at every Nside, those below the same lmax / theta, the first group
// always.
__host__ __device__ inline bool grid_never(int p0, int npair, int lmax) {
  if (2 * lmax >= 3 * npair) return 196608LL * p0 < (long long)(lmax + 1) * npair;
  return npair >= 1024 && p0 < npair / 32;
}
// the aligned grid start of a group whose recorded one is lg
__host__ __device__ inline int grid_start(int m, int lg) {
  return m + (lg - m + kGridBlock - 1) / kGridBlock * kGridBlock;
}

struct GridState {
  float s1, f1, s2, f2;
};
__device__ __forceinline__ void grid_split(Df x, float C, float& s, float& f) {
  const float h = __fmul_rn(x.hi, 0x1p-104f);  // exact: |mu| >= 2^-4 here, and n2 has grown alongside
  s = __fsub_rn(__fadd_rn(h, C), C);
  f = __fadd_rn(__fsub_rn(h, s), __fmul_rn(x.lo, 0x1p-104f));
}
__device__ __forceinline__ GridState grid_enter(Df n1, Df n2, float C) {
  GridState g;
  grid_split(n1, C, g.s1, g.f1);
  grid_split(n2, C, g.s2, g.f2);
  return g;
}
__device__ __forceinline__ void regrid(GridState& g, float C) {
  const float k1 = __fsub_rn(__fadd_rn(g.f1, C), C), k2 = __fsub_rn(__fadd_rn(g.f2, C), C);
  g.s1 = __fadd_rn(g.s1, k1);
  g.f1 = __fsub_rn(g.f1, k1);
  g.s2 = __fadd_rn(g.s2, k2);
  g.f2 = __fsub_rn(g.f2, k2);
}
__device__ __forceinline__ float grid_step(GridState& g, Df t, float C) {  // t = c_l z
  const float q = __fsub_rn(__fmaf_rn(t.hi, g.s1, C), C);
  float r = __fmaf_rn(t.hi, g.s1, -q);
  const float s = __fsub_rn(q, g.s2);
  r = __fmaf_rn(t.hi, g.f1, r);
  r = __fmaf_rn(t.lo, g.s1, r);
  const float f = __fsub_rn(r, g.f2);
  g.s2 = g.s1;
  g.f2 = g.f1;
  g.s1 = s;
  g.f1 = f;
  return __fadd_rn(s, f);
}

// Two chains a thread, packed: each operation is one instruction for both
// (f32x2), rounded as the scalar one.
using F2 = unsigned long long;
__device__ __forceinline__ F2 pk2(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpk2(F2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ F2 neg2(F2 v) {
  float a, b;
  unpk2(v, a, b);
  return pk2(-a, -b);
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
struct GridState2 {
  F2 s1 = 0, f1 = 0, s2 = 0, f2 = 0;
};
__device__ __forceinline__ GridState2 grid_pack(const GridState& a, const GridState& b) {
  return GridState2{pk2(a.s1, b.s1), pk2(a.f1, b.f1), pk2(a.s2, b.s2), pk2(a.f2, b.f2)};
}
__device__ __forceinline__ void grid_unpack(const GridState2& g, GridState& a, GridState& b) {
  unpk2(g.s1, a.s1, b.s1);
  unpk2(g.f1, a.f1, b.f1);
  unpk2(g.s2, a.s2, b.s2);
  unpk2(g.f2, a.f2, b.f2);
}
__device__ __forceinline__ void regrid(GridState2& g, F2 C) {
  const F2 nC = neg2(C), k1 = add2(add2(g.f1, C), nC), k2 = add2(add2(g.f2, C), nC);
  g.s1 = add2(g.s1, k1);
  g.f1 = add2(g.f1, neg2(k1));
  g.s2 = add2(g.s2, k2);
  g.f2 = add2(g.f2, neg2(k2));
}
// c4: the step's coefficient pair, each part twice (hi, hi, lo, lo)
__device__ __forceinline__ F2 grid_step(GridState2& g, float4 c4, F2 zh, F2 zl, F2 C) {
  const F2 ch = pk2(c4.x, c4.y), cl = pk2(c4.z, c4.w);
  const F2 p = mul2(ch, zh);
  F2 e = fma2(ch, zh, neg2(p));
  e = fma2(ch, zl, e);
  e = fma2(cl, zh, e);
  const F2 q = add2(fma2(p, g.s1, C), neg2(C));
  F2 r = fma2(p, g.s1, neg2(q));
  const F2 s = add2(q, neg2(g.s2));
  r = fma2(p, g.f1, r);
  r = fma2(e, g.s1, r);
  const F2 f = add2(r, neg2(g.f2));
  g.s2 = g.s1;
  g.f2 = g.f1;
  g.s1 = s;
  g.f1 = f;
  return add2(s, f);
}

// the general phase of one chain
struct RecurG {
  Df n1{0.f, 0.f}, n2{0.f, 0.f};
  __device__ __forceinline__ float step(float2 c, Df z) { return step(df_mul(Df{c.x, c.y}, z)); }
  __device__ __forceinline__ float step(Df t) {  // t = c_l z
    const Df mu = df_step(t, n1, n2);
    n2 = n1;
    n1 = mu;
    return df_real(mu);
  }
  // the step l == lc, from the stored (mu_{lc-1}, mu_lc) 2^104 as (hi, lo, hi, lo)
  __device__ __forceinline__ float start(float4 st) {
    n2 = Df{st.x, st.y};
    n1 = Df{st.z, st.w};
    return df_real(n1);
  }
};

// One chain through both phases, step by step from some l = m + 32 k at or
// before its start (table fills): the scalar form of what the kernels do.
struct Chain {
  RecurG rc;
  GridState g{0.f, 0.f, 0.f, 0.f};
  float4 st{0.f, 0.f, 0.f, 0.f};
  Df z{0.f, 0.f};
  float C = kGridC;
  int m = 0, lc = 0x7fffffff, lg = 0x7fffffff;  // lg: aligned grid start of the chain's group
  const float2* c = nullptr;
  __device__ __forceinline__ float step(int l) {
    if (l < lg) return l == lc ? rc.start(st) : rc.step(c[l], z);
    if (l == lg) g = grid_enter(rc.n1, rc.n2, C);
    else if (((l - m) & (kRegrid - 1)) == 0) regrid(g, C);
    return grid_step(g, df_mul(Df{c[l].x, c[l].y}, z), C);
  }
  // l .. l + 7, l - m a multiple of 8 (lg and the regrids lie on such l); zeros
  // past lmax.  On the grid the coefficients' loads and products do not wait on
  // the chain.
  __device__ __forceinline__ void steps8(int l, int lmax, float (&v)[8]) {
    if (l >= lg) {
      float2 q[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) q[u] = c[min(l + u, lmax)];
      if (l == lg) g = grid_enter(rc.n1, rc.n2, C);
      else if (((l - m) & (kRegrid - 1)) == 0) regrid(g, C);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float x = grid_step(g, df_mul(Df{q[u].x, q[u].y}, z), C);
        v[u] = l + u <= lmax ? x : 0.f;
      }
    } else {
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = l + u <= lmax ? step(l + u) : 0.f;
    }
  }
};

__host__ __device__ inline long long alm_base(int lmax, int m) {  // index(l = 0, m); index(l, m) = alm_base + l
  return (long long)m * (2 * lmax + 1 - m) / 2;
}

// the chain (m, p) with values scaled by S (a power of two); zeros for p >= npair
template <int S>
__device__ __forceinline__ Chain chain_at(const RingInfo* __restrict__ rings, const float2* __restrict__ coef_cf,
                                          const int* __restrict__ lc_tab, const float4* __restrict__ start,
                                          const int* __restrict__ lgrid, int ngrid, int lmax, int npair, int m, int p) {
  Chain ch;
  ch.m = m;
  ch.c = coef_cf + alm_base(lmax, m);
  ch.C = kGridC * S;
  if (p < npair) {
    const long long ci = (long long)m * npair + p;
    ch.lc = lc_tab[ci];
    ch.lg = grid_start(m, lgrid[(long long)m * ngrid + (p >> 6)]);
    ch.z = df_of(rings[p].z);
    const float4 v = start[ci];
    ch.st = make_float4(S * v.x, S * v.y, S * v.z, S * v.w);
  }
  return ch;
}

// G_m(y) = w_y exp(-i m phi_{0,y}) X_y[m mod N_y], with X_y[N - k] = conj X_y[k]
// (the m-aliasing fold of Eq. 26 for m >= N_y / 2).
template <typename T>
__device__ __forceinline__ C2<T> ring_coef(const C2<T>* __restrict__ spec, const C2<T>* __restrict__ etab,
                                           const RingInfo& R, int m, int b, long long nspec, int use_w) {
  const int N = R.nphi, H = N >> 1;
  const int k = m % N;
  const C2<T>* X = spec + (long long)b * nspec + R.specoff;
  const C2<T> x = (k <= H) ? X[k] : cconj(X[N - k]);
  C2<T> g = cmul(x, etab[R.etab + ((long long)R.sigma * m) % (2LL * N)]);
  if (use_w) g = cscale(g, (T)R.w);
  return g;
}

// A general step of a chain in the state registers of both phases (n1, n2 as
// hi and lo parts).  A chain that has not started (l < lc) holds its start
// values there and gives zero; at lc it gives the second of them.  WAIT false:
// the chain is past its start.
template <bool WAIT>
__device__ __forceinline__ float general_step(GridState& g, Df t, int l, int lc) {  // t = c_l z
  RecurG r{Df{g.s1, g.f1}, Df{g.s2, g.f2}};
  float v = r.step(t);
  if constexpr (WAIT) {
    const bool run = l > lc;
    if (run) g = GridState{r.n1.hi, r.n1.lo, r.n2.hi, r.n2.lo};
    v = run ? v : l == lc ? df_real(Df{g.s1, g.f1}) : 0.f;
  } else {
    g = GridState{r.n1.hi, r.n1.lo, r.n2.hi, r.n2.lo};
  }
  return v;
}
// the state before the start, from the stored (mu_{lc-1}, mu_lc) as (hi, lo, hi, lo)
__device__ __forceinline__ GridState start_state(float4 st, float scale) {
  return GridState{scale * st.z, scale * st.w, scale * st.x, scale * st.y};
}

// The two chains of one lane.  One state serves both phases: general before
// the group's grid start, grid (s, f) from it on.  Grid steps take both chains
// packed (f32x2).  Values are scaled by S, a power of two.
template <int S>
struct Chains2 {
  static constexpr float kC = kGridC * S;
  GridState2 g;
  F2 zh, zl;
  int lca = 0x7fffffff, lcb = 0x7fffffff;  // starts (INT_MAX: none)
  int lmin, lmax_c;  // the warp's earliest and latest start
  int lg = 0x7fffffff;  // the group's aligned grid start
  int m;

  __device__ __forceinline__ void init(const float2* __restrict__ zf, const int* __restrict__ lc_tab,
                                       const float4* __restrict__ start, const int* __restrict__ lgrid, int ngrid,
                                       int npair, int lmax, int m_, int grp, int lane) {
    m = m_;
    const int pa = grp * 64 + lane, pb = pa + 32;
    const long long ca = (long long)m * npair + pa;
    float2 za = make_float2(0.f, 0.f), zb = za;
    GridState a{0.f, 0.f, 0.f, 0.f}, b = a;
    if (pa < npair) {
      lca = lc_tab[ca];
      za = zf[pa];
      a = start_state(start[ca], (float)S);
      lg = grid_start(m, lgrid[(long long)m * ngrid + grp]);
    }
    if (pb < npair) {
      lcb = lc_tab[ca + 32];
      zb = zf[pb];
      b = start_state(start[ca + 32], (float)S);
    }
    if (lca > lmax) lca = 0x7fffffff;
    if (lcb > lmax) lcb = 0x7fffffff;
    zh = pk2(za.x, zb.x);
    zl = pk2(za.y, zb.y);
    g = grid_pack(a, b);
    lmin = __reduce_min_sync(0xffffffffu, min(lca, lcb));
    lmax_c = __reduce_max_sync(0xffffffffu, max(lca, lcb));
    lg = __reduce_min_sync(0xffffffffu, lg);  // lanes past npair follow the group
  }

  // mu_l .. mu_{l+7} of both chains, l - m a multiple of 8; cz: c_l .. c_{l+7}
  // as (hi, hi, lo, lo)
  __device__ __forceinline__ void steps8(const float4* cz, int l, float (&va)[8], float (&vb)[8]) {
    const F2 C = pk2(kC, kC);
    if (l > lg) {
      if (((l - m) & (kRegrid - 1)) == 0) regrid(g, C);
#pragma unroll
      for (int u = 0; u < 8; ++u) unpk2(grid_step(g, cz[u], zh, zl, C), va[u], vb[u]);
      return;
    }
    GridState a, b;
    grid_unpack(g, a, b);
    if (l == lg) {
      g = grid_pack(grid_enter(Df{a.s1, a.f1}, Df{a.s2, a.f2}, kC), grid_enter(Df{b.s1, b.f1}, Df{b.s2, b.f2}, kC));
#pragma unroll
      for (int u = 0; u < 8; ++u) unpk2(grid_step(g, cz[u], zh, zl, C), va[u], vb[u]);
      return;
    }
    Df za, zb;
    unpk2(zh, za.hi, zb.hi);
    unpk2(zl, za.lo, zb.lo);
    // the products c z first: they do not wait on the chains
    Df ta[8], tb[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const Df c{cz[u].x, cz[u].z};
      ta[u] = df_mul(c, za);
      tb[u] = df_mul(c, zb);
    }
    if (lmax_c >= l) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        va[u] = general_step<true>(a, ta[u], l + u, lca);
        vb[u] = general_step<true>(b, tb[u], l + u, lcb);
      }
    } else {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        va[u] = general_step<false>(a, ta[u], l + u, lca);
        vb[u] = general_step<false>(b, tb[u], l + u, lcb);
      }
    }
    g = grid_pack(a, b);
  }
};

// The plan-resident lambda table (HPX_PLAN_LAMBDA_TABLE): for every m and
// every group g of 32 consecutive ring pairs, rows l = lstart(m,g)..lmax of 32
// values mu_l (one per pair of the group), lstart = the group's earliest chain
// start; row r of (m, g) at tab[off(m,g) + 32 r].  Written once at plan time
// by the steps of the recomputing kernels (FP64 plans RecurD, the others Chain).
template <typename T> struct LamTab {
  const T* tab;
  const long long* off;
  const int* lstart;
  int ngroup;
};

template <typename T>
inline LamTab<T> lam_tab(const hpx_plan_s* p) {
  LamTab<T> tb;
  tb.tab = static_cast<const T*>(p->d_tab);
  tb.off = p->d_tab_off;
  tb.lstart = p->d_tab_lstart;
  tb.ngroup = p->ngroup;
  return tb;
}

// From this Nside the ring launches are split by size and run on two streams;
// below it they are bound by launch latency, and all rings are one launch (an FP64
// analysis + synthesis at Nside 32: 96 us with the belt and the caps apart, 78 us
// together).
constexpr int kRingSplitNside = 512;

// The launches of the second stream run beside those on the caller's
// stream: forked from the caller's stream before the launches and joined
// back after them, so the call stays ordered on the caller's stream (and
// captures into a graph as a fork and a join).  `which` picks the stream and
// events of the analysis (0) or the synthesis (1).
struct RingFork {
  cudaStream_t s, side;
  cudaEvent_t join_ev = nullptr;
  RingFork(const hpx_plan_s* p, int which, cudaStream_t s_, cudaError_t& e) : s(s_), side(s_) {
    if (!p->fft_streams || p->nside < kRingSplitNside || e != cudaSuccess) return;
    // a stream with a priority of its own keeps all its launches: on the second
    // stream, of default priority, the belt rings would wait behind the work that
    // the caller's is to overtake
    int prio = 0;
    if (cudaStreamGetPriority(s, &prio) != cudaSuccess || prio != 0) {
      cudaGetLastError();
      return;
    }
    cudaStream_t st = static_cast<cudaStream_t*>(p->fft_streams)[which];
    cudaEvent_t* ev = static_cast<cudaEvent_t*>(p->fft_events) + 2 * which;
    e = cudaEventRecord(ev[0], s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, ev[0], 0);
    if (e == cudaSuccess) {
      side = st;
      join_ev = ev[1];
    }
  }
  cudaError_t join(cudaError_t e) {
    if (!join_ev) return e;
    cudaError_t e2 = cudaEventRecord(join_ev, side);
    if (e2 == cudaSuccess) e2 = cudaStreamWaitEvent(s, join_ev, 0);
    return e != cudaSuccess ? e : e2;
  }
};

// launchers (FP64: hpx_fft.cu, hpx_legendre.cu; FP32: hpx_fft_f32.cu, hpx_legendre_f32.cu)
template <typename T>
cudaError_t launch_r2c(const hpx_plan_s* p, const T* map, cudaStream_t s);
template <typename T>
cudaError_t launch_c2r(const hpx_plan_s* p, T* map, bool scale_by_weight, cudaStream_t s);
// mfac multiplies every coefficient with m > 0 on its way out (analysis) or
// in (synthesis): 1 for the transforms, 2 and 1/2 for the gradients.
template <typename T>
cudaError_t launch_analysis(const hpx_plan_s* p, T* alm, bool use_weight, double mfac, cudaStream_t s,
                            int* nlaunch);
template <typename T>
cudaError_t launch_synthesis(const hpx_plan_s* p, const T* alm, double mfac, cudaStream_t s, int* nlaunch);
template <> cudaError_t launch_r2c<double>(const hpx_plan_s*, const double*, cudaStream_t);
template <> cudaError_t launch_r2c<float>(const hpx_plan_s*, const float*, cudaStream_t);
cudaError_t launch_r2c16(const hpx_plan_s* p, const float* map, cudaStream_t s);  // 16-bit single-product plans
template <> cudaError_t launch_c2r<double>(const hpx_plan_s*, double*, bool, cudaStream_t);
template <> cudaError_t launch_c2r<float>(const hpx_plan_s*, float*, bool, cudaStream_t);
// ring launches of a stage
template <typename T> int ring_launch_count(const hpx_plan_s* p);
template <> int ring_launch_count<double>(const hpx_plan_s*);
template <> int ring_launch_count<float>(const hpx_plan_s*);
template <> cudaError_t launch_analysis<double>(const hpx_plan_s*, double*, bool, double, cudaStream_t, int*);
template <> cudaError_t launch_analysis<float>(const hpx_plan_s*, float*, bool, double, cudaStream_t, int*);
template <> cudaError_t launch_synthesis<double>(const hpx_plan_s*, const double*, double, cudaStream_t, int*);
template <> cudaError_t launch_synthesis<float>(const hpx_plan_s*, const float*, double, cudaStream_t, int*);

// plan-time table builders (hpx_fft.cu, hpx_legendre.cu)
template <typename T>
cudaError_t build_fft_tables(hpx_plan_s* p, cudaStream_t s);
template <> cudaError_t build_fft_tables<double>(hpx_plan_s*, cudaStream_t);
template <> cudaError_t build_fft_tables<float>(hpx_plan_s*, cudaStream_t);
cudaError_t build_fft_tables16(hpx_plan_s* p, cudaStream_t s);
cudaError_t build_recurrence_tables(hpx_plan_s* p, cudaStream_t s);
template <typename T>
cudaError_t build_lambda_table(hpx_plan_s* p, cudaStream_t s);

// tensor-core Legendre stages (hpx_tc.cu): plan-time column table, operand
// buffers and TMA descriptors; per launch of up to tc_channels_per_launch
// channels from b0, an operand pack and then the tile kernel.  The analysis
// pack reads the ring spectra and the tile kernel writes alm; the synthesis
// pack reads alm and the tile kernel writes the ring workspace d_F.  Both
// stages pack every channel group of the transform (launch_pack_tc per group,
// launch_pack_at_tc all, into the groups' Gt / At regions) and then run
// one tile launch over all of them (launch_tile_tc / launch_synthesis_tc with
// nb up to the plan's nbatch).
// The 16-bit dtypes (HPX_F32_BF16 ...) have only this path; their tables
// (row and column, hi and for x3 lo parts) are built here too.
int tc_columns(int nbatch, int cap);  // N of a tile for nbatch channels, at most cap per launch
int tc_mode_of(int dtype, unsigned flags);  // 0 3xTF32, 1 one 16-bit product, 2 16-bit x3; -1 none
size_t tc_extra_bytes_estimate(int nside, int lmax, int mmax, int nbatch, int mode, bool host_tables, bool streamed);
cudaError_t build_tc(hpx_plan_s* p, cudaStream_t s);
int tc_channels_per_launch(const hpx_plan_s* p, bool synthesis);
cudaError_t launch_pack_tc(hpx_plan_s* p, int b0, int nb, bool use_weight, cudaStream_t s);
cudaError_t launch_tile_tc(hpx_plan_s* p, float* alm, int b0, int nb, double mfac, cudaStream_t s);
cudaError_t launch_pack_at_tc(hpx_plan_s* p, const float* alm, double mfac, cudaStream_t s);
cudaError_t launch_synthesis_tc(hpx_plan_s* p, int b0, int nb, cudaStream_t s);
// lambda generated in the kernel (hpx_gen.cu): the analysis reads the packed
// operand Gt (launch_pack_tc; launch_pack_gen for the FP32 plans, whose operand
// buffers build_gen makes), the synthesis At, as the table tiles do
cudaError_t build_gen(hpx_plan_s* p, int parts, cudaStream_t s);
size_t gen_extra_bytes_estimate(int nside, int mmax, int nbatch, int parts);
int gen_parts_of(int nside, int lmax, int mmax, int nbatch, int dtype, unsigned flags);
bool gen_analysis_pays(int nside, int lmax, int mmax, int n);
// whether this call's analysis (of p->nbatch channels, of a view fewer than the plan's) takes them
inline bool gen_analysis(const hpx_plan_s* p) {
  return p->gen_parts == 3 && gen_analysis_pays(p->nside, p->lmax, p->mmax, p->nbatch);
}
// the plan as the staged wide analysis of a streamed split-product plan sees it; false if this call does not take it
bool staged_view(const hpx_plan_s* p, cudaStream_t s, hpx_plan_s* view);
cudaError_t launch_pack_gen(hpx_plan_s* p, int b0, int nb, bool use_weight, cudaStream_t s);
cudaError_t launch_gen_analysis(const hpx_plan_s* p, float* alm, double mfac, cudaStream_t s);
cudaError_t launch_gen_synthesis(const hpx_plan_s* p, cudaStream_t s);
void free_tc_host(hpx_plan_s* p);  // out-of-core resources (pinned tables, stream, events)

}  // namespace hpx
