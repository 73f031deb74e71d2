// Ring Fourier stage of the FP32 plans (Sec. III-D Eq. 13 and 24, Sec. III-E).
//
// A ring of N = 4i real values is two complex transforms of length i:
//   z_e[n] = x[4n] + i x[4n+2],  z_o[n] = x[4n+1] + i x[4n+3],
// and the four real subsequences' spectra A, B, C, D that these hold give the
// ring's by one radix-4 step,
//   X[k + t i] = sum_r (-i)^(rt) W_N^(rk) A_r[k],  t = 0..3, k < i,
// in which t = 2 and 3 are the conjugates of X[2i-k] and X[i-k]: one thread
// forms all four bins from elements k and i - k.  The two transforms share
// every twiddle, chirp factor, kernel value, address and barrier, an element
// of both is one 16-byte word that a map's float4 already is, and additions
// are one instruction for both (f32x2).
//
// Length-i transforms: M = A A R points in shared memory, in place, radix A = 4
// (M to 128), 8 (to 512) or 16 twice, then radix R.  Powers of two directly;
// other i by Bluestein's convolution with M >= 2i - 1 and R any of 2..8, 10, 12,
// 14, 16 (M is 13% above 2i - 1 on average at Nside 1024; a power of two 40%).
// The convolution's forward transform leaves the spectrum in digit-reversed
// order, and the inverse (the same forward kernels on conjugates, digits in
// reverse) starts from that order: the radix-R pass, the product with the
// kernel spectrum and the inverse's radix-R pass happen in registers, and the
// kernel table is stored in the order in which the threads read it.  Half of
// the input is zero and half of the output unwanted; the first and the last
// radix-A passes are pruned to those halves.  What a pass reads from tables is
// loaded before the barrier that it starts with.
//
// Element n = (n1, n2, n3) of a transform (n3 < R) lives at n1 S1 + n2 S2 + n3,
// S2 odd and S1 = R mod 8: the lanes of every pass fall on distinct 16-byte bank
// groups, except in the first pass for R = 2, 4, 6, ... (two-way), and a
// thread's addresses are one base and one stride.  Rings of at most 32 pixels
// are direct sums.  Rings start on multiples of four pixels (and maps on 16
// bytes): whole float4 everywhere.
//
// Measured at Nside 1024, analysis and synthesis stage: 8 channels, lmax 3071,
// 0.446 -> 0.315 and 0.651 -> 0.53 ms; 64 channels, lmax 2047, 3.25 -> 2.16 and
// 4.22 -> 2.86 ms (map and spectra once: 0.12 and 0.97 ms), against radix-16
// Stockham passes over one transform of length 2i, M a power of two.  That one
// was bound by instruction issue (70% of slots; 90 million warp instructions for
// the larger cap rings of 4 channels, here 40); this one waits, at 16 warps a
// multiprocessor, on table and map loads (a third of the time), instruction
// fetch (a fifth: long straight code) and shared memory.  Measured and not kept:
// 96 or 80 registers for 5 or 6 CTAs (spills: 2.79 / 3.59 and 3.10 / 4.08 ms),
// two to four units a CTA behind common barriers (3.05 / 3.51 ms).
#include <type_traits>

#include "hpx_internal.cuh"

namespace hpx {
namespace {

__device__ __forceinline__ F2 sub2(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ F2 mulr2(F2 a, float c) {
  float x, y;
  unpk2(a, x, y);
  return pk2(x * c, y * c);
}
__device__ __forceinline__ F2 fmar2(F2 a, float c, F2 d) {
  float x, y, u, v;
  unpk2(a, x, y);
  unpk2(d, u, v);
  return pk2(fmaf(x, c, u), fmaf(y, c, v));
}

// Kernel builds by launch: the belt (a power of two, no convolution), cap rings
// of at most 128 threads, larger ones (radices from 10).  Threads of a CTA at
// most, and CTAs of that size a multiprocessor: 128 registers a thread.
enum Kind { kBelt, kCaps, kBigCaps };
constexpr int max_threads(Kind k) { return k == kBigCaps ? 256 : 128; }
constexpr int min_ctas(Kind k) { return k == kBigCaps ? 2 : 4; }

// An element of the two transforms.
struct __align__(16) X2 {
  F2 re, im;
};
using C64 = double2;  // of one FP64 transform (the kernel spectra, once per plan)

__device__ __forceinline__ X2 xadd(X2 a, X2 b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ X2 xsub(X2 a, X2 b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
__device__ __forceinline__ X2 xaddi(X2 a, X2 b) { return {add2(a.re, b.im), sub2(a.im, b.re)}; }  // a - i b
__device__ __forceinline__ X2 xsubi(X2 a, X2 b) { return {sub2(a.re, b.im), add2(a.im, b.re)}; }  // a + i b
__device__ __forceinline__ X2 xmulr(X2 a, double c) { return {mulr2(a.re, (float)c), mulr2(a.im, (float)c)}; }
__device__ __forceinline__ X2 xfmar(X2 a, double c, X2 d) { return {fmar2(a.re, (float)c, d.re), fmar2(a.im, (float)c, d.im)}; }
// a (c - i s)
__device__ __forceinline__ X2 xrot(X2 a, double c, double s) {
  const F2 cc = pk2((float)c, (float)c), ss = pk2((float)s, (float)s), ns = pk2((float)-s, (float)-s);
  return {fma2(a.im, ss, mul2(a.re, cc)), fma2(a.re, ns, mul2(a.im, cc))};
}
// a factor of both
struct W2 {
  F2 x, y;
};
__device__ __forceinline__ W2 wide2(float2 w) { return {pk2(w.x, w.x), pk2(w.y, w.y)}; }
__device__ __forceinline__ X2 xcmul(X2 a, W2 w) {
  return {fma2(a.im, neg2(w.y), mul2(a.re, w.x)), fma2(a.re, w.y, mul2(a.im, w.x))};
}
__device__ __forceinline__ X2 xcmul(X2 a, float2 w) { return xcmul(a, wide2(w)); }
__device__ __forceinline__ X2 xcmulc(X2 a, float2 f) {  // conj(a) f
  const W2 w = wide2(f);
  return {fma2(a.im, w.y, mul2(a.re, w.x)), fma2(a.re, w.y, mul2(a.im, neg2(w.x)))};
}

__device__ __forceinline__ C64 xadd(C64 a, C64 b) { return cadd(a, b); }
__device__ __forceinline__ C64 xsub(C64 a, C64 b) { return csub(a, b); }
__device__ __forceinline__ C64 xaddi(C64 a, C64 b) { return cmk<C64>(a.x + b.y, a.y - b.x); }
__device__ __forceinline__ C64 xsubi(C64 a, C64 b) { return cmk<C64>(a.x - b.y, a.y + b.x); }
__device__ __forceinline__ C64 xmulr(C64 a, double c) { return cscale(a, c); }
__device__ __forceinline__ C64 xfmar(C64 a, double c, C64 d) { return cmk<C64>(fma(a.x, c, d.x), fma(a.y, c, d.y)); }
__device__ __forceinline__ C64 xrot(C64 a, double c, double s) { return cmk<C64>(a.x * c + a.y * s, a.y * c - a.x * s); }

// Forward DFTs of length R in registers, natural order in and out.
template <typename X> __device__ __forceinline__ void dft4(X& a, X& b, X& c, X& d) {
  const X u0 = xadd(a, c), u1 = xadd(b, d), w0 = xsub(a, c), w1 = xsub(b, d);
  a = xadd(u0, u1);
  c = xsub(u0, u1);
  b = xaddi(w0, w1);
  d = xsubi(w0, w1);
}
// Q = 3, 5, 7: sums and differences of the mirrored inputs
template <int Q, typename X> __device__ __forceinline__ void dft_odd(X (&v)[Q]) {
  constexpr double c3[1] = {-0.5}, s3[1] = {0.86602540378443864676};
  constexpr double c5[2] = {0.30901699437494742410, -0.80901699437494742410},
                   s5[2] = {0.95105651629515357212, 0.58778525229247312917};
  constexpr double c7[3] = {0.62348980185873353053, -0.22252093395631440429, -0.90096886790241912624},
                   s7[3] = {0.78183148246802980871, 0.97492791218182360702, 0.43388373911755812048};
  constexpr int H = (Q - 1) / 2;
  X t[H], s[H], y0 = v[0];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    t[j] = xadd(v[j + 1], v[Q - 1 - j]);
    s[j] = xsub(v[j + 1], v[Q - 1 - j]);
    y0 = xadd(y0, t[j]);
  }
#pragma unroll
  for (int k = 1; k <= H; ++k) {
    X a = v[0], b = s[0];
#pragma unroll
    for (int j = 0; j < H; ++j) {
      const int e = (j + 1) * k % Q, f = (e <= H ? e : Q - e) - 1;
      const double c = Q == 3 ? c3[f % 1] : Q == 5 ? c5[f % 2] : c7[f];
      const double sn = (e <= H ? 1.0 : -1.0) * (Q == 3 ? s3[f % 1] : Q == 5 ? s5[f % 2] : s7[f]);
      a = xfmar(t[j], c, a);
      b = j == 0 ? xmulr(s[0], sn) : xfmar(s[j], sn, b);
    }
    v[k] = xaddi(a, b);
    v[Q - k] = xsubi(a, b);
  }
  v[0] = y0;
}
// Even radices 2 Q: prime-factor map n = Q n1 + 2 n2, k = k1 mod 2, k2 mod Q
template <int Q, typename X> __device__ __forceinline__ void dft_2odd(X (&v)[2 * Q]) {
  X a[Q], b[Q];
#pragma unroll
  for (int n = 0; n < Q; ++n) {
    const X p = v[2 * n], q = v[(Q + 2 * n) % (2 * Q)];
    a[n] = xadd(p, q);
    b[n] = xsub(p, q);
  }
  dft_odd<Q>(a);
  dft_odd<Q>(b);
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    v[k % 2 == 0 ? k : k + Q] = a[k];  // k1 = 0: the even index that is k mod Q
    v[k % 2 == 1 ? k : k + Q] = b[k];
  }
}
// Radix 16 = 4 x 4.  NZ = 8: inputs 8..15 are zero.
template <int NZ, typename X> __device__ __forceinline__ void dft16(X (&v)[16]) {
  constexpr double h = 0.70710678118654752440, c1 = 0.92387953251128675613, s1 = 0.38268343236508977173;
  X y[4][4];
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) {
    if constexpr (NZ == 8) {
      const X a = v[n2], b = v[4 + n2];
      y[n2][0] = xadd(a, b);
      y[n2][1] = xaddi(a, b);
      y[n2][2] = xsub(a, b);
      y[n2][3] = xsubi(a, b);
    } else {
#pragma unroll
      for (int n1 = 0; n1 < 4; ++n1) y[n2][n1] = v[4 * n1 + n2];
      dft4(y[n2][0], y[n2][1], y[n2][2], y[n2][3]);
    }
  }
  // times W_16^(n2 k1); exponent 4 (-i) goes into the sums below
  y[1][1] = xrot(y[1][1], c1, s1);
  y[1][2] = xrot(y[1][2], h, h);
  y[1][3] = xrot(y[1][3], s1, c1);
  y[2][1] = xrot(y[2][1], h, h);
  y[2][3] = xrot(y[2][3], -h, h);
  y[3][1] = xrot(y[3][1], s1, c1);
  y[3][2] = xrot(y[3][2], -h, h);
  y[3][3] = xrot(y[3][3], -c1, -s1);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    const X u0 = k1 == 2 ? xaddi(y[0][k1], y[2][k1]) : xadd(y[0][k1], y[2][k1]);
    const X w0 = k1 == 2 ? xsubi(y[0][k1], y[2][k1]) : xsub(y[0][k1], y[2][k1]);
    const X u1 = xadd(y[1][k1], y[3][k1]), w1 = xsub(y[1][k1], y[3][k1]);
    v[k1] = xadd(u0, u1);
    v[k1 + 4] = xaddi(w0, w1);
    v[k1 + 8] = xsub(u0, u1);
    v[k1 + 12] = xsubi(w0, w1);
  }
}
// NZ < R (R = 4, 8, 16): inputs R / 2 .. are zero.
template <int R, int NZ = R, typename X> __device__ __forceinline__ void dft_r(X (&v)[R]) {
  if constexpr (R == 4 && NZ == 2) {
    const X a = v[0], b = v[1];
    v[0] = xadd(a, b);
    v[1] = xaddi(a, b);
    v[2] = xsub(a, b);
    v[3] = xsubi(a, b);
  } else if constexpr (R == 2) {
    const X a = v[0];
    v[0] = xadd(a, v[1]);
    v[1] = xsub(a, v[1]);
  } else if constexpr (R == 3 || R == 5 || R == 7) {
    dft_odd<R>(v);
  } else if constexpr (R == 4) {
    dft4(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 6 || R == 10 || R == 14) {
    dft_2odd<R / 2>(v);
  } else if constexpr (R == 8) {
    constexpr double h = 0.70710678118654752440;
    X u[4], w[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      u[r] = NZ == 4 ? v[r] : xadd(v[r], v[r + 4]);
      w[r] = NZ == 4 ? v[r] : xsub(v[r], v[r + 4]);
    }
    w[1] = xrot(w[1], h, h);
    w[3] = xrot(w[3], -h, h);
    dft4(u[0], u[1], u[2], u[3]);
    // w[2] times -i
    const X p0 = xaddi(w[0], w[2]), q0 = xsubi(w[0], w[2]), p1 = xadd(w[1], w[3]), q1 = xsub(w[1], w[3]);
    v[0] = u[0];
    v[2] = u[1];
    v[4] = u[2];
    v[6] = u[3];
    v[1] = xadd(p0, p1);
    v[5] = xsub(p0, p1);
    v[3] = xaddi(q0, q1);
    v[7] = xsubi(q0, q1);
  } else if constexpr (R == 12) {  // prime-factor map n = 3 n1 + 4 n2, k = k1 mod 4, k2 mod 3
    X a[4][3];
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < 4; ++n1) a[n1][n2] = v[(3 * n1 + 4 * n2) % 12];
      dft4(a[0][n2], a[1][n2], a[2][n2], a[3][n2]);
    }
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      dft_odd<3>(a[k1]);
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2) v[(9 * k1 + 4 * k2) % 12] = a[k1][k2];
    }
  } else if constexpr (R == 16) {
    dft16<NZ>(v);
  }
}

// The transform of a ring's length (fft32_shape) and its layout, radix A first.
template <int A> struct Shape {
  static constexpr int kTasks = A * A;  // of the radix-R pass
  int rad, nb;                          // nb = M / A = A rad
  int S1, S2;
  unsigned inv;  // j / rad = j inv >> 16 for j < 256
  __device__ __forceinline__ explicit Shape(int rad_) : rad(rad_), nb(A * rad_) {
    S2 = rad | 1;
    S1 = A * S2 + ((rad + (A == 4 ? 4 : 0)) & 7);
    inv = 65536u / (unsigned)rad + 1;
  }
  __device__ __forceinline__ int div(int j) const { return (int)(((unsigned)j * inv) >> 16); }
  // position of elements j + r nb (r S1 further on)
  __device__ __forceinline__ int first(int j) const {
    const int n2 = div(j);
    return n2 * S2 + (j - n2 * rad);
  }
  __device__ __forceinline__ int mid(int j) const { return (j / A) * S1 + (j % A) * S2; }
};
// natural order: one unused element after every 16
__device__ __forceinline__ int npos(int n) { return n + (n >> 4); }

template <int A> __device__ __forceinline__ void twiddle(X2 (&v)[A], float2 w) {  // v[r] w^r, at most four products deep
  const float2 w2 = cmul(w, w), w3 = cmul(w2, w);
  v[1] = xcmul(v[1], w);
  v[2] = xcmul(v[2], w2);
  v[3] = xcmul(v[3], w3);
  if constexpr (A >= 8) {
    const float2 w4 = cmul(w2, w2);
    v[4] = xcmul(v[4], w4);
    const float2 w5 = cmul(w3, w2), w6 = cmul(w3, w3), w7 = cmul(w4, w3);
    v[5] = xcmul(v[5], w5);
    v[6] = xcmul(v[6], w6);
    v[7] = xcmul(v[7], w7);
    if constexpr (A == 16) {
      const float2 w8 = cmul(w4, w4);
      v[8] = xcmul(v[8], w8);
      v[9] = xcmul(v[9], cmul(w8, w));
      v[10] = xcmul(v[10], cmul(w8, w2));
      v[11] = xcmul(v[11], cmul(w8, w3));
      v[12] = xcmul(v[12], cmul(w8, w4));
      v[13] = xcmul(v[13], cmul(w8, w5));
      v[14] = xcmul(v[14], cmul(w8, w6));
      v[15] = xcmul(v[15], cmul(w8, w7));
    }
  }
}
// Second pass of a forward transform (DIF: products, then twiddles) or last but
// one of an inverse (twiddles first), in place; w = W_(A R)^n3 of the thread.
template <int A, bool DIF>
__device__ __forceinline__ void pass2(X2* buf, const Shape<A>& sh, float2 w) {
  const int j = threadIdx.x;
  if (j >= sh.nb) return;
  const int n1 = sh.div(j), n3 = j - n1 * sh.rad;
  X2* at = buf + n1 * sh.S1 + n3;
  X2 v[A];
#pragma unroll
  for (int r = 0; r < A; ++r) v[r] = at[r * sh.S2];
  if (!DIF) twiddle<A>(v, w);
  dft_r<A>(v);
  if (DIF) twiddle<A>(v, w);
#pragma unroll
  for (int r = 0; r < A; ++r) at[r * sh.S2] = v[r];
}
// Radix-R pass, from its barrier on.  Bluestein: the spectrum's last digit, its
// product with the kernel's (both conjugated) and the inverse's first pass, in
// place.
template <int A, int R>
__device__ __forceinline__ void mid_blue(X2* buf, const Shape<A>& sh, const float2* __restrict__ bk) {
  constexpr int n = A * A;
  float2 k[R];
  int j = threadIdx.x;
  if (j < n) {
#pragma unroll
    for (int r = 0; r < R; ++r) k[r] = __ldg(bk + r * n + j);
  }
  __syncthreads();
  while (j < n) {
    X2* at = buf + sh.mid(j);
    X2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = at[r];
    dft_r<R>(v);
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = xcmulc(v[r], k[r]);
    j += blockDim.x;
    if (j < n) {
#pragma unroll
      for (int r = 0; r < R; ++r) k[r] = __ldg(bk + r * n + j);
    }
    dft_r<R>(v);
#pragma unroll
    for (int r = 0; r < R; ++r) at[r] = v[r];
  }
}
// Power of two: the last digit, to natural order.  blockDim.x >= A R and at
// least 64.
template <int A, int R>
__device__ __forceinline__ void mid_pow2(X2* buf, const Shape<A>& sh) {
  constexpr int n = A * A, Q = A < 16 ? 1 : R == 8 ? 2 : 4;
  __syncthreads();
  X2 v[Q][R];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int j = threadIdx.x + q * blockDim.x;
    if (j < n) {
      const X2* at = buf + sh.mid(j);
#pragma unroll
      for (int r = 0; r < R; ++r) v[q][r] = at[r];
      dft_r<R>(v[q]);
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int j = threadIdx.x + q * blockDim.x;
    if (j < n) {
      X2* at = buf + npos(j / A + A * (j % A));  // digits reversed
#pragma unroll
      for (int r = 0; r < R; ++r) at[r * (n + n / 16)] = v[q][r];
    }
  }
}

// A ring's transforms.  load(n) gives element n < i, before its chirp factor;
// in_buf if it reads buf.  Powers of two are left in natural order in buf, past a
// barrier; Bluestein's go, times the chirp and conjugated back, to put(n, x)
// (to_buf if that writes buf, which then ends with a barrier).
template <int A, Kind K, typename Load, typename Put>
__device__ __forceinline__ void ring_dft(X2* buf, int rad, int n4, const float2* __restrict__ tw_all,
                                         const float2* __restrict__ bk, const float2* __restrict__ C, bool in_buf,
                                         bool to_buf, Load load, Put put) {
  const Shape<A> sh(rad);
  const float2* tw = tw_all + fft32_tw_offset(A, rad);
  const int j = threadIdx.x;
  const bool mine = j < sh.nb, blue = K != kBelt && bk != nullptr;
  X2* at = buf + sh.first(j);
  float2 w1, w2;
  {
    X2 v[A];
    if (mine) {
      w1 = __ldg(tw + j);
      w2 = __ldg(tw + A * (j - sh.div(j) * rad));
      if (blue) {
        float2 c[A / 2];
#pragma unroll
        for (int r = 0; r < A / 2; ++r) {
          const int n = j + r * sh.nb;
          c[r] = n < n4 ? __ldg(C + n) : make_float2(0.f, 0.f);
          v[r] = n < n4 ? load(n) : X2{0, 0};
        }
#pragma unroll
        for (int r = 0; r < A / 2; ++r) v[r] = xcmul(v[r], c[r]);
        dft_r<A, A / 2>(v);
      } else {
#pragma unroll
        for (int r = 0; r < A; ++r) v[r] = load(j + r * sh.nb);
        dft_r<A>(v);
      }
      twiddle<A>(v, w1);
    }
    if (in_buf) __syncthreads();
    if (mine) {
#pragma unroll
      for (int r = 0; r < A; ++r) at[r * sh.S1] = v[r];
    }
  }
  __syncthreads();
  pass2<A, true>(buf, sh, w2);
  if (blue) {
    switch (rad) {
      case 2: mid_blue<A, 2>(buf, sh, bk); break;
      case 3: mid_blue<A, 3>(buf, sh, bk); break;
      case 4: mid_blue<A, 4>(buf, sh, bk); break;
      case 5: mid_blue<A, 5>(buf, sh, bk); break;
      case 6: mid_blue<A, 6>(buf, sh, bk); break;
      case 7: mid_blue<A, 7>(buf, sh, bk); break;
      case 8: mid_blue<A, 8>(buf, sh, bk); break;
      default:
        if constexpr (A == 16 && K == kBigCaps) {
          switch (rad) {
            case 10: mid_blue<A, 10>(buf, sh, bk); break;
            case 12: mid_blue<A, 12>(buf, sh, bk); break;
            case 14: mid_blue<A, 14>(buf, sh, bk); break;
            case 16: mid_blue<A, 16>(buf, sh, bk); break;
          }
        }
    }
    __syncthreads();
    pass2<A, false>(buf, sh, w2);
    float2 c[A / 2];
    if (mine) {
#pragma unroll
      for (int r = 0; r < A / 2; ++r) {
        const int n = j + r * sh.nb;
        c[r] = n < n4 ? __ldg(C + n) : make_float2(0.f, 0.f);
      }
    }
    __syncthreads();
    X2 v[A];
    if (mine) {
#pragma unroll
      for (int r = 0; r < A; ++r) v[r] = at[r * sh.S1];
      twiddle<A>(v, w1);
      dft_r<A>(v);
    }
    if (to_buf) __syncthreads();
    if (mine) {
#pragma unroll
      for (int r = 0; r < A / 2; ++r) {
        const int n = j + r * sh.nb;
        if (n < n4) put(n, xcmulc(v[r], c[r]));
      }
    }
    if (to_buf) __syncthreads();
  } else {
    switch (rad) {
      case 1: mid_pow2<A, 1>(buf, sh); break;
      case 2: mid_pow2<A, 2>(buf, sh); break;
      case 4: mid_pow2<A, 4>(buf, sh); break;
      case 8: mid_pow2<A, 8>(buf, sh); break;
    }
    __syncthreads();
  }
}

__device__ __forceinline__ X2 pair_of(float4 x) { return {pk2(x.x, x.y), pk2(x.z, x.w)}; }
// d + a w, d - a w: two roundings a component (a product first has three)
__device__ __forceinline__ float2 cfma(float2 a, float2 w, float2 d) {
  return make_float2(fmaf(a.x, w.x, fmaf(-a.y, w.y, d.x)), fmaf(a.x, w.y, fmaf(a.y, w.x, d.y)));
}
__device__ __forceinline__ float2 cfms(float2 a, float2 w, float2 d) {
  return make_float2(fmaf(-a.x, w.x, fmaf(a.y, w.y, d.x)), fmaf(-a.x, w.y, fmaf(-a.y, w.x, d.y)));
}
// (e, o) components of a pair
__device__ __forceinline__ float2 lo_of(X2 a) {
  float x, y, u, v;
  unpk2(a.re, x, y);
  unpk2(a.im, u, v);
  return make_float2(x, u);
}
__device__ __forceinline__ float2 hi_of(X2 a) {
  float x, y, u, v;
  unpk2(a.re, x, y);
  unpk2(a.im, u, v);
  return make_float2(y, v);
}

constexpr int kDirect = 8;  // rings of at most 4 kDirect pixels: direct sums

// A launch takes the belt (caps = 0), the two cap rings of every length 4i, i =
// ihi - blockIdx.y (1; the longest first), or all rings, the caps' from the longest,
// then the belt's (2).  blockIdx.x counts (ring, channel), the channels of a ring
// side by side, so that its tables are read from HBM once.
struct Ring32Args {
  const RingInfo* rings;
  const float2 *etab, *btab, *chirp, *tw;
  long long npix, nspec;
  int caps, ihi, nside, nb;
  __device__ __forceinline__ int ring(int r) const {
    if (caps == 0) return nside - 1 + r;
    const int i = ihi - (caps == 1 ? (int)blockIdx.y : r >> 1);
    if (i < 1) return nside - 1 + (r - 2 * (nside - 1));
    return (r & 1) ? 4 * nside - 1 - i : i - 1;
  }
};

// ---------------------------------------------------------------------------
// analysis: real ring -> half spectrum X_y[k], k = 0..N/2 (Eq. 13)
// ---------------------------------------------------------------------------
template <Kind K>
__global__ void __launch_bounds__(max_threads(K), min_ctas(K))
k_ring_r2c_f32(const float* __restrict__ map, float2* __restrict__ spec, const Ring32Args a,
               unsigned* __restrict__ bmax) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  X2* buf = reinterpret_cast<X2*>(smem_raw);
  const int t = threadIdx.x, b = blockIdx.x % a.nb, y = a.ring(blockIdx.x / a.nb);
  const RingInfo R = a.rings[y];
  const int N = R.nphi, n4 = N >> 2;
  const float2* E = a.etab + R.etab;
  const float* x = map + (long long)b * a.npix + R.start;
  float2* out = spec + (long long)b * a.nspec + R.specoff;
  float amax = 0.f;  // largest |component| written by this thread
  auto put = [&](int k, float2 X) {
    out[k] = X;
    amax = fmaxf(amax, fmaxf(fabsf(X.x), fabsf(X.y)));
  };
  if (n4 <= kDirect) {
    float* xs = reinterpret_cast<float*>(buf);
    if (t < N) xs[t] = x[t];
    __syncthreads();
    if (t <= 2 * n4) {
      float2 s[4] = {};
      for (int n = 0; n < N; n += 4)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float2 e = E[(2 * t * (n + u)) % (2 * N)];
          s[u] = make_float2(fmaf(xs[n + u], e.x, s[u].x), fmaf(xs[n + u], e.y, s[u].y));
        }
      put(t, cadd(cadd(s[0], s[1]), cadd(s[2], s[3])));
    }
  } else {
    const bool blue = K != kBelt && R.btab >= 0;
    const float2 *bk = blue ? a.btab + R.btab : nullptr, *C = blue ? a.chirp + fft32_chirp_offset(n4) : nullptr;
    auto load = [&](int n) { return pair_of(__ldg(reinterpret_cast<const float4*>(x) + n)); };
    auto keep = [&](int n, X2 z) { buf[npos(n)] = z; };
    const int rad = R.logm & 255;
    switch (R.logm >> 8) {
      case 4: ring_dft<4, K>(buf, rad, n4, a.tw, bk, C, false, true, load, keep); break;
      case 8: ring_dft<8, K>(buf, rad, n4, a.tw, bk, C, false, true, load, keep); break;
      case 16: ring_dft<16, K>(buf, rad, n4, a.tw, bk, C, false, true, load, keep); break;
    }
    // (e, o) of p = (Z[k] + conj Z[n4-k]) / 2 are A and B, of q = (Z[k] - conj
    // Z[n4-k]) / 2i C and D
    constexpr int U = 2;  // k in flight
    for (int k0 = t; k0 <= n4 / 2; k0 += U * blockDim.x) {
      float2 e[U][3];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = min(k0 + u * (int)blockDim.x, n4 / 2);
#pragma unroll
        for (int r = 0; r < 3; ++r) e[u][r] = __ldg(E + 2 * (r + 1) * k);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = k0 + u * blockDim.x;
        if (k > n4 / 2) break;
        const X2 z = buf[npos(k)], m = buf[npos(k ? n4 - k : 0)];
        const X2 p = {mulr2(add2(z.re, m.re), 0.5f), mulr2(sub2(z.im, m.im), 0.5f)};
        const X2 q = {mulr2(add2(z.im, m.im), 0.5f), mulr2(sub2(m.re, z.re), 0.5f)};
        const float2 A = lo_of(p), B = cmul(hi_of(p), e[u][0]), Cc = lo_of(q), D = hi_of(q);
        const float2 u0 = cfma(Cc, e[u][1], A), w0 = cfms(Cc, e[u][1], A), u1 = cfma(D, e[u][2], B), w1 = cfms(D, e[u][2], B);
        put(k, cadd(u0, u1));
        put(k + n4, make_float2(w0.x + w1.y, w0.y - w1.x));
        if (2 * k != n4) {
          put(2 * n4 - k, cconj(csub(u0, u1)));
          if (k) put(n4 - k, make_float2(w0.x - w1.y, -(w0.y + w1.x)));
        }
      }
    }
  }
  // the channel's largest spectrum component, for the 16-bit operand scale
  // of the tensor-core analysis (blockDim is a multiple of 32)
  if (bmax) {
    const unsigned wmax = __reduce_max_sync(0xffffffffu, __float_as_uint(amax));  // of non-negative floats
    if ((t & 31) == 0) atomicMax(bmax + b, wmax);
  }
}

// ---------------------------------------------------------------------------
// synthesis: F_m(y), m = 0..mmax -> ring values (Eq. 24)
// ---------------------------------------------------------------------------
// The ring's values are p_x = sum_{k<N} D[k] exp(2 pi i k x / N) with
// D[k] = sum_{m = k mod N} F_m e^{i m phi0} + sum_{m = -k mod N, m >= 1}
// conj(F_m e^{i m phi0}) (the aliasing fold; m = 0 contributes Re F_0).
// With m phi0 = pi sigma m / N every alias of bin k carries the phase of k and a
// sign: D[k] = e^(i pi sigma k / N) g(k),
//   g(k) = sum_t s^t F_(k + t N) + s sum_t s^t conj F_((t+1) N - k),  s = (-1)^sigma.
struct Fold {
  const float2* F;
  int N, mmax;
  float s;
  __device__ __forceinline__ float2 f(int m) const {  // F_m, with Im F_0 dropped (real maps)
    float2 v = F[m];
    if (m == 0) v.y = 0;
    return v;
  }
  // bins k0 .. of this thread (blockDim.x apart) into out; every load unconditional
  template <int U> __device__ __forceinline__ void bins(float2* out, int k0, int last) const {
    float2 g[U], c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) g[u] = c[u] = make_float2(0.f, 0.f);
    for (int m0 = 0; m0 <= mmax; m0 += 2 * N) {  // even and odd t, the latter with their sign
      float2 v[U][4];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = min(k0 + u * (int)blockDim.x, last);
        const int m[4] = {k + m0, k + N + m0, N - k + m0, 2 * N - k + m0};
#pragma unroll
        for (int r = 0; r < 4; ++r) v[u][r] = __ldg(F + min(m[r], mmax));
        if (m[0] == 0) v[u][0].y = 0.f;  // Im F_0 is dropped (real maps)
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (m[r] > mmax) v[u][r] = make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        g[u] = make_float2(g[u].x + fmaf(s, v[u][1].x, v[u][0].x), g[u].y + fmaf(s, v[u][1].y, v[u][0].y));
        c[u] = make_float2(c[u].x + fmaf(s, v[u][3].x, v[u][2].x), c[u].y + fmaf(s, v[u][3].y, v[u][2].y));
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (k0 + u * (int)blockDim.x <= last) out[k0 + u * blockDim.x] = join(g[u], c[u]);
  }
  __device__ __forceinline__ float2 join(float2 sa, float2 sb) const {
    return make_float2(fmaf(s, sb.x, sa.x), fmaf(-s, sb.y, sa.y));
  }
};

template <Kind K>
__global__ void __launch_bounds__(max_threads(K), min_ctas(K))
k_ring_c2r_f32(const float2* __restrict__ F, float* __restrict__ map, const Ring32Args a, int nring, int mmax,
               int scale_by_weight, int bins_at) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  X2* buf = reinterpret_cast<X2*>(smem_raw);
  float2* bins = reinterpret_cast<float2*>(smem_raw + bins_at);
  const int t = threadIdx.x, b = blockIdx.x % a.nb, y = a.ring(blockIdx.x / a.nb);
  const RingInfo R = a.rings[y];
  const int N = R.nphi, n4 = N >> 2;
  const float2* E = a.etab + R.etab;
  const int sig = R.sigma;
  const Fold fold{F + ((long long)b * nring + y) * (mmax + 1), N, mmax, sig ? -1.f : 1.f};
  const float sc = scale_by_weight ? (float)R.w : 1.f;
  float* out = map + (long long)b * a.npix + R.start;
  const bool staged = mmax >= N || n4 <= kDirect;  // folded into bins first
  if ((mmax + N) / N > 8) {                         // few bins, many aliases: one warp per bin
    const int lane = t & 31, nw = blockDim.x >> 5;
    // lane l takes the aliases t = l, l + 32, ...: all of one sign
    const float sgn = (lane & 1) ? fold.s : 1.f;
    for (int k = t >> 5; k <= 2 * n4; k += nw) {
      float2 sa = make_float2(0.f, 0.f), sb = sa;
      for (int m = k + lane * N; m <= mmax; m += 32 * N) sa = cadd(sa, fold.f(m));
      for (int m = (lane + 1) * N - k; m <= mmax; m += 32 * N) sb = cadd(sb, fold.F[m]);
      sa = cscale(sa, sgn);
      sb = cscale(sb, sgn);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        sa.x += __shfl_xor_sync(0xffffffffu, sa.x, off);
        sa.y += __shfl_xor_sync(0xffffffffu, sa.y, off);
        sb.x += __shfl_xor_sync(0xffffffffu, sb.x, off);
        sb.y += __shfl_xor_sync(0xffffffffu, sb.y, off);
      }
      if (lane == 0) bins[k] = fold.join(sa, sb);
    }
  } else if (staged) {
    for (int k = t; k <= 2 * n4; k += 4 * blockDim.x) fold.bins<4>(bins, k, 2 * n4);
  }
  if (staged) __syncthreads();
  if (n4 <= kDirect) {
    if (t < N) {
      float s0 = bins[0].x, s1 = 0.f, s2 = 0.f;
      for (int k = 1; k <= 2 * n4; ++k) {  // e^(i pi sigma k / N) e^(2 pi i k t / N)
        const float2 d = bins[k], e = E[((2 * t + sig) * k) % (2 * N)];
        if (k < 2 * n4) {
          s1 = fmaf(d.x, e.x, s1);
          s2 = fmaf(d.y, e.y, s2);
        } else {
          s0 += fmaf(d.x, e.x, d.y * e.y);
        }
      }
      out[t] = sc * (s0 + 2.f * (s1 + s2));
    }
    return;
  }
  // A_r[k] = W_N^(-rk) sum_t i^(rt) D[k + t n4]; the transforms of conj(A + i C)
  // and conj(B + i D) give the conjugates of p[4n] + i p[4n+2], p[4n+1] + i p[4n+3].
  // The four D share the phase of k but for e^(i pi sigma t / 4) (t = 0, 1) and
  // its conjugates (t = 2, 3: conj g(2 n4 - k), conj g(n4 - k)), so A_r takes the
  // one table value at (sigma + 2 r) k.
  constexpr int U = 4;  // k in flight (16 loads of F)
  const bool alias = mmax >= 2 * n4;
  for (int k0 = t; k0 <= n4 / 2; k0 += U * blockDim.x) {
    float2 e[U][4], g[U][4];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = min(k0 + u * (int)blockDim.x, n4 / 2);
#pragma unroll
      for (int r = 0; r < 4; ++r) e[u][r] = __ldg(E + (sig + 2 * r) * k);
      const int q[4] = {k, k + n4, 2 * n4 - k, n4 - k};
      if (staged) {
#pragma unroll
        for (int r = 0; r < 4; ++r) g[u][r] = bins[q[r]];
      } else {  // at most one alias of each kind; every load unconditional
#pragma unroll
        for (int r = 0; r < 4; ++r) g[u][r] = __ldg(fold.F + min(q[r], mmax));
      }
    }
    if (!staged) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = min(k0 + u * (int)blockDim.x, n4 / 2);
        const int q[4] = {k, k + n4, 2 * n4 - k, n4 - k};
        if (k == 0) g[u][0].y = 0.f;
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (q[r] > mmax) g[u][r] = make_float2(0.f, 0.f);
        if (alias) {
          float2 c[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) c[r] = __ldg(fold.F + min(N - q[r], mmax));
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (N - q[r] <= mmax) g[u][r] = fold.join(g[u][r], c[r]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = k0 + u * blockDim.x;
      if (k > n4 / 2) break;
      const float h = 0.70710678118654752440f;
      const float2 d0 = g[u][0];
      float2 d1 = g[u][1], d2 = cconj(g[u][2]), d3 = cconj(g[u][3]);
      if (sig) {
        d1 = make_float2(h * (d1.x - d1.y), h * (d1.x + d1.y));
        d2 = make_float2(d2.y, -d2.x);
        d3 = make_float2(h * (d3.x + d3.y), h * (d3.y - d3.x));
      }
      const float2 u0 = cadd(d0, d2), u1 = cadd(d1, d3), w0 = csub(d0, d2), w1 = csub(d1, d3);
      const float2 A = cmul(cadd(u0, u1), cconj(e[u][0])), Cc = cmul(csub(u0, u1), cconj(e[u][2]));
      const float2 B = cmul(make_float2(w0.x - w1.y, w0.y + w1.x), cconj(e[u][1]));
      const float2 D = cmul(make_float2(w0.x + w1.y, w0.y - w1.x), cconj(e[u][3]));
      // conj(A + i C) and, at n4 - k (where A and C are conjugated), A - i C
      const F2 ar = pk2(A.x, B.x), ai = pk2(A.y, B.y), cr = pk2(Cc.x, D.x), ci = pk2(Cc.y, D.y);
      buf[npos(k)] = X2{sub2(ar, ci), sub2(0, add2(ai, cr))};
      if (k > 0 && 2 * k != n4) buf[npos(n4 - k)] = X2{add2(ar, ci), sub2(ai, cr)};
    }
  }
  __syncthreads();
  const bool blue = K != kBelt && R.btab >= 0;
  const float2 *bk = blue ? a.btab + R.btab : nullptr, *C = blue ? a.chirp + fft32_chirp_offset(n4) : nullptr;
  auto load = [&](int n) { return buf[npos(n)]; };
  auto emit = [&](int n, X2 f) {
    const float2 e = lo_of(f), o = hi_of(f);
    reinterpret_cast<float4*>(out)[n] = make_float4(e.x * sc, o.x * sc, -e.y * sc, -o.y * sc);
  };
  const int rad = R.logm & 255;
  switch (R.logm >> 8) {
    case 4: ring_dft<4, K>(buf, rad, n4, a.tw, bk, C, true, false, load, emit); break;
    case 8: ring_dft<8, K>(buf, rad, n4, a.tw, bk, C, true, false, load, emit); break;
    case 16: ring_dft<16, K>(buf, rad, n4, a.tw, bk, C, true, false, load, emit); break;
  }
  if (!blue) {
#pragma unroll 4
    for (int n = t; n < n4; n += blockDim.x) emit(n, buf[npos(n)]);
  }
}

// ---------------------------------------------------------------------------
// plan-time tables
// ---------------------------------------------------------------------------
__global__ void k_tables32(int nside, float2* tw, float2* chirp, float2* etab) {
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
  if (blockIdx.y == 0) {
    for (int A = 4; A <= 16; A *= 2)
      for (int rad = 1; rad <= 16; ++rad)
        for (int j = tid; j < A * rad; j += step) {  // exp(-2 pi i j / M)
          double sn, cs;
          sincospi(-2.0 * (double)j / (double)(A * A * rad), &sn, &cs);
          tw[fft32_tw_offset(A, rad) + j] = make_float2((float)cs, (float)sn);
        }
  }
  for (int i = 1 + blockIdx.y; i <= nside; i += gridDim.y) {
    // E_N[r] = exp(-i pi r / N), r < 2N, of every ring length N = 4i
    float2* e = etab + 4LL * i * (i - 1);
    for (int r = tid; r < 8 * i; r += step) {
      double sn, cs;
      sincospi((double)r / (double)(4 * i), &sn, &cs);
      e[r] = make_float2((float)cs, (float)(-sn));
    }
    if (i == nside) break;
    for (int n = tid; n < i; n += step) {  // exp(-pi i n^2 / i), reduced exactly
      double sn, cs;
      sincospi(-(double)(((long long)n * n) % (2 * i)) / (double)i, &sn, &cs);
      chirp[fft32_chirp_offset(i) + n] = make_float2((float)cs, (float)sn);
    }
  }
}
// FFT of the kernel b[j] = exp(+pi i j^2 / i), |j| < i, zero elsewhere, over M
// points in FP64 (the passes of ring_dft); its conjugate over M is stored in the
// order that mid_blue reads.
template <int R>
__device__ __forceinline__ void mid64(const C64* buf, int ntask, float2* out, double scale) {
  for (int j = threadIdx.x; j < ntask; j += blockDim.x) {
    C64 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = buf[j * R + r];
    dft_r<R>(v);
#pragma unroll
    for (int r = 0; r < R; ++r) out[r * ntask + j] = make_float2((float)(v[r].x * scale), (float)(-v[r].y * scale));
  }
}
__global__ void k_kernel32(const RingInfo* __restrict__ rings, float2* btab) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C64* buf = reinterpret_cast<C64*>(smem_raw);
  const RingInfo R = rings[blockIdx.x];  // north cap ring i = blockIdx.x + 1
  const int i = R.nphi >> 2;
  if (R.btab < 0 || i <= kDirect) return;  // uniform over the block
  const int A = R.logm >> 8, rad = R.logm & 255, M = A * A * rad;
  for (int j = threadIdx.x; j < M; j += blockDim.x) {
    const long long jj = j < i ? j : (M - j < i ? M - j : -1);
    C64 v = cmk<C64>(0.0, 0.0);
    if (jj >= 0) {
      double sn, cs;
      sincospi((double)((jj * jj) % (2 * i)) / (double)i, &sn, &cs);
      v = cmk<C64>(cs, sn);
    }
    buf[j] = v;
  }
  __syncthreads();
  auto pass = [&](auto radix, int len) {  // within blocks of len
    constexpr int P = decltype(radix)::value;
    const int st = len / P;
    for (int j = threadIdx.x; j < M / P; j += blockDim.x) {
      const int blk = j / st, n0 = j - blk * st;
      C64* at = buf + blk * len + n0;
      C64 v[P];
#pragma unroll
      for (int r = 0; r < P; ++r) v[r] = at[r * st];
      dft_r<P>(v);
#pragma unroll
      for (int r = 0; r < P; ++r) {
        double sn, cs;
        sincospi(-2.0 * (double)(n0 * r) / (double)len, &sn, &cs);
        at[r * st] = cmul(v[r], cmk<C64>(cs, sn));
      }
    }
    __syncthreads();
  };
  for (int len = M; len > rad; len /= A) {
    if (A == 4) pass(std::integral_constant<int, 4>{}, len);
    if (A == 8) pass(std::integral_constant<int, 8>{}, len);
    if (A == 16) pass(std::integral_constant<int, 16>{}, len);
  }
  const int n = A * A;
  const double scale = 1.0 / (double)M;
  float2* out = btab + R.btab;
  switch (rad) {
    case 2: mid64<2>(buf, n, out, scale); break;
    case 3: mid64<3>(buf, n, out, scale); break;
    case 4: mid64<4>(buf, n, out, scale); break;
    case 5: mid64<5>(buf, n, out, scale); break;
    case 6: mid64<6>(buf, n, out, scale); break;
    case 7: mid64<7>(buf, n, out, scale); break;
    case 8: mid64<8>(buf, n, out, scale); break;
    case 10: mid64<10>(buf, n, out, scale); break;
    case 12: mid64<12>(buf, n, out, scale); break;
    case 14: mid64<14>(buf, n, out, scale); break;
    case 16: mid64<16>(buf, n, out, scale); break;
  }
}

// ---------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------
// Shared memory of ring length 4i: both layouts of its transform.
size_t shape_bytes(int i) {
  if (i <= kDirect) return 4 * kDirect * sizeof(float);
  const int code = fft32_shape(i), A = code >> 8, rad = code & 255, M = A * A * rad;
  const int a = A * (A * (rad | 1) + ((rad + (A == 4 ? 4 : 0)) & 7)), b = M + M / 16 + 1;
  return sizeof(X2) * (size_t)(a > b ? a : b);
}
int shape_threads(int i) {
  if (i <= kDirect) return 64;
  const int code = fft32_shape(i), nb = (code >> 8) * (code & 255);
  return nb < 64 ? 64 : (nb + 31) / 32 * 32;
}

struct Launch32 {
  int caps, ilo, n, threads, side;
  size_t smem, bins;  // bins: of the synthesis's fold
  dim3 grid(const hpx_plan_s* p) const {
    const int rings = caps == 0 ? 2 * p->nside + 1 : caps == 1 ? 2 : 4 * p->nside - 1;
    return dim3(rings * p->nbatch, caps == 1 ? n : 1);
  }
};
// Launch shapes.  From Nside 512 the belt rings (i = nside) are one launch and the
// cap rings three, by size (i up to nside / 2, 3/4 nside and nside - 1), each with
// the threads and shared memory of its own longest transform; the belt launch
// runs on the plan's second stream beside them.  Below, one launch of all rings
// (two to four CTAs of any one ring would fit anyway, and the second launch's
// latency is as long as the rings': Nside 64, 17 channels, 23 / 25 -> 19 / 20 us).
int ring_launches32(const hpx_plan_s* p, Launch32* out) {
  const int ns = p->nside;
  const bool split = ns >= kRingSplitNside;
  int k = 0;
  auto add = [&](int caps, int lo, int hi, int side) {  // lengths 4 lo .. 4 hi
    if (lo > hi) return;
    Launch32 L{caps, lo, hi - lo + 1, 64, side, 0, 0};
    for (int i = lo; i <= hi; ++i) {
      if (shape_bytes(i) > L.smem) L.smem = shape_bytes(i);
      if (shape_threads(i) > L.threads) L.threads = shape_threads(i);
      const size_t bytes = sizeof(float2) * (size_t)(2 * i + 2);  // a multiple of 16
      if ((p->mmax >= 4 * i || i <= kDirect) && bytes > L.bins) L.bins = bytes;
    }
    out[k++] = L;
  };
  if (split) {
    add(0, ns, ns, 1);
    add(1, 3 * ns / 4 + 1, ns - 1, 0);
    add(1, ns / 2 + 1, 3 * ns / 4, 0);
    add(1, 1, ns / 2, 0);
  } else {
    add(2, 1, ns, 0);
  }
  return k;
}
Ring32Args ring_args(const hpx_plan_s* p, const Launch32& L) {
  return {p->d_ring, (const float2*)p->d_etab, (const float2*)p->d_btab, (const float2*)p->d_chirp, (const float2*)p->d_tw,
          p->npix, p->nspec, L.caps, L.caps == 2 ? p->nside - 1 : L.ilo + L.n - 1, p->nside, p->nbatch};
}

}  // namespace

template <> int ring_launch_count<float>(const hpx_plan_s* p) {
  Launch32 ls[4];
  return ring_launches32(p, ls);
}

template <> cudaError_t build_fft_tables<float>(hpx_plan_s* p, cudaStream_t s) {
  const int ns = p->nside;
  k_tables32<<<dim3(4, ns < 256 ? ns : 256), 256, 0, s>>>(ns, (float2*)p->d_tw, (float2*)p->d_chirp, (float2*)p->d_etab);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && ns > kDirect + 1) {
    e = allow_max_smem(k_kernel32);
    if (e != cudaSuccess) return e;
    size_t smem = 0;
    for (int i = kDirect + 1; i < ns; ++i) {
      const size_t b = sizeof(C64) * (size_t)fft32_len(i);
      if (b > smem) smem = b;
    }
    k_kernel32<<<ns - 1, 256, smem, s>>>(p->d_ring, (float2*)p->d_btab);
    e = cudaGetLastError();
  }
  return e;
}

template <> cudaError_t launch_r2c<float>(const hpx_plan_s* p, const float* map, cudaStream_t s) {
  if (p->d_ring16) return launch_r2c16(p, map, s);  // 16-bit single products (hpx_fft.cu)
  cudaError_t e = allow_max_smem(k_ring_r2c_f32<kBelt>);
  if (e == cudaSuccess) e = allow_max_smem(k_ring_r2c_f32<kCaps>);
  if (e == cudaSuccess) e = allow_max_smem(k_ring_r2c_f32<kBigCaps>);
  // analyses with 16-bit operands or parts record each channel's largest
  // spectrum component here (zeroed first; for the parts the analysis that read the
  // last ones has left zeros)
  unsigned* bmax = p->tc_mode > 0 || gen_analysis(p) ? p->d_bmax : nullptr;
  if (e == cudaSuccess && bmax && p->tc_mode > 0) e = cudaMemsetAsync(bmax, 0, sizeof(unsigned) * p->nbatch, s);
  RingFork f(p, 0, s, e);
  Launch32 ls[4];
  const int nl = ring_launches32(p, ls);
  for (int i = 0; i < nl; ++i) {
    const Launch32& L = ls[i];
    if (e != cudaSuccess) continue;
    auto kern = !L.caps ? k_ring_r2c_f32<kBelt> : L.threads <= 128 ? k_ring_r2c_f32<kCaps> : k_ring_r2c_f32<kBigCaps>;
    kern<<<L.grid(p), L.threads, L.smem, L.side ? f.side : s>>>(
        map, (float2*)p->d_spec, ring_args(p, L), bmax);
    e = cudaGetLastError();
  }
  return f.join(e);
}

template <> cudaError_t launch_c2r<float>(const hpx_plan_s* p, float* map, bool scale_by_weight, cudaStream_t s) {
  cudaError_t e = allow_max_smem(k_ring_c2r_f32<kBelt>);
  if (e == cudaSuccess) e = allow_max_smem(k_ring_c2r_f32<kCaps>);
  if (e == cudaSuccess) e = allow_max_smem(k_ring_c2r_f32<kBigCaps>);
  RingFork f(p, 1, s, e);
  Launch32 ls[4];
  const int nl = ring_launches32(p, ls);
  for (int i = 0; i < nl; ++i) {
    const Launch32& L = ls[i];
    if (e != cudaSuccess) continue;
    auto kern = !L.caps ? k_ring_c2r_f32<kBelt> : L.threads <= 128 ? k_ring_c2r_f32<kCaps> : k_ring_c2r_f32<kBigCaps>;
    kern<<<L.grid(p), L.threads, L.smem + L.bins, L.side ? f.side : s>>>(
        (const float2*)p->d_F, map, ring_args(p, L), p->nring, p->mmax, scale_by_weight ? 1 : 0, (int)L.smem);
    e = cudaGetLastError();
  }
  return f.join(e);
}

}  // namespace hpx
