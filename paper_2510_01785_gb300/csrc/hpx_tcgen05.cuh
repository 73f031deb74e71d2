// Device helpers shared by the tensor-core kernels (hpx_tc.cu, hpx_gen.cu):
// mbarriers with bounded waits, TMA loads, tcgen05 products and tensor-memory
// access in inline PTX, and the operand element types.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "hpx_internal.cuh"

namespace hpx {
namespace {

constexpr unsigned long long kWaitNs = 1000000000ull;  // 1 s per wait
// 16-bit lambda tables hold 2^9 lambda (|lambda_lm| <= sqrt((2l+1)/4pi) < 64
// for l < 25000, so 2^9 |lambda| < 2^15 stays in FP16 range), which keeps
// the FP16 remainder parts of small values out of the subnormal range; the
// epilogues multiply by 2^-9.
constexpr double kLamScale = 512.0;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Wait for the phase of `bar` with the given parity.  Gives up (false) when
// another thread of the CTA has raised the abort flag (if watch_abort) or
// after kWaitNs, raising the flag itself.
__device__ bool wait_phase(uint64_t* bar, uint32_t parity, volatile int* abort_flag, bool watch_abort) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  for (unsigned i = 1; i < (1u << 31); ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 63u) == 0) {
      if (watch_abort && *abort_flag) return false;
      if (global_ns() - t0 > kWaitNs) break;
    }
  }
  *abort_flag = 1;
  return false;
}
__device__ __forceinline__ void tma_load_2d(void* dst, const void* map, int c0, int c1, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(smem_u32(bar))
      : "memory");
}
// Shared-memory matrix descriptor of a K-major operand in the 128-byte
// swizzle: rows of 128 bytes, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
__device__ __forceinline__ void umma_tf32(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void umma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
// The same product twice with one A: the first keeps A's slice in the collector
// buffer, the second takes it from there (one read of A from shared memory).
__device__ __forceinline__ void umma_f16_pair(uint32_t d, uint64_t a, uint64_t b0, uint64_t b1, uint32_t idesc,
                                              uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %5, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], %1, %2, %4, p;\n"
      " tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%0], %1, %3, %4, 1;\n}" ::"r"(d),
      "l"(a), "l"(b0), "l"(b1), "r"(idesc), "r"(acc));
}
// A operand in tensor memory (lane = row, one 32-bit column per K element)
__device__ __forceinline__ void umma_tf32_ta(uint32_t d, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}" ::"r"(d),
      "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
// 16 consecutive accumulator columns of this warp's 32 TMEM lanes (complete
// after tmem_wait_ld).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// 32 consecutive columns of this warp's 32 TMEM lanes, complete on return.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
      "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]),
      "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]),
      "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// x rounded to the nearest TF32 value (ties away from zero): the 13 low
// mantissa bits rounded into the upper 19.  Finite inputs of table and
// spectrum magnitude only (no overflow to infinity can occur there).
__device__ __forceinline__ float tf32_rn(float x) {
  return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
}
// The part of x the tensor cores drop (they read the TF32 truncation of x),
// exact in FP32, itself rounded to TF32.
__device__ __forceinline__ float tf32_rem(float x) {
  return tf32_rn(x - __uint_as_float(__float_as_uint(x) & 0xFFFFE000u));
}
__device__ __forceinline__ float4 tf32_rem4(float4 x) {
  return make_float4(tf32_rem(x.x), tf32_rem(x.y), tf32_rem(x.z), tf32_rem(x.w));
}

// ---------------------------------------------------------------------------
// operand element types
// ---------------------------------------------------------------------------
// float: FP32 tables and operands; the products are 3xTF32 with the
//   remainders made in shared memory (mode 0).
// __nv_bfloat16 / __half: 16-bit tables and operands (kind::f16 products,
//   FP32 accumulation); the hi part, and for the x3 modes the lo part
//   lo = x - hi rounded again, are stored (modes 1 and 2).
// A row of any operand tile is 128 bytes: 32 floats or 64 16-bit values.
template <typename E> struct Elt;
template <> struct Elt<float> {
  static constexpr int kw = 32;
  static __device__ __forceinline__ float from_float(float v) { return v; }
  static __device__ __forceinline__ float to_float(float v) { return v; }
};
template <> struct Elt<__nv_bfloat16> {
  static constexpr int kw = 64;
  static __device__ __forceinline__ __nv_bfloat16 from_float(float v) { return __float2bfloat16_rn(v); }
  static __device__ __forceinline__ float to_float(__nv_bfloat16 v) { return __bfloat162float(v); }
};
template <> struct Elt<__half> {
  static constexpr int kw = 64;
  static __device__ __forceinline__ __half from_float(float v) { return __float2half_rn(v); }
  static __device__ __forceinline__ float to_float(__half v) { return __half2float(v); }
};

// Operand value v (already scaled) into row n of a tile column: hi at row n,
// and for x3 the remainder at row NN + n.
template <typename E>
__device__ __forceinline__ void put(E* col, int n, int NN, float v, bool x3) {
  constexpr int KW = Elt<E>::kw;
  const E h = Elt<E>::from_float(v);
  col[(long long)n * KW] = h;
  if (x3) col[(long long)(NN + n) * KW] = Elt<E>::from_float(v - Elt<E>::to_float(h));
}

// Power of two s with s * bound <= 2^14, from the channel's recorded largest
// component |x| (bit pattern of a non-negative float) times sfac, so that
// FP16 operands stay in range; 1 without a record (FP32 operands) or for an
// all-zero channel.
__device__ __forceinline__ float chan_scale(const unsigned* bmax, int b, float sfac) {
  if (!bmax) return 1.f;
  const float amax = __uint_as_float(bmax[b]) * sfac;
  if (!(amax > 0.f) || !(amax < 3.0e38f)) return 1.f;
  int e;
  frexpf(amax, &e);  // amax < 2^e
  return ldexpf(1.f, min(14 - e, 126));  // 2^126 at most, so that the scale and its inverse are normal
}

}  // namespace
}  // namespace hpx
