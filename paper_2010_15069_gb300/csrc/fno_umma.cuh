// tcgen05 building blocks shared by the Fourier neural operator's tensor-core
// kernels (fno_tc.cu, fno_dft.cu, fno_layer.cu, fno_head.cu): K-major bfloat16
// operands in shared memory with the 128-byte swizzle, MMA issue and commit,
// tensor-memory allocation and loads, and the split of float32 values into
// bfloat16 terms.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "async_copy.cuh"

namespace spgpe {
namespace fno {

constexpr int kTcRows = 128;              // points per tile (MMA M)
constexpr int kKBlock = 64;               // bfloat16 per 128-byte swizzled row
constexpr int kRowBytes = 128;

__device__ __forceinline__ uint32_t sw128(int row, int chunk) {
  return (uint32_t)row * kRowBytes + ((uint32_t)(chunk ^ (row & 7)) << 4);
}

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (stride byte offset), descriptor version 1.
__device__ __forceinline__ uint64_t sw128_desc(const void *base) {
  const uint64_t a = smem_addr(base);
  return ((a >> 4) & 0x3FFFull) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}

// Instruction descriptor of kind::f16: float32 accumulator, bfloat16 A and
// B, both K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_bf16(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(slot)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D (TMEM) [+]= A (smem) x B (smem)
__device__ __forceinline__ void umma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive on the mbarrier once every MMA this thread issued has completed.
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}

// 16 consecutive 32-bit columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// 8 columns.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16(__nv_bfloat16 a, __nv_bfloat16 b) {
  return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

// Eight float32 values as three bfloat16 terms each (v = h + m + l, h =
// bf16(v), m = bf16(v - h), l = bf16(v - h - m): all 24 bits), packed into the
// 16-byte chunks of the three operand terms.
__device__ __forceinline__ uint32_t cvt_bf16x2(float lo, float hi) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&p);
}
__device__ __forceinline__ void split3(const float (&v)[8], uint4 &h, uint4 &m, uint4 &l) {
  uint32_t hw[4], mw[4], lw[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float a = v[2 * i], b = v[2 * i + 1];
    hw[i] = cvt_bf16x2(a, b);
    const float a1 = a - __uint_as_float(hw[i] << 16), b1 = b - __uint_as_float(hw[i] & 0xffff0000u);
    mw[i] = cvt_bf16x2(a1, b1);
    lw[i] = cvt_bf16x2(a1 - __uint_as_float(mw[i] << 16), b1 - __uint_as_float(mw[i] & 0xffff0000u));
  }
  h = make_uint4(hw[0], hw[1], hw[2], hw[3]);
  m = make_uint4(mw[0], mw[1], mw[2], mw[3]);
  l = make_uint4(lw[0], lw[1], lw[2], lw[3]);
}

// The same split with the first term on a fixed grid, for products whose sum
// must not pick up the tensor cores' rounding: with |v| <= 128, h = v to the
// nearest integer (8 bits, exact in bfloat16), m and l the rest.  Against a
// second operand split likewise on a grid of 2^-7, every h h' product and
// every partial sum of up to 1024 of them is a multiple of 2^-7 below 2^17:
// exact in float32 whatever the accumulator's rounding (which truncates: the
// errors of a plain split all have one sign, and a transform adds them up).
// The other products carry 2^-8 of the weight and go to an accumulator of
// their own.
__device__ __forceinline__ float grid_round(float v) { return __fadd_rn(__fadd_rn(v, 12582912.f), -12582912.f); }
__device__ __forceinline__ void split3_grid(const float (&v)[8], float c, uint4 &h, uint4 &m, uint4 &l) {
  uint32_t hw[4], mw[4], lw[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float a = v[2 * i] * c, b = v[2 * i + 1] * c;
    const float ah = grid_round(a), bh = grid_round(b);
    hw[i] = cvt_bf16x2(ah, bh);
    const float a1 = a - ah, b1 = b - bh;
    mw[i] = cvt_bf16x2(a1, b1);
    lw[i] = cvt_bf16x2(a1 - __uint_as_float(mw[i] << 16), b1 - __uint_as_float(mw[i] & 0xffff0000u));
  }
  h = make_uint4(hw[0], hw[1], hw[2], hw[3]);
  m = make_uint4(mw[0], mw[1], mw[2], mw[3]);
  l = make_uint4(lw[0], lw[1], lw[2], lw[3]);
}
// The power of two c that brings values of magnitude up to vmax below 128
// (from vmax's exponent; values below 2^-118 keep fewer bits), and 1/c.
__device__ __forceinline__ float grid_scale(float vmax) {
  const int e = max(8, (__float_as_int(vmax) >> 23) & 255);
  return __int_as_float((260 - e) << 23);
}
__device__ __forceinline__ float grid_unscale(float vmax) {
  const int e = max(8, (__float_as_int(vmax) >> 23) & 255);
  return __int_as_float((e - 6) << 23);
}

// D [+]= A B over one 64-wide K block with both operands split into three
// terms (term t of A at a + t aterm; the terms of B as 3 N consecutive rows),
// into three accumulators of N columns: the leading products h h' at d, h m' +
// m h' at d + N, h l' + m m' + l h' at d + 2N (the products dropped are below
// 2^-24 of the result).  B's terms lie side by side, so each term of A is
// multiplied by all it needs in one MMA of up to 3 N columns: three MMAs per
// step of 16 instead of six, each term of A read once.  3 N <= 256.  One
// thread issues it.
template <int N>
__device__ __forceinline__ void umma_split33(uint32_t d, const unsigned char *a, size_t aterm, const unsigned char *b,
                                             bool accumulate) {
  const uint64_t a0 = sw128_desc(a), a1 = sw128_desc(a + aterm), a2 = sw128_desc(a + 2 * aterm), bd = sw128_desc(b);
#pragma unroll
  for (int kk = 0; kk < kKBlock / 16; ++kk) {  // 16 bfloat16 = 32 bytes per step
    umma_bf16(d, a0 + 2 * kk, bd + 2 * kk, idesc_bf16(kTcRows, 3 * N), accumulate || kk > 0);
    umma_bf16(d + N, a1 + 2 * kk, bd + 2 * kk, idesc_bf16(kTcRows, 2 * N), 1);
    umma_bf16(d + 2 * N, a2 + 2 * kk, bd + 2 * kk, idesc_bf16(kTcRows, N), 1);
  }
}

}  // namespace fno
}  // namespace spgpe
