// Warp-level matrix fragments and packed float32 arithmetic shared by the kernels whose
// tiles of 16 rows belong to one warp (eloc.cu).
//
// Products run as mma.sync m16n8k16 (BF16 operands, FP32 accumulation).  Measured on GB300:
// bit-identical to tcgen05.mma for the same operands in the same order of 16-wide K steps,
// at 604 TFLOP/s over all SMs (about a third of tcgen05) -- far above what tiles of 16 x F
// can use, and without the round trip through shared memory, an mbarrier and tensor memory.
//
// Feature order.  A thread (g = lane / 4, q = lane % 4) of a tile owns rows g and g + 8 and,
// of every 16-feature chunk c, the four features 16 c + 4 q .. + 3.  As the A operand they
// are the K slots (2q, 2q+1, 2q+8, 2q+9) of K step c; as results they are columns (2q, 2q+1)
// of the column tiles 2c and 2c + 1.  The B fragments of load_wfrag() are permuted to match,
// so a result is the next product's A operand without leaving its thread.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace gna {

// ---- pairs of float32 in one 64-bit register (one instruction does both halves) ----
__device__ __forceinline__ uint64_t f2_pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t r, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t f2_dup(float a) { return f2_pack(a, a); }

// D (16 x 8) += A (16 x 16) B (16 x 8)
__device__ __forceinline__ void mma_16816(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// D (16 x 8) = A (16 x 16) B (16 x 8)
__device__ __forceinline__ void mma_16816_first(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

// Two float32 as packed BF16 hi = bf16(x) and lo = bf16(x - hi); m1 = (-1, -1).
__device__ __forceinline__ void split2(uint64_t m1, float a, float b, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  float ra, rb;
  f2_unpack(f2_fma(f2_pack(__uint_as_float(hi << 16), __uint_as_float(hi & 0xFFFF0000u)), m1, f2_pack(a, b)), ra,
            rb);
  const __nv_bfloat162 l = __floats2bfloat162_rn(ra, rb);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// Two float32 as packed BF16 hi + mid + lo: all 24 bits.
__device__ __forceinline__ void split3(uint64_t m1, float a, float b, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  float ra, rb;
  f2_unpack(f2_fma(f2_pack(__uint_as_float(hi << 16), __uint_as_float(hi & 0xFFFF0000u)), m1, f2_pack(a, b)), ra,
            rb);
  split2(m1, ra, rb, mid, lo);
}

// B fragments of W (2F x F, row-major float32, rounded to BF16), FC = F / 16: entry
// ((kc * FC + c) * 32 + lane) holds, for K step kc (16 rows of W) and output chunk c, the
// registers (b0, b1) of column tile 2c and (b0, b1) of column tile 2c + 1.
// term: 0 = bf16(w), 1 = bf16 of what that leaves, 2 = bf16 of what both leave.
// (an infinite w of a split in terms becomes one that saturates tanh as well, so that the terms stay numbers)
constexpr float kSaturatingW = 1e30f;
__device__ __forceinline__ float finite_w(float w) { return fabsf(w) == INFINITY ? copysignf(kSaturatingW, w) : w; }
__device__ __forceinline__ float wterm(float w, int term) {
  for (int t = 0; t < term; ++t) w -= __bfloat162float(__float2bfloat16_rn(w));
  return w;
}
template <int FC, bool TERMS = false>
__device__ __forceinline__ uint4 make_wfrag(const float* W, int kc, int c, int lane, int term) {
  constexpr int F = 16 * FC;
  const int n = lane >> 2, q = lane & 3;
  uint32_t r[4];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float* w = W + (size_t)(16 * kc + 4 * q) * F + 16 * c + 4 * (n >> 1) + 2 * h + (n & 1);
    float t[4] = {w[0], w[F], w[2 * F], w[3 * F]};
    if (TERMS)
#pragma unroll
      for (int i = 0; i < 4; ++i) t[i] = finite_w(t[i]);
    const __nv_bfloat162 x = __floats2bfloat162_rn(wterm(t[0], term), wterm(t[1], term));
    const __nv_bfloat162 y = __floats2bfloat162_rn(wterm(t[2], term), wterm(t[3], term));
    r[2 * h] = *reinterpret_cast<const uint32_t*>(&x);
    r[2 * h + 1] = *reinterpret_cast<const uint32_t*>(&y);
  }
  return make_uint4(r[0], r[1], r[2], r[3]);
}

template <typename T>
__device__ __forceinline__ T warp_sum_f(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---- asynchronous 16-byte copies global -> shared ----
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

}  // namespace gna
