// Shared device helpers of the q4decode kernels (sm_100a).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels.h"

namespace q4d {

// ---- bf16 <-> f32 by bit pattern ------------------------------------------------
__device__ __forceinline__ float bf16_lo(uint32_t pair) { return __uint_as_float(pair << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t pair) { return __uint_as_float(pair & 0xffff0000u); }
__device__ __forceinline__ float bf16_to_f32(uint16_t h) { return __uint_as_float(((uint32_t)h) << 16); }

// round-to-nearest-even f32 -> bf16 bits
__device__ __forceinline__ uint16_t f32_to_bf16(float f) {
  uint16_t r;
  asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(r) : "f"(f));
  return r;
}
// {lo, hi} -> packed bf16x2 (lo in the low half)
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// ---- async copies ------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem_dst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gsrc) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(smem_dst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---- programmatic dependent launch (no-ops when the launch has no such attribute) ----
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---- tensor-core MMA: D(16x8,f32) += A(16x16,bf16,row) * B(16x8,bf16,col) -----------
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The same with a zero accumulator: D = A * B.
__device__ __forceinline__ void mma_bf16_first(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                               uint32_t b0, uint32_t b1) {
  const float z = 0.0f;
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(z));
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], const void* smem_row) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(smem_row)));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], const void* smem_row) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(smem_row)));
}

// ---- fragment-ordered GEMM operand ---------------------------------------------------
// The GEMM reads its activations as bf16 with every aligned chunk of 8 elements stored in the order {0,4,1,5,2,6,3,7}
// (so that a lane's 16 bytes are its B fragments of two k-steps), plus the sum of every group of 64 elements.
// Producers build both with these helpers, always with the same summation tree: ((e0+e1)+(e2+e3))+((e4+e5)+(e6+e7))
// per chunk, then a pairwise tree over the 8 chunks of the group.
//
// Scaling (the mma.sync kernels, OPERAND_FRAG).  Those kernels hand the packed codes to the tensor cores as they
// lie in the word: a 4-bit code in bits 0..3 of a half-word IS the bf16 subnormal q * 2^-133, and one in bits 4..7 is
// 16 q * 2^-133 (bits 0..7 of bf16 count in steps of 2^-133: the first normal binade has the subnormals' spacing), so
// unpacking is one AND.  The powers of two go into the activations, exactly: elements 0, 2, 4, 6 of a chunk are stored
// times 2^64, elements 1, 3, 5, 7 times 2^60.  A product then counts in 2^-69, which the fp32 result loses at the end;
// activations from 2^-50 to 2^63 keep every bit.  The group sums (times 2^-69) are three bf16 terms, 24 bits, laid out as
// a B fragment against the biases: 16 values per (256 features, request), 4 per lane t of a fragment row.
constexpr float kOperandUnscale = 590295810358705651712.0f;            // 2^69
constexpr float kOperandSumScale = 1.0f / 590295810358705651712.0f;    // 2^-69
constexpr int kOperandSumBytes = 32;                                    // per (256 features, request)
// Element offset of chunk c (8 features) of request r in an operand of K features: OPERAND_BLOCKED is [K/8][16][8] (all requests of a chunk side by side: the tcgen05 kernel copies a K-range as one
// block); OPERAND_FRAG is [K/64][2][2][32][8]: per group of 64 features and 8 requests, the two 16-byte halves that lane
// 4 (r % 8) + (c % 8) / 2 of a warp holds as its B fragments, 512 contiguous bytes per half.
__device__ __forceinline__ size_t operand_chunk_offset(int layout, int K, int r, int c) {
  if (layout == OPERAND_FRAG) return (((size_t)(c >> 3) * 4 + (r >> 3) * 2 + (c & 1)) * 32 + (r & 7) * 4 + ((c & 7) >> 1)) * 8;
  return ((size_t)c * 16 + r) * 8;
}
__device__ __forceinline__ uint4 permute_chunk(const uint4 v) {
  uint4 o;
  o.x = __byte_perm(v.x, v.z, 0x5410);
  o.y = __byte_perm(v.x, v.z, 0x7632);
  o.z = __byte_perm(v.y, v.w, 0x5410);
  o.w = __byte_perm(v.y, v.w, 0x7632);
  return o;
}
// one register of a permuted chunk times 2^64, or 2^60 for an odd register (exact)
__device__ __forceinline__ uint32_t scale_pair(uint32_t a, bool odd) {
  uint32_t f = odd ? ((127u + 60u) << 7) * 0x10001u : ((127u + 64u) << 7) * 0x10001u;
  __nv_bfloat162 r = __hmul2(*reinterpret_cast<__nv_bfloat162*>(&a), *reinterpret_cast<__nv_bfloat162*>(&f));
  return *reinterpret_cast<uint32_t*>(&r);
}
// a permuted chunk times {2^64, 2^60, 2^64, 2^60} by register (exact)
__device__ __forceinline__ uint4 scale_chunk(const uint4 v) {
  return make_uint4(scale_pair(v.x, false), scale_pair(v.y, true), scale_pair(v.z, false), scale_pair(v.w, true));
}
// sum of the 8 elements of a chunk that scale_chunk has scaled, times 2^64
__device__ __forceinline__ float scaled_chunk_sum(const uint4 v) {
  const float even = (__uint_as_float(v.x << 16) + __uint_as_float(v.x & 0xffff0000u)) + (__uint_as_float(v.z << 16) + __uint_as_float(v.z & 0xffff0000u));
  const float odd = (__uint_as_float(v.y << 16) + __uint_as_float(v.y & 0xffff0000u)) + (__uint_as_float(v.w << 16) + __uint_as_float(v.w & 0xffff0000u));
  return fmaf(16.0f, odd, even);
}
// what lane t of a fragment row holds of those 16 values: groups P, P + 1 with sums v0, v1 (times 2^-69); lanes 0, 1 (`outer`)
// the first and third terms, lanes 2, 3 the second terms and zeros
__device__ __forceinline__ uint2 sum_terms_fragment(float v0, float v1, bool outer) {
  const uint32_t t1 = pack_bf16x2(v0, v1);
  v0 -= bf16_lo(t1), v1 -= bf16_hi(t1);
  const uint32_t t2 = pack_bf16x2(v0, v1);
  v0 -= bf16_lo(t2), v1 -= bf16_hi(t2);
  return outer ? make_uint2(t1, pack_bf16x2(v0, v1)) : make_uint2(t2, 0u);
}
// group gi (0..3) of the 32 bytes of one (256 features, request): the sum, already times 2^-69, in three bf16 terms
__device__ __forceinline__ void store_sum_terms(unsigned char* dst, int gi, float v) {
  uint16_t* d = reinterpret_cast<uint16_t*>(dst) + (gi >> 1) * 4 + (gi & 1);
  const uint16_t t1 = f32_to_bf16(v);
  v -= bf16_to_f32(t1);
  const uint16_t t2 = f32_to_bf16(v);
  v -= bf16_to_f32(t2);
  d[0] = t1, d[2] = f32_to_bf16(v), d[8] = t2, d[10] = 0;
}
__device__ __forceinline__ float chunk_sum(const uint4 v) {  // v in natural order
  return ((bf16_lo(v.x) + bf16_hi(v.x)) + (bf16_lo(v.y) + bf16_hi(v.y))) +
         ((bf16_lo(v.z) + bf16_hi(v.z)) + (bf16_lo(v.w) + bf16_hi(v.w)));
}
// Sum over the 8 lanes of an aligned lane group (each lane holds one chunk of the same 64-element group).
__device__ __forceinline__ float group_sum_8lanes(float s) {
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  s += __shfl_xor_sync(0xffffffffu, s, 4);
  return s;
}

// Chunk c (8 features, natural order) of request r, and the sum of 64-feature group `group`, in the given layout.
__device__ __forceinline__ void store_operand_chunk(int layout, uint16_t* xp, int K, int r, int c, const uint4 v) {
  const uint4 pv = permute_chunk(v);
  *reinterpret_cast<uint4*>(xp + operand_chunk_offset(layout, K, r, c)) = layout == OPERAND_BLOCKED ? pv : scale_chunk(pv);
}
__device__ __forceinline__ void store_operand_sum(int layout, void* xs, int r, int group, float sum) {
  if (layout == OPERAND_BLOCKED)
    reinterpret_cast<float*>(xs)[(size_t)group * 16 + r] = sum;
  else
    store_sum_terms(reinterpret_cast<unsigned char*>(xs) + ((size_t)(group >> 2) * 16 + r) * kOperandSumBytes, group & 3, sum * kOperandSumScale);
}

// ---- warp reductions ----------------------------------------------------------------
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

}  // namespace q4d
