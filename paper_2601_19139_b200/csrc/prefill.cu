// Prompt processing: the projections, the rotary embedding with the append of K and V, and causal attention for many
// tokens of one request at once.
//
// Projections.  y[t][j] = sum_k (s_jg q_jk + b_jg) x[t][k].  With the codes centred, s q + b = s (q - 8) + (b + 8 s): the
// scale has 8 significant bits and q - 8 needs 3 (or is a power of two), so s (q - 8) is EXACT in f16 (11 bits), as is
// a bf16 activation.  The products are therefore exact in an f16 tensor-core MMA with fp32 accumulation over the whole
// of K, and no group of 64 needs an accumulator of its own.  The second term, (b + 8 s) times the sum of the group's
// activations, joins the same accumulation as extra features: per group the pairs (b, X1), (b, X2), (8 s, X1),
// (8 s, X2) with X1 + X2 the fp32 sum in two f16 terms (6 % more features).  The range of f16 is met with powers of two:
// one per weight row (from the row's largest scale and bias) and one per token (from the row's largest activation and
// group sum), both taken out of the fp32 result.
#include <cuda_fp16.h>
#include <math.h>

#include "common.cuh"
#include "kernels.h"
#include "launch.h"
#include "tcgen05.cuh"

namespace q4d {

namespace {

// exponent e with 2^14 <= m * 2^e < 2^15 for a positive normal m (0 for m = 0), and 2^e as a float
__device__ __forceinline__ int range_exponent(float m) {
  if (!(m > 0.0f)) return 0;
  const int e = 14 - ((int)((__float_as_uint(m) >> 23) & 0xffu) - 127);
  return e < -110 ? -110 : (e > 110 ? 110 : e);
}
__device__ __forceinline__ float pow2f(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }
__device__ __forceinline__ uint32_t half2_bits(__half2 h) { return *reinterpret_cast<uint32_t*>(&h); }
__device__ __forceinline__ uint32_t pack_f16x2(float lo, float hi) { return half2_bits(__floats2half2_rn(lo, hi)); }

// ---- operand ---------------------------------------------------------------------------------------------------
// One CTA per row.  The row is held in registers (NCH chunks of 8 elements per thread).
template <int NCH, bool NORM>
__global__ void __launch_bounds__(256) prefill_pack_kernel(const uint16_t* x, int x_stride, const uint16_t* w, float eps, int K,
                                                            uint16_t* y, uint16_t* operand, float* inv_scale) {
  extern __shared__ float s_sums[];  // [K / 64]
  __shared__ float red[8];
  grid_launch_dependents();
  const int r = blockIdx.x, nch = K >> 3, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  grid_dependency_wait();
  uint4 v[NCH];
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    const int c = threadIdx.x + i * 256;
    v[i] = c < nch ? *reinterpret_cast<const uint4*>(x + (size_t)r * x_stride + c * 8) : make_uint4(0u, 0u, 0u, 0u);
  }
  auto block_reduce = [&](float a, bool is_max) -> float {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float b = __shfl_xor_sync(0xffffffffu, a, o);
      a = is_max ? fmaxf(a, b) : a + b;
    }
    if (lane == 0) red[warp] = a;
    __syncthreads();
    a = red[0];
#pragma unroll
    for (int i = 1; i < 8; ++i) a = is_max ? fmaxf(a, red[i]) : a + red[i];
    __syncthreads();
    return a;
  };
  if (NORM) {
    float ss = 0.0f;
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      const uint32_t e[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
      for (int j = 0; j < 4; ++j) ss = fmaf(bf16_lo(e[j]), bf16_lo(e[j]), ss), ss = fmaf(bf16_hi(e[j]), bf16_hi(e[j]), ss);
    }
    ss = block_reduce(ss, false);
    const float inv = 1.0f / sqrtf(ss / (float)K + eps);
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      const int c = threadIdx.x + i * 256;
      if (c < nch) {
        const uint4 wv = *reinterpret_cast<const uint4*>(w + c * 8);
        const uint32_t e[4] = {v[i].x, v[i].y, v[i].z, v[i].w}, ww[4] = {wv.x, wv.y, wv.z, wv.w};
        uint32_t o[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) o[j] = pack_bf16x2(bf16_lo(e[j]) * inv * bf16_lo(ww[j]), bf16_hi(e[j]) * inv * bf16_hi(ww[j]));
        v[i] = make_uint4(o[0], o[1], o[2], o[3]);
        if (y) *reinterpret_cast<uint4*>(y + (size_t)r * K + c * 8) = v[i];
      }
    }
  }
  float top = 0.0f;
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    const int c = threadIdx.x + i * 256;
    const uint32_t e[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
    for (int j = 0; j < 4; ++j) top = fmaxf(top, fmaxf(fabsf(bf16_lo(e[j])), fabsf(bf16_hi(e[j]))));
    const float gsum = group_sum_8lanes(chunk_sum(v[i]));  // 8 lanes hold one group of 64
    top = fmaxf(top, fabsf(gsum));
    if (c < nch && (c & 7) == 0) s_sums[c >> 3] = gsum;
  }
  top = block_reduce(top, true);
  const int ex = range_exponent(top);
  const float sc = pow2f(ex);
  if (threadIdx.x == 0) inv_scale[r] = pow2f(-ex);
  uint16_t* row = operand + (size_t)r * prefill_operand_stride(K);
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    const int c = threadIdx.x + i * 256;
    if (c < nch) {
      const uint4 pv = permute_chunk(v[i]);
      const uint32_t e[4] = {pv.x, pv.y, pv.z, pv.w};
      uint32_t o[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) o[j] = pack_f16x2(bf16_lo(e[j]) * sc, bf16_hi(e[j]) * sc);
      *reinterpret_cast<uint4*>(row + c * 8) = make_uint4(o[0], o[1], o[2], o[3]);
    }
  }
  // group sums in two f16 terms: per 16 groups {X1, X2, X1, X2}
  const int groups = K >> 6;
  for (int i = threadIdx.x; i < ((groups + 15) & ~15); i += 256) {
    const float X = i < groups ? s_sums[i] * sc : 0.0f;
    const __half x1 = __float2half_rn(X), x2 = __float2half_rn(X - __half2float(x1));
    uint16_t* d = row + K + (i >> 4) * 64 + (i & 15);
    d[0] = d[32] = __half_as_ushort(x1);
    d[16] = d[48] = __half_as_ushort(x2);
  }
}

// ---- projections -------------------------------------------------------------------------------------------------
// Persistent, one CTA per SM.  A tile is 128 weight rows (the lanes of tensor memory) x up to 256 tokens (columns); two
// accumulators of 256 columns let the epilogue of a tile run under the MMAs of the next.  Roles:
//   warp 0      producer: TMA loads of the tokens' operand, 64 features a stage (128-byte swizzle)
//   warp 1      MMA issue (one thread); owns the tensor-memory allocation
//   warps 2, 3  the power of two of each weight row of the next tile, the tokens' inverse scales
//   warps 4..7  epilogue (one per lane quarter of tensor memory)
//   warps 8..15 dequantisation: two threads per weight row, 32 codes each per stage, straight from global memory
//               (four stages of codes in registers ahead) into the swizzled A stage
// A dequantised code costs ~1.6 instructions, so a stage (128 x 64) costs the eight warps about 130 issue cycles per
// scheduler against 512 cycles of tensor time at 256 tokens.  Measured at 2048 tokens, gate/up of the 8B shape (24576 x
// 4096): 453 us = 0.91 PFLOP/s; as 128 passes of sixteen tokens the same projection took 3560 us.
constexpr int kPgThreads = 512;
constexpr int kPgStages = 4;
constexpr int kPgAStage = 128 * 128;  // 128 rows x 64 f16
constexpr int kPgBStage = 256 * 128;  // 256 tokens x 64 f16
constexpr int kPgSmem = kPgStages * (kPgAStage + kPgBStage) + 1024;

struct PgParams {
  const uint32_t* qw;
  const uint16_t* scales;
  const uint16_t* biases;
  const float* inv_scale;
  uint16_t* out;
  unsigned int* status;
  const int4* units;
  const int* n_units;
  int N, K, rows, n_tile, row_tiles, tok_tiles, out_stride, epilogue;
};

// D (128 x N, f32, tensor memory) (+)= A (128 x 16 f16) * B (N x 16 f16), both K-major in shared memory
__device__ __forceinline__ void umma_f16_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// K-major operand with 128-byte rows and the 128-byte swizzle: 8-row atoms 1024 bytes apart
__device__ __forceinline__ uint64_t desc_sw128(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(1024u >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void tmem_ld16f(uint32_t taddr, float (&v)[16]) {
  uint32_t u[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]), "=r"(u[9]),
        "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(u[i]);
}
__device__ __forceinline__ uint4 ldg_stream(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// 8 codes -> 8 f16 values s (q - 8) in the order 0,4,1,5,2,6,3,7
__device__ __forceinline__ uint4 dequant_word(uint32_t w, __half2 s2) {
  const __half2 c1032 = __float2half2_rn(1032.0f), c16th = __float2half2_rn(0.0625f), c72 = __float2half2_rn(-72.0f);
  auto f = [](uint32_t u) -> __half2 { return *reinterpret_cast<__half2*>(&u); };
  const uint32_t w8 = w >> 8;
  const __half2 a = __hsub2(f((w & 0x000f000fu) | 0x64006400u), c1032);            // 1024 + q - 1032
  const __half2 b = __hfma2(f((w & 0x00f000f0u) | 0x64006400u), c16th, c72);       // (1024 + 16 q) / 16 - 72
  const __half2 c = __hsub2(f((w8 & 0x000f000fu) | 0x64006400u), c1032);
  const __half2 d = __hfma2(f((w8 & 0x00f000f0u) | 0x64006400u), c16th, c72);
  return make_uint4(half2_bits(__hmul2(a, s2)), half2_bits(__hmul2(b, s2)), half2_bits(__hmul2(c, s2)), half2_bits(__hmul2(d, s2)));
}

struct PgTile {
  int row_tile, tok0, valid, expert;
};

__global__ void __launch_bounds__(kPgThreads, 1) prefill_gemm_kernel(const PgParams p, const __grid_constant__ CUtensorMap map_b) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[kPgStages], empty[kPgStages];
  __shared__ __align__(8) uint64_t d_full[2], d_empty[2], rs_full[2], rs_empty[2];
  __shared__ uint32_t s_tmem_base;
  __shared__ int s_rexp[2][128];
  __shared__ __align__(16) float s_inv[2][256];

  grid_launch_dependents();

  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* sA = smem;
  unsigned char* sB = smem + kPgStages * kPgAStage;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool grouped = p.units != nullptr, silu = p.epilogue == EPI_SILU_PACK;
  const int half_n = p.N >> 1, K = p.K;
  const int kb_main = K >> 6, kb_all = prefill_operand_stride(K) >> 6;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kPgStages; ++s) um_mbar_init(&full[s], 9), um_mbar_init(&empty[s], 1);
    for (int b = 0; b < 2; ++b)
      um_mbar_init(&d_full[b], 1), um_mbar_init(&d_empty[b], 4), um_mbar_init(&rs_full[b], 2), um_mbar_init(&rs_empty[b], 12);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)), "n"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = s_tmem_base;

  if (grouped) grid_dependency_wait();  // the list of units is the preceding kernel's
  const int total = p.row_tiles * (grouped ? *p.n_units : p.tok_tiles);
  auto tile_at = [&](int idx) -> PgTile {
    PgTile t;
    if (grouped) {
      const int u = idx / p.row_tiles;
      const int4 un = p.units[u];
      t.row_tile = idx - u * p.row_tiles, t.expert = un.x, t.tok0 = un.y, t.valid = un.z;
    } else {
      t.row_tile = idx / p.tok_tiles;
      t.tok0 = (idx - t.row_tile * p.tok_tiles) * p.n_tile;
      t.valid = min(p.n_tile, p.rows - t.tok0), t.expert = 0;
    }
    return t;
  };
  // row `lrow` of a tile in the tensor: with the SiLU epilogue each quarter holds 16 gate rows and the 16 matching up rows
  auto tensor_row = [&](const PgTile& t, int lrow) -> size_t {
    int r = t.row_tile * 128 + lrow;
    if (silu) {
      const int f = t.row_tile * 64 + (lrow >> 5) * 16 + (lrow & 15);
      r = (lrow & 16) ? half_n + f : f;
    }
    return (size_t)t.expert * p.N + r;
  };

  bool ok = true;
  if (warp == 0) {
    // ---- producer ----
    if (lane == 0) {
      if (!grouped) grid_dependency_wait();
      int kb = 0;
      for (int idx = blockIdx.x; idx < total && ok; idx += gridDim.x) {
        const PgTile t = tile_at(idx);
        for (int j = 0; j < kb_all; ++j, ++kb) {
          const int s = kb % kPgStages;
          if (!um_mbar_wait(&empty[s], (uint32_t)(((kb / kPgStages) & 1) ^ 1))) {
            ok = false;
            break;
          }
          um_mbar_expect_tx(&full[s], (uint32_t)(p.n_tile * 128));
          um_tma_2d(sB + s * kPgBStage, &map_b, j * 64, t.tok0, &full[s]);
        }
      }
      if (!ok && p.status) atomicExch(p.status, 3u);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---- MMA issue ----
    if (lane == 0) {
      // D f32, A and B f16, both K-major, M = 128
      const uint32_t idesc = (1u << 4) | ((uint32_t)(p.n_tile >> 3) << 17) | ((128u >> 4) << 24);
      int kb = 0, it = 0;
      for (int idx = blockIdx.x; idx < total && ok; idx += gridDim.x, ++it) {
        const int buf = it & 1;
        if (!um_mbar_wait(&d_empty[buf], (uint32_t)(((it >> 1) & 1) ^ 1))) ok = false;
        tc_fence_after();
        for (int j = 0; j < kb_all && ok; ++j, ++kb) {
          const int s = kb % kPgStages;
          if (!um_mbar_wait(&full[s], (uint32_t)((kb / kPgStages) & 1))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t da = desc_sw128(smem_u32(sA + s * kPgAStage)), db = desc_sw128(smem_u32(sB + s * kPgBStage));
#pragma unroll
          for (int ks = 0; ks < 4; ++ks)
            umma_f16_ss(tbase + (uint32_t)(buf * 256), da + (uint64_t)(ks * 2), db + (uint64_t)(ks * 2), idesc, (j | ks) != 0);
          umma_commit(&empty[s]);
        }
        if (ok) umma_commit(&d_full[buf]);
      }
      if (!ok && p.status) atomicExch(p.status, 3u);
    }
    __syncwarp();
  } else if (warp < 4) {
    // ---- row exponents and token scales, a tile ahead ----
    const int tid = threadIdx.x - 64;
    int it = 0;
    for (int idx = blockIdx.x; idx < total && ok; idx += gridDim.x, ++it) {
      const PgTile t = tile_at(idx);
      const int buf = it & 1;
      int ex[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const size_t off = tensor_row(t, tid + 64 * h) * (size_t)(K >> 6);
        uint32_t ms = 0, mb = 0;
#pragma unroll 8
        for (int g = 0; g < (K >> 6); g += 4) {
          const uint2 a = *reinterpret_cast<const uint2*>(p.scales + off + g), b = *reinterpret_cast<const uint2*>(p.biases + off + g);
          ms = __vmaxu2(ms, __vmaxu2(a.x & 0x7fff7fffu, a.y & 0x7fff7fffu));
          mb = __vmaxu2(mb, __vmaxu2(b.x & 0x7fff7fffu, b.y & 0x7fff7fffu));
        }
        const float fs = fmaxf(bf16_lo(ms), bf16_hi(ms)), fb = fmaxf(bf16_lo(mb), bf16_hi(mb));
        ex[h] = range_exponent(fmaxf(8.0f * fs, fb));
      }
      if (it == 0 && !grouped) grid_dependency_wait();
      if (!um_mbar_wait_warp(&rs_empty[buf], (uint32_t)(((it >> 1) & 1) ^ 1))) ok = false;
      s_rexp[buf][tid] = ex[0], s_rexp[buf][tid + 64] = ex[1];
      for (int i = tid; i < p.n_tile; i += 64) s_inv[buf][i] = i < t.valid ? p.inv_scale[t.tok0 + i] : 0.0f;
      __syncwarp();
      if (lane == 0) um_mbar_arrive(&rs_full[buf]);
    }
    if (!ok && lane == 0 && p.status) atomicExch(p.status, 3u);
  } else if (warp < 8) {
    // ---- epilogue ----
    const int q = warp - 4;
    const uint32_t lane_addr = tbase + ((uint32_t)(q * 32) << 16);
    if (!grouped) grid_dependency_wait();  // the output may still be read by the preceding kernels
    int it = 0;
    for (int idx = blockIdx.x; idx < total && ok; idx += gridDim.x, ++it) {
      const PgTile t = tile_at(idx);
      const int buf = it & 1;
      const uint32_t par = (uint32_t)((it >> 1) & 1);
      if (!um_mbar_wait_warp(&rs_full[buf], par) || !um_mbar_wait_warp(&d_full[buf], par)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const float rinv = pow2f(-s_rexp[buf][q * 32 + lane]);
      for (int c0 = 0; c0 < t.valid; c0 += 16) {
        float v[16];
        tmem_ld16f(lane_addr + (uint32_t)(buf * 256 + c0), v);
#pragma unroll
        for (int i = 0; i < 16; i += 4) {
          const float4 cs = *reinterpret_cast<const float4*>(&s_inv[buf][c0 + i]);
          v[i] = v[i] * rinv * cs.x, v[i + 1] = v[i + 1] * rinv * cs.y;
          v[i + 2] = v[i + 2] * rinv * cs.z, v[i + 3] = v[i + 3] * rinv * cs.w;
        }
        if (silu) {
          // lanes 0..15 hold gate rows, 16..31 the up rows of the same features.  Of columns c, c + 1 the lower half
          // takes c, the upper c + 1; then neighbours pair up so that a lane stores two features of one token.
#pragma unroll
          for (int i = 0; i < 16; i += 4) {
            float h[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              const float v0 = bf16_to_f32(f32_to_bf16(v[i + 2 * j])), v1 = bf16_to_f32(f32_to_bf16(v[i + 2 * j + 1]));
              const float got = __shfl_xor_sync(0xffffffffu, lane < 16 ? v1 : v0, 16);
              const float gt = lane < 16 ? v0 : got, up = lane < 16 ? got : v1;
              h[j] = (gt / (1.0f + expf(-gt))) * up;
            }
            const float other = __shfl_xor_sync(0xffffffffu, (lane & 1) ? h[0] : h[1], 1);
            const uint32_t o = (lane & 1) ? pack_bf16x2(other, h[1]) : pack_bf16x2(h[0], other);
            const int col = c0 + i + ((lane & 1) ? 2 : 0) + (lane >> 4);
            if (col < t.valid)
              *reinterpret_cast<uint32_t*>(p.out + (size_t)(t.tok0 + col) * p.out_stride + t.row_tile * 64 + q * 16 + (lane & 14)) = o;
          }
        } else {
          uint16_t* base = p.out + (size_t)t.tok0 * p.out_stride + t.row_tile * 128 + q * 32 + (lane & 30);
          uint32_t old[8];
          if (p.epilogue == EPI_RESIDUAL) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int col = c0 + 2 * i + (lane & 1);
              old[i] = col < t.valid ? *reinterpret_cast<const uint32_t*>(base + (size_t)col * p.out_stride) : 0u;
            }
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            // columns 2i, 2i + 1: even lanes keep the first, odd lanes the second, for two neighbouring rows each
            const float other = __shfl_xor_sync(0xffffffffu, (lane & 1) ? v[2 * i] : v[2 * i + 1], 1);
            uint32_t o = (lane & 1) ? pack_bf16x2(other, v[2 * i + 1]) : pack_bf16x2(v[2 * i], other);
            const int col = c0 + 2 * i + (lane & 1);
            if (p.epilogue == EPI_RESIDUAL) o = pack_bf16x2(bf16_lo(old[i]) + bf16_lo(o), bf16_hi(old[i]) + bf16_hi(o));
            if (col < t.valid) *reinterpret_cast<uint32_t*>(base + (size_t)col * p.out_stride) = o;
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) um_mbar_arrive(&d_empty[buf]), um_mbar_arrive(&rs_empty[buf]);
    }
    if (!ok && lane == 0 && p.status) atomicExch(p.status, 3u);
  } else {
    // ---- dequantisation ----
    const int tid = threadIdx.x - 256, lrow = tid >> 1, h = tid & 1;
    const int nsb = K >> 8;  // superblocks of four stages: 128 bytes of codes per row
    const uint32_t* qrow = nullptr;
    const uint16_t *srow = nullptr, *brow = nullptr;
    auto set_row = [&](const PgTile& t) {
      const size_t r = tensor_row(t, lrow);
      qrow = p.qw + r * (size_t)(K >> 3) + h * 4;
      srow = p.scales + r * (size_t)(K >> 6), brow = p.biases + r * (size_t)(K >> 6);
    };
    uint4 nxt[4];
    uint2 nsc;
    auto load_sb = [&](int sb) {
#pragma unroll
      for (int j = 0; j < 4; ++j) nxt[j] = ldg_stream(qrow + sb * 32 + j * 8);
      nsc = *reinterpret_cast<const uint2*>(srow + sb * 4);
    };
    if (blockIdx.x < total) {
      set_row(tile_at(blockIdx.x));
      load_sb(0);
    }
    // where this thread's four 16-byte chunks of a stage go
    unsigned char* a_row = sA + lrow * 128;
    int a_off[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) a_off[i] = ((h * 4 + i) ^ (lrow & 7)) << 4;
    int kb = 0, it = 0;
    for (int idx = blockIdx.x; idx < total && ok; idx += gridDim.x, ++it) {
      const int buf = it & 1;
      if (!um_mbar_wait_warp(&rs_full[buf], (uint32_t)((it >> 1) & 1))) {
        ok = false;
        break;
      }
      const float rs = pow2f(s_rexp[buf][lrow]);
      const uint16_t* my_sb = h ? srow : brow;  // the bias stages: biases (h = 0) or 8 x scales (h = 1)
      const float my_f = h ? 8.0f * rs : rs;
      for (int sb = 0; sb < nsb && ok; ++sb) {
        const uint4 cur[4] = {nxt[0], nxt[1], nxt[2], nxt[3]};
        const uint2 csc = nsc;
        if (sb + 1 < nsb) {
          load_sb(sb + 1);
        } else if (idx + (int)gridDim.x < total) {
          set_row(tile_at(idx + gridDim.x));
          load_sb(0);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j, ++kb) {
          const int s = kb % kPgStages;
          const uint32_t sw = j < 2 ? csc.x : csc.y;
          const __half2 s2 = __float2half2_rn(((j & 1) ? bf16_hi(sw) : bf16_lo(sw)) * rs);
          uint4 a[4];
          a[0] = dequant_word(cur[j].x, s2), a[1] = dequant_word(cur[j].y, s2);
          a[2] = dequant_word(cur[j].z, s2), a[3] = dequant_word(cur[j].w, s2);
          if (ok && !um_mbar_wait_warp(&empty[s], (uint32_t)(((kb / kPgStages) & 1) ^ 1))) ok = false;
          if (!ok) break;
#pragma unroll
          for (int i = 0; i < 4; ++i) *reinterpret_cast<uint4*>(a_row + s * kPgAStage + a_off[i]) = a[i];
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) um_mbar_arrive(&full[s]);
        }
      }
      for (int e = 0; e < kb_all - kb_main && ok; ++e, ++kb) {
        const int s = kb % kPgStages;
        uint2 w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          w[i] = e * 16 + i * 4 < kb_main ? *reinterpret_cast<const uint2*>(my_sb + e * 16 + i * 4) : make_uint2(0u, 0u);
        uint4 c[2];
#pragma unroll
        for (int i = 0; i < 2; ++i)
          c[i] = make_uint4(pack_f16x2(bf16_lo(w[2 * i].x) * my_f, bf16_hi(w[2 * i].x) * my_f),
                            pack_f16x2(bf16_lo(w[2 * i].y) * my_f, bf16_hi(w[2 * i].y) * my_f),
                            pack_f16x2(bf16_lo(w[2 * i + 1].x) * my_f, bf16_hi(w[2 * i + 1].x) * my_f),
                            pack_f16x2(bf16_lo(w[2 * i + 1].y) * my_f, bf16_hi(w[2 * i + 1].y) * my_f));
        if (!um_mbar_wait_warp(&empty[s], (uint32_t)(((kb / kPgStages) & 1) ^ 1))) {
          ok = false;
          break;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) *reinterpret_cast<uint4*>(a_row + s * kPgAStage + a_off[i]) = c[i & 1];
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) um_mbar_arrive(&full[s]);
      }
      if (ok && lane == 0) um_mbar_arrive(&rs_empty[buf]);
    }
    if (!ok && lane == 0 && p.status) atomicExch(p.status, 3u);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "n"(512) : "memory");
}

// ---- rotary embedding and append ---------------------------------------------------------------------------------
// One warp per (token, head of qkv): optional RMSNorm over the head, rotary embedding at the token's position, then
// q -> q, k and v -> the token's slot of the pool.
__global__ void __launch_bounds__(256) prefill_rope_kernel(const PrefillAttnArgs p) {
  grid_launch_dependents();
  grid_dependency_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int heads = p.nq + 2 * p.nkv, r = blockIdx.x, pos = p.start + r;
  const float4 cs = *reinterpret_cast<const float4*>(p.rope + ((size_t)pos * 64 + 2 * lane) * 2);  // c0 s0 c1 s1
  const int blk = p.block_table[pos / kBlockSize], slot = pos % kBlockSize;
  for (int hd = warp; hd < heads; hd += 8) {
    const uint16_t* src = p.qkv + ((size_t)r * heads + hd) * kHeadDim;
    // lane holds elements 2*lane, 2*lane+1 and their rotary partners 64 + 2*lane, 64 + 2*lane + 1
    const uint32_t wa = *reinterpret_cast<const uint32_t*>(src + 2 * lane), wb = *reinterpret_cast<const uint32_t*>(src + 64 + 2 * lane);
    uint32_t oa = wa, ob = wb;
    if (hd < p.nq + p.nkv) {
      float a0 = bf16_lo(wa), a1 = bf16_hi(wa), b0 = bf16_lo(wb), b1 = bf16_hi(wb);
      const uint16_t* nw = hd < p.nq ? p.q_norm : p.k_norm;
      if (nw) {
        const float ss = warp_sum(a0 * a0 + a1 * a1 + b0 * b0 + b1 * b1);
        const float inv = 1.0f / sqrtf(ss * (1.0f / kHeadDim) + p.eps);
        const uint32_t na = *reinterpret_cast<const uint32_t*>(nw + 2 * lane), nb = *reinterpret_cast<const uint32_t*>(nw + 64 + 2 * lane);
        a0 = bf16_to_f32(f32_to_bf16(a0 * inv * bf16_lo(na))), a1 = bf16_to_f32(f32_to_bf16(a1 * inv * bf16_hi(na)));
        b0 = bf16_to_f32(f32_to_bf16(b0 * inv * bf16_lo(nb))), b1 = bf16_to_f32(f32_to_bf16(b1 * inv * bf16_hi(nb)));
      }
      oa = pack_bf16x2(a0 * cs.x - b0 * cs.y, a1 * cs.z - b1 * cs.w);
      ob = pack_bf16x2(b0 * cs.x + a0 * cs.y, b1 * cs.z + a1 * cs.w);
    }
    uint16_t* dst;
    if (hd < p.nq) {
      dst = p.q + ((size_t)r * p.nq + hd) * kHeadDim;
    } else {
      const int kvh = (hd - p.nq) % p.nkv;
      dst = (hd >= p.nq + p.nkv ? p.vpool : p.kpool) + (((size_t)blk * p.nkv + kvh) * kBlockSize + slot) * kHeadDim;
    }
    *reinterpret_cast<uint32_t*>(dst + 2 * lane) = oa;
    *reinterpret_cast<uint32_t*>(dst + 64 + 2 * lane) = ob;
  }
}

// ---- causal attention ----------------------------------------------------------------------------------------------
// A CTA of four warps takes 64 consecutive tokens of one query head (a warp 16 rows) and walks the keys 0..position in
// tiles of 64 (four blocks of the pool), double buffered with cp.async.  Scores and P V run on m16n8k16 MMAs with the
// online softmax in fp32 and P in two bf16 terms, as in the decode kernel.  Later tokens see more keys: their CTAs
// come first in the grid.
constexpr int kPaTile = 64;
constexpr int kPaStage = 2 * kPaTile * 256;  // K then V, 64 tokens x 256 bytes each
constexpr int kPaSmem = 2 * kPaStage;
constexpr float kPaScaleLog2 = 0.08838834764831845f * 1.4426950408889634f;  // log2(e) / sqrt(128)

__device__ __forceinline__ void cp_async16_zfill(void* smem_dst, const void* gsrc, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(smem_dst)), "l"(gsrc), "r"(valid ? 16 : 0) : "memory");
}

__global__ void __launch_bounds__(128, 2) prefill_attention_kernel(const PrefillAttnArgs p) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int head = blockIdx.x, kvh = head / (p.nq / p.nkv);
  const int q0 = ((int)gridDim.y - 1 - (int)blockIdx.y) * 64;  // first row of the CTA
  grid_launch_dependents();
  grid_dependency_wait();

  const int keys = p.start + min(q0 + 64, p.rows);  // keys 0..keys-1 are visible to some row of the CTA
  const int tiles = (keys + kPaTile - 1) / kPaTile;
  auto issue = [&](int tile) {
    unsigned char* dst = smem + (tile & 1) * kPaStage;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int c = i * 128 + threadIdx.x, tok = c >> 4, c16 = c & 15;
      const int key = tile * kPaTile + tok;
      const bool valid = key < keys;
      const int blk = p.block_table[(valid ? key : 0) >> 4];
      const size_t src = (((size_t)blk * p.nkv + kvh) * kBlockSize + (key & 15)) * kHeadDim + c16 * 8;
      const int off = tok * 256 + ((c16 ^ (tok & 7)) << 4);
      cp_async16_zfill(dst + off, p.kpool + src, valid);
      cp_async16_zfill(dst + kPaTile * 256 + off, p.vpool + src, valid);
    }
    cp_async_commit();
  };
  issue(0);

  // Q fragments: rows g, g + 8 of the warp's 16 tokens
  const int row0 = q0 + warp * 16;
  uint32_t qa[8][4];
  {
    const uint16_t* r0 = p.q + ((size_t)min(row0 + g, p.rows - 1) * p.nq + head) * kHeadDim;
    const uint16_t* r1 = p.q + ((size_t)min(row0 + g + 8, p.rows - 1) * p.nq + head) * kHeadDim;
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      qa[ks][0] = *reinterpret_cast<const uint32_t*>(r0 + 16 * ks + 2 * t), qa[ks][1] = *reinterpret_cast<const uint32_t*>(r1 + 16 * ks + 2 * t);
      qa[ks][2] = *reinterpret_cast<const uint32_t*>(r0 + 16 * ks + 2 * t + 8), qa[ks][3] = *reinterpret_cast<const uint32_t*>(r1 + 16 * ks + 2 * t + 8);
    }
  }
  float o[16][4];
#pragma unroll
  for (int j = 0; j < 16; ++j) o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.0f;
  float m_lo = -INFINITY, m_hi = -INFINITY, l_lo = 0.0f, l_hi = 0.0f;
  const int pos_lo = p.start + row0 + g, pos_hi = pos_lo + 8;

  for (int tile = 0; tile < tiles; ++tile) {
    if (tile + 1 < tiles) issue(tile + 1);
    else cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    const unsigned char* sK = smem + (tile & 1) * kPaStage;
    const unsigned char* sV = sK + kPaTile * 256;
    if (tile * kPaTile <= p.start + row0 + 15) {  // else every key of the tile lies after every row of the warp
      float s[8][4];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        s[j][0] = s[j][1] = s[j][2] = s[j][3] = 0.0f;
        const int tok = 8 * j + (lane & 7);
#pragma unroll
        for (int kp = 0; kp < 4; ++kp) {
          uint32_t kb[4];
          ldmatrix_x4(kb, sK + tok * 256 + (((4 * kp + (lane >> 3)) ^ (tok & 7)) << 4));
          mma_bf16(s[j], qa[2 * kp][0], qa[2 * kp][1], qa[2 * kp][2], qa[2 * kp][3], kb[0], kb[1]);
          mma_bf16(s[j], qa[2 * kp + 1][0], qa[2 * kp + 1][1], qa[2 * kp + 1][2], qa[2 * kp + 1][3], kb[2], kb[3]);
        }
      }
      if (tile * kPaTile + kPaTile - 1 > p.start + row0) {  // some key of the tile lies after some row of the warp
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int key = tile * kPaTile + 8 * j + 2 * t + (c & 1);
            if (key > (c < 2 ? pos_lo : pos_hi) || key >= keys) s[j][c] = -INFINITY;
          }
      }
      float mx_lo = -INFINITY, mx_hi = -INFINITY;
#pragma unroll
      for (int j = 0; j < 8; ++j) mx_lo = fmaxf(mx_lo, fmaxf(s[j][0], s[j][1])), mx_hi = fmaxf(mx_hi, fmaxf(s[j][2], s[j][3]));
      mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 1)), mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 2));
      mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 1)), mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 2));
      const float mn_lo = fmaxf(m_lo, mx_lo * kPaScaleLog2), mn_hi = fmaxf(m_hi, mx_hi * kPaScaleLog2);  // key 0 is visible: finite
      if (__any_sync(0xffffffffu, mn_lo > m_lo || mn_hi > m_hi)) {
        const float c_lo = exp2f(m_lo - mn_lo), c_hi = exp2f(m_hi - mn_hi);
        l_lo *= c_lo, l_hi *= c_hi;
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j][0] *= c_lo, o[j][1] *= c_lo, o[j][2] *= c_hi, o[j][3] *= c_hi;
        m_lo = mn_lo, m_hi = mn_hi;
      }
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {  // 16 keys at a time: P as A fragments in two bf16 terms, then P V
        uint32_t ph[4], pl[4];
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          const float (&sv)[4] = s[2 * kk + hf];
          const float p0 = exp2f(fmaf(sv[0], kPaScaleLog2, -m_lo)), p1 = exp2f(fmaf(sv[1], kPaScaleLog2, -m_lo));
          const float p2 = exp2f(fmaf(sv[2], kPaScaleLog2, -m_hi)), p3 = exp2f(fmaf(sv[3], kPaScaleLog2, -m_hi));
          l_lo += p0 + p1, l_hi += p2 + p3;
          const uint32_t h01 = pack_bf16x2(p0, p1), h23 = pack_bf16x2(p2, p3);
          ph[2 * hf] = h01, ph[2 * hf + 1] = h23;
          pl[2 * hf] = pack_bf16x2(p0 - bf16_lo(h01), p1 - bf16_hi(h01));
          pl[2 * hf + 1] = pack_bf16x2(p2 - bf16_lo(h23), p3 - bf16_hi(h23));
        }
        const int i = lane >> 3, tok = kk * 16 + (i & 1) * 8 + (lane & 7);
#pragma unroll
        for (int jp = 0; jp < 8; ++jp) {
          uint32_t vb[4];
          ldmatrix_x4_trans(vb, sV + tok * 256 + (((2 * jp + (i >> 1)) ^ (tok & 7)) << 4));
          mma_bf16(o[2 * jp], ph[0], ph[1], ph[2], ph[3], vb[0], vb[1]);
          mma_bf16(o[2 * jp + 1], ph[0], ph[1], ph[2], ph[3], vb[2], vb[3]);
          mma_bf16(o[2 * jp], pl[0], pl[1], pl[2], pl[3], vb[0], vb[1]);
          mma_bf16(o[2 * jp + 1], pl[0], pl[1], pl[2], pl[3], vb[2], vb[3]);
        }
      }
    }
    __syncthreads();  // the buffer is refilled two tiles on
  }
  l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 1), l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 2);
  l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 1), l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 2);
#pragma unroll
  for (int hf = 0; hf < 2; ++hf) {
    const int row = row0 + g + 8 * hf;
    const float l = hf ? l_hi : l_lo;
    if (row < p.rows) {
      uint16_t* d = p.out + ((size_t)row * p.nq + head) * kHeadDim + 2 * t;
#pragma unroll
      for (int j = 0; j < 16; ++j)
        *reinterpret_cast<uint32_t*>(d + 8 * j) = pack_bf16x2(o[j][2 * hf] / l, o[j][2 * hf + 1] / l);
    }
  }
}

int g_prefill_sms = 0;

}  // namespace

cudaError_t prefill_init() {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(prefill_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPgSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(prefill_attention_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPaSmem);
  if (e == cudaSuccess) g_prefill_sms = sms;
  return e;
}

cudaError_t launch_prefill_pack(const uint16_t* x, int x_stride, const uint16_t* norm_w, float eps, int rows, int K, uint16_t* y,
                                uint16_t* operand, float* inv_scale, cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  if (K % 256 || K > kPrefillMaxWidth || x_stride % 8) return cudaErrorInvalidValue;
  const size_t smem = (size_t)(K >> 6) * sizeof(float);
  auto go = [&](auto kernel) { return launch_kernel(kernel, dim3(rows), dim3(256), smem, s, x, x_stride, norm_w, eps, K, y, operand, inv_scale); };
  const int nch = (K + 2047) / 2048;
  if (norm_w) {
    if (nch <= 1) return go(prefill_pack_kernel<1, true>);
    if (nch <= 2) return go(prefill_pack_kernel<2, true>);
    if (nch <= 4) return go(prefill_pack_kernel<4, true>);
    return nch <= 8 ? go(prefill_pack_kernel<8, true>) : go(prefill_pack_kernel<16, true>);
  }
  if (nch <= 1) return go(prefill_pack_kernel<1, false>);
  if (nch <= 2) return go(prefill_pack_kernel<2, false>);
  if (nch <= 4) return go(prefill_pack_kernel<4, false>);
  return nch <= 8 ? go(prefill_pack_kernel<8, false>) : go(prefill_pack_kernel<16, false>);
}

cudaError_t launch_prefill_gemm(const PrefillGemmArgs& a, cudaStream_t s) {
  if (g_prefill_sms == 0) {
    cudaError_t e = prefill_init();
    if (e != cudaSuccess) return e;
  }
  if (a.rows <= 0) return cudaSuccess;
  const bool grouped = a.units != nullptr;
  if (a.N % 128 || a.K % 256 || a.K > kPrefillMaxWidth || (grouped && (!a.n_units || a.unit_rows % 16 || a.unit_rows < 16 || a.unit_rows > 256)))
    return cudaErrorInvalidValue;
  PgParams p;
  p.qw = a.qw, p.scales = a.scales, p.biases = a.biases, p.inv_scale = a.inv_scale, p.out = a.out, p.status = a.status;
  p.units = a.units, p.n_units = a.n_units;
  p.N = a.N, p.K = a.K, p.rows = a.rows, p.out_stride = a.out_stride, p.epilogue = a.epilogue;
  p.row_tiles = a.N / 128;
  if (grouped) {
    p.n_tile = a.unit_rows, p.tok_tiles = 0;
  } else {  // equal token tiles of at most 256, a multiple of 16 each
    p.tok_tiles = (a.rows + 255) / 256;
    p.n_tile = ((a.rows + p.tok_tiles - 1) / p.tok_tiles + 15) & ~15;
  }
  EncodeTiledFn encode = nullptr;
  cudaError_t e = encode_tiled_fn(&encode);
  if (e != cudaSuccess) return e;
  const int stride = prefill_operand_stride(a.K);
  const cuuint64_t dims[2] = {(cuuint64_t)stride, (cuuint64_t)a.operand_rows}, strides[1] = {(cuuint64_t)stride * 2};
  const cuuint32_t box[2] = {64u, (cuuint32_t)p.n_tile}, elem[2] = {1u, 1u};
  CUtensorMap map;
  if (encode(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<uint16_t*>(a.operand), dims, strides, box, elem,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  int ctas = g_prefill_sms;
  if (!grouped) ctas = p.row_tiles * p.tok_tiles < ctas ? p.row_tiles * p.tok_tiles : ctas;
  return launch_kernel(prefill_gemm_kernel, dim3(ctas), dim3(kPgThreads), kPgSmem, s, p, map);
}

cudaError_t launch_prefill_rope_append(const PrefillAttnArgs& a, cudaStream_t s) {
  if (a.rows <= 0) return cudaSuccess;
  return launch_kernel(prefill_rope_kernel, dim3(a.rows), dim3(256), 0, s, a);
}

cudaError_t launch_prefill_attention(const PrefillAttnArgs& a, cudaStream_t s) {
  if (a.rows <= 0) return cudaSuccess;
  return launch_kernel(prefill_attention_kernel, dim3(a.nq, (a.rows + 63) / 64), dim3(128), kPaSmem, s, a);
}

}  // namespace q4d
