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
// fp32 results of a projection whose K was cut into parts, in part order: elements i, i + 1
__device__ __forceinline__ float2 add_parts(const float* sums, size_t i, int parts, size_t stride) {
  float2 v = *reinterpret_cast<const float2*>(sums + i);
#pragma unroll 4
  for (int q = 1; q < parts; ++q) {
    const float2 a = *reinterpret_cast<const float2*>(sums + q * stride + i);
    v.x += a.x, v.y += a.y;
  }
  return v;
}
// eight of them, the parts' loads side by side
__device__ __forceinline__ void add_parts8(const float* sums, size_t i, int parts, size_t stride, float (&v)[8]) {
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = 0.0f;
#pragma unroll 4
  for (int q = 0; q < parts; ++q) {
    const float4 a = *reinterpret_cast<const float4*>(sums + q * stride + i), b = *reinterpret_cast<const float4*>(sums + q * stride + i + 4);
    v[0] += a.x, v[1] += a.y, v[2] += a.z, v[3] += a.w, v[4] += b.x, v[5] += b.y, v[6] += b.z, v[7] += b.w;
  }
}

template <int NCH, bool NORM>
__global__ void __launch_bounds__(256) prefill_pack_kernel(const PrefillPackArgs p) {
  extern __shared__ float s_sums[];  // [K / 64]
  __shared__ float red[8];
  grid_launch_dependents();
  const int K = p.K, r = blockIdx.x, nch = K >> 3, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint16_t* w = p.norm_w;
  uint16_t* y = p.y;
  grid_dependency_wait();
  uint4 v[NCH];
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    const int c = threadIdx.x + i * 256;
    v[i] = make_uint4(0u, 0u, 0u, 0u);
    if (c >= nch) continue;
    uint16_t* px = p.x + (size_t)r * p.x_stride + c * 8;
    if (!p.sums) {
      v[i] = *reinterpret_cast<const uint4*>(px);
      continue;
    }
    float a[8];
    uint32_t o[4];
    if (p.silu) {  // h = bf16(silu(bf16(gate)) * bf16(up))
      float b[8];
      const size_t at = (size_t)r * 2 * K + c * 8, stride = (size_t)p.rows * 2 * K;
      add_parts8(p.sums, at, p.parts, stride, a);
      add_parts8(p.sums, at + K, p.parts, stride, b);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float h[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const float gt = bf16_to_f32(f32_to_bf16(a[2 * k + q])), up = bf16_to_f32(f32_to_bf16(b[2 * k + q]));
          h[q] = (gt / (1.0f + expf(-gt))) * up;
        }
        o[k] = pack_bf16x2(h[0], h[1]);
      }
      v[i] = make_uint4(o[0], o[1], o[2], o[3]);
    } else {  // the residual stream takes the projection's result
      add_parts8(p.sums, (size_t)r * K + c * 8, p.parts, (size_t)p.rows * K, a);
      const uint4 old = *reinterpret_cast<const uint4*>(px);
      const uint32_t ow[4] = {old.x, old.y, old.z, old.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t d = pack_bf16x2(a[2 * k], a[2 * k + 1]);
        o[k] = pack_bf16x2(bf16_lo(ow[k]) + bf16_lo(d), bf16_hi(ow[k]) + bf16_hi(d));
      }
      v[i] = make_uint4(o[0], o[1], o[2], o[3]);
      *reinterpret_cast<uint4*>(px) = v[i];
    }
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
    const float inv = 1.0f / sqrtf(ss / (float)K + p.eps);
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
  if (threadIdx.x == 0) p.inv_scale[r] = pow2f(-ex);
  uint16_t* row = p.operand + (size_t)r * prefill_operand_stride(K);
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
// accumulators of 256 columns let the epilogue of a tile run under the MMAs of the next.  K goes by in blocks of 64
// features: 128 rows and the tokens as f16 with the 128-byte swizzle, in a ring of four to six stages.  Roles:
//   warp 0      producer: TMA loads of the packed codes (128 rows x 128 features at a time) and of the tokens' operand
//   warp 1      MMA issue; owns the tensor-memory allocation
//   warps 2, 3  the power of two of each weight row of the next tile, the tokens' inverse scales
//   warps 4..7  epilogue (one per lane quarter of tensor memory)
//   warps 8..15 dequantisation, shared memory to shared memory: four pairs, each of which fills every fourth block, a
//               thread two of its rows
// A dequantised code costs ~1.6 instructions, a block about 145 issue cycles per scheduler against 512 cycles of tensor
// time at 256 tokens.  The chain wait - convert - store - fence - arrive - MMA - commit is several times longer than a
// block, so four blocks are in the making at once and a pair converts its first row before it waits for the stage (all
// eight warps on one block after another: 513 ns per block whatever the tile's width, 1.07 PFLOP/s on the gate/up
// projection of the 8B shape at 2048 tokens; a single thread issuing under `lane == 0`: 605 ns, 0.91).  The codes come by
// TMA: from global memory, 16 rows per load instruction, they cost 110 ns per block.
// A projection with few tiles is cut along K as well: the parts' fp32 sums go to global memory, and the kernel that reads
// the result (which exists anyway) adds them up.
constexpr int kPgThreads = 512;
constexpr int kPgBlockCycles = 600;   // a block takes about this many cycles and one more per token (48 tokens: 650, 256: 840)
constexpr int kPgABlock = 128 * 128;  // 128 rows x 64 f16
constexpr int kPgCodes = 128 * 64;    // the codes of two blocks
constexpr int kPgMaxStages = 6, kPgMaxCodes = 8;
// Tiles whose exponents and token scales are kept: a narrow tile of a mixture of experts is through before the epilogue of
// the one before has given its set back (four sets instead of two: the down projection's tiles 5.5 -> 5.0 us).
__host__ __device__ constexpr int pg_scale_sets(bool grouped) { return grouped ? 4 : 2; }
constexpr int kPgSmemBudget = 225 * 1024;
constexpr int kPgUnits = 448;         // units kept in shared memory (with one and a half shares each, 256 experts are 427 at most)

struct PgParams {
  const uint16_t* scales;
  const uint16_t* biases;
  const float* inv_scale;
  uint16_t* out;
  unsigned int* status;
  const int4* units;
  const int* n_units;
  int N, K, rows, n_tile, row_tiles, tok_tiles, out_stride, epilogue;
  int stages, code_slots;  // depths of the rings
  int parts;               // of K; `sums` given: the results are fp32 sums [part][rows][N] there
  float* sums;
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

// The largest of four scales or biases, folded into a pair of running maxima of magnitudes.
__device__ __forceinline__ uint32_t max_magnitude(uint32_t m, const uint2 v) {
  return __vmaxu2(m, __vmaxu2(v.x & 0x7fff7fffu, v.y & 0x7fff7fffu));
}

struct PgTile {
  int row_tile, tok0, valid, expert;
};

// GROUPED: the tiles are those of a list of units, 16 to 240 tokens of one expert each.
template <bool GROUPED>
__global__ void __launch_bounds__(kPgThreads, 1)
prefill_gemm_kernel(const PgParams p, const __grid_constant__ CUtensorMap map_b, const __grid_constant__ CUtensorMap map_codes) {
  constexpr int SETS = pg_scale_sets(GROUPED);
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[kPgMaxStages], empty[kPgMaxStages];      // operands of a stage
  __shared__ __align__(8) uint64_t c_full[kPgMaxCodes], c_empty[kPgMaxCodes];    // codes of two blocks
  __shared__ __align__(8) uint64_t d_full[2], d_empty[2], rs_full[SETS], rs_empty[SETS];
  __shared__ uint32_t s_tmem_base;
  __shared__ signed char s_rexp[SETS][128];             // powers of two of the weight rows
  __shared__ __align__(16) signed char s_inv[SETS][256];  // and of the tokens (as exponents: shared memory is full)

  grid_launch_dependents();

  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int NS = p.stages, NC = p.code_slots, b_block = p.n_tile * 128, stage_bytes = kPgABlock + b_block;
  unsigned char* sC = smem + NS * stage_bytes;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const bool silu = p.epilogue == EPI_SILU_PACK;
  const int half_n = p.N >> 1, K = p.K;
  const int kb_main = K >> 6, kb_all = prefill_operand_stride(K) >> 6, kst = (kb_all + 1) >> 1;  // blocks, pairs of blocks

  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) um_mbar_init(&full[s], 3), um_mbar_init(&empty[s], 1);
    for (int s = 0; s < NC; ++s) um_mbar_init(&c_full[s], 1), um_mbar_init(&c_empty[s], 4);
    for (int b = 0; b < 2; ++b) um_mbar_init(&d_full[b], 1), um_mbar_init(&d_empty[b], 4);
    for (int b = 0; b < SETS; ++b) um_mbar_init(&rs_full[b], 2), um_mbar_init(&rs_empty[b], 12);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)), "n"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // The list of units is the preceding kernel's.  Every role looks a tile up when it comes to it: from shared memory, for a
  // tile of the down projection (K = 768) is through in the time of a few loads.
  int4* s_units = reinterpret_cast<int4*>(sC + NC * kPgCodes);
  int n_units = 0;
  if (GROUPED) {
    grid_dependency_wait();
    n_units = *p.n_units;
    for (int i = threadIdx.x; i < min(n_units, kPgUnits); i += kPgThreads) s_units[i] = p.units[i];
    __syncthreads();
  }
  const int total = p.row_tiles * (GROUPED ? n_units : p.tok_tiles) * p.parts;
  // with K in parts, the parts of a tile are neighbours in the list; a part is whole pairs of blocks
  auto tile_kb0 = [&](int idx) -> int { return p.parts == 1 ? 0 : kst * (idx % p.parts) / p.parts * 2; };
  auto tile_kb1 = [&](int idx) -> int { return p.parts == 1 ? kb_all : min(kb_all, kst * (idx % p.parts + 1) / p.parts * 2); };
  auto tile_at = [&](int idx) -> PgTile {
    PgTile t;
    if (p.parts > 1) idx /= p.parts;
    if (GROUPED) {
      const int u = idx / p.row_tiles;
      const int4 un = u < kPgUnits ? s_units[u] : p.units[u];
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
  // exponent of a row over the scales and biases of its whole K, by four neighbouring lanes
  auto exponent_of = [&](uint32_t ms, uint32_t mb) -> int {
    float m = fmaxf(8.0f * fmaxf(bf16_lo(ms), bf16_hi(ms)), fmaxf(bf16_lo(mb), bf16_hi(mb)));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
    return range_exponent(m);
  };
  auto row_exponent = [&](const PgTile& t, int lrow) -> int {
    const size_t off = tensor_row(t, lrow) * (size_t)kb_main + (lane & 3) * 4;
    uint32_t ms = 0, mb = 0;
#pragma unroll 4
    for (int g = 0; g + (lane & 3) * 4 < kb_main; g += 16) {
      ms = max_magnitude(ms, __ldg(reinterpret_cast<const uint2*>(p.scales + off + g)));
      mb = max_magnitude(mb, __ldg(reinterpret_cast<const uint2*>(p.biases + off + g)));
    }
    return exponent_of(ms, mb);
  };
  // the first tile's exponents, by everybody at once: nothing can be dequantised without them
  if ((int)blockIdx.x < total) {
    const int ex = row_exponent(tile_at(blockIdx.x), threadIdx.x >> 2);
    if ((lane & 3) == 0) s_rexp[0][threadIdx.x >> 2] = (signed char)ex;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = s_tmem_base;

  bool ok = true;
  if (warp == 0) {
    // ---- producer: the whole warp walks, one lane issues.  Codes run ahead of the operand by their ring's depth; they
    // do not depend on the preceding kernel. ----
    int c_idx = blockIdx.x, c_kb, c_slot = 0;
    uint32_t c_phase = 1u;
    PgTile ct = tile_at(c_idx < total ? c_idx : 0);
    int c_kb1 = tile_kb1(c_idx);
    c_kb = tile_kb0(c_idx);
    // Issues what fits: pairs up to `want` pairs from the start.  A slot that is still being read is left for later; it is
    // free by the time the operand ring has turned, before anyone can be waiting for it.
    int want = NC, issued = 0;
    auto issue_codes = [&]() {
      while (issued < want && c_idx < total) {
        // (blocks of group sums have no codes; K is a multiple of 256, so no pair is half weights)
        if (c_kb < kb_main) {
          if (!um_mbar_test_warp(&c_empty[c_slot], c_phase)) return;
          const int row0 = __shfl_sync(0xffffffffu, ct.expert * p.N + (silu ? ct.row_tile * 64 : ct.row_tile * 128), 0);
          const int row1 = row0 + (silu ? half_n : 64), x = c_kb * 32;
          if (elect_one()) {
            um_mbar_expect_tx(&c_full[c_slot], (uint32_t)kPgCodes);
            um_tma_2d(sC + c_slot * kPgCodes, &map_codes, x, row0, &c_full[c_slot]);
            um_tma_2d(sC + c_slot * kPgCodes + 64 * 64, &map_codes, x, row1, &c_full[c_slot]);
          }
          __syncwarp();
          if (++c_slot == NC) c_slot = 0, c_phase ^= 1u;
        }
        ++issued;
        c_kb += 2;
        if (c_kb >= c_kb1) {
          c_idx += gridDim.x;
          if (c_idx < total) ct = tile_at(c_idx), c_kb = tile_kb0(c_idx), c_kb1 = tile_kb1(c_idx);
        }
      }
    };
    issue_codes();
    if (!GROUPED) grid_dependency_wait();
    int s = 0;
    uint32_t phase = 1u;
    for (int idx = blockIdx.x; idx < total && ok; idx += gridDim.x) {
      const PgTile t = tile_at(idx);
      const int tok0 = __shfl_sync(0xffffffffu, t.tok0, 0);
      const int kb0 = tile_kb0(idx), kb1 = tile_kb1(idx);
      for (int j = kb0; j < kb1 && ok; ++j) {
        if (!um_mbar_wait_warp(&empty[s], phase)) {
          ok = false;
          break;
        }
        if (elect_one()) {
          um_mbar_expect_tx(&full[s], (uint32_t)b_block);
          um_tma_2d(smem + s * stage_bytes + kPgABlock, &map_b, j * 64, tok0, &full[s]);
        }
        __syncwarp();
        if (++s == NS) s = 0, phase ^= 1u;
        if (j & 1) ++want;
        issue_codes();
      }
      if ((kb1 - kb0) & 1) ++want;
    }
    if (!ok && lane == 0 && p.status) atomicExch(p.status, 3u);
  } else if (warp == 1) {
    // ---- MMA issue: the whole warp walks, one lane issues ----
    // D f32, A and B f16, both K-major, M = 128
    const uint32_t idesc = (1u << 4) | ((uint32_t)(p.n_tile >> 3) << 17) | ((128u >> 4) << 24);
    const uint32_t smem_a = smem_u32(smem);
    int s = 0, it = 0;
    uint32_t phase = 0u;
    for (int idx = blockIdx.x; idx < total && ok; idx += gridDim.x, ++it) {
      const int buf = it & 1, kb0 = tile_kb0(idx), kb1 = tile_kb1(idx);
      if (!um_mbar_wait_warp(&d_empty[buf], (uint32_t)(((it >> 1) & 1) ^ 1))) ok = false;
      for (int j = kb0; j < kb1 && ok; ++j) {
        if (!um_mbar_wait_warp(&full[s], phase)) {
          ok = false;
          break;
        }
        tc_fence_after();
        if (elect_one()) {
          const uint32_t base = smem_a + (uint32_t)(s * stage_bytes);
          const uint64_t da = desc_sw128(base), db = desc_sw128(base + kPgABlock);
#pragma unroll
          for (int ks = 0; ks < 4; ++ks)
            umma_f16_ss(tbase + (uint32_t)(buf * 256), da + (uint64_t)(ks * 2), db + (uint64_t)(ks * 2), idesc, j != kb0 || ks != 0);
          umma_commit(&empty[s]);
          if (j == kb1 - 1) umma_commit(&d_full[buf]);
        }
        __syncwarp();
        if (++s == NS) s = 0, phase ^= 1u;
      }
    }
    if (!ok && lane == 0 && p.status) atomicExch(p.status, 3u);
  } else if (warp < 4) {
    // ---- token scales of a tile, and the row exponents of the next one ----
    const int tid = threadIdx.x - 64;
    if (!GROUPED) grid_dependency_wait();
    int it = 0;
    for (int idx = blockIdx.x; idx < total && ok; idx += gridDim.x, ++it) {
      const PgTile t = tile_at(idx);
      const int set = it % SETS;
      int ex[8];
      if (it > 0) {
        if (GROUPED) {
          // eight rows side by side: one after another their loads took as long as a narrow tile (12 us at K = 2048)
          const uint16_t *sp[8], *bp[8];
          uint32_t ms[8], mb[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const size_t off = tensor_row(t, i * 16 + (tid >> 2)) * (size_t)kb_main + (lane & 3) * 4;
            sp[i] = p.scales + off, bp[i] = p.biases + off, ms[i] = mb[i] = 0u;
          }
          for (int g = 0; g + (lane & 3) * 4 < kb_main; g += 16) {
            uint2 a[8], b[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) a[i] = __ldg(reinterpret_cast<const uint2*>(sp[i] + g)), b[i] = __ldg(reinterpret_cast<const uint2*>(bp[i] + g));
#pragma unroll
            for (int i = 0; i < 8; ++i) ms[i] = max_magnitude(ms[i], a[i]), mb[i] = max_magnitude(mb[i], b[i]);
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) ex[i] = exponent_of(ms[i], mb[i]);
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) ex[i] = row_exponent(t, i * 16 + (tid >> 2));
        }
      }
      if (!um_mbar_wait_warp(&rs_empty[set], (uint32_t)((it / SETS & 1) ^ 1))) ok = false;
      if (it > 0 && (lane & 3) == 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) s_rexp[set][i * 16 + (tid >> 2)] = (signed char)ex[i];
      }
      for (int i = tid; i < p.n_tile; i += 64) s_inv[set][i] = i < t.valid ? (signed char)((int)(__float_as_uint(p.inv_scale[t.tok0 + i]) >> 23) - 127) : (signed char)0;
      __syncwarp();
      if (lane == 0) um_mbar_arrive(&rs_full[set]);
    }
    if (!ok && lane == 0 && p.status) atomicExch(p.status, 3u);
  } else if (warp < 8) {
    // ---- epilogue ----
    const int q = warp - 4;
    const uint32_t lane_addr = tbase + ((uint32_t)(q * 32) << 16);
    if (!GROUPED) grid_dependency_wait();  // the output may still be read by the preceding kernels
    int it = 0;
    for (int idx = blockIdx.x; idx < total && ok; idx += gridDim.x, ++it) {
      const PgTile t = tile_at(idx);
      const int buf = it & 1, set = it % SETS;
      const uint32_t par = (uint32_t)((it >> 1) & 1);
      if (!um_mbar_wait_warp(&rs_full[set], (uint32_t)(it / SETS & 1)) || !um_mbar_wait_warp(&d_full[buf], par)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const float rinv = pow2f(-s_rexp[set][q * 32 + lane]);
      for (int c0 = 0; c0 < t.valid; c0 += 16) {
        float v[16];
        tmem_ld16f(lane_addr + (uint32_t)(buf * 256 + c0), v);
#pragma unroll
        for (int i = 0; i < 16; i += 4) {
          const char4 ce = *reinterpret_cast<const char4*>(&s_inv[set][c0 + i]);
          const float4 cs = make_float4(pow2f(ce.x), pow2f(ce.y), pow2f(ce.z), pow2f(ce.w));
          v[i] = v[i] * rinv * cs.x, v[i + 1] = v[i + 1] * rinv * cs.y;
          v[i + 2] = v[i + 2] * rinv * cs.z, v[i + 3] = v[i + 3] * rinv * cs.w;
        }
        if (p.sums) {
          float* d = p.sums + ((size_t)(idx % p.parts) * p.rows + t.tok0 + c0) * p.N + tensor_row(t, q * 32 + lane);
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (c0 + i < t.valid) d[(size_t)i * p.N] = v[i];
        } else if (silu) {
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
      if (lane == 0) um_mbar_arrive(&d_empty[buf]), um_mbar_arrive(&rs_empty[set]);
    }
    if (!ok && lane == 0 && p.status) atomicExch(p.status, 3u);
  } else {
    // ---- dequantisation: pair `grp` fills blocks b with b % 4 == grp (counted over all tiles), thread i rows i, i + 64 ----
    const int grp = (warp - 8) >> 1, tid = (warp & 1) * 32 + lane;
    // where the codes of tensor_row(row) are: with the SiLU epilogue a code slot holds 64 gate rows, then 64 up rows
    const unsigned char* c_row[2];
    int c_swz[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int row = tid + 64 * i, crow = silu ? (row >> 5) * 16 + (row & 15) + ((row & 16) ? 64 : 0) : row;
      c_row[i] = sC + crow * 64, c_swz[i] = (crow >> 1) & 3;  // (64-byte swizzle)
    }
    unsigned char* a_row = smem + tid * 128;
    int a_off[8];  // rows 64 apart share the swizzle
#pragma unroll
    for (int i = 0; i < 8; ++i) a_off[i] = (i ^ (tid & 7)) << 4;
    const uint16_t* srow[2];
    const ptrdiff_t to_biases = p.biases - p.scales;
    uint16_t nsc[2] = {0, 0};
    auto set_tile = [&](const PgTile& t) {
#pragma unroll
      for (int i = 0; i < 2; ++i) srow[i] = p.scales + tensor_row(t, tid + 64 * i) * (size_t)kb_main;
    };
    auto load_scales = [&](int j) {
#pragma unroll
      for (int i = 0; i < 2; ++i) nsc[i] = __ldg(srow[i] + j);
    };
    int base = 0;  // blocks before this tile, modulo 4
    int s = grp, it = 0, c_slot = 0, c_seen = 0;  // c_seen: the code slot the pair looks at, counted from the tile's first
    uint32_t phase = 1u, c_phase = 0u;
    while (s >= NS) s -= NS, phase ^= 1u;
    auto next_code_slot = [&](int n) {
      for (int i = 0; i < n; ++i)
        if (++c_slot == NC) c_slot = 0, c_phase ^= 1u;
    };
    for (int idx = blockIdx.x; idx < total && ok; idx += gridDim.x, ++it) {
      const int set = it % SETS, kb0 = tile_kb0(idx), kb1 = tile_kb1(idx), kc1 = min(kb1, kb_main);
      int j = kb0 + ((grp - base) & 3);
      set_tile(tile_at(idx));
      if (j < kc1) load_scales(j);
      if (it > 0 && !um_mbar_wait_warp(&rs_full[set], (uint32_t)(it / SETS & 1))) {
        ok = false;
        break;
      }
      float rs[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) rs[i] = pow2f(s_rexp[set][tid + 64 * i]);
      c_seen = 0;
      for (; j < kb1; j += 4) {
        unsigned char* dst = a_row + s * stage_bytes;
        if (j < kb_main) {
          const int slot_of = (j - kb0) >> 1;
          next_code_slot(slot_of - c_seen);
          c_seen = slot_of;
          __half2 s2[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) s2[i] = __float2half2_rn(bf16_to_f32(nsc[i]) * rs[i]);
          if (j + 4 < kc1) load_scales(j + 4);
          if (!um_mbar_wait_warp(&c_full[c_slot], c_phase)) {
            ok = false;
            break;
          }
          uint4 w[2][2];
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int c = 0; c < 2; ++c)
              w[i][c] = *reinterpret_cast<const uint4*>(c_row[i] + c_slot * kPgCodes + ((((j & 1) * 2 + c) ^ c_swz[i]) << 4));
          uint4 a[8];
          auto convert = [&](const uint4 (&v)[2], const __half2 sc) {
            a[0] = dequant_word(v[0].x, sc), a[1] = dequant_word(v[0].y, sc), a[2] = dequant_word(v[0].z, sc), a[3] = dequant_word(v[0].w, sc);
            a[4] = dequant_word(v[1].x, sc), a[5] = dequant_word(v[1].y, sc), a[6] = dequant_word(v[1].z, sc), a[7] = dequant_word(v[1].w, sc);
          };
          convert(w[0], s2[0]);
          if (!um_mbar_wait_warp(&empty[s], phase)) {
            ok = false;
            break;
          }
#pragma unroll
          for (int c = 0; c < 8; ++c) *reinterpret_cast<uint4*>(dst + a_off[c]) = a[c];
          convert(w[1], s2[1]);
#pragma unroll
          for (int c = 0; c < 8; ++c) *reinterpret_cast<uint4*>(dst + 64 * 128 + a_off[c]) = a[c];
          // The slot goes back when its codes have been used: loads that are merely issued do not hold back the arrival, and
          // the next codes overtook those of the second row.
          __syncwarp();
          if (lane == 0) um_mbar_arrive(&c_empty[c_slot]);
        } else {
          // 16 groups: {b, b} against {X1, X2}, {8 s, 8 s} against the same.  Narrow tiles: all loads go out together, before
          // the wait for the stage.
          const int e = (j - kb_main) * 16;
          auto load_groups = [&](int i, int q, int c) {  // row, biases or scales, four groups
            return e + c * 4 < kb_main ? __ldg(reinterpret_cast<const uint2*>(srow[i] + (q ? 0 : to_biases) + e + c * 4)) : make_uint2(0u, 0u);
          };
          uint2 v[2][2][4];
          if (GROUPED) {
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k >> 3][(k >> 2) & 1][k & 3] = load_groups(k >> 3, (k >> 2) & 1, k & 3);
          }
          if (!um_mbar_wait_warp(&empty[s], phase)) {
            ok = false;
            break;
          }
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const float f = q ? 8.0f * rs[i] : rs[i];
              uint32_t o[8];
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                const uint2 w = GROUPED ? v[i][q][c] : load_groups(i, q, c);
                o[2 * c] = pack_f16x2(bf16_lo(w.x) * f, bf16_hi(w.x) * f), o[2 * c + 1] = pack_f16x2(bf16_lo(w.y) * f, bf16_hi(w.y) * f);
              }
#pragma unroll
              for (int c = 0; c < 4; ++c)
                *reinterpret_cast<uint4*>(dst + i * (64 * 128) + a_off[q * 4 + c]) =
                    make_uint4(o[(c & 1) * 4], o[(c & 1) * 4 + 1], o[(c & 1) * 4 + 2], o[(c & 1) * 4 + 3]);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) um_mbar_arrive(&full[s]);
        s += 4;
        while (s >= NS) s -= NS, phase ^= 1u;
      }
      base = (base + kb1 - kb0) & 3;
      // the tile's code slots this pair did not look at go by as well
      if (kc1 > kb0) next_code_slot(((kc1 - kb0) >> 1) - c_seen);
      __syncwarp();
      if (ok && lane == 0) um_mbar_arrive(&rs_empty[set]);
    }
    if (!ok && lane == 0 && p.status) atomicExch(p.status, 3u);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "n"(512) : "memory");
}

// ---- rotary embedding and append ---------------------------------------------------------------------------------
// One warp per (token, head of qkv): optional RMSNorm over the head, rotary embedding at the token's position, then
// q -> q, k and v -> the token's slot of the pool.  A head is a chain of two round trips: with few tokens their heads are
// spread over CTAs (blockIdx.y) until the chip has a wave of them (77 tokens of the 0.6B shape: 9.9 us with four heads per warp).
__global__ void __launch_bounds__(256) prefill_rope_kernel(const PrefillAttnArgs p) {
  grid_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int heads = p.nq + 2 * p.nkv, r = blockIdx.x, pos = p.start + r;
  const float4 cs = *reinterpret_cast<const float4*>(p.rope + ((size_t)pos * 64 + 2 * lane) * 2);  // c0 s0 c1 s1
  const int blk = p.block_table[pos / kBlockSize], slot = pos % kBlockSize;
  grid_dependency_wait();  // the rotary table and the block table are older than the preceding kernel
  for (int hd = blockIdx.y * 8 + warp; hd < heads; hd += 8 * gridDim.y) {
    const size_t at = ((size_t)r * heads + hd) * kHeadDim + 2 * lane;
    // lane holds elements 2*lane, 2*lane+1 and their rotary partners 64 + 2*lane, 64 + 2*lane + 1
    uint32_t wa, wb;
    if (p.sums) {
      const size_t stride = (size_t)p.rows * heads * kHeadDim;
      const float2 a = add_parts(p.sums, at, p.parts, stride), b = add_parts(p.sums, at + 64, p.parts, stride);
      wa = pack_bf16x2(a.x, a.y), wb = pack_bf16x2(b.x, b.y);
    } else {
      wa = *reinterpret_cast<const uint32_t*>(p.qkv + at), wb = *reinterpret_cast<const uint32_t*>(p.qkv + at + 64);
    }
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
  if (e == cudaSuccess) e = cudaFuncSetAttribute(prefill_gemm_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPgSmemBudget);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(prefill_gemm_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPgSmemBudget);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(prefill_attention_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPaSmem);
  if (e == cudaSuccess) g_prefill_sms = sms;
  return e;
}

cudaError_t launch_prefill_pack(const PrefillPackArgs& a, cudaStream_t s) {
  if (a.rows <= 0) return cudaSuccess;
  const int K = a.K;
  if (K % 256 || K > kPrefillMaxWidth || a.x_stride % 8) return cudaErrorInvalidValue;
  const size_t smem = (size_t)(K >> 6) * sizeof(float);
  auto go = [&](auto kernel) { return launch_kernel(kernel, dim3(a.rows), dim3(256), smem, s, a); };
  const int nch = (K + 2047) / 2048;
  if (a.norm_w) {
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

// Token tiles of equal width (a multiple of 16, at most 256) so that waves x time per block is smallest.  Parts of K where
// even so under half of the SMs get a tile: at least four blocks each.
PrefillTiling prefill_tiling(int N, int K, int rows) {
  const int sms = g_prefill_sms > 0 ? g_prefill_sms : 148, row_tiles = N / 128;
  PrefillTiling best = {1, 16, 1};
  long long best_cost = -1;
  for (int k = (rows + 255) / 256; k <= (rows + 95) / 96 + 1; ++k) {
    const int n = ((rows + k - 1) / k + 15) & ~15, tiles = (rows + n - 1) / n;
    const long long waves = ((long long)row_tiles * tiles + sms - 1) / sms, cost = waves * (kPgBlockCycles + n);
    if (best_cost < 0 || cost < best_cost) best_cost = cost, best.tok_tiles = tiles, best.n_tile = n;
  }
  const int tiles = row_tiles * best.tok_tiles, stages = (prefill_operand_stride(K) / 64 + 1) / 2;
  if (tiles * 2 <= sms) {
    best.parts = sms / tiles;
    if (best.parts > stages / 2) best.parts = stages / 2;
    if (best.parts > kPrefillMaxParts) best.parts = kPrefillMaxParts;
    if (best.parts < 1) best.parts = 1;
  }
  return best;
}

cudaError_t launch_prefill_gemm(const PrefillGemmArgs& a, cudaStream_t s) {
  if (g_prefill_sms == 0) {
    cudaError_t e = prefill_init();
    if (e != cudaSuccess) return e;
  }
  if (a.rows <= 0) return cudaSuccess;
  const bool grouped = a.units != nullptr;
  if (a.N % 128 || a.K % 256 || a.K > kPrefillMaxWidth || (grouped && (!a.n_units || a.sums || a.unit_rows % 16 || a.unit_rows < 16 || a.unit_rows > 240)))
    return cudaErrorInvalidValue;
  PgParams p;
  p.scales = a.scales, p.biases = a.biases, p.inv_scale = a.inv_scale, p.out = a.out, p.status = a.status;
  p.units = a.units, p.n_units = a.n_units;
  p.N = a.N, p.K = a.K, p.rows = a.rows, p.out_stride = a.out_stride, p.epilogue = a.epilogue;
  p.row_tiles = a.N / 128, p.parts = 1, p.sums = a.sums;
  if (grouped) {
    p.n_tile = a.unit_rows, p.tok_tiles = 0;
  } else {
    const PrefillTiling t = prefill_tiling(a.N, a.K, a.rows);
    p.tok_tiles = t.tok_tiles, p.n_tile = t.n_tile;
    if (a.sums) p.parts = t.parts;
  }
  // Narrow tiles pass through a stage faster, and their smaller operand leaves room for more codes ahead.  A wait on a ring
  // tells a phase from the one before it only, so whoever reads a ring has to meet every turn of it.  A pair reads every
  // second slot of codes: their number is even, or a pair would meet a slot every second turn and could take codes that
  // are a turn old for its own.  And it fills every fourth stage: there are at least four.
  const int stage = kPgABlock + p.n_tile * 128;
  const int units_bytes = grouped ? kPgUnits * (int)sizeof(int4) : 0;
  auto stages_with = [&](int slots) { return (kPgSmemBudget - 1024 - units_bytes - slots * kPgCodes) / stage; };
  p.code_slots = p.n_tile <= 128 ? kPgMaxCodes : 4;
  p.stages = stages_with(p.code_slots);
  if (p.stages < 4) return cudaErrorInvalidValue;
  if (p.stages > kPgMaxStages) p.stages = kPgMaxStages;
  const size_t smem = 1024 + (size_t)p.stages * stage + (size_t)p.code_slots * kPgCodes + units_bytes;
  EncodeTiledFn encode = nullptr;
  cudaError_t e = encode_tiled_fn(&encode);
  if (e != cudaSuccess) return e;
  const int stride = prefill_operand_stride(a.K);
  const cuuint32_t elem[2] = {1u, 1u};
  CUtensorMap map_b, map_codes;
  {
    const cuuint64_t dims[2] = {(cuuint64_t)stride, (cuuint64_t)a.operand_rows}, strides[1] = {(cuuint64_t)stride * 2};
    const cuuint32_t box[2] = {64u, (cuuint32_t)p.n_tile};
    if (encode(&map_b, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<uint16_t*>(a.operand), dims, strides, box, elem,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  {
    const cuuint64_t dims[2] = {(cuuint64_t)(a.K / 2), (cuuint64_t)a.N * a.experts}, strides[1] = {(cuuint64_t)(a.K / 2)};
    const cuuint32_t box[2] = {64u, 64u};
    if (encode(&map_codes, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint32_t*>(a.qw), dims, strides, box, elem,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  int ctas = g_prefill_sms;
  if (!grouped && p.row_tiles * p.tok_tiles * p.parts < ctas) ctas = p.row_tiles * p.tok_tiles * p.parts;
  auto go = [&](auto kernel) { return launch_kernel(kernel, dim3(ctas), dim3(kPgThreads), smem, s, p, map_b, map_codes); };
  return grouped ? go(prefill_gemm_kernel<true>) : go(prefill_gemm_kernel<false>);
}

cudaError_t launch_prefill_rope_append(const PrefillAttnArgs& a, cudaStream_t s) {
  if (a.rows <= 0) return cudaSuccess;
  const int most = (a.nq + 2 * a.nkv + 7) / 8, fit = g_prefill_sms * 8 / a.rows;  // CTAs of a token's heads; of a wave
  return launch_kernel(prefill_rope_kernel, dim3(a.rows, fit < 1 ? 1 : (fit < most ? fit : most)), dim3(256), 0, s, a);
}

cudaError_t launch_prefill_attention(const PrefillAttnArgs& a, cudaStream_t s) {
  if (a.rows <= 0) return cudaSuccess;
  return launch_kernel(prefill_attention_kernel, dim3(a.nq, (a.rows + 63) / 64), dim3(128), kPaSmem, s, a);
}

}  // namespace q4d
