// Fused dequantise-and-multiply of 4-bit affine group-64 weights against bf16
// activations for 1..16 requests (the QKV, O, gate/up, down and LM-head
// projections of the decode step).
//
// y[r][j] = sum_k (scale[j][k/64] * q[j][k] + bias[j][k/64]) * x[r][k]
//         = sum_g scale[j][g] * (sum_{k in g} q[j][k] x[r][k]) + bias[j][g] * (sum_{k in g} x[r][k])
//
// The inner sums run on the tensor cores with the 4-bit codes taken as bf16 subnormals q * 2^-133 straight from the
// packed word and the activations scaled up to match (common.cuh): products are exact, accumulation is fp32, no
// dequantised weight is ever rounded to bf16.  The scale multiplies the fp32 group sums; the bias term is one more MMA
// per 256 features, biases against the group sums of the activations in three bf16 terms.
//
// Dense projections: q4_slice_kernel (K split over the warps of a CTA, operand in registers).  Mixture of experts:
// q4_expert_kernel (the same over a list of routed experts).
#include <stdlib.h>
#include <string.h>

#include "common.cuh"
#include "kernels.h"
#include "launch.h"
#include "tcgen05.cuh"

namespace q4d {

namespace {


// float of element i of four packed bf16
__device__ __forceinline__ float bf16_at(const uint2& v, int i) {
  uint32_t w = (i >> 1) ? v.y : v.x;
  return (i & 1) ? bf16_hi(w) : bf16_lo(w);
}

// MMAs the compiler may move: the multiplication below has registers to spare for overlapping its groups.
__device__ __forceinline__ void mma_free(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_free_first(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.0f));
}

// shared-memory accesses by 32-bit address (a generic pointer costs 64-bit arithmetic on the busiest pipe here)
__device__ __forceinline__ uint32_t lds32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}

// acc += 16 rows x 256 features with the operand's fragments in registers.  codes: shared address of this lane's first 8
// bytes of the stage's row g (a group further is an XOR with 32 in the swizzled, 1024-byte-aligned stage; row g + 8 is 1024
// bytes on).  bi: address of this lane's pair of biases (8 rows are 128 bytes); sc_lo, sc_hi: the 4 scales of rows g, g + 8.
// The pipe that shifts and masks issues every other cycle and is the busiest one here, so nothing but the unpacking is
// left to it: scalar FMAs instead of packed ones (whose operand pairs cost moves), no address arithmetic.
template <int NT>
__device__ __forceinline__ void multiply_regs(uint32_t codes, uint32_t bi, const uint2 sc_lo, const uint2 sc_hi,
                                              const uint4 (&bf)[4][NT][2], const uint2 (&x)[NT], float (&acc)[NT][4]) {
  const uint32_t b_lo = lds32(bi), b_hi = lds32(bi + 128);
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) mma_free(acc[nt], b_lo, b_hi, b_lo, b_hi, x[nt].x, x[nt].y);
  // The four MMAs of a group and 8 requests are a chain; four chains side by side hide the pipe's latency.
  constexpr int GP = 4 / NT;  // groups at a time
#pragma unroll
  for (int g0 = 0; g0 < 4; g0 += GP) {
    uint2 wl[GP], wh[GP];
    float pc[GP][NT][4];
#pragma unroll
    for (int i = 0; i < GP; ++i) {
      const uint32_t at = codes ^ (uint32_t)((g0 + i) << 5);
      wl[i] = lds64(at), wh[i] = lds64(at + 1024);
    }
#pragma unroll
    for (int step = 0; step < 4; ++step) {
#pragma unroll
      for (int i = 0; i < GP; ++i) {
        const uint32_t wa = step < 2 ? wl[i].x : wl[i].y, wb = step < 2 ? wh[i].x : wh[i].y;
        const uint32_t l = (step & 1) ? wa >> 8 : wa, h = (step & 1) ? wb >> 8 : wb;
        const uint32_t a0 = l & 0x000f000fu, a1 = h & 0x000f000fu, a2 = l & 0x00f000f0u, a3 = h & 0x00f000f0u;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          const uint4& bv = bf[g0 + i][nt][step >> 1];
          const uint32_t b0 = (step & 1) ? bv.z : bv.x, b1 = (step & 1) ? bv.w : bv.y;
          if (step == 0) mma_free_first(pc[i][nt], a0, a1, a2, a3, b0, b1);
          else mma_free(pc[i][nt], a0, a1, a2, a3, b0, b1);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < GP; ++i) {
      const float s_lo = bf16_at(sc_lo, g0 + i), s_hi = bf16_at(sc_hi, g0 + i);
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        acc[nt][0] = fmaf(s_lo, pc[i][nt][0], acc[nt][0]), acc[nt][1] = fmaf(s_lo, pc[i][nt][1], acc[nt][1]);
        acc[nt][2] = fmaf(s_hi, pc[i][nt][2], acc[nt][2]), acc[nt][3] = fmaf(s_hi, pc[i][nt][3], acc[nt][3]);
      }
    }
  }
}

// ---- dense projections -------------------------------------------------------------------------------------------
// One CTA per SM owns a contiguous range of 16-row tiles (and, for K > 4096, one part of K).  K is split over the WARPS:
// warp (kslice, row group) owns 256 or 512 input features and keeps the operand of those features in registers, as the B
// fragments of all their MMAs, while it walks the tiles of its row group.  The operand is read once per CTA, straight
// from global memory in fragment order, and shared memory holds nothing but the weight stream and the warps' partial
// tiles.  (With the operand in shared memory its fragment loads were 64 of 106 shared-memory wavefronts per stage, which
// bounded the multiply at 3.5 TB/s of weights on the LM head of the 8B shape; kept in registers they cost nothing.)
// The warps of a row group read one row's pieces side by side.  The partial tiles of a batch of rounds (a round = one
// tile per row group) meet in shared memory: one warp per (tile, 8 requests) adds them in kslice order and applies the
// epilogue, a batch behind the multiplication so that no warp waits for another (a CTA barrier per batch and an epilogue
// through shared memory made 143 us of the LM head's 108).
// A ring slot is 16 rows of 128 or 256 bytes of codes (TMA boxes of 128 bytes a row, 128-byte swizzle) and the rows' scales and biases (boxes of
// 16 bytes a row; where a row of scales is no multiple of 16 bytes, SB_TMA = false,
// 8-byte asynchronous copies instead).  TMA keeps the feed off the issue slots and off the load/store unit, whose time
// an asynchronous copy of 16 scattered 8-byte pieces takes 16 wavefronts of.
struct SliceParams {
  const uint16_t* scales;
  const uint16_t* biases;
  const uint16_t* xp;       // operand, OPERAND_FRAG
  const unsigned char* xs;  // its group sums, or NULL: every warp adds up its own
  void* out;
  uint16_t* out_xp;        // EPI_SILU_PACK: the next projection's operand, OPERAND_FRAG
  float2* argmax_partial;  // [warps of the grid][16]
  unsigned int* status;    // set to 3 when a wait gives up (may be NULL)
  float* partial;          // [parts][T][16 * 8 NT] sums of a tile over one part of K (parts > 1 only)
  int* counters;           // [T], zero between launches (parts > 1 only)
  int N, K, n, out_stride, epilogue;
  int T;       // row tiles of 16 rows (SiLU epilogue: 8 gate rows and the 8 matching up rows)
  int kw, rg;  // kslices and row groups of a CTA: kw * rg warps
  int batch;   // rounds between two meetings
  int slots;   // ring slots of a warp in use (kSliceSlots, or fewer where a warp has fewer stages)
  int vec_ok;
};
// A CTA covers at most 4096 features: 16 warps of one stage (256 features) each, or with 16 requests, whose operand takes 64
// registers per stage, 8 warps of two stages: half as many partial tiles, and registers to overlap the groups' MMAs
// (with 16 warps of 128 registers the LM head took 110 instead of 101 us).
__host__ __device__ constexpr int slice_sub(int nt) { return nt; }
__host__ __device__ constexpr int slice_max_warps(int nt) { return 16 / slice_sub(nt); }
constexpr int kSliceSlots = 3;  // ring slots per warp
__host__ __device__ constexpr int slice_slot_codes(int nt) { return slice_sub(nt) * 16 * 128; }
constexpr int kSliceSb = 2 * 16 * 16;  // of a slot: scales, then biases, 16 bytes a row

__device__ __forceinline__ void mbar_expect_tx_addr(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// the box at (x, row y, plane z) of the map (this GPU's memory only, no multicast)
__device__ __forceinline__ void tma_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
               "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
               : "memory");
}
// Waits for the phase of the given parity of the barrier at a shared address; gives up (false) after about two seconds.
__device__ __forceinline__ bool mbar_wait_addr(uint32_t bar, uint32_t parity) {
  for (int tries = 0; tries < 20000; ++tries) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity), "r"(100000u)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ uint32_t transpose_8x8(uint32_t v) {  // of b16: lane (g, t) gives row g, columns 2t, 2t + 1
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
  return r;
}

// h = bf16(silu(bf16(gate)) * bf16(up)) of 8 features (rows g are gate rows, rows g + 8 the matching up rows) x 8 requests, as
// chunk `tile` of an OPERAND_FRAG of K features; lane (g, t) writes a part of request 8 nt + g (if `valid`).
__device__ __forceinline__ void silu_epilogue(const float (&v)[4], uint16_t* out_xp, int K, int tile, int g, int t, bool valid, int nt = 0) {
  float h[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float gt = bf16_to_f32(f32_to_bf16(v[j])), up = bf16_to_f32(f32_to_bf16(v[2 + j]));
    h[j] = (gt / (1.0f + expf(-gt))) * up;
  }
  const uint32_t f = transpose_8x8(pack_bf16x2(h[0], h[1]));
  // the operand pairs features (j, j + 4) in word order 0: (0, 4), 1: (1, 5), 2: (2, 6), 3: (3, 7): lanes t < 2 take
  // (2t, 2t + 4), lanes t + 2 take (2t + 1, 2t + 5); odd words are stored times 2^60
  const uint32_t other = __shfl_xor_sync(0xffffffffu, t < 2 ? f >> 16 : f & 0xffffu, 2);
  const uint32_t pair = t < 2 ? (f & 0xffffu) | (other << 16) : other | (f & 0xffff0000u);
  const int word = t < 2 ? 2 * t : 2 * t - 3;
  if (valid)
    *reinterpret_cast<uint32_t*>(out_xp + operand_chunk_offset(OPERAND_FRAG, K, nt * 8 + g, tile) + word * 2) = scale_pair(pair, word & 1);
}

// Epilogue of 16 rows x 8 requests (nt: which 8) from an accumulator fragment (lane holds rows g, g + 8 and requests 2t,
// 2t + 1), without a detour through shared memory: fp32 results leave in 32-byte pieces as they lie, bf16 results are
// transposed in registers.  best, bidx: the lane's running argmax for its two requests (EPI_F32).
// old: the residual stream's values there, where the caller has them already (EPI_RESIDUAL).
__device__ __forceinline__ void slice_epilogue(const SliceParams& p, float (&v)[4], int tile, int nt, int g, int t, bool have_old,
                                               const uint32_t (&old_pair)[2], float (&best)[2], int (&bidx)[2]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) v[c] *= kOperandUnscale;
  if (p.epilogue == EPI_F32) {
    float* out = reinterpret_cast<float*>(p.out);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int row = tile * 16 + g + 8 * (c >> 1), req = nt * 8 + 2 * t + (c & 1);
      if (row < p.N && req < p.n) {
        out[(size_t)req * p.out_stride + row] = v[c];
        if (v[c] > best[c & 1]) best[c & 1] = v[c], bidx[c & 1] = row;  // a lane's rows ascend: the lowest among equals
      }
    }
    return;
  }
  const int req = nt * 8 + g;  // after the transposition: request g, rows (or features) 2t, 2t + 1
  if (p.epilogue == EPI_SILU_PACK) {
    silu_epilogue(v, p.out_xp, p.N >> 1, tile, g, t, req < p.n && tile * 8 < (p.N >> 1), nt);
    return;
  }
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    uint32_t y = transpose_8x8(pack_bf16x2(v[2 * half], v[2 * half + 1]));
    const int row = tile * 16 + half * 8 + 2 * t;
    if (req < p.n && row < p.N) {
      uint16_t* o = reinterpret_cast<uint16_t*>(p.out) + (size_t)req * p.out_stride + row;
      if (row + 1 < p.N && p.vec_ok) {
        if (p.epilogue == EPI_RESIDUAL) {
          const uint32_t old = have_old ? old_pair[half] : *reinterpret_cast<const uint32_t*>(o);
          y = pack_bf16x2(bf16_lo(old) + bf16_lo(y), bf16_hi(old) + bf16_hi(y));
        }
        *reinterpret_cast<uint32_t*>(o) = y;
      } else {
#pragma unroll
        for (int i = 0; i < 2; ++i)
          if (row + i < p.N) {
            uint16_t e = (uint16_t)(i ? y >> 16 : y);
            if (p.epilogue == EPI_RESIDUAL) e = f32_to_bf16(bf16_to_f32(o[i]) + bf16_to_f32(e));
            o[i] = e;
          }
      }
    }
  }
}

// The bound on registers for 8 requests is that of more threads than a CTA has (92 a thread instead of 106): it leaves the
// register file room for a CTA of the norm before, which this one is to stand beside, not behind (3B shape, eight requests:
// 5940 -> 5720 us).  With 16 requests it cannot (a bound of 208 costs the LM head 9 us).
template <int NT, bool SB_TMA>
__global__ void __launch_bounds__(NT == 1 ? 608 : 256, 1) q4_slice_kernel(const SliceParams p, const __grid_constant__ GemmMaps maps) {
  constexpr int SUB = slice_sub(NT), kSliceCodes = slice_slot_codes(NT);
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t s_bar[slice_max_warps(NT)][kSliceSlots];
  __shared__ __align__(8) uint64_t s_full[2], s_free[2];  // a buffer of partial tiles: written by, and read by, every warp

  grid_launch_dependents();

  // the warp's number from lane 0: known to be uniform, so that the coordinates and addresses of its copies are
  // uniform registers (a TMA instruction takes nothing else; from vector registers each one cost a loop of ~15)
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int warps = blockDim.x >> 5, rg = p.rg, slots = p.slots;
  const int ksl = warp / rg, rgi = warp - ksl * rg;
  const bool silu = p.epilogue == EPI_SILU_PACK;
  const int half_n = p.N >> 1;

  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* ring = smem + warp * (slots * kSliceCodes);
  unsigned char* ring_sb = smem + warps * (slots * kSliceCodes) + warp * (slots * kSliceSb);
  float4* sP = reinterpret_cast<float4*>(smem + warps * (slots * (kSliceCodes + kSliceSb)));  // two buffers of [tile of the batch][kslice][NT][32]

  // this CTA's tiles and part of K; this warp's stages of K (SUB, or one less at the end) and tiles
  const int stages = p.K >> 8, m = (stages + SUB - 1) / SUB, parts = gridDim.y;
  const int j0 = (int)((long long)blockIdx.y * m / parts), nks = (int)((long long)(blockIdx.y + 1) * m / parts) - j0;
  const int t0 = (int)((long long)blockIdx.x * p.T / gridDim.x), Tc = (int)((long long)(blockIdx.x + 1) * p.T / gridDim.x) - t0;
  const int j = j0 + ksl;
  const bool both = SUB == 2 && 2 * j + 1 < stages;  // the slice has its second stage
  const int my_n = ksl < nks && rgi < Tc ? (Tc - rgi + rg - 1) / rg : 0;

  const uint32_t ring_a = smem_u32(ring), sb_a = smem_u32(ring_sb), bar_a = smem_u32(&s_bar[warp][0]);
  // scale boxes hold 8 groups: two stages, of which a one-stage slice is the first or the second
  const int gx = (j * SUB * 4) & ~7, sb_half = SB_TMA && SUB == 1 ? (j & 1) * 8 : 0;
  const int kg = p.K >> 6;
  auto issue = [&](int tile, int slot) {
    const int y0 = silu ? tile * 8 : tile * 16, y1 = silu ? half_n + tile * 8 : tile * 16 + 8;
    if (elect_one()) {
      const uint32_t bar = bar_a + slot * 8, dst = ring_a + slot * kSliceCodes;
      mbar_expect_tx_addr(bar, (both ? 4096 : 2048) + (SB_TMA ? kSliceSb : 0));
      tma_3d(dst, &maps.codes, j * (SUB * 128), y0, 0, bar);
      if (both) tma_3d(dst + 2048, &maps.codes, j * 256 + 128, y0, 0, bar);
      if (SB_TMA) {
        const uint32_t sb = sb_a + slot * kSliceSb;
        tma_3d(sb, &maps.scales, gx, y0, 0, bar);
        tma_3d(sb + 256, &maps.biases, gx, y0, 0, bar);
      }
    }
    if (!SB_TMA && lane < 16) {
      const size_t off = (size_t)min(lane < 8 ? y0 + lane : y1 + lane - 8, p.N - 1) * kg + j * (SUB * 4);
      unsigned char* dst = ring_sb + slot * kSliceSb + lane * 16;
      cp_async8(dst, p.scales + off);
      cp_async8(dst + 256, p.biases + off);
      if (both) cp_async8(dst + 8, p.scales + off + 4), cp_async8(dst + 264, p.biases + off + 4);
    }
  };
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < kSliceSlots; ++i) um_mbar_init(&s_bar[warp][i], 1);
    if (warp == 0) {
#pragma unroll
      for (int i = 0; i < 2; ++i) um_mbar_init(&s_full[i], warps), um_mbar_init(&s_free[i], warps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (!SB_TMA && SUB == 2 && !both) {  // the scales and biases of a stage that does not exist are zeros too
    for (int i = lane; i < slots * 32; i += 32) *reinterpret_cast<uint2*>(ring_sb + i * 16 + 8) = make_uint2(0u, 0u);
  }
  __syncwarp();
  // Weights do not depend on the preceding kernel: fill the ring before waiting for it.
#pragma unroll
  for (int i = 0; i < kSliceSlots; ++i) {
    if (i < my_n && i < slots) issue(t0 + i * rg + rgi, i);
    if (!SB_TMA) cp_async_commit();
  }

  // Everything up to the first multiplication that does not need the operand is done before the preceding kernel is
  // awaited: what comes after it is the step's critical path, a few hundred nanoseconds at a time.
  bool ok = true;
  auto wait = [&](uint32_t bar, uint32_t parity) {
    if (!mbar_wait_addr(bar, parity)) {
      ok = false;  // a copy or a warp that never came: report, results are void
      if (p.status) atomicExch(p.status, 3u);
    }
  };
  const uint32_t full_a = smem_u32(&s_full[0]), free_a = smem_u32(&s_free[0]);
  const int buf_f4 = p.batch * rg * p.kw * (NT * 32);  // float4 of a buffer
  // this lane's addresses in slot 0: codes of row g, its scales and its pair of biases
  const uint32_t codes0 = ring_a + g * 128 + (((t >> 1) ^ g) << 4) + (t & 1) * 8;
  const uint32_t sc0 = sb_a + g * 16 + sb_half, bi0 = sc0 + 256 + (t & 1) * 4;
  const int part_step = rg * p.kw * (NT * 32);
  const int batches = (Tc + p.batch * rg - 1) / (p.batch * rg);
  const uint4* op_src = reinterpret_cast<const uint4*>(p.xp) + (size_t)j * (SUB * 16 * 32) + lane;
  __syncthreads();  // the barriers of the partial tiles exist
  if (my_n > 0) wait(bar_a, 0u);  // the first stage's codes
  grid_dependency_wait();

  // the operand of this warp's features, as B fragments, and the terms of its group sums
  uint4 bf[SUB][4][NT][2];
  uint2 x[SUB][NT];
  // Only the fragments of requests that exist are read: with one request a warp's 4 KB are 512 bytes, and the time is the
  // bytes' (148 CTAs x 16 warps).  The other columns' results are never stored.
#pragma unroll
  for (int sub = 0; sub < SUB; ++sub)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const bool in = my_n > 0 && (sub == 0 || both) && nt * 8 + g < p.n;
#pragma unroll
      for (int gi = 0; gi < 4; ++gi)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          bf[sub][gi][nt][h] = in ? __ldcg(op_src + (sub * 16 + (gi * 2 + nt) * 2 + h) * 32) : make_uint4(0u, 0u, 0u, 0u);
      x[sub][nt] = make_uint2(0u, 0u);
      if (p.xs && in)
        x[sub][nt] = __ldcg(reinterpret_cast<const uint2*>(p.xs + ((size_t)(SUB * j + sub) * 16 + nt * 8 + g) * kOperandSumBytes + t * 8));
    }
  if (!p.xs && my_n > 0) {
    // the producer left no group sums: the four lanes of a request hold a group's 64 elements
#pragma unroll
    for (int sub = 0; sub < SUB; ++sub)
      if (sub == 0 || both) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          float v[4];
#pragma unroll
          for (int gi = 0; gi < 4; ++gi) {
            float s = scaled_chunk_sum(bf[sub][gi][nt][0]) + scaled_chunk_sum(bf[sub][gi][nt][1]);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            v[gi] = s * kOperandSumScale * 0x1p-64f;
          }
          x[sub][nt] = sum_terms_fragment((t & 1) ? v[2] : v[0], (t & 1) ? v[3] : v[1], t < 2);
        }
      }
  }

  // the residual stream under the warp's first tile of the first batch, so that its epilogue waits for no load
  uint32_t old_pair[2] = {0u, 0u};
  if (p.epilogue == EPI_RESIDUAL && p.vec_ok && warp < min(p.batch * rg, Tc) * NT) {
    const int req = (warp % NT) * 8 + g;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int row = (t0 + warp / NT) * 16 + half * 8 + 2 * t;
      if (req < p.n && row + 1 < p.N)
        old_pair[half] = __ldcg(reinterpret_cast<const uint32_t*>(reinterpret_cast<const uint16_t*>(p.out) + (size_t)req * p.out_stride + row));
    }
  }

  float best[NT][2];
  int bidx[NT][2];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) best[nt][0] = best[nt][1] = -INFINITY, bidx[nt][0] = bidx[nt][1] = 0x7fffffff;

  // The tiles of batch b, one warp per (tile, 8 requests), dealt round robin over the batches: the kslices' sums in
  // kslice order, then the epilogue.
  int task = warp;  // of the coming batch, dealt round robin over the batches
  auto finish_batch = [&](int b) {
    const int first = b * p.batch * rg, tiles = min(p.batch * rg, Tc - first), buf = b & 1;
    wait(full_a + buf * 8, (uint32_t)((b >> 1) & 1));
    __syncwarp();
    const int all = tiles * NT;
    auto add_kslices = [&](int tl, int nt, float (&v)[4]) {
      v[0] = v[1] = v[2] = v[3] = 0.0f;
      const float4* src = sP + buf * buf_f4 + tl * (p.kw * NT * 32) + nt * 32 + lane;
      for (int k0 = 0; k0 < nks; k0 += 4) {  // four at a time: their loads go out together
        float4 a[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = k0 + k < nks ? src[(k0 + k) * (NT * 32)] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int k = 0; k < 4; ++k) v[0] += a[k].x, v[1] += a[k].y, v[2] += a[k].z, v[3] += a[k].w;
      }
    };
    // Where several CTAs hold parts of a tile's sums they publish them, and the last to arrive adds them in part order.  The
    // warp publishes all its tiles of the batch before it counts any (a lane per tile, 28 at most): one fence and one round
    // trip of the counters, not one of each per tile.
    unsigned last = 0u;
    const size_t stride = (size_t)p.T * (NT * 32);
    if (parts > 1) {
      int mine = 0;
      for (int tk = task; tk < all; tk += warps, ++mine) {
        const int tl = tk / NT, nt = tk - tl * NT;
        float v[4];
        add_kslices(tl, nt, v);
        reinterpret_cast<float4*>(p.partial)[blockIdx.y * stride + (size_t)(t0 + first + tl) * (NT * 32) + nt * 32 + lane] = make_float4(v[0], v[1], v[2], v[3]);
      }
      __threadfence();
      __syncwarp();
      bool is_last = false;
      if (lane < mine) {
        const int tk = task + lane * warps, tl = tk / NT, sh = (tk - tl * NT) * 16;  // a tile's two halves count in the halves of its counter
        int* counter = p.counters + t0 + first + tl;
        is_last = ((atomicAdd(counter, 1 << sh) >> sh) & 0xffff) == parts - 1;
        if (is_last) atomicSub(counter, parts << sh);
        __threadfence();
      }
      last = __ballot_sync(0xffffffffu, is_last);
    }
    for (int i = 0; task < all; task += warps, ++i) {
      const int tl = task / NT, nt = task - tl * NT, tile = t0 + first + tl;
      float v[4];
      if (parts == 1) {
        add_kslices(tl, nt, v);
      } else {
        if (!((last >> i) & 1u)) continue;
        const float4* part = reinterpret_cast<const float4*>(p.partial) + (size_t)tile * (NT * 32) + nt * 32 + lane;
        v[0] = v[1] = v[2] = v[3] = 0.0f;
        for (int y0 = 0; y0 < parts; y0 += 4) {  // four parts at a time: their loads go out together
          float4 a[4];
#pragma unroll
          for (int y = 0; y < 4; ++y) a[y] = y0 + y < parts ? __ldcg(part + (y0 + y) * stride) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
          for (int y = 0; y < 4; ++y) v[0] += a[y].x, v[1] += a[y].y, v[2] += a[y].z, v[3] += a[y].w;
        }
      }
#pragma unroll
      for (int q = 0; q < NT; ++q)
        if (q == nt) slice_epilogue(p, v, tile, q, g, t, i == 0 && b == 0, old_pair, best[q], bidx[q]);
    }
    task -= tiles * NT;  // the next batch's first task of this warp
    __syncwarp();
    if (lane == 0) um_mbar_arrive(&s_free[buf]);
  };

  int it = 0, slot = 0, next_tile = t0 + slots * rg + rgi;
  uint32_t phase = 0;
  for (int b = 0; b < batches; ++b) {
    const int buf = b & 1;
    if (b >= 2) wait(free_a + buf * 8, (uint32_t)(((b >> 1) - 1) & 1));
    float4* dst = sP + buf * buf_f4 + (rgi * p.kw + ksl) * (NT * 32) + lane;
    const int it_end = min(my_n, (b + 1) * p.batch);
    for (; it < it_end; ++it, dst += part_step) {
      if (!SB_TMA) cp_async_wait<kSliceSlots - 1>();
      if (it > 0) wait(bar_a + slot * 8, phase);
      __syncwarp();
      float acc[NT][4];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.0f;
      const uint32_t codes = codes0 + slot * kSliceCodes, bi = bi0 + slot * kSliceSb;
      const uint32_t sc = sc0 + slot * kSliceSb;
      if (SUB == 1) {
        multiply_regs<NT>(codes, bi, lds64(sc), lds64(sc + 128), bf[0], x[0], acc);
      } else {
        const uint4 sc_lo = lds128(sc), sc_hi = lds128(sc + 128);
        multiply_regs<NT>(codes, bi, make_uint2(sc_lo.x, sc_lo.y), make_uint2(sc_hi.x, sc_hi.y), bf[0], x[0], acc);
        // a slice without its second stage multiplies it with an operand of zeros: no branch between the halves
          multiply_regs<NT>(codes + 2048, bi + 8, make_uint2(sc_lo.z, sc_lo.w), make_uint2(sc_hi.z, sc_hi.w), bf[SUB - 1], x[SUB - 1], acc);
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) dst[nt * 32] = make_float4(acc[nt][0], acc[nt][1], acc[nt][2], acc[nt][3]);
      __syncwarp();
      if (it + slots < my_n) {  // refill the slot just multiplied
        if (ok) issue(next_tile, slot);
        next_tile += rg;
      }
      if (!SB_TMA) cp_async_commit();
      if (++slot == slots) slot = 0, phase ^= 1u;
    }
    __syncwarp();
    if (lane == 0) um_mbar_arrive(&s_full[buf]);
    if (b > 0) finish_batch(b - 1);  // a batch behind: the other warps' sums are there by now, nobody waits for anybody
  }
  if (batches > 0) finish_batch(batches - 1);
  if (!SB_TMA) cp_async_wait<0>();

  if (p.epilogue == EPI_F32 && p.argmax_partial) {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int c = 0; c < 2; ++c) {  // over the lanes of a request
        float v = best[nt][c];
        int i = bidx[nt][c];
#pragma unroll
        for (int o = 4; o <= 16; o <<= 1) {
          const float ov = __shfl_xor_sync(0xffffffffu, v, o);
          const int oi = __shfl_xor_sync(0xffffffffu, i, o);
          if (ov > v || (ov == v && oi < i)) v = ov, i = oi;
        }
        if (g == 0)
          p.argmax_partial[((size_t)(blockIdx.y * gridDim.x + blockIdx.x) * warps + warp) * 16 + nt * 8 + 2 * t + c] = make_float2(v, __int_as_float(i));
      }
  }
}

struct SlicePlan {
  int nt, parts, kw, rg, T, ctas, batch, slots;
  size_t smem, partial_bytes;
};

SlicePlan plan_slices(int N, int K, int n, int epilogue, int sm_count) {
  SlicePlan t;
  t.nt = n <= 8 ? 1 : 2;
  const int max_warps = slice_max_warps(t.nt), m = (K / 256 + slice_sub(t.nt) - 1) / slice_sub(t.nt);
  t.parts = (m + max_warps - 1) / max_warps;  // a warp holds the operand of one slice
  t.kw = (m + t.parts - 1) / t.parts;
  t.T = epilogue == EPI_SILU_PACK ? (N / 2 + 7) / 8 : (N + 15) / 16;
  int ctas = sm_count / t.parts;
  if (ctas < 1) ctas = 1;
  // A small projection runs on half the warps: then the next kernel's CTAs fit on the SMs beside it (the register file is
  // what they share) and have their first codes by the time they are released, which is worth more than a shorter
  // multiplication (1024 -> 6144 at one request, launch to launch: 4.31 us with 12 warps, which leave the next CTA no
  // room, so that its codes arrive 1.8 us after the release; 3.67 with 8).  It is not worth a third stage per warp, nor a
  // second one with 16 requests, where a stage takes twice as long (2048 -> 5120, 1024 -> 6144: slower).
  const int half = max_warps / 2 / t.kw;
  t.ctas = t.T < ctas ? t.T : ctas;
  const int per_cta = (t.T + t.ctas - 1) / t.ctas;
  t.rg = max_warps / t.kw;
  if (half >= 1 && (per_cta + half - 1) / half <= (t.nt == 1 ? 2 : 1)) t.rg = half;
  if (t.rg > per_cta) t.rg = per_cta;
  const int warps = t.kw * t.rg, rounds = (per_cta + t.rg - 1) / t.rg;
  t.slots = rounds < kSliceSlots ? rounds : kSliceSlots;
  const size_t fixed = 1024 + (size_t)warps * t.slots * (slice_slot_codes(t.nt) + kSliceSb);
  const size_t per_round = 2 * (size_t)warps * t.nt * 512;  // two buffers
  const int most = (int)((220 * 1024 - fixed) / per_round);  // rounds whose partial tiles fit
  const int batches = (rounds + most - 1) / most;
  t.batch = (rounds + batches - 1) / batches;
  t.smem = fixed + t.batch * per_round;
  t.partial_bytes = t.parts > 1 ? (size_t)t.parts * t.T * 16 * (8 * t.nt) * sizeof(float) : 0;
  return t;
}

// ---- mixture-of-experts projections --------------------------------------------------------------------------------
// The same multiplication over a list of units, a unit being up to eight requests that were routed to one expert: with
// sixteen requests and 128 experts an expert serves one or two of them, so eight columns are enough where the earlier
// kernel multiplied all sixteen requests with every touched expert.  The row tiles of all units form one list, cut into
// equal contiguous ranges, one per CTA; a warp exchanges its operand fragments when its range enters the next unit (the
// weight ring runs on across the border).  Gate/up reads the fragments of a unit's requests from the step's operand;
// its output is the unit's own operand for the down projection.  Measured (30B-A3B shape, 16 requests, between events):
// gate/up 62 -> 39 us, down with the combination 2 x 22.7 -> 2 x 18.2 us.
struct ExpertParams {
  const uint16_t* scales;
  const uint16_t* biases;
  const uint16_t* xp;        // OPERAND_FRAG: of the step (gate/up), or one per unit, unit_stride elements apart (down)
  const unsigned char* xs;   // group sums of the step's operand (gate/up)
  uint16_t* out;             // down: bf16 [unit][8][N]
  uint16_t* out_xp;          // gate/up: OPERAND_FRAG per unit
  unsigned int* status;
  const int4* units;         // {expert, requests, request ids as bytes (two words)}
  const int* n_units;
  size_t unit_stride, out_unit_stride;  // elements
  int N, K, tiles;           // rows and row tiles of an expert
  unsigned tiles_inv;        // 2^32 / tiles, rounded up: the high word of a product with it divides a tile's number
  int kw, rg, batch;
};

template <bool GATE_UP, bool SB_TMA>
__global__ void __launch_bounds__(32 * slice_max_warps(1), 1) q4_expert_kernel(const ExpertParams p, const __grid_constant__ GemmMaps maps) {
  constexpr int kCodes = 16 * 128;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t s_bar[slice_max_warps(1)][kSliceSlots];
  __shared__ __align__(8) uint64_t s_full[2], s_free[2];
  __shared__ int4 s_units[kMaxExpertUnits];

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int warps = blockDim.x >> 5, rg = p.rg;
  const int j = warp / rg, rgi = warp - j * rg;  // 256-feature slice, row group
  const int half_n = p.N >> 1, kg = p.K >> 6;

  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* ring = smem + warp * (kSliceSlots * kCodes);
  unsigned char* ring_sb = smem + warps * (kSliceSlots * kCodes) + warp * (kSliceSlots * kSliceSb);
  float4* sP = reinterpret_cast<float4*>(smem + warps * (kSliceSlots * (kCodes + kSliceSb)));
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < kSliceSlots; ++i) um_mbar_init(&s_bar[warp][i], 1);
    if (warp == 0) {
#pragma unroll
      for (int i = 0; i < 2; ++i) um_mbar_init(&s_full[i], warps), um_mbar_init(&s_free[i], warps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // The list of units is the router's.  Gate/up follows the router and waits for it; only then does it let the down
  // projection start, which may therefore read the list at once and fetch its first weights under gate/up's tail.
  if (GATE_UP) {
    grid_dependency_wait();
    grid_launch_dependents();
  } else {
    grid_launch_dependents();
  }
  // the whole list without waiting for its length: one round trip
  const int n_units = min(__ldcg(p.n_units), kMaxExpertUnits);
  for (int i = threadIdx.x; i < kMaxExpertUnits; i += blockDim.x) s_units[i] = __ldcg(p.units + i);
  __syncthreads();
  const int total = n_units * p.tiles;
  const int t0 = (int)((long long)blockIdx.x * total / gridDim.x), Tc = (int)((long long)(blockIdx.x + 1) * total / gridDim.x) - t0;
  const int my_n = rgi < Tc ? (Tc - rgi + rg - 1) / rg : 0;

  const uint32_t ring_a = smem_u32(ring), sb_a = smem_u32(ring_sb), bar_a = smem_u32(&s_bar[warp][0]);
  const int gx = (j * 4) & ~7, sb_half = SB_TMA ? (j & 1) * 8 : 0;
  auto issue = [&](int gt, int slot) {  // tile gt of the list
    const int unit = (int)__umulhi((unsigned)gt, p.tiles_inv), tile = gt - unit * p.tiles;
    const int e = __shfl_sync(0xffffffffu, s_units[unit].x, 0);
    const int y = GATE_UP ? tile * 8 : e * p.N + tile * 16, z = GATE_UP ? 2 * e : 0;
    if (elect_one()) {
      const uint32_t bar = bar_a + slot * 8;
      mbar_expect_tx_addr(bar, kCodes + (SB_TMA ? kSliceSb : 0));
      tma_3d(ring_a + slot * kCodes, &maps.codes, j * 128, y, z, bar);
      if (SB_TMA) {
        tma_3d(sb_a + slot * kSliceSb, &maps.scales, gx, y, z, bar);
        tma_3d(sb_a + slot * kSliceSb + 256, &maps.biases, gx, y, z, bar);
      }
    }
    if (!SB_TMA && lane < 16) {
      const int r = GATE_UP ? (lane < 8 ? tile * 8 + lane : half_n + tile * 8 + lane - 8) : tile * 16 + lane;
      const size_t off = ((size_t)e * p.N + r) * kg + j * 4;
      unsigned char* dst = ring_sb + slot * kSliceSb + lane * 16;
      cp_async8(dst, p.scales + off);
      cp_async8(dst + 256, p.biases + off);
    }
  };
#pragma unroll
  for (int i = 0; i < kSliceSlots; ++i) {
    if (i < my_n) issue(t0 + i * rg + rgi, i);
    if (!SB_TMA) cp_async_commit();
  }
  if (!GATE_UP) grid_dependency_wait();

  uint4 bf[4][1][2];
  uint2 x[1];
  auto load_operand = [&](int unit) {
    const int4 u = s_units[unit];
    int r = g;
    const uint16_t* base = p.xp;
    if (GATE_UP) r = ((g < 4 ? u.z : u.w) >> ((g & 3) * 8)) & 15;
    else base += (size_t)unit * p.unit_stride;
    const uint4* src = reinterpret_cast<const uint4*>(base) + (size_t)j * 16 * 32 + (r >> 3) * 64 + (r & 7) * 4 + t;
    const bool in = g < u.y;  // only the unit's requests are read
#pragma unroll
    for (int gi = 0; gi < 4; ++gi)
#pragma unroll
      for (int h = 0; h < 2; ++h) bf[gi][0][h] = in ? __ldcg(src + (gi * 4 + h) * 32) : make_uint4(0u, 0u, 0u, 0u);
    if (GATE_UP) {
      x[0] = make_uint2(0u, 0u);
      if (in) x[0] = __ldcg(reinterpret_cast<const uint2*>(p.xs + ((size_t)j * 16 + r) * kOperandSumBytes + t * 8));
    } else {
      float v[4];
#pragma unroll
      for (int gi = 0; gi < 4; ++gi) {
        float s = scaled_chunk_sum(bf[gi][0][0]) + scaled_chunk_sum(bf[gi][0][1]);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        v[gi] = s * kOperandSumScale * 0x1p-64f;
      }
      x[0] = sum_terms_fragment((t & 1) ? v[2] : v[0], (t & 1) ? v[3] : v[1], t < 2);
    }
  };

  bool ok = true;
  auto wait = [&](uint32_t bar, uint32_t parity) {
    if (!mbar_wait_addr(bar, parity)) {
      ok = false;  // a copy or a warp that never came: report, results are void
      if (p.status) atomicExch(p.status, 3u);
    }
  };
  const uint32_t full_a = smem_u32(&s_full[0]), free_a = smem_u32(&s_free[0]);
  const int buf_f4 = p.batch * rg * p.kw * 32;  // float4 of a buffer

  int task = warp;  // of the coming batch, dealt round robin over the batches
  auto finish_batch = [&](int b) {
    const int first = b * p.batch * rg, tiles = min(p.batch * rg, Tc - first), buf = b & 1;
    wait(full_a + buf * 8, (uint32_t)((b >> 1) & 1));
    __syncwarp();
    for (; task < tiles; task += warps) {
      const int gt = t0 + first + task, unit = (int)__umulhi((unsigned)gt, p.tiles_inv), tile = gt - unit * p.tiles;
      const int count = s_units[unit].y;
      float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      const float4* src = sP + buf * buf_f4 + task * (p.kw * 32) + lane;
      for (int k0 = 0; k0 < p.kw; k0 += 4) {  // four at a time: their loads go out together
        float4 a[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = k0 + k < p.kw ? src[(k0 + k) * 32] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int k = 0; k < 4; ++k) v[0] += a[k].x, v[1] += a[k].y, v[2] += a[k].z, v[3] += a[k].w;
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] *= kOperandUnscale;
      if (GATE_UP) {
        silu_epilogue(v, p.out_xp + (size_t)unit * p.out_unit_stride, half_n, tile, g, t, g < count);
      } else {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const uint32_t y = transpose_8x8(pack_bf16x2(v[2 * half], v[2 * half + 1]));
          if (g < count)
            *reinterpret_cast<uint32_t*>(p.out + ((size_t)unit * 8 + g) * p.N + tile * 16 + half * 8 + 2 * t) = y;
        }
      }
    }
    task -= tiles;
    __syncwarp();
    if (lane == 0) um_mbar_arrive(&s_free[buf]);
  };

  int it = 0, slot = 0, gt = t0 + rgi, unit = -1, unit_end = 0;
  uint32_t phase = 0;
  const uint32_t codes0 = ring_a + g * 128 + (((t >> 1) ^ g) << 4) + (t & 1) * 8;
  const uint32_t sc0 = sb_a + g * 16 + sb_half, bi0 = sc0 + 256 + (t & 1) * 4;
  const int part_step = rg * p.kw * 32;
  const int batches = (Tc + p.batch * rg - 1) / (p.batch * rg);
  for (int b = 0; b < batches; ++b) {
    const int buf = b & 1;
    if (b >= 2) wait(free_a + buf * 8, (uint32_t)(((b >> 1) - 1) & 1));
    float4* dst = sP + buf * buf_f4 + (rgi * p.kw + j) * 32 + lane;
    const int it_end = min(my_n, (b + 1) * p.batch);
    for (; it < it_end; ++it, dst += part_step, gt += rg) {
      if (gt >= unit_end) {
        unit = (int)__umulhi((unsigned)gt, p.tiles_inv), unit_end = (unit + 1) * p.tiles;
        load_operand(unit);
      }
      if (!SB_TMA) cp_async_wait<kSliceSlots - 1>();
      wait(bar_a + slot * 8, phase);
      __syncwarp();
      float acc[1][4] = {{0.0f, 0.0f, 0.0f, 0.0f}};
      const uint32_t sc = sc0 + slot * kSliceSb;
      multiply_regs<1>(codes0 + slot * kCodes, bi0 + slot * kSliceSb, lds64(sc),
                       lds64(sc + 128), bf, x, acc);
      dst[0] = make_float4(acc[0][0], acc[0][1], acc[0][2], acc[0][3]);
      __syncwarp();
      if (ok && it + kSliceSlots < my_n) issue(gt + kSliceSlots * rg, slot);  // refill the slot just multiplied
      if (!SB_TMA) cp_async_commit();
      if (++slot == kSliceSlots) slot = 0, phase ^= 1u;
    }
    __syncwarp();
    if (lane == 0) um_mbar_arrive(&s_full[buf]);
    if (b > 0) finish_batch(b - 1);
  }
  if (batches > 0) finish_batch(batches - 1);
  if (!SB_TMA) cp_async_wait<0>();
}

struct ExpertPlan {
  int tiles, kw, rg, batch;
  size_t smem;
};
ExpertPlan plan_experts(int N, int K) {
  ExpertPlan t;
  t.tiles = N / 16;
  t.kw = K / 256;
  t.rg = slice_max_warps(1) / t.kw;
  const int warps = t.kw * t.rg;
  const size_t fixed = 1024 + (size_t)warps * kSliceSlots * (slice_slot_codes(1) + kSliceSb), per_round = 2 * (size_t)warps * 512;
  t.batch = 4;  // tiles of a row group between two meetings
  t.smem = fixed + t.batch * per_round;
  return t;
}

int g_sm_count = 0;

int sm_count_or_default() {
  if (g_sm_count == 0) {
    if (gemm_init() != cudaSuccess) {
      (void)cudaGetLastError();
      return 148;  // sizing only: no device in this process
    }
  }
  return g_sm_count;
}

// next[r] = the best of the row-block partial results, lowest index among equals.
__global__ void __launch_bounds__(256) argmax_finish_kernel(const float2* partial, int row_blocks, int32_t* next) {
  __shared__ float sv[8];
  __shared__ int si[8];
  grid_launch_dependents();
  grid_dependency_wait();
  const int req = blockIdx.x;
  float best = -INFINITY;
  int bidx = 0x7fffffff;
  for (int b = threadIdx.x; b < row_blocks; b += blockDim.x) {
    const float2 v = partial[(size_t)b * 16 + req];
    const int i = __float_as_int(v.y);
    if (v.x > best || (v.x == best && i < bidx)) best = v.x, bidx = i;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bidx, o);
    if (ov > best || (ov == best && oi < bidx)) best = ov, bidx = oi;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) sv[warp] = best, si[warp] = bidx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w)
      if (sv[w] > best || (sv[w] == best && si[w] < bidx)) best = sv[w], bidx = si[w];
    next[req] = bidx == 0x7fffffff ? 0 : bidx;
  }
}

}  // namespace

// Dense projections run on the slice kernel; Q4D_GEMM_KERNEL=tcgen05 (read once per process) selects the
// tcgen05 kernel of q4_umma.cu instead, which is correct on every shape but, as measured, not yet faster.
static bool g_legacy = true;
static bool use_umma(int N, int K, int epilogue) { return !g_legacy && umma_supported(N, K, epilogue); }

size_t gemm_partial_bytes(int N, int K, int epilogue) {
  const int sms = sm_count_or_default();
  if (use_umma(N, K, epilogue)) return plan_umma(N, K, epilogue, sms).partial_bytes;
  const size_t a = plan_slices(N, K, 8, epilogue, sms).partial_bytes, b = plan_slices(N, K, 16, epilogue, sms).partial_bytes;
  return a > b ? a : b;
}

int gemm_counters_needed(int N) { return (N + 15) / 16 + 1; }

int gemm_row_blocks(int N, int K, int n, int epilogue) {
  if (use_umma(N, K, epilogue)) return plan_umma(N, K, epilogue, sm_count_or_default()).tiles * 4;  // one per warp of a tile
  const SlicePlan t = plan_slices(N, K, n, epilogue, sm_count_or_default());
  return t.ctas * t.parts * t.kw * t.rg;  // one argmax partial per warp of the grid
}

int gemm_operand_layout() {
  (void)sm_count_or_default();
  return g_legacy ? OPERAND_FRAG : OPERAND_BLOCKED;
}

cudaError_t gemm_init() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int sms = 0;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // 227 KB is the per-CTA limit for static + dynamic shared memory; leave room for the static part.
  const int big = 220 * 1024;
  auto big_smem = [&](auto kernel) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
  };
  big_smem(q4_expert_kernel<true, true>), big_smem(q4_expert_kernel<true, false>);
  big_smem(q4_expert_kernel<false, true>), big_smem(q4_expert_kernel<false, false>);
  big_smem(q4_slice_kernel<1, true>), big_smem(q4_slice_kernel<2, true>);
  big_smem(q4_slice_kernel<1, false>), big_smem(q4_slice_kernel<2, false>);
  if (e != cudaSuccess) return e;
  if (const char* f = getenv("Q4D_GEMM_KERNEL")) g_legacy = strcmp(f, "tcgen05") != 0;
  g_sm_count = sms;
  return cudaSuccess;
}

// The packed codes as bytes [N][K / 2], boxes of 16 rows x 128 bytes (256 codes) with the 128-byte swizzle; scales and biases
// as [N][K / 64], boxes of 16 rows x 8 groups (only where a row is a multiple of 16 bytes: K a multiple of 512).  For a
// gate/up tensor the two halves of the rows are two planes, and a box is 8 rows of both; stacked experts continue the
// planes (gate/up) or the rows.
cudaError_t gemm_make_maps(const uint32_t* qw, const uint16_t* scales, const uint16_t* biases, long long N, int K, bool gate_up,
                           GemmMaps* out, int experts) {
  EncodeTiledFn encode = nullptr;
  const cudaError_t e = encode_tiled_fn(&encode);
  if (e != cudaSuccess) return e;
  auto make = [&](CUtensorMap* m, CUtensorMapDataType type, const void* base, int row_elems, int elem_bytes, unsigned box_x,
                  CUtensorMapSwizzle swizzle) {
    const long long planes = gate_up ? 2 * experts : 1, rows = gate_up ? N / 2 : N * experts;
    const cuuint64_t dims[3] = {(cuuint64_t)row_elems, (cuuint64_t)rows, (cuuint64_t)planes};
    const cuuint64_t strides[2] = {(cuuint64_t)row_elems * elem_bytes, (cuuint64_t)row_elems * elem_bytes * rows};
    const cuuint32_t box[3] = {box_x, gate_up ? 8u : 16u, gate_up ? 2u : 1u}, elem[3] = {1u, 1u, 1u};
    return encode(m, type, 3, const_cast<void*>(base), dims, strides, box, elem, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                  CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  };
  out->sb_tma = K % 512 == 0 && reinterpret_cast<uintptr_t>(scales) % 16 == 0 && reinterpret_cast<uintptr_t>(biases) % 16 == 0;
  bool ok = make(&out->codes, CU_TENSOR_MAP_DATA_TYPE_UINT8, qw, K / 2, 1, 128, CU_TENSOR_MAP_SWIZZLE_128B);
  if (out->sb_tma) {
    ok = ok && make(&out->scales, CU_TENSOR_MAP_DATA_TYPE_UINT16, scales, K / 64, 2, 8, CU_TENSOR_MAP_SWIZZLE_NONE);
    ok = ok && make(&out->biases, CU_TENSOR_MAP_DATA_TYPE_UINT16, biases, K / 64, 2, 8, CU_TENSOR_MAP_SWIZZLE_NONE);
  }
  return ok ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t launch_q4_gemm(const GemmArgs& a, cudaStream_t s) {
  if (g_sm_count == 0) {
    cudaError_t e = gemm_init();
    if (e != cudaSuccess) return e;
  }
  if (a.n <= 0) return cudaSuccess;
  if (a.N <= 0 || a.K <= 0 || (a.K % 256) || a.n > kMaxBatch) return cudaErrorInvalidValue;
  if (a.epilogue == EPI_SILU_PACK && ((a.N % 16) || !a.out_xp)) return cudaErrorInvalidValue;
  if (use_umma(a.N, a.K, a.epilogue)) return launch_q4_umma(a, g_sm_count, s);
  const SlicePlan t = plan_slices(a.N, a.K, a.n, a.epilogue, g_sm_count);
  SliceParams p;
  p.scales = a.scales, p.biases = a.biases, p.xp = a.xp, p.xs = static_cast<const unsigned char*>(a.xs), p.out = a.out;
  p.out_xp = a.out_xp, p.argmax_partial = a.argmax_partial, p.status = a.status;
  p.N = a.N, p.K = a.K, p.n = a.n, p.out_stride = a.out_stride, p.epilogue = a.epilogue;
  p.T = t.T, p.kw = t.kw, p.rg = t.rg, p.batch = t.batch, p.slots = t.slots;
  p.partial = a.partial, p.counters = a.counters;
  if (t.parts > 1 && (!a.partial || !a.counters || t.partial_bytes > a.partial_bytes || t.T > a.counters_len))
    return cudaErrorInvalidValue;
  const int elem = a.epilogue == EPI_F32 ? 4 : 2;
  p.vec_ok = a.out && (reinterpret_cast<uintptr_t>(a.out) % 16 == 0) && ((size_t)a.out_stride * elem % 16 == 0);
  GemmMaps made;
  const GemmMaps* maps = a.maps;
  if (!maps) {
    const cudaError_t e = gemm_make_maps(a.qw, a.scales, a.biases, a.N, a.K, a.epilogue == EPI_SILU_PACK, &made);
    if (e != cudaSuccess) return e;
    maps = &made;
  }
  const dim3 grid(t.ctas, t.parts), block(32 * t.kw * t.rg);
  auto go = [&](auto kernel) { return launch_kernel(kernel, grid, block, t.smem, s, p, *maps); };
  if (t.nt == 2) return maps->sb_tma ? go(q4_slice_kernel<2, true>) : go(q4_slice_kernel<2, false>);
  return maps->sb_tma ? go(q4_slice_kernel<1, true>) : go(q4_slice_kernel<1, false>);
}

cudaError_t launch_q4_experts(const ExpertArgs& a, cudaStream_t s) {
  if (g_sm_count == 0) {
    cudaError_t e = gemm_init();
    if (e != cudaSuccess) return e;
  }
  if (a.N % 16 || a.K % 256 || a.K / 256 > slice_max_warps(1) || !a.maps || !a.units || !a.n_units) return cudaErrorInvalidValue;
  const ExpertPlan t = plan_experts(a.N, a.K);
  if (t.tiles < 2 || t.tiles > 3600) return cudaErrorInvalidValue;  // where tiles_inv is exact for every tile of the list
  ExpertParams p;
  p.scales = a.scales, p.biases = a.biases, p.xp = a.xp, p.xs = static_cast<const unsigned char*>(a.xs), p.out = a.out, p.out_xp = a.out_xp;
  p.status = a.status, p.units = a.units, p.n_units = a.n_units, p.unit_stride = a.unit_stride, p.out_unit_stride = a.out_unit_stride;
  p.N = a.N, p.K = a.K, p.tiles = t.tiles, p.kw = t.kw, p.rg = t.rg, p.batch = t.batch;
  p.tiles_inv = (unsigned)((((unsigned long long)1 << 32) + t.tiles - 1) / t.tiles);
  const dim3 grid(g_sm_count), block(32 * t.kw * t.rg);
  auto go = [&](auto kernel) { return launch_kernel(kernel, grid, block, t.smem, s, p, *a.maps); };
  if (a.gate_up) return a.maps->sb_tma ? go(q4_expert_kernel<true, true>) : go(q4_expert_kernel<true, false>);
  return a.maps->sb_tma ? go(q4_expert_kernel<false, true>) : go(q4_expert_kernel<false, false>);
}

cudaError_t launch_argmax_finish(const float2* partial, int row_blocks, int n, int32_t* next, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  return launch_kernel(argmax_finish_kernel, dim3(n), dim3(256), 0, s, partial, row_blocks, next);
}

}  // namespace q4d
