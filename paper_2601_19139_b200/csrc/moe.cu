// Mixture-of-experts routing for the decode step: router logits, softmax, top-k, the list of experts
// touched by the batch, and the weighted combination of the expert outputs into the residual stream.
//
//   z = Wr y (bf16 dense router, fp32 accumulation);  pi = softmax(z) over all experts;
//   the top_k experts by z (lower index wins a tie), weights pi_k, renormalised to sum 1 if asked;
//   x = bf16(x + bf16(sum_k pi_k * bf16(expert_k output)))
//
// The expert projections themselves run as grouped 4-bit GEMMs over the touched-expert list
// (q4_gemm.cu); every touched expert is evaluated for all requests of the batch and the routing
// weights select what is used, so the packed weights of an expert are streamed once per step.
#include <math.h>

#include "common.cuh"
#include "kernels.h"
#include "launch.h"

namespace q4d {

namespace {

constexpr int kMaxExperts = 256;

// Softmax over the E logits in sz and the top_k experts by logit (lower index wins a tie), by one warp: lane k gets the
// k-th expert and its weight (renormalised to sum 1 if norm).  Logits as integers of the same order, so that the best of
// the warp is one instruction (with ten shuffles and an exponential per expert eight experts took 4.5 us, this 1.1).
__device__ __forceinline__ void select_experts(const float* sz, int E, int top_k, int norm, int lane, int& my_e, float& my_w) {
  // each lane owns experts lane, lane + 32, ...
  float v[kMaxExperts / 32];
  uint32_t key[kMaxExperts / 32];  // 0: none, or taken
  float m = -INFINITY;
#pragma unroll
  for (int i = 0; i < kMaxExperts / 32; ++i) {
    const int e = lane + 32 * i;
    v[i] = e < E ? sz[e] + 0.0f : -INFINITY;  // -0 ties with 0
    m = fmaxf(m, v[i]);
    const uint32_t b = __float_as_uint(v[i]);
    key[i] = e < E ? max((b >> 31) ? ~b : b | 0x80000000u, 1u) : 0u;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  float Z = 0.0f;
#pragma unroll
  for (int i = 0; i < kMaxExperts / 32; ++i)
    if (lane + 32 * i < E) Z += expf(v[i] - m);
  Z = warp_sum(Z);
  my_e = 0;
#pragma unroll 1
  for (int k = 0; k < top_k; ++k) {
    uint32_t best = key[0];
    int e = lane;
#pragma unroll
    for (int i = 1; i < kMaxExperts / 32; ++i)
      if (key[i] > best) best = key[i], e = lane + 32 * i;
    const uint32_t top = __reduce_max_sync(0xffffffffu, best);
    e = (int)__reduce_min_sync(0xffffffffu, best == top ? (uint32_t)e : 0xffffu);
    if (lane == k) my_e = e;
#pragma unroll
    for (int i = 0; i < kMaxExperts / 32; ++i)
      if (e == lane + 32 * i) key[i] = 0u;
  }
  my_w = lane < top_k ? expf(sz[my_e] - m) / Z : 0.0f;
  if (norm) my_w = my_w / warp_sum(my_w);
}

constexpr int kRouterThreads = 512;  // a warp per 128 features, and per request
constexpr int kRouterWarps = kRouterThreads / 32;
constexpr int kExpertWarps = kMaxExperts / 32;

// One CTA per 8 experts, for all requests at once: the warps split the features (128 each), multiply their part of the
// requests (MMA rows) with their part of the 8 router rows (columns) straight from global memory, all loads in flight
// together, and add up in shared memory in feature order.  The CTA that finishes last selects every request's experts (a
// warp per request) and turns the choices into the list of units the expert projections walk.  (One CTA per 8 experts and
// request, with a second hand-over between CTAs to build the list, made the 30B-A3B step at one request 10.68 ms per four
// steps against 10.11.)
__global__ void __launch_bounds__(kRouterThreads) moe_router_kernel(const MoeRouteArgs p, int n) {
  __shared__ float s_part[kRouterWarps][16][8];
  __shared__ float sz[kMaxBatch][kMaxExperts];
  __shared__ int s_last, s_base[kMaxExperts], s_warp_units[kExpertWarps], s_warp_touched[kExpertWarps];
  __shared__ uint32_t s_mask[kMaxExperts];      // requests of an expert
  __shared__ short s_idx[kMaxBatch * 32];       // [request][top_k]
  grid_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int e0 = blockIdx.x * 8;
  const bool active = warp * 128 < p.H;
  uint4 wv[4];
  if (active) {  // the router does not depend on the preceding kernel
    const uint16_t* w = p.router + (size_t)min(e0 + g, p.E - 1) * p.H + warp * 128 + t * 8;
#pragma unroll
    for (int i = 0; i < 4; ++i) wv[i] = __ldg(reinterpret_cast<const uint4*>(w + i * 32));
  }
  if (threadIdx.x < kMaxExperts) s_mask[threadIdx.x] = 0u;
  grid_dependency_wait();
  float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  if (active) {
    const uint16_t* y = p.y + warp * 128 + t * 8;
    const uint16_t *lo = y + (size_t)min(g, n - 1) * p.H, *hi = y + (size_t)min(g + 8, n - 1) * p.H;
    uint4 a[4], b[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const uint4*>(lo + i * 32), b[i] = *reinterpret_cast<const uint4*>(hi + i * 32);
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // a 16-byte load is two k-steps of the same permutation of k on both sides
      mma_bf16(acc, a[i].x, b[i].x, a[i].y, b[i].y, wv[i].x, wv[i].y);
      mma_bf16(acc, a[i].z, b[i].z, a[i].w, b[i].w, wv[i].z, wv[i].w);
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) s_part[warp][g + 8 * (c >> 1)][2 * t + (c & 1)] = acc[c];
  __syncthreads();
  if (threadIdx.x < 128) {
    const int r = threadIdx.x >> 3, e = threadIdx.x & 7;
    float z = 0.0f;
#pragma unroll
    for (int w = 0; w < kRouterWarps; ++w) z += s_part[w][r][e];
    if (r < n && e0 + e < p.E) p.logits[(size_t)r * p.E + e0 + e] = z;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(p.counter, 1) == (int)gridDim.x - 1;
    if (s_last) *p.counter = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int i = threadIdx.x; i < n * p.E; i += kRouterThreads) {
    const int r = i / p.E;
    sz[r][i - r * p.E] = __ldcg(p.logits + i);
  }
  __syncthreads();
  for (int r = warp; r < n; r += kRouterWarps) {
    int my_e;
    float my_w;
    select_experts(sz[r], p.E, p.top_k, p.norm, lane, my_e, my_w);
    if (lane < p.top_k) {
      s_idx[r * p.top_k + lane] = (short)my_e;
      p.wgt[r * p.top_k + lane] = my_w;
      atomicOr(&s_mask[my_e], 1u << r);
    }
  }
  __syncthreads();
  // units in ascending expert order, an expert's requests in ascending order: thread e serves expert e
  const int e = threadIdx.x;
  uint32_t left = e < kMaxExperts ? s_mask[e] : 0u;
  const int count = __popc(left), mine = (count + 7) >> 3;
  int units = mine;  // inclusive prefix sum over the experts
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int a = __shfl_up_sync(0xffffffffu, units, o);
    if (lane >= o) units += a;
  }
  const unsigned touched = __ballot_sync(0xffffffffu, count > 0);
  if (lane == 31 && warp < kExpertWarps) s_warp_units[warp] = units, s_warp_touched[warp] = __popc(touched);
  __syncthreads();
  if (e < kMaxExperts) {
#pragma unroll
    for (int w = 0; w < kExpertWarps; ++w) units += w < warp ? s_warp_units[w] : 0;
    s_base[e] = units - mine;
    for (int u = 0; u < mine; ++u) {
      uint32_t ids[2] = {0u, 0u};
      int k = 0;
      for (; k < 8 && left; ++k, left &= left - 1u) ids[k >> 2] |= (uint32_t)(__ffs(left) - 1) << ((k & 3) * 8);
      p.units[units - mine + u] = make_int4(e, k, (int)ids[0], (int)ids[1]);
    }
    if (e == kMaxExperts - 1) {
      *p.n_units = units;
      int tot = 0;
#pragma unroll
      for (int w = 0; w < kExpertWarps; ++w) tot += s_warp_touched[w];
      if (p.touched_total) atomicAdd(p.touched_total, tot);  // nobody waits for it
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n * p.top_k; i += kRouterThreads) {
    const int ex = s_idx[i], r = i / p.top_k;
    p.pos[i] = s_base[ex] * 8 + __popc(s_mask[ex] & ((1u << r) - 1u));  // full units of 8 follow one another
  }
}

// acc += w * the 8 bf16 values of v
__device__ __forceinline__ void add_weighted(float (&acc)[8], float w, const uint4 v) {
  const uint32_t vw[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    acc[2 * i] = fmaf(w, bf16_lo(vw[i]), acc[2 * i]);
    acc[2 * i + 1] = fmaf(w, bf16_hi(vw[i]), acc[2 * i + 1]);
  }
}
// bf16(x + bf16(acc)) of 8 elements
__device__ __forceinline__ uint4 add_to_residual(const uint4 xv, const float (&acc)[8]) {
  const uint32_t xw[4] = {xv.x, xv.y, xv.z, xv.w};
  uint32_t ow[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float d0 = bf16_to_f32(f32_to_bf16(acc[2 * i])), d1 = bf16_to_f32(f32_to_bf16(acc[2 * i + 1]));
    ow[i] = pack_bf16x2(bf16_lo(xw[i]) + d0, bf16_hi(xw[i]) + d1);
  }
  return make_uint4(ow[0], ow[1], ow[2], ow[3]);
}

// x[r] = bf16(x[r] + bf16(sum_k wgt[r][k] * o[pos[r][k]])), and the next norm of it as the next projection's operand: one
// CTA per request, a thread per 8 consecutive elements.  Everything but the experts' outputs (the router's choice, the
// residual stream, the norm weights: all from kernels that had ended before the preceding one started) is read before
// that one is awaited, the outputs eight at a time.  (As two kernels: 4.6 and 2.0 us a layer at one request.)
__global__ void __launch_bounds__(256) moe_combine_norm_kernel(const MoeCombineArgs p) {
  __shared__ float red[8];
  grid_launch_dependents();
  const int r = blockIdx.x, c = threadIdx.x, lane = c & 31, warp = c >> 5;
  const bool in = c < (p.H >> 3);
  uint16_t* x = p.x + (size_t)r * p.H + c * 8;
  uint4 xv = make_uint4(0u, 0u, 0u, 0u), wv = xv;
  if (in) xv = __ldcg(reinterpret_cast<const uint4*>(x)), wv = __ldg(reinterpret_cast<const uint4*>(p.norm + c * 8));
  int pos = 0;
  float wgt = 0.0f;
  if (lane < p.top_k) pos = __ldcg(p.pos + r * p.top_k + lane), wgt = __ldcg(p.wgt + r * p.top_k + lane);
  grid_dependency_wait();
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
  for (int k0 = 0; k0 < p.top_k; k0 += 8) {
    uint4 o[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int at = __shfl_sync(0xffffffffu, pos, (k0 + k) & 31);
      o[k] = make_uint4(0u, 0u, 0u, 0u);
      if (in && k0 + k < p.top_k) o[k] = __ldcg(reinterpret_cast<const uint4*>(p.o + (size_t)at * p.H + c * 8));
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float w = __shfl_sync(0xffffffffu, wgt, (k0 + k) & 31);
      if (k0 + k < p.top_k) add_weighted(acc, w, o[k]);
    }
  }
  const uint4 xn = add_to_residual(xv, acc);
  if (in) *reinterpret_cast<uint4*>(x) = xn;
  const uint32_t e[4] = {xn.x, xn.y, xn.z, xn.w}, ww[4] = {wv.x, wv.y, wv.z, wv.w};
  float ss = 0.0f;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float a = bf16_lo(e[j]), b = bf16_hi(e[j]);
    if (in) ss = fmaf(a, a, ss), ss = fmaf(b, b, ss);
  }
  ss = warp_sum(ss);
  if (lane == 0) red[warp] = ss;
  __syncthreads();
  float tot = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) tot += red[i];
  const float inv = 1.0f / sqrtf(tot / (float)p.H + p.eps);
  uint32_t y[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) y[j] = pack_bf16x2(bf16_lo(e[j]) * inv * bf16_lo(ww[j]), bf16_hi(e[j]) * inv * bf16_hi(ww[j]));
  const uint4 v = make_uint4(y[0], y[1], y[2], y[3]);
  const float gsum = group_sum_8lanes(chunk_sum(v));
  if (in) {
    store_operand_chunk(p.layout, p.yp, p.H, r, c, v);
    if ((c & 7) == 0) store_operand_sum(p.layout, p.ys, r, c >> 3, gsum);
  }
}

// ---- many tokens (prompt processing) -------------------------------------------------------------------------------
constexpr int kPrefillRouterThreads = 512;
constexpr int kPrefillRouterWarps = kPrefillRouterThreads / 32;
// Parts of the features, so that sixteen warps have a tile of 16 experts each (128 experts: two parts).
__host__ __device__ inline int prefill_router_parts(int E) { return E <= 64 ? 4 : E <= 128 ? 2 : 1; }

// Router of 16 tokens per CTA: logits on m16n8k16 MMAs with fp32 accumulation (rows = experts, columns = tokens; a lane's
// 16-byte loads hold two k-steps of the same permutation of k on both sides), then one warp per token selects.  A warp's
// time is the latency of its router loads, one batch after another: sixteen of them in flight, and the features split
// over the warps that the experts leave (eight loads, unsplit, and two tokens per warp: 31 us for 500 tokens).
__global__ void __launch_bounds__(kPrefillRouterThreads) prefill_router_kernel(const PrefillMoeArgs p) {
  extern __shared__ __align__(16) unsigned char router_smem[];
  const int stride = p.H * 2 + 16;                                      // bytes per token row: 16 apart modulo 128
  float* sz = reinterpret_cast<float*>(router_smem + 16 * stride);      // [part][16][E]
  grid_launch_dependents();
  grid_dependency_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int t0 = blockIdx.x * 16, chunks = p.H >> 3, parts = prefill_router_parts(p.E), len = p.H / parts;
  for (int r = warp; r < 16; r += kPrefillRouterWarps) {
    const uint4* src = reinterpret_cast<const uint4*>(p.y + (size_t)min(t0 + r, p.rows - 1) * p.H);
#pragma unroll 8
    for (int k = lane; k < chunks; k += 32) *reinterpret_cast<uint4*>(router_smem + r * stride + k * 16) = src[k];
  }
  __syncthreads();
  const int tiles = (p.E + 15) >> 4;
  for (int w = warp; w < tiles * parts; w += kPrefillRouterWarps) {
    const int part = w / tiles, e0 = (w - part * tiles) * 16, k1 = (part + 1) * len;
    const uint16_t* w_lo = p.router + (size_t)min(e0 + g, p.E - 1) * p.H + t * 8;
    const uint16_t* w_hi = p.router + (size_t)min(e0 + g + 8, p.E - 1) * p.H + t * 8;
    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll 8
    for (int k = part * len; k < k1; k += 32) {
      const uint4 a = __ldg(reinterpret_cast<const uint4*>(w_lo + k)), b = __ldg(reinterpret_cast<const uint4*>(w_hi + k));
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        const uint4 x = *reinterpret_cast<const uint4*>(router_smem + (nt * 8 + g) * stride + k * 2 + t * 16);
        mma_bf16(acc[nt], a.x, b.x, a.y, b.y, x.x, x.y);
        mma_bf16(acc[nt], a.z, b.z, a.w, b.w, x.z, x.w);
      }
    }
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int e = e0 + g + 8 * (c >> 1);
        if (e < p.E) sz[(part * 16 + nt * 8 + 2 * t + (c & 1)) * p.E + e] = acc[nt][c];
      }
  }
  __syncthreads();
  for (int i = warp; i < 16 && t0 + i < p.rows; i += kPrefillRouterWarps) {
    for (int e = lane; e < p.E; e += 32) {  // the parts in order; a lane reads what it has added up
      float z = sz[i * p.E + e];
      for (int q = 1; q < parts; ++q) z += sz[(q * 16 + i) * p.E + e];
      sz[i * p.E + e] = z;
    }
    __syncwarp();
    int e;
    float w;
    select_experts(sz + i * p.E, p.E, p.top_k, p.norm, lane, e, w);
    if (lane < p.top_k) {
      p.idx[(size_t)(t0 + i) * p.top_k + lane] = e;
      p.wgt[(size_t)(t0 + i) * p.top_k + lane] = w;
      atomicAdd(p.counts + e, 1);
    }
  }
}

// Rows of the sorted operand per expert (cursor = its first row) and the list of units; counts return to zero.
__global__ void __launch_bounds__(kMaxExperts) prefill_units_kernel(const PrefillMoeArgs p) {
  __shared__ int s_rows[kMaxExperts / 32], s_units[kMaxExperts / 32];
  grid_launch_dependents();
  grid_dependency_wait();
  const int e = threadIdx.x, warp = e >> 5, lane = e & 31;
  const int cnt = e < p.E ? p.counts[e] : 0, un = (cnt + p.unit_rows - 1) / p.unit_rows;
  int rows = cnt, units = un;  // inclusive prefix sums over the experts
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int a = __shfl_up_sync(0xffffffffu, rows, o), b = __shfl_up_sync(0xffffffffu, units, o);
    if (lane >= o) rows += a, units += b;
  }
  if (lane == 31) s_rows[warp] = rows, s_units[warp] = units;
  __syncthreads();
  for (int w = 0; w < warp; ++w) rows += s_rows[w], units += s_units[w];
  if (e < p.E) p.cursor[e] = rows - cnt, p.counts[e] = 0;
  for (int i = 0; i < un; ++i)
    p.units[units - un + i] = make_int4(e, rows - cnt + i * p.unit_rows, min(p.unit_rows, cnt - i * p.unit_rows), 0);
  if (e == kMaxExperts - 1) *p.n_units = units;
}

// Copies a token's operand row to the next free row of each of its experts (the order within an expert is arbitrary:
// a row's results do not depend on its neighbours).  One CTA per token, one warp per expert.
__global__ void __launch_bounds__(256) prefill_scatter_kernel(const PrefillMoeArgs p) {
  grid_launch_dependents();
  grid_dependency_wait();
  const int r = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunks = prefill_operand_stride(p.H) >> 3;
  const uint4* src = reinterpret_cast<const uint4*>(p.operand) + (size_t)r * chunks;
  for (int k = warp; k < p.top_k; k += 8) {
    int row = 0;
    if (lane == 0) {
      row = atomicAdd(p.cursor + p.idx[(size_t)r * p.top_k + k], 1);
      p.pos[(size_t)r * p.top_k + k] = row;
      p.sorted_inv_scale[row] = p.inv_scale[r];
    }
    row = __shfl_sync(0xffffffffu, row, 0);
    uint4* dst = reinterpret_cast<uint4*>(p.sorted) + (size_t)row * chunks;
    for (int c = lane; c < chunks; c += 32) dst[c] = src[c];
  }
}

// x[r] = bf16(x[r] + bf16(sum_k wgt[r][k] * o[pos[r][k]]))
__global__ void __launch_bounds__(256) prefill_combine_kernel(const PrefillMoeArgs p) {
  grid_launch_dependents();
  grid_dependency_wait();
  const int r = blockIdx.x;
  for (int c = threadIdx.x; c < (p.H >> 3); c += 256) {
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int k = 0; k < p.top_k; ++k) {
      const float w = p.wgt[(size_t)r * p.top_k + k];
      add_weighted(acc, w, *reinterpret_cast<const uint4*>(p.o + (size_t)p.pos[(size_t)r * p.top_k + k] * p.H + c * 8));
    }
    uint4* x = reinterpret_cast<uint4*>(p.x + (size_t)r * p.H + c * 8);
    *x = add_to_residual(*x, acc);
  }
}

}  // namespace

cudaError_t launch_moe_router(const MoeRouteArgs& a, int n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (a.E < 1 || a.E > kMaxExperts || a.top_k < 1 || a.top_k > 32 || a.top_k > a.E || a.H % 8) return cudaErrorInvalidValue;
  if (a.H % 128 || a.H > kRouterWarps * 128 || n > kMaxBatch || !a.logits) return cudaErrorInvalidValue;
  return launch_kernel(moe_router_kernel, dim3((a.E + 7) / 8), dim3(kRouterThreads), 0, s, a, n);
}

cudaError_t launch_moe_combine_norm(const MoeCombineArgs& a, int n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (a.H % 64 || a.H > 2048 || a.top_k > 32) return cudaErrorInvalidValue;
  return launch_kernel(moe_combine_norm_kernel, dim3(n), dim3(256), 0, s, a);
}

cudaError_t launch_prefill_route(const PrefillMoeArgs& a, cudaStream_t s) {
  if (a.rows <= 0) return cudaSuccess;
  if (a.E < 1 || a.E > kMaxExperts || a.top_k < 1 || a.top_k > 32 || a.top_k > a.E || a.H % 256) return cudaErrorInvalidValue;
  const size_t smem = 16 * ((size_t)a.H * 2 + 16) + (size_t)prefill_router_parts(a.E) * 16 * a.E * sizeof(float);
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(prefill_router_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  if (smem > 160 * 1024) return cudaErrorInvalidValue;
  cudaError_t e = launch_kernel(prefill_router_kernel, dim3((a.rows + 15) / 16), dim3(kPrefillRouterThreads), smem, s, a);
  if (e == cudaSuccess) e = launch_kernel(prefill_units_kernel, dim3(1), dim3(kMaxExperts), 0, s, a);
  if (e == cudaSuccess) e = launch_kernel(prefill_scatter_kernel, dim3(a.rows), dim3(256), 0, s, a);
  return e;
}

cudaError_t launch_prefill_combine(const PrefillMoeArgs& a, cudaStream_t s) {
  if (a.rows <= 0) return cudaSuccess;
  return launch_kernel(prefill_combine_kernel, dim3(a.rows), dim3(256), 0, s, a);
}

}  // namespace q4d
