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
// k-th expert and its weight (renormalised to sum 1 if norm).
__device__ __forceinline__ void select_experts(const float* sz, int E, int top_k, int norm, int lane, int& my_e, float& my_w) {
  // each lane owns experts lane, lane + 32, ...
  float v[kMaxExperts / 32];
  float m = -INFINITY;
#pragma unroll
  for (int i = 0; i < kMaxExperts / 32; ++i) {
    const int e = lane + 32 * i;
    v[i] = e < E ? sz[e] : -INFINITY;
    m = fmaxf(m, v[i]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  float Z = 0.0f;
#pragma unroll
  for (int i = 0; i < kMaxExperts / 32; ++i)
    if (lane + 32 * i < E) Z += expf(v[i] - m);
  Z = warp_sum(Z);
  float sel_sum = 0.0f;
  my_w = 0.0f, my_e = 0;
  for (int k = 0; k < top_k; ++k) {
    float best = -INFINITY;
    int bidx = 0x7fffffff;
#pragma unroll
    for (int i = 0; i < kMaxExperts / 32; ++i) {
      const int e = lane + 32 * i;
      if (v[i] > best || (v[i] == best && v[i] != -INFINITY && e < bidx)) best = v[i], bidx = e;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bidx, o);
      if (ov > best || (ov == best && oi < bidx)) best = ov, bidx = oi;
    }
    if (bidx == 0x7fffffff) bidx = k;  // logits that are not numbers: some expert
    const float wk = expf(best - m) / Z;
    sel_sum += wk;
    if (lane == k) my_e = bidx, my_w = wk;
    if ((bidx & 31) == lane) {  // remove the winner from its owner's candidates
#pragma unroll
      for (int i = 0; i < kMaxExperts / 32; ++i)
        if (i == (bidx >> 5)) v[i] = -INFINITY;
    }
  }
  if (norm) my_w = my_w / sel_sum;
}

constexpr int kRouterThreads = 256;
constexpr int kRouterWarps = kRouterThreads / 32;

// CTA (slice, request): the request's row is staged in shared memory and each warp computes the logits of one or
// more experts of the slice, keeping eight 16-byte loads of a router row in flight per lane (the router matrix is
// small, 512 KB for 128 experts of width 2048, so it is spread over many SMs and the loads overlap).  A lane adds
// its chunks lane, lane + 32, ... in ascending order.  The logits go to global memory; the CTA that finishes a
// request's last slice selects its experts, and the CTA that finishes the last request compacts the touched-expert
// flags into a list.
__global__ void __launch_bounds__(kRouterThreads) moe_router_kernel(const MoeRouteArgs p) {
  extern __shared__ __align__(16) unsigned char router_smem[];
  uint4* sy = reinterpret_cast<uint4*>(router_smem);  // the row: H / 8 chunks of 8 bf16
  __shared__ float sz[kMaxExperts];
  __shared__ int s_last;
  __shared__ int s_warp_base[kRouterWarps];
  grid_launch_dependents();
  const int r = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunks = p.H >> 3;
  const int per_slice = (p.E + (int)gridDim.x - 1) / (int)gridDim.x;
  const int e_begin = blockIdx.x * per_slice, e_end = min(p.E, e_begin + per_slice);
  grid_dependency_wait();
  {
    const uint4* y = reinterpret_cast<const uint4*>(p.y + (size_t)r * p.H);
    for (int c = threadIdx.x; c < chunks; c += kRouterThreads) sy[c] = y[c];
  }
  __syncthreads();
  for (int e = e_begin + warp; e < e_end; e += kRouterWarps) {
    const uint4* wr = reinterpret_cast<const uint4*>(p.router + (size_t)e * p.H);
    float acc = 0.0f;
    for (int c0 = lane; c0 < chunks; c0 += 32 * 8) {
      uint4 a[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int c = c0 + 32 * i;
        a[i] = c < chunks ? __ldg(wr + c) : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int c = c0 + 32 * i;
        if (c < chunks) {
          const uint4 b = sy[c];
          const uint32_t aw[4] = {a[i].x, a[i].y, a[i].z, a[i].w}, bw[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            acc = fmaf(bf16_lo(aw[j]), bf16_lo(bw[j]), acc);
            acc = fmaf(bf16_hi(aw[j]), bf16_hi(bw[j]), acc);
          }
        }
      }
    }
    acc = warp_sum(acc);
    if (lane == 0) p.logits[(size_t)r * p.E + e] = acc;
  }
  // ---- the CTA with the request's last slice selects the experts ----
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = (atomicAdd(p.slice_counter + r, 1) == (int)gridDim.x - 1);
    if (s_last) p.slice_counter[r] = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int e = threadIdx.x; e < p.E; e += kRouterThreads) sz[e] = __ldcg(p.logits + (size_t)r * p.E + e);
  __syncthreads();
  if (warp == 0) {
    int my_e;
    float my_w;
    select_experts(sz, p.E, p.top_k, p.norm, lane, my_e, my_w);
    if (lane < p.top_k) {
      p.idx[r * p.top_k + lane] = my_e;
      p.wgt[r * p.top_k + lane] = my_w;
      p.flags[my_e] = 1;
    }
  }
  // ---- the last CTA builds the list of touched experts, in ascending expert order ----
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = (atomicAdd(p.counter, 1) == (int)gridDim.y - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int e = threadIdx.x;
  const int f = (e < p.E) ? __ldcg(p.flags + e) : 0;
  const unsigned ball = __ballot_sync(0xffffffffu, f != 0);
  if (lane == 0) s_warp_base[warp] = __popc(ball);
  __syncthreads();
  int base = 0;
  for (int w = 0; w < warp; ++w) base += s_warp_base[w];
  if (f) {
    const int pos = base + __popc(ball & ((1u << lane) - 1u));
    p.expert_ids[pos] = e;
    p.slot_of[e] = pos;
  }
  if (e < p.E) p.flags[e] = 0;
  if (threadIdx.x == 0) {
    int tot = 0;
    for (int w = 0; w < kMaxExperts / 32; ++w) tot += s_warp_base[w];
    *p.n_touched = tot;
    *p.counter = 0;
    if (p.touched_total) *p.touched_total += tot;  // one CTA per launch, launches of a step are stream-ordered
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
// x[0..8) = bf16(x + bf16(acc))
__device__ __forceinline__ void add_to_residual(uint16_t* x, const float (&acc)[8]) {
  const uint4 xv = *reinterpret_cast<const uint4*>(x);
  const uint32_t xw[4] = {xv.x, xv.y, xv.z, xv.w};
  uint32_t ow[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float d0 = bf16_to_f32(f32_to_bf16(acc[2 * i])), d1 = bf16_to_f32(f32_to_bf16(acc[2 * i + 1]));
    ow[i] = pack_bf16x2(bf16_lo(xw[i]) + d0, bf16_hi(xw[i]) + d1);
  }
  *reinterpret_cast<uint4*>(x) = make_uint4(ow[0], ow[1], ow[2], ow[3]);
}

// x[r] = bf16(x[r] + bf16(sum_k wgt[r][k] * o[slot_of[idx[r][k]]][r])); a thread takes 8 consecutive elements.
__global__ void __launch_bounds__(256) moe_combine_kernel(const MoeCombineArgs p) {
  grid_launch_dependents();
  grid_dependency_wait();
  const int r = blockIdx.y;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= (p.H >> 3)) return;
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (int k = 0; k < p.top_k; ++k) {
    const int slot = p.slot_of[p.idx[r * p.top_k + k]];
    const float w = p.wgt[r * p.top_k + k];
    add_weighted(acc, w, *reinterpret_cast<const uint4*>(p.o + ((size_t)slot * 16 + r) * p.H + c * 8));
  }
  add_to_residual(p.x + (size_t)r * p.H + c * 8, acc);
}

// ---- many tokens (prompt processing) -------------------------------------------------------------------------------
// Router of 16 tokens per CTA: logits on m16n8k16 MMAs with fp32 accumulation (rows = experts, columns = tokens; a lane's
// 16-byte loads hold two k-steps of the same permutation of k on both sides), then one warp per token selects.
__global__ void __launch_bounds__(kRouterThreads) prefill_router_kernel(const PrefillMoeArgs p) {
  extern __shared__ __align__(16) unsigned char router_smem[];
  const int stride = p.H * 2 + 16;                                      // bytes per token row: 16 apart modulo 128
  float* sz = reinterpret_cast<float*>(router_smem + 16 * stride);      // [16][E]
  grid_launch_dependents();
  grid_dependency_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int t0 = blockIdx.x * 16, chunks = p.H >> 3;
  for (int c = threadIdx.x; c < 16 * chunks; c += kRouterThreads) {
    const int r = c / chunks, k = c - r * chunks;
    *reinterpret_cast<uint4*>(router_smem + r * stride + k * 16) =
        *reinterpret_cast<const uint4*>(p.y + (size_t)min(t0 + r, p.rows - 1) * p.H + k * 8);
  }
  __syncthreads();
  for (int e0 = warp * 16; e0 < p.E; e0 += kRouterWarps * 16) {
    const uint16_t* w_lo = p.router + (size_t)min(e0 + g, p.E - 1) * p.H + t * 8;
    const uint16_t* w_hi = p.router + (size_t)min(e0 + g + 8, p.E - 1) * p.H + t * 8;
    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll 4
    for (int k = 0; k < p.H; k += 32) {
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
        if (e < p.E) sz[(nt * 8 + 2 * t + (c & 1)) * p.E + e] = acc[nt][c];
      }
  }
  __syncthreads();
  for (int i = warp; i < 16 && t0 + i < p.rows; i += kRouterWarps) {
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
    add_to_residual(p.x + (size_t)r * p.H + c * 8, acc);
  }
}

}  // namespace

cudaError_t launch_moe_router(const MoeRouteArgs& a, int n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (a.E < 1 || a.E > kMaxExperts || a.top_k < 1 || a.top_k > 32 || a.top_k > a.E || a.H % 8) return cudaErrorInvalidValue;
  if ((size_t)a.H * 2 > 48 * 1024 || !a.logits || !a.slice_counter) return cudaErrorInvalidValue;
  const int slices = (a.E + kRouterWarps - 1) / kRouterWarps;  // one expert per warp while that gives at most 32 slices
  return launch_kernel(moe_router_kernel, dim3(slices < 32 ? slices : 32, n), dim3(kRouterThreads), (size_t)a.H * 2, s, a);
}

cudaError_t launch_moe_combine(const MoeCombineArgs& a, int n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int chunks = a.H >> 3;
  return launch_kernel(moe_combine_kernel, dim3((chunks + 255) / 256, n), dim3(256), 0, s, a);
}

cudaError_t launch_prefill_route(const PrefillMoeArgs& a, cudaStream_t s) {
  if (a.rows <= 0) return cudaSuccess;
  if (a.E < 1 || a.E > kMaxExperts || a.top_k < 1 || a.top_k > 32 || a.top_k > a.E || a.H % 256) return cudaErrorInvalidValue;
  const size_t smem = 16 * ((size_t)a.H * 2 + 16) + (size_t)16 * a.E * sizeof(float);
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(prefill_router_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  if (smem > 160 * 1024) return cudaErrorInvalidValue;
  cudaError_t e = launch_kernel(prefill_router_kernel, dim3((a.rows + 15) / 16), dim3(kRouterThreads), smem, s, a);
  if (e == cudaSuccess) e = launch_kernel(prefill_units_kernel, dim3(1), dim3(kMaxExperts), 0, s, a);
  if (e == cudaSuccess) e = launch_kernel(prefill_scatter_kernel, dim3(a.rows), dim3(256), 0, s, a);
  return e;
}

cudaError_t launch_prefill_combine(const PrefillMoeArgs& a, cudaStream_t s) {
  if (a.rows <= 0) return cudaSuccess;
  return launch_kernel(prefill_combine_kernel, dim3(a.rows), dim3(256), 0, s, a);
}

}  // namespace q4d
