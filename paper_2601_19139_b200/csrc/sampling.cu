// Seeded temperature / top-k / top-p sampling of the next token from fp32 logits (GenerateToken beyond greedy).
//
// Definition (per request; l = logits, T = temperature > 0, V = vocabulary):
//   w_j    = rint(2^40 * exp((l_j - max l) / T))                     integer weights: sums are exact in any order
//   top-k  : keep { j : l_j >= the k-th largest logit }              (k <= 0 or k >= V: keep all; ties at the cut stay)
//   top-p  : with W_k the kept weight, keep { j : l_j >= c } for the largest value c whose set weighs >= top_p * W_k
//   draw   : W = weight of the kept set, t = floor(u * W) for the given u in [0, 1); walk the kept tokens by
//            descending logit, ascending index among equal logits, and take the first whose running weight exceeds t.
// T <= 0 selects the greedy token (largest logit, lowest index among equals).
//
// A cluster of eight CTAs per request: every CTA keeps an eighth of the logits in shared memory, so they are read from
// global memory once, and 128 SMs work on sixteen requests (one CTA per request, five to twelve passes over the logits
// in L2, took 345 us at V = 151936; this takes the time of one launch and a few cluster barriers).  The cut that comes
// first (top-k by counts, else top-p or the draw by weights) is narrowed by one histogram over the leading 11 bits of the
// order-preserving image of the logits; the tokens at or above the bin where it falls, usually a few hundred, are gathered
// into the first CTA, sorted, and everything else is a prefix sum there.  Only when more than 4096 tokens are left does
// the descent go on to the next bits, and past the last bit to the next cut, over the whole vocabulary.
#include <cooperative_groups.h>
#include <math.h>

#include "common.cuh"
#include "kernels.h"
#include "launch.h"

namespace q4d {

namespace {

namespace cg = cooperative_groups;

constexpr int kSampleCtas = 8;  // CTAs per request: one cluster
constexpr int kSampleThreads = 1024;
constexpr int kSampleBins = 2048;
constexpr int kSampleList = 4096;       // tokens the first CTA sorts
constexpr int kSampleSlice = 32 * 1024;  // logits a CTA keeps in shared memory; longer slices are read again from global memory
constexpr int kSampleWide = 1 << 17;    // slices beyond this could overflow 32-bit sums of 14-bit pieces

// larger float <=> larger key
__device__ __forceinline__ uint32_t order_key(float l) {
  const uint32_t u = __float_as_uint(l);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_value(uint32_t k) { return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k); }

struct SampleShared {
  uint32_t cnt[kSampleBins];               // this CTA's histogram: counts, and weights in three pieces of 14 bits
  uint32_t part[3][kSampleBins];           // (slices beyond kSampleWide: 64-bit sums in the first two)
  unsigned long long mass[kSampleBins];    // first CTA: the cluster's totals
  uint32_t total[kSampleBins];
  unsigned long long list[kSampleList];    // first CTA: (key, ~index) of the gathered tokens
  unsigned long long red[32];
  // results of the first CTA's scan, read by all
  unsigned long long w_all, w_gt, w_bin;
  uint32_t bin, c_gt, c_bin, list_count;
  float best;
  int best_idx;
  uint32_t equal;
};

// the draw's target over a set of weight W: t + 1 for t = floor(u * W)
__device__ __forceinline__ unsigned long long draw_target(float u, unsigned long long W) {
  unsigned long long t = (unsigned long long)((double)u * (double)W);
  if (t >= W) t = W - 1ull;
  return t + 1ull;
}
// top-p's target: ceil(p * W) within [1, W]
__device__ __forceinline__ unsigned long long top_p_target(float p, unsigned long long W) {
  unsigned long long t = (unsigned long long)ceil((double)p * (double)W);
  if (t < 1ull) t = 1ull;
  return t > W ? W : t;
}

// Exclusive prefix sum over the block's threads (red: 32 words of scratch); *all gets the total.
__device__ __forceinline__ unsigned long long block_scan(unsigned long long v, unsigned long long* red, unsigned long long* all) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long a = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += a;
  }
  if (lane == 31) red[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    unsigned long long w = red[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long a = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += a;
    }
    red[lane] = w;
  }
  __syncthreads();
  const unsigned long long before = (warp ? red[warp - 1] : 0ull) + incl - v;
  *all = red[31];
  __syncthreads();
  return before;
}

enum { CUT_K = 0, CUT_P = 1, CUT_DRAW = 2 };

__global__ void __cluster_dims__(kSampleCtas, 1, 1) __launch_bounds__(kSampleThreads) sample_kernel(const SampleArgs a) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  SampleShared& s = *reinterpret_cast<SampleShared*>(dyn_smem);
  float* kept = reinterpret_cast<float*>(dyn_smem + sizeof(SampleShared));
  cg::cluster_group cluster = cg::this_cluster();

  grid_launch_dependents();
  grid_dependency_wait();

  const int r = blockIdx.x / kSampleCtas, rank = (int)cluster.block_rank(), V = a.vocab, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  SampleShared& lead = *cluster.map_shared_rank(&s, 0);
  const int per = (V + kSampleCtas - 1) / kSampleCtas, j0 = min(V, rank * per), L = min(V, j0 + per) - j0;
  const float* row = a.logits + (size_t)r * V + j0;
  const float* src = per <= kSampleSlice ? kept : row;
  const float T = a.temperature[r];

  // ---- the slice into shared memory; largest logit and its first index ----
  float best = -INFINITY;
  int bidx = 0x7fffffff;
  for (int j = tid; j < L; j += kSampleThreads) {
    const float v = row[j];
    if (per <= kSampleSlice) kept[j] = v;
    if (v > best) best = v, bidx = j0 + j;
  }
  auto better = [](float ov, int oi, float bv, int bi) { return ov > bv || (ov == bv && oi < bi); };
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bidx, o);
    if (better(ov, oi, best, bidx)) best = ov, bidx = oi;
  }
  float* redf = reinterpret_cast<float*>(s.part[0]);
  int* redi = reinterpret_cast<int*>(s.part[1]);
  if (lane == 0) redf[warp] = best, redi[warp] = bidx;
  __syncthreads();
  if (warp == 0) {
    best = redf[lane], bidx = redi[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bidx, o);
      if (better(ov, oi, best, bidx)) best = ov, bidx = oi;
    }
    if (lane == 0) s.best = best, s.best_idx = bidx, s.list_count = 0u;
  }
  cluster.sync();
  best = -INFINITY, bidx = 0x7fffffff;
#pragma unroll
  for (int q = 0; q < kSampleCtas; ++q) {
    const SampleShared& o = *cluster.map_shared_rank(&s, q);
    const float ov = o.best;
    const int oi = o.best_idx;
    if (better(ov, oi, best, bidx)) best = ov, bidx = oi;
  }
  if (!(T > 0.0f)) {
    if (rank == 0 && tid == 0) a.next[r] = bidx == 0x7fffffff ? 0 : bidx;
    cluster.sync();  // nobody leaves while its shared memory is read
    return;
  }
  const float m = best, inv_t = 1.0f / T;
  auto weight = [&](float l) -> unsigned long long {
    return (unsigned long long)__float2ull_rn(expf((l - m) * inv_t) * 1099511627776.0f);  // 2^40
  };
  const bool wide = per > kSampleWide;
  unsigned long long* wide_mass = reinterpret_cast<unsigned long long*>(s.part[0]);

  // ---- one cut after another over the whole vocabulary, until the tokens that are left fit the list ----
  const int k = a.top_k[r];
  const float p = a.top_p[r];
  int cut = k > 0 && k < V ? CUT_K : (p < 1.0f ? CUT_P : CUT_DRAW);
  uint32_t floor_key = 0u;        // tokens below are out
  unsigned long long W = 0;       // weight of the tokens at or above floor_key, once known
  bool know_w = false, listed = false;
  unsigned long long target = 0;
  while (!listed) {
    uint32_t prefix = 0u;
    unsigned long long w_gt = 0ull;
    uint32_t c_gt = 0u;
    for (int d = 0; d < 3; ++d) {
      const int shift = d == 0 ? 21 : (d == 1 ? 10 : 0), bins = d == 2 ? 1024 : 2048;
      const uint32_t hi_mask = d == 0 ? 0u : (d == 1 ? 0xffe00000u : 0xfffffc00u);
      for (int b = tid; b < kSampleBins; b += kSampleThreads) s.cnt[b] = s.part[0][b] = s.part[1][b] = s.part[2][b] = 0u;
      __syncthreads();
      for (int j = tid; j < L; j += kSampleThreads) {
        const float l = src[j];
        const uint32_t key = order_key(l);
        if (key < floor_key || (key & hi_mask) != prefix) continue;
        const uint32_t b = (key >> shift) & (bins - 1);
        atomicAdd(&s.cnt[b], 1u);
        if (cut == CUT_K) continue;  // by counts alone
        const unsigned long long w = weight(l);
        if (wide) {
          atomicAdd(&wide_mass[b], w);
        } else if (w) {
          atomicAdd(&s.part[0][b], (uint32_t)w & 0x3fffu);
          atomicAdd(&s.part[1][b], (uint32_t)(w >> 14) & 0x3fffu);
          atomicAdd(&s.part[2][b], (uint32_t)(w >> 28));
        }
      }
      cluster.sync();
      // each CTA adds up an eighth of the bins for the first one
      if (tid < kSampleBins / kSampleCtas) {
        const int b = rank * (kSampleBins / kSampleCtas) + tid;
        uint32_t c = 0u;
        unsigned long long mm = 0ull;
#pragma unroll
        for (int q = 0; q < kSampleCtas; ++q) {
          const SampleShared& o = *cluster.map_shared_rank(&s, q);
          c += o.cnt[b];
          if (cut != CUT_K)
            mm += wide ? reinterpret_cast<const unsigned long long*>(o.part[0])[b]
                       : (unsigned long long)o.part[0][b] + ((unsigned long long)o.part[1][b] << 14) + ((unsigned long long)o.part[2][b] << 28);
        }
        lead.total[b] = c, lead.mass[b] = mm;
      }
      cluster.sync();
      if (rank == 0) {
        // thread i: bins `bins` - 1 - 2i and the one below, in descending order
        const int b1 = bins - 1 - 2 * tid, b0 = b1 - 1;
        const bool in = b0 >= 0;
        const unsigned long long m1 = in ? s.mass[b1] : 0ull, m0 = in ? s.mass[b0] : 0ull;
        const uint32_t c1 = in ? s.total[b1] : 0u, c0 = in ? s.total[b0] : 0u;
        unsigned long long all_w, all_c;
        const unsigned long long before_w = block_scan(m1 + m0, s.red, &all_w) + w_gt;
        const uint32_t before_c = (uint32_t)block_scan(c1 + c0, s.red, &all_c) + c_gt;
        if (d == 0) {
          if (cut != CUT_K && !know_w) W = all_w;
          if (cut == CUT_K) {
            target = (unsigned long long)k;
          } else if (cut == CUT_P) {
            target = top_p_target(p, W);
          } else {
            target = draw_target(a.u[r], W);
          }
        }
        // the bin in which the running total first reaches the target
        const unsigned long long have = cut == CUT_K ? before_c : before_w;
        const unsigned long long h1 = have + (cut == CUT_K ? c1 : m1), h0 = h1 + (cut == CUT_K ? c0 : m0);
        if (have < target && target <= h1) s.bin = b1, s.w_gt = before_w, s.c_gt = before_c, s.w_bin = m1, s.c_bin = c1;
        else if (h1 < target && target <= h0) s.bin = b0, s.w_gt = before_w + m1, s.c_gt = before_c + c1, s.w_bin = m0, s.c_bin = c0;
        if (tid == 0) s.w_all = W;
      }
      cluster.sync();
      prefix |= lead.bin << shift, w_gt = lead.w_gt, c_gt = lead.c_gt;
      W = lead.w_all;
      if (c_gt + lead.c_bin <= (uint32_t)kSampleList) {
        listed = true;
        break;
      }
    }
    if (listed) {
      if (prefix > floor_key) floor_key = prefix;  // everything at or above the bin's lower edge
      if (cut != CUT_K) know_w = true;
      break;
    }
    // the cut is the exact key `prefix`
    floor_key = prefix;
    if (cut == CUT_DRAW) break;
    know_w = cut == CUT_P;
    if (know_w) W = lead.w_gt + lead.w_bin;
    cut = cut == CUT_K && p < 1.0f ? CUT_P : CUT_DRAW;
    cluster.sync();  // the results are read before the next pass writes them
  }

  if (listed) {
    for (int j = tid; j < L; j += kSampleThreads) {
      const uint32_t key = order_key(src[j]);
      if (key >= floor_key) {
        const uint32_t pos = atomicAdd(&lead.list_count, 1u);
        if (pos < (uint32_t)kSampleList) lead.list[pos] = ((unsigned long long)key << 32) | (uint32_t)~(j0 + j);
      }
    }
    cluster.sync();
    if (rank != 0) return;  // nobody reads the other CTAs' shared memory any more
    const int M = min((int)s.list_count, kSampleList);
    int P2 = 32;
    while (P2 < M) P2 <<= 1;
    for (int i = M + tid; i < P2; i += kSampleThreads) s.list[i] = 0ull;
    __syncthreads();
    // bitonic sort, descending logit, ascending index among equals
    for (int size = 2; size <= P2; size <<= 1)
      for (int stride = size >> 1; stride > 0; stride >>= 1) {
        for (int i = tid; i < P2 / 2; i += kSampleThreads) {
          const int x = 2 * i - (i & (stride - 1)), y = x + stride;
          const unsigned long long vx = s.list[x], vy = s.list[y];
          if (((x & size) == 0) ? vx < vy : vx > vy) s.list[x] = vy, s.list[y] = vx;
        }
        // strides below 32 stay within the 64 elements of a warp's 32 pairs
        if (stride > 32 || stride == 1) __syncthreads();
        else __syncwarp();
      }
    __syncthreads();
    // running weights: thread tid owns kSampleList / 1024 consecutive places
    constexpr int kOwn = kSampleList / kSampleThreads;
    unsigned long long* run = reinterpret_cast<unsigned long long*>(s.cnt);  // [kSampleList], over the histogram
    unsigned long long w[kOwn], sum = 0ull, all;
#pragma unroll
    for (int i = 0; i < kOwn; ++i) {
      const int at = tid * kOwn + i;
      sum += at < M ? weight(key_value((uint32_t)(s.list[at] >> 32))) : 0ull;
      w[i] = sum;
    }
    const unsigned long long before = block_scan(sum, s.red, &all);
#pragma unroll
    for (int i = 0; i < kOwn; ++i) run[tid * kOwn + i] = before + w[i];
    __syncthreads();
    // first place whose running weight reaches `goal` (1 <= goal <= run[M - 1]), and the end of a place's ties
    auto reach = [&](unsigned long long goal) -> int {
      int lo = 0, hi = M - 1;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (run[mid] >= goal) hi = mid; else lo = mid + 1;
      }
      return lo;
    };
    auto ties_end = [&](int i) -> int {  // one past the last place with the key of place i
      const uint32_t key = (uint32_t)(s.list[i] >> 32);
      int lo = i, hi = M - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((uint32_t)(s.list[mid] >> 32) == key) lo = mid; else hi = mid - 1;
      }
      return lo + 1;
    };
    if (tid == 0) {
      if (cut == CUT_K) {
        W = run[ties_end(min(k, M) - 1) - 1];
        cut = p < 1.0f ? CUT_P : CUT_DRAW;
      }
      if (cut == CUT_P) {
        W = run[ties_end(reach(top_p_target(p, W))) - 1];
      }
      a.next[r] = (int)~(uint32_t)s.list[reach(draw_target(a.u[r], W))];
    }
    return;
  }

  // ---- the draw fell on a logit that more than a list of tokens share or exceed: its place among equals, by index ----
  const unsigned long long each = lead.c_bin ? lead.w_bin / lead.c_bin : 1ull;
  const unsigned long long rho = draw_target(a.u[r], W) - lead.w_gt;  // 1 .. w_bin
  uint32_t want = each ? (uint32_t)((rho + each - 1ull) / each) : 1u;
  if (want < 1u) want = 1u;
  if (want > lead.c_bin) want = lead.c_bin;
  // thread tid owns the slice's elements [tid * n, (tid + 1) * n)
  const int n = (L + kSampleThreads - 1) / kSampleThreads, e0 = min(L, tid * n), e1 = min(L, e0 + n);
  uint32_t mine = 0u;
  for (int j = e0; j < e1; ++j) mine += order_key(src[j]) == floor_key;
  unsigned long long all;
  uint32_t before = (uint32_t)block_scan(mine, s.red, &all);
  if (tid == 0) s.equal = (uint32_t)all;
  cluster.sync();
  for (int q = 0; q < rank; ++q) before += cluster.map_shared_rank(&s, q)->equal;
  if (mine && before < want && want <= before + mine) {
    uint32_t seen = before;
    for (int j = e0; j < e1; ++j)
      if (order_key(src[j]) == floor_key && ++seen == want) a.next[r] = j0 + j;
  }
  cluster.sync();  // nobody leaves while its shared memory is read
}

}  // namespace

cudaError_t launch_sample(const SampleArgs& a, int n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (n > kMaxBatch || a.vocab < 1 || !a.logits || !a.next) return cudaErrorInvalidValue;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(sample_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SampleShared) + kSampleSlice * 4);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  const int per = (a.vocab + kSampleCtas - 1) / kSampleCtas;
  const size_t smem = sizeof(SampleShared) + (per <= kSampleSlice ? (size_t)per * 4 : 0);
  return launch_kernel(sample_kernel, dim3(n * kSampleCtas), dim3(kSampleThreads), smem, s, a);
}

}  // namespace q4d
