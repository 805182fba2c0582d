// Host-side launch interface of the q4decode kernels (internal to the library).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace q4d {

constexpr int kMaxBatch = 16;
constexpr int kHeadDim = 128;
constexpr int kBlockSize = 16;

// ---- launch helper -----------------------------------------------------------------
// Launches with the programmatic-dependent-launch attribute when `pdl` is set: the kernel may start while its
// predecessor on the stream drains; every kernel of the library waits (griddepcontrol.wait) before it touches
// memory that another kernel writes.
void set_pdl_enabled(bool on);
bool pdl_enabled();

// ---- fragment-ordered GEMM operand ---------------------------------------------------
// xp bf16 [16][K] (chunks of 8 permuted, scaled), xs the group sums; see common.cuh.
// Layouts of the bf16 elements: OPERAND_BLOCKED (the tcgen05 kernel) and OPERAND_FRAG (the mma.sync kernels: a warp's
// fragments as contiguous 512-byte pieces).  Both keep the order 0,4,1,5,2,6,3,7 inside a chunk of 8 and take 16 K elements.
enum GemmPrologue { PRO_PLAIN = 0, PRO_SILU_MUL = 1 };
enum OperandLayout { OPERAND_BLOCKED = 1, OPERAND_FRAG = 2 };
__host__ __device__ __forceinline__ size_t operand_sums_bytes(int K) { return (size_t)(K / 256) * 16 * 32; }  // any layout

cudaError_t launch_pack_operand(const uint16_t* x, int x_stride, int K, int n, int prologue, uint16_t* xp, void* xs,
                                int layout, cudaStream_t s);

// ---- 4-bit skinny GEMM ------------------------------------------------------------
// EPI_SILU_PACK: the tensor has 2*I rows (gate rows then up rows); the output is the operand of the next GEMM,
// h = bf16(silu(bf16(gate)) * bf16(up)), written as an operand to out_xp and out_xs.
enum GemmEpilogue { EPI_BF16 = 0, EPI_RESIDUAL = 1, EPI_F32 = 2, EPI_SILU_PACK = 3 };

// Tensor maps of a dense projection (gemm_make_maps).
struct GemmMaps {
  CUtensorMap codes, scales, biases;
  bool sb_tma;  // scales and biases have maps
};
struct GemmArgs {
  const uint32_t* qw;      // [N][K/8]
  const GemmMaps* maps = nullptr;  // of a dense projection, or NULL: made for the call
  const uint16_t* scales;  // [N][K/64]
  const uint16_t* biases;  // [N][K/64]
  int N, K;
  const uint16_t* xp;  // fragment-ordered operand
  const void* xs;      // group sums (NULL: the kernel adds them up itself)
  int n;
  int epilogue;
  void* out;
  int out_stride;
  uint16_t* out_xp;  // EPI_SILU_PACK only
  void* out_xs;
  float2* argmax_partial;  // EPI_F32 only, optional: [row blocks][16] = (max, index as float bits) per request
  float* partial;          // split-K partial sums
  size_t partial_bytes;
  int* counters;  // zero between launches
  int counters_len;
  unsigned int* status = nullptr;  // device word set non-zero when a bounded wait inside the kernel gives up
};

// Bytes of split-K scratch a GEMM of this shape may use (upper bound over batch sizes).
size_t gemm_partial_bytes(int N, int K, int epilogue);
int gemm_counters_needed(int N);
int gemm_row_blocks(int N, int K, int n, int epilogue);  // grid.x of the launch (size of argmax_partial)
cudaError_t launch_q4_gemm(const GemmArgs& a, cudaStream_t s);
int gemm_operand_layout();  // the operand layout launch_q4_gemm expects
cudaError_t gemm_make_maps(const uint32_t* qw, const uint16_t* scales, const uint16_t* biases, long long N, int K, bool gate_up,
                           GemmMaps* out, int experts = 1);

// Mixture of experts: the projection of every unit, a unit being up to 8 requests routed to one expert.
constexpr int kMaxExpertUnits = 256 + 64;  // one partly filled unit for each of 256 experts, plus 16 x 32 pairs in eights
struct ExpertArgs {
  const uint16_t* scales;  // stacked tensors: N rows per expert
  const uint16_t* biases;
  const GemmMaps* maps;
  bool gate_up;            // SiLU epilogue into out_xp (OPERAND_FRAG per unit), else bf16 rows out [unit][8][N]
  int N, K;
  const uint16_t* xp;      // gate_up: the step's operand (OPERAND_FRAG, 16 requests) with its group sums xs; else per unit
  const void* xs;
  uint16_t* out;
  uint16_t* out_xp;
  size_t unit_stride, out_unit_stride;  // elements between the units' operands
  const int4* units;       // device list {expert, requests, request ids as bytes in two words}
  const int* n_units;
  unsigned int* status;
};
cudaError_t launch_q4_experts(const ExpertArgs& a, cudaStream_t s);

// tcgen05 kernel (q4_umma.cu): tiles of 128 rows, K in `parts` across CTAs, stages of 256 features.
struct UmmaPlan {
  int tiles, parts, ns;
  size_t partial_bytes;
};
UmmaPlan plan_umma(int N, int K, int epilogue, int sm_count);
bool umma_supported(int N, int K, int epilogue);
cudaError_t launch_q4_umma(const GemmArgs& a, int sm_count, cudaStream_t s);
cudaError_t gemm_init();  // sets the dynamic shared memory limits once per process/device
cudaError_t launch_argmax_finish(const float2* partial, int row_blocks, int n, int32_t* next, cudaStream_t s);

// ---- paged decode attention -------------------------------------------------------
struct AttnPlan {   // filled on the host from the request lengths
  int n_work;       // (request, chunk) items
  int n_slots;      // partial-result slots = n_work
  int chunk_tiles;  // tiles (16 tokens) per chunk
};
// work: int4 {request, first tile, end tile, slot}; slot_base/nchunks per request.
// wave_ctas: CTAs resident at once (attention_wave_ctas); the automatic chunk size fills one such wave.
AttnPlan plan_attention(const int32_t* lens, int n, int nkv, int chunk_tokens, int wave_ctas, int4* work,
                        int32_t* slot_base, int32_t* nchunks, int max_work);
int attention_wave_ctas(int nq, int nkv);
int attention_max_work(int max_batch, int max_positions);

struct AttnArgs {
  const uint16_t* q;  // [n][nq][128]
  const uint16_t* kpool;
  const uint16_t* vpool;  // this layer: [blocks][nkv][16][128]
  const int32_t* block_tables;
  const int32_t* lens;
  const int4* work;
  const int32_t* slot_base;
  const int32_t* nchunks;
  int n_work, n, nq, nkv, max_blocks;
  float* part_acc;  // [slots][nq][128]
  float* part_ml;   // [slots][nq][2]
  uint16_t* out;    // plain [n][nq][128], or NULL
  uint16_t* out_xp; // fragment-ordered operand [16][nq*128] of the O projection, or NULL
  void* out_xs;     // its group sums
  int out_layout = OPERAND_FRAG;  // layout of out_xp
  int* merge_counters = nullptr;  // [16][nkv], zero between launches: the attention kernel merges the chunks itself
  // The kernel requests its first K, V tiles before it waits for the preceding kernel (cached K, V do not depend on
  // it).  Set when they do (the preceding kernel appends tokens this launch reads): the launch then carries no
  // programmatic-dependent-launch attribute and starts only after the preceding kernel has completed.
  bool after_predecessor = false;
  // With qkv given (bf16 [n][(nq+2nkv)*128], the QKV projection's output) the kernel prepares q itself (qk-norm,
  // rotary embedding) and appends k, v of the new token to the pool; `q` is then unused.
  const uint16_t* qkv = nullptr;
  const uint16_t* q_norm = nullptr;  // bf16 [128] or NULL
  const uint16_t* k_norm = nullptr;
  float eps = 0.0f;
  const float* rope = nullptr;  // f32 [positions][64][2]
  uint16_t* kpool_w = nullptr;  // this layer of the pool, writable
  uint16_t* vpool_w = nullptr;
};
cudaError_t launch_paged_attention(const AttnArgs& a, cudaStream_t s);
cudaError_t launch_attention_merge(const AttnArgs& a, cudaStream_t s);
cudaError_t attention_init();

struct RopeArgs {
  const uint16_t* qkv;
  const uint16_t* q_norm;
  const uint16_t* k_norm;
  float eps;
  const float* rope;
  int n, nq, nkv;
  const int32_t* lens;
  const int32_t* block_tables;
  int max_blocks;
  uint16_t* kpool;
  uint16_t* vpool;
  uint16_t* q_out;
};
cudaError_t launch_rope_append(const RopeArgs& a, cudaStream_t s);

// ---- mixture of experts ------------------------------------------------------------
struct MoeRouteArgs {
  const uint16_t* y;       // plain normed hidden state bf16 [n][H]
  const uint16_t* router;  // bf16 [E][H]
  int H, E, top_k, norm;
  float* wgt;           // [16][top_k] weights of the selected experts, by decreasing logit
  int32_t* pos;         // [16][top_k]: 8 x unit + place in the unit
  int32_t* counter;     // zero between launches
  int4* units;          // the list the expert projections walk (ExpertArgs)
  int32_t* n_units;
  float* logits;           // [16][E] scratch
  int32_t* touched_total = nullptr;  // optional: running sum of the touched experts over the launches of a step
};
struct MoeCombineArgs {
  uint16_t* x;        // residual stream bf16 [n][H], updated in place
  const uint16_t* o;  // expert outputs bf16 [unit][8][H]
  const int32_t* pos;
  const float* wgt;
  int H, top_k;
  const uint16_t* norm;  // the next norm's weights; its output is the operand yp, ys
  float eps;
  uint16_t* yp;
  void* ys;
  int layout;
};
cudaError_t launch_moe_router(const MoeRouteArgs& a, int n, cudaStream_t s);
cudaError_t launch_moe_combine_norm(const MoeCombineArgs& a, int n, cudaStream_t s);

// ---- prompt processing (prefill.cu): many tokens of one request at once ------------------
// Operand of a prompt projection: f16 [rows][prefill_operand_stride(K)], every row scaled by a power of two of its own
// (inv_scale[row] undoes it): K features (chunks of 8 in the order 0,4,1,5,2,6,3,7), then the sums of every group of 64
// features as two f16 terms, laid out against the biases and scales of the weights (see prefill.cu).
constexpr int kPrefillChunk = 2048;      // tokens per pass over the weights
constexpr int kPrefillMaxWidth = 32768;  // widest operand row
__host__ __device__ __forceinline__ int prefill_operand_stride(int K) { return K + 64 * ((K + 1023) / 1024); }
// rows of bf16 x (optionally RMS-normalised with norm_w first, the normalised row also written to y) -> operand
struct PrefillPackArgs {
  uint16_t* x;
  int x_stride;
  const uint16_t* norm_w;
  float eps;
  int rows, K;
  uint16_t* y;  // or NULL
  uint16_t* operand;
  float* inv_scale;
  // the result of a projection cut into parts of K, fp32 [parts][rows][..]: added to x, which takes the sum (silu: the row
  // is h = silu(gate) * up of its [2 K] results, x is not used)
  const float* sums = nullptr;
  int parts = 0;
  bool silu = false;
};
cudaError_t launch_prefill_pack(const PrefillPackArgs& a, cudaStream_t s);
struct PrefillGemmArgs {
  const uint32_t* qw;
  const uint16_t* scales;
  const uint16_t* biases;
  int N, K;                // N a multiple of 128
  const uint16_t* operand;
  int operand_rows;        // rows the operand buffer holds (bound of the tensor map)
  const float* inv_scale;
  int rows;                // tokens
  int epilogue;            // EPI_BF16, EPI_RESIDUAL, or EPI_SILU_PACK: h = silu(gate) * up, plain bf16 [rows][N / 2]
  uint16_t* out;
  int out_stride;
  unsigned int* status;
  // grouped mode (mixture of experts): `units` is a device list of {expert, first operand row, rows <= unit_rows, 0}
  const int4* units = nullptr;
  const int* n_units = nullptr;
  int unit_rows = 0;
  int experts = 1;         // experts stacked in the tensors
  float* sums = nullptr;   // given: the results go there instead, as fp32 [parts][rows][N] (parts: prefill_tiling)
};
cudaError_t launch_prefill_gemm(const PrefillGemmArgs& a, cudaStream_t s);
constexpr int kPrefillMaxParts = 16;
struct PrefillTiling {
  int tok_tiles, n_tile;
  int parts;  // of K, worth using where the reader of the result can add fp32 sums up (1: none)
};
PrefillTiling prefill_tiling(int N, int K, int rows);
// Bytes of `sums` any projection with parts > 1 needs (a part of K is used only while all tiles fit one wave).
constexpr size_t kPrefillSumsBytes = (size_t)148 * 128 * 256 * 4;
struct PrefillAttnArgs {
  const uint16_t* qkv;     // bf16 [rows][(nq + 2 nkv) * 128], or as fp32 parts of K [parts][rows][..] in sums
  const float* sums;
  int parts;
  uint16_t* q;             // bf16 [rows][nq][128] scratch: prepared queries
  const uint16_t* q_norm;  // or NULL
  const uint16_t* k_norm;
  float eps;
  const float* rope;
  int rows, start;         // row r is the token at position start + r
  int nq, nkv;
  const int32_t* block_table;
  uint16_t* kpool;         // this layer of the pool
  uint16_t* vpool;
  uint16_t* out;           // bf16 [rows][nq][128]
};
cudaError_t launch_prefill_rope_append(const PrefillAttnArgs& a, cudaStream_t s);
cudaError_t launch_prefill_attention(const PrefillAttnArgs& a, cudaStream_t s);
cudaError_t prefill_init();

// Routing of many tokens: the experts of each token, then every (token, expert) pair as a row of an operand sorted by
// expert, and the list of units (runs of at most unit_rows rows of one expert) the grouped projections walk.
struct PrefillMoeArgs {
  const uint16_t* y;       // normed hidden state bf16 [rows][H]
  const uint16_t* router;  // bf16 [E][H]
  int rows, H, E, top_k, norm;
  int32_t* idx;            // [rows][top_k]
  float* wgt;              // [rows][top_k]
  int32_t* pos;            // [rows][top_k]: row of the pair in the sorted operand
  int32_t* counts;         // [E], zero between calls
  int32_t* cursor;         // [E]
  int4* units;
  int* n_units;
  int unit_rows;
  const uint16_t* operand; // operand of the tokens and its scales
  const float* inv_scale;
  uint16_t* sorted;        // operand of the pairs and its scales
  float* sorted_inv_scale;
  const uint16_t* o;       // expert outputs bf16 [pairs][H]
  uint16_t* x;             // residual stream bf16 [rows][H], updated in place
};
cudaError_t launch_prefill_route(const PrefillMoeArgs& a, cudaStream_t s);    // idx, wgt, counts -> units -> sorted operand
cudaError_t launch_prefill_combine(const PrefillMoeArgs& a, cudaStream_t s);

// ---- sampling ------------------------------------------------------------------------
struct SampleArgs {  // passed to the kernel by value: the per-request settings travel with the launch
  const float* logits;  // f32 [n][vocab]
  int32_t* next;        // [n]
  int vocab;
  float temperature[kMaxBatch];  // <= 0: greedy
  int top_k[kMaxBatch];          // <= 0 or >= vocab: off
  float top_p[kMaxBatch];        // >= 1: off
  float u[kMaxBatch];            // the draw, in [0, 1)
};
cudaError_t launch_sample(const SampleArgs& a, int n, cudaStream_t s);

// ---- small kernels ----------------------------------------------------------------
cudaError_t launch_embed(const uint32_t* q, const uint16_t* scales, const uint16_t* biases, int vocab, int H,
                         const int32_t* tokens, int n, uint16_t* x, cudaStream_t s);
// y (plain, optional) and/or the fragment-ordered operand (yp, ys) of the next GEMM.
cudaError_t launch_rmsnorm(const uint16_t* x, const uint16_t* w, float eps, int n, int H, uint16_t* y,
                           uint16_t* yp, void* ys, int layout, cudaStream_t s);
cudaError_t launch_argmax(const float* logits, int n, int vocab, int32_t* next, cudaStream_t s);
cudaError_t launch_dequant(const uint32_t* q, const uint16_t* scales, const uint16_t* biases, int N, int K,
                           float* out, cudaStream_t s);
cudaError_t launch_kv_gather(const uint16_t* kpool, const uint16_t* vpool, int nkv, const int32_t* block_table,
                             int len, uint16_t* k_out, uint16_t* v_out, cudaStream_t s);

}  // namespace q4d
