// Internal definition of the model handle and of the GEMM entry used by the verify forward.
#pragma once
#include <vector>

#include "state.cuh"

namespace laser { struct GenHost; }

struct laser_model {
  laser_model_cfg cfg{};
  int rows_per_seq = 0;  // max_draft + 1
  int R = 0;             // max_batch * rows_per_seq
  int R_pad = 0;         // R rounded up to a multiple of 16
  int R_cap = 0;         // rows of the workspace: R_pad, or those of a prefill pass where that is more
  int dq = 0, dkv = 0, dqkv = 0;
  const __nv_bfloat16 *tok_emb = nullptr, *lm_head = nullptr, *final_norm = nullptr;
  std::vector<const __nv_bfloat16*> wqkv, wo, wgu, wdown, attn_norm, ffn_norm;
  std::vector<void*> owned;  // device allocations released with the model
  // workspace (all device, one allocation)
  float* resid = nullptr;          // [R_cap, d] residual stream, fp32
  __nv_bfloat16* xn = nullptr;     // [R_cap, d] normalised activations (GEMM operand)
  __nv_bfloat16* q = nullptr;      // [R_cap, dq] rotated queries
  float* qf = nullptr;             // [R_cap, dq] the same in fp32 (precise mode only)
  bool precise = false;            // activations handed to the contractions as hi + lo bf16 pairs: xn, attn, act are
                                   // [R_cap, 2 x width] with the lo parts in the second half of a row
  __nv_bfloat16* attn = nullptr;   // [R_cap, dq] attention output
  __nv_bfloat16* act = nullptr;    // [R_cap, f] SwiGLU output
  float* sumsq = nullptr;          // [ceil(d/128)][R_cap] per-tile sums of squares of the residual
  float* rope = nullptr;           // [R_cap, head_dim/2, 2] cos, sin of each row's position
  int32_t* row_pos = nullptr;      // [R_cap] position of the row, -1 = inactive
  int32_t* row_seq = nullptr;      // [R_cap] cache slot of the row
  int32_t* row_ctx = nullptr;      // [row groups] cached tokens before each sequence of the step (a prompt chunk's start in a prefill)
  int32_t* row_n = nullptr;        // [row groups] effective rows of each
  unsigned long long* row_mask = nullptr;  // [R_pad] token tree: rows of its sequence a row attends to (bit j = row j)
  // acceptance fused into the LM head: what its epilogue leaves per (row, 128-token vocabulary tile)
  int32_t* row_draft = nullptr;    // [R_pad] token whose verdict the row gives, -1 = none
  float* draft_logit = nullptr;    // [R_pad] logit of that token
  float4* top_val = nullptr;       // [R_pad][vocab tiles] the tile's four largest logits, in order
  int4* top_idx = nullptr;         // [R_pad][vocab tiles] their token ids
  float* tile_sum = nullptr;       // [R_pad][vocab tiles] sum over the tile of exp(l - tile max)
  int32_t* status = nullptr;       // first device-side error of the stream, 0 = none
  float* attn_part = nullptr;      // partial attention results where a sequence's pages are split, and arrivals per (sequence, head, tile)
  int32_t* attn_arrived = nullptr;
  float* pair_scratch = nullptr;   // partial sums of the contractions for many rows (gemm_pair.cu), and the cut tiles' state
  int32_t* pair_state = nullptr;
  int peer_cycles = 200000;        // how long they wait for each other: about 0.1 ms, many times the skew between pairs that are running
  std::vector<double> prefill_us{0.0};  // [chunks] what a layer of a prefill pass of that many chunks is estimated to take, as far as needed so far
  void* gemm_state = nullptr;      // tensor-map cache of the tensor-core GEMM
  void* gen_buf = nullptr;         // work buffers of laser_generate, kept between calls (in `owned`)
  size_t gen_bytes = 0;
  laser::GenHost* gen_host = nullptr;  // pinned memory and events of laser_generate, kept between calls
  // optional per-class kernel timing (class 0 = GEMM, 1 = attention)
  bool profile = false;
  std::vector<cudaEvent_t> prof_events[2];  // begin/end pairs
  size_t prof_used[2] = {0, 0};
};

namespace laser {

// A prefill pass runs the contractions over up to this many prompt tokens: enough rows for the tensor pipe to be the bound
// (7B, 4 layers: 3.6 us a row at 144 rows, 1.6 us at 1024), and to fill whole waves of tiles: 16 tiles of 256 weight rows, as the O and down
// projections of 4096 features have, leave 14 % of the last wave idle at 1024 rows (64 of 74 pairs), 3 % at 2304 (144 of 148).  A
// model of few weights a layer gains nothing by that, and would only be created more slowly.
constexpr int prefill_rows(int64_t layer_weights) { return layer_weights >= (int64_t(16) << 20) ? 2304 : 1024; }
constexpr int kAttnSplitCtas = 3 * 148; // most CTAs of an attention launch that splits pages: three an SM
constexpr int kPrefillChunk = 32;   // rows of a chunk of a prompt
constexpr int kPrefillShare = 4;    // consecutive chunks that share each staged K/V page in the attention kernel

void gen_host_free(laser_model* m);

// Chunks of each pass of a prefill of n_chunks, in order: the division whose estimated time is least.
std::vector<int> prefill_passes(laser_model* m, int n_chunks);

// The entry points of the same names; `stamp` (optional): the device clock at the end of the rows' making, at the start of the verdict.
laser_status make_rows(const int32_t* last_token, const int32_t* draft, const int32_t* draft_len, int32_t B, int32_t K, int32_t* tokens,
                       int32_t* n_rows, unsigned long long* stamp, cudaStream_t stream);
laser_status make_rows_tree(const int32_t* last_token, const int32_t* draft, const int32_t* draft_parents, const int32_t* draft_len,
                            int32_t B, int32_t K, int32_t* tokens, int32_t* parents, int32_t* n_rows, unsigned long long* stamp,
                            cudaStream_t stream);
laser_status accept_commit(laser_kv* kv, const int32_t* seq_ids, const float* logits, const int32_t* tokens, const int32_t* n_rows,
                           int32_t B, int32_t V, const laser_params* p, int32_t* n_accept, int32_t* out_tokens, int32_t* n_out,
                           unsigned long long* stamp, cudaStream_t stream);
laser_status accept_tree(laser_kv* kv, const int32_t* seq_ids, const float* logits, const int32_t* tokens, const int32_t* parents,
                         const int32_t* n_rows, int32_t B, int32_t V, const laser_params* p, int32_t* n_accept, int32_t* out_tokens,
                         int32_t* n_out, int32_t* path_rows, unsigned long long* stamp, cudaStream_t stream);

// What the GEMM does with a finished 128-feature x NT-row accumulator tile.
enum { EPI_PLAIN = 0, EPI_RESID = 1, EPI_SWIGLU = 2, EPI_QKV = 3, EPI_VERDICT = 4 };

struct GemmEpilogue {
  int R_rows = 0;                    // rows of the step: a token tile may overhang them, and what lies beyond is not finished
  // Operands as hi + lo bf16 pairs (the precise mode): the A operand's rows are [hi | lo] with lo starting at column
  // a_lo_off (0 = plain bf16 operand); out_split = the bf16 activations this epilogue writes (xb, act) are pairs too
  int a_lo_off = 0, out_split = 0;
  // RMSNorm of the A operand, applied as a per-row scale of the result: the producer left
  // x * gain in bf16 and one sum of squares per (128-feature tile, row); null = no scale
  const float* sumsq_in = nullptr;
  int sumsq_in_tiles = 0, sumsq_ld = 0;
  float inv_d = 0.f, eps = 0.f;
  // EPI_PLAIN: out[r][n] = scale * acc (fp32), rows < R_store
  float* out = nullptr;
  int ldo = 0, R_store = 0;
  // EPI_VERDICT: the scaled row is a row of logits; per (row, weight tile) the tile's top_n largest of them with
  // their ids (ties: smaller id first), the sum of exp(l - tile max) when tile_sum is given, and the logit of the
  // row's draft token from the tile that holds it; `out` may be null (logits never stored)
  const int32_t* row_draft = nullptr;
  float* draft_logit = nullptr;
  float4* top_val = nullptr;
  int4* top_idx = nullptr;
  float* tile_sum = nullptr;
  int top_n = 0, n_vtiles = 0;
  // EPI_RESID: resid[r][n] += acc; xb = bf16(resid * gain_next); sumsq_out[tile][r]
  float* resid = nullptr;
  __nv_bfloat16* xb = nullptr;
  const __nv_bfloat16* gain_next = nullptr;
  float* sumsq_out = nullptr;
  // EPI_SWIGLU: W is [gate rows | up rows] (f each); act[r][j] = silu(gate_j) * up_j
  __nv_bfloat16* act = nullptr;
  int f = 0;
  // EPI_QKV: rotary embedding, Q store (bf16, or fp32 into qf when given), K/V page write
  __nv_bfloat16* q = nullptr;
  float* qf = nullptr;
  __nv_bfloat16* pages_layer = nullptr;
  size_t page_elems = 0;
  const int32_t* page_table = nullptr;
  int pages_per_seq = 0;
  const int32_t* row_pos = nullptr;
  const int32_t* row_seq = nullptr;
  const float* rope = nullptr;
  int H = 0, Hkv = 0, dh = 0;
};

// Whether contractions of that many rows run on pairs of SMs (gemm_pair.cu).
bool gemm_by_pairs(laser_model* m, int R_pad);
// acc[r][n] = sum_k A[r][k] * W[n][k] (A bf16 [R_pad, K], W bf16 [N, K], both row-major),
// finished by the epilogue `epi`.  N and K must be multiples of 8.
laser_status gemm_fused(laser_model* m, const __nv_bfloat16* A, const __nv_bfloat16* W, int R_pad, int N, int K, int epi,
                        const GemmEpilogue& e, cudaStream_t stream);
void gemm_state_free(laser_model* m);

// Brackets one launch with events when profiling is on.
struct ProfScope {
  laser_model* m; int cls; cudaStream_t st; bool on;
  ProfScope(laser_model* m_, int cls_, cudaStream_t st_) : m(m_), cls(cls_), st(st_), on(m_->profile) { mark(); }
  ~ProfScope() { mark(); }
  void mark() {
    if (!on) return;
    auto& ev = m->prof_events[cls];
    size_t& used = m->prof_used[cls];
    if (used == ev.size()) { cudaEvent_t e; if (cudaEventCreate(&e) != cudaSuccess) { on = false; return; } ev.push_back(e); }
    cudaEventRecord(ev[used++], st);
  }
};


// TMA-fed paged attention (head_dim 64 or 128 and a cache small enough for 32-bit row
// coordinates); the verify forward falls back to a plain kernel otherwise.
bool attention_tma_supported(const laser_model* m, const laser_kv* kv);
// fresh: pages below a sequence's row_ctx may be written by the kernel right before (prompt chunks of one prefill pass).
laser_status attention_tma_launch(laser_model* m, laser_kv* kv, int layer, const int32_t* seq_ids, int B, int Rs, bool tree, bool fresh,
                                  cudaStream_t stream);
// The same for the chunks of a prefill pass (default mode; head_dim 64 or 128 as above).
laser_status attention_prefill_launch(laser_model* m, laser_kv* kv, int layer, const int32_t* seq_ids, int n_chunks, cudaStream_t stream);

// Prompt processing: the verify forward without the LM head over chunks of up to kPrefillChunk prompt tokens.  Chunk i is
// n_rows[i] tokens of cache slot seq_ids[i] from position start[i] on; chunks of one prompt may share a call, in any order:
// every layer caches the K and V of all of them before its attention.  K and V of the rows go to the cache, lengths are not
// changed.  n_chunks * kPrefillChunk rows at most m->R_cap.
laser_status prefill_chunks(laser_model* m, laser_kv* kv, const int32_t* seq_ids, const int32_t* start, const int32_t* tokens,
                            const int32_t* n_rows, int32_t n_chunks, cudaStream_t stream);

// The verify forward with acceptance fused into the LM head: per (row, 128-token vocabulary tile) the tile's
// top_n (1..4) largest logits and ids, with `sums` the tile's sum of exp(l - tile max), and per row the logit of
// its draft token, all in the model's buffers; logits (may be null) are stored only when given.
laser_status verify_fused(laser_model* m, laser_kv* kv, const int32_t* seq_ids, const int32_t* tokens,
                          const int32_t* n_rows, int32_t B, float* logits, int top_n, bool sums, cudaStream_t stream);

}  // namespace laser
