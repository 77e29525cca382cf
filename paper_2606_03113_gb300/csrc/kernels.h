// kernels.h -- host-side launchers of the engine's kernels (internal).
#pragma once

#include "common.cuh"

namespace ssd {

// Statistics of one chunk of a row's logits (exit head), merged by the row's
// last chunk.
struct HeadPart {
  float mx;  // max logit
  float S;   // sum exp(z - mx)
  float T;   // sum exp(z - mx) (z - mx)
  float tv[kTopK];
  int32_t ti[kTopK];
};
constexpr int kHeadParts = 256;  // chunks of a row, at most

// Per-block partial slots of the streamed kernels (running + split), for up
// to kMaxBlocks blocks.
constexpr int kMaxBlocks = 512;
inline int head_tiles(int V) { return (V + 15) / 16; }

// Tensor maps of the split input rows (high and low planes [2][kMaxM][K]), read
// by the bf16 tensor-core kernels one 64-column box per unit.
struct TileMaps {
  CUtensorMap h[3], attn_out[3], act[3];  // boxes of 8, 16, 24 rows
};

// Encodes the tensor map of a bf16 weight matrix [rows][cols] (64 x 64 boxes,
// 128-byte swizzle) or of split input rows.
bool encode_weight_map(CUtensorMap* m, const void* W, int rows, int cols);
bool encode_input_maps(CUtensorMap (&m)[3], const void* xs, int cols);
// h of the rows as a matrix with norm weights gnorm reads it, where the kernel
// that wrote h did not know them.
cudaError_t launch_resplit(const Dims& D, const Bufs& B, const void* gnorm, RowSel sel, int mrows,
                           cudaStream_t st);
cudaError_t prepare_tile_kernels();
// Resident blocks per SM of the tensor-core kernels (0: cannot be resident).
int tile_blocks_per_sm();
// Floats of the tensor-core kernels' split-tile partials for `num_sms` blocks.
size_t tile_part_floats(int num_sms);
cudaError_t launch_tile_part(const Dims& D, const Bufs& B, const TileMaps& tm, const LayerW& w,
                             int layer, int part, const void* next_norm, RowSel sel, int mrows,
                             cudaStream_t st);
// One launch of a layer's O projection, gate/up and down (and, with next, the
// next layer's QKV) as the phases of one persistent kernel.
cudaError_t launch_tile_chain(const Dims& D, const Bufs& B, const TileMaps& tm, const LayerW& w,
                              const LayerW* next, const void* final_norm, int layer, RowSel sel,
                              int mrows, cudaStream_t st);
cudaError_t launch_tile_head(const Dims& D, const Bufs& B, const TileMaps& tm,
                             const CUtensorMap& lm, RowSel sel, int mrows, cudaStream_t st);
cudaError_t launch_tile_plain(const Dims& D, const Bufs& B, const CUtensorMap& wm, int rows,
                              int cols, const float* x, int M, float* y, cudaStream_t st);

// Prompt chunks of the bf16 decoder (wide.cu): up to kWideCap rows a pass.
constexpr int kWideCap = 1024;
struct WideMaps {
  CUtensorMap xn[3], xo[3], xa[3];  // hi/lo input planes, boxes of 32, 64, 128 tokens
};
// Tensor map of an input's hi and lo planes ([2][cap][cols] bf16), boxes of
// 64 columns x box_rows tokens x both planes.
bool encode_split_map(CUtensorMap* m, const void* x, int cols, int cap, int box_rows);
bool encode_wide_maps(CUtensorMap (&m)[3], const void* x, int cols, int cap);
cudaError_t prepare_wide_kernels();
long long wide_layer_cost(const Dims& D, int M);
cudaError_t launch_embed_wide(const Dims& D, const Bufs& B, const WideBufs& P, const void* embed,
                              const void* gnorm, const int32_t* toks, int M, cudaStream_t st);
// One layer over the chunk's M rows at positions pos0..; next_norm: the norm
// weights of the layer after it (null: none).
cudaError_t launch_layer_wide(const Dims& D, const Bufs& B, const WideBufs& P, const WideMaps& xm,
                              const LayerW& w, const void* next_norm, int layer, int M, int pos0,
                              cudaStream_t st);
// Logits of the chunk's rows row0 .. row0 + M - 1 (at most kHeadRows) after its
// last layer, whose next_norm was the final norm.
cudaError_t launch_head_wide(const Dims& D, const Bufs& B, const WideBufs& P, const WideMaps& xm,
                             const CUtensorMap& lm, int row0, int M, cudaStream_t st);

// fp32 decoders (fp32.cu): the matrices of a layer (0 QKV, 2 O, 3 gate/up,
// 4 down) and the LM head.
cudaError_t launch_f32_part(const Dims& D, const Bufs& B, const LayerW& w, int layer, int part,
                              RowSel sel, int mrows, cudaStream_t st);
cudaError_t launch_f32_head(const Dims& D, const Bufs& B, const void* lm, const void* final_norm,
                              RowSel sel, int mrows, cudaStream_t st);

// mrows is the largest number of rows a launch may see.  It picks the instance:
// fp32 matrices 1, 8 or 17 input rows, bf16 products 8, 16 or 24 token rows
// (the smallest that holds mrows), bf16 attention the row groups of a block.
// gnorm: norm weights of the first layer.  big: a block for each of kMaxM rows,
// else for one.
cudaError_t launch_embed(const Dims& D, const Bufs& B, int dtype, const void* embed,
                         const void* gnorm, RowSel sel, bool big,
                         cudaGraphConditionalHandle set_lstar_switch, cudaStream_t st);
cudaError_t launch_attention(const Dims& D, const Bufs& B, int dtype, int layer, RowSel sel,
                             int mrows, cudaStream_t st);
cudaError_t launch_head_stats(const Dims& D, const Bufs& B, int topk, RowSel sel, int mrows,
                              cudaStream_t st);
cudaError_t prepare_attention_kernels(int dtype);
// Keys per split of the bf16 decode attention.
int attn_split_keys(int n_kv_heads, int max_seq, int sms);
cudaError_t launch_round_begin(const Dims& D, const Bufs& B, cudaGraphConditionalHandle draft_if,
                               cudaStream_t st);
cudaError_t launch_decide(const Dims& D, const Bufs& B, int mode, int cand_idx, int is_last,
                          int layer, const void* final_norm, int dtype,
                          cudaGraphConditionalHandle next_if,
                          cudaGraphConditionalHandle draft_while, cudaStream_t st);
cudaError_t launch_draft_begin(const Bufs& B, cudaGraphConditionalHandle draft_while,
                               cudaStream_t st);
cudaError_t launch_accept(const Dims& D, const Bufs& B, cudaGraphConditionalHandle gen_while,
                          cudaStream_t st);
// Sampled decoding: weight sums of the logits rows row0 .. mrows - 1 (keep_mode 1,
// 2: also the row as the round's draft 0 or k), then those of the first rejected
// draft's residual.
cudaError_t launch_row_weights(const Dims& D, const Bufs& B, RowSel sel, int row0, int mrows,
                               int keep_mode, cudaStream_t st);
cudaError_t launch_residual_weights(const Dims& D, const Bufs& B, cudaStream_t st);
cudaError_t launch_begin_call(const Bufs& B, int max_new, cudaStream_t st);
cudaError_t launch_reset_sequence(const Bufs& B, cudaStream_t st);
cudaError_t launch_trace_push(const Bufs& B, int first_row, int n_rows, cudaStream_t st);
cudaError_t launch_set_pending(const Dims& D, const Bufs& B, int stats_row, int token, int pos,
                               cudaStream_t st);
cudaError_t launch_qnet_eval(const Bufs& B, int hidden, const float* states, int n, float* q,
                             cudaStream_t st);
cudaError_t launch_gemv_plain(const Dims& D, const Bufs& B, int dtype, const void* W, int rows,
                              int cols, const float* x, int M, float* y, cudaStream_t st);
// Raises the dynamic shared-memory limit of every streamed-kernel instance.
cudaError_t prepare_gemv_kernels();
cudaError_t launch_synth_fill(void* dst, int dtype, uint64_t n, uint32_t seed, uint32_t tid,
                              double sigma, cudaStream_t st);
cudaError_t launch_read_probe(const void* src, uint64_t bytes, uint32_t* sink, cudaStream_t st);
cudaError_t launch_kv_to_f32(const Dims& D, const Bufs& B, int dtype, int layer, int kind,
                             int head, int p0, int n, float* out, cudaStream_t st);

enum DecideMode : int { kDecideWalk = 0, kDecideDraft = 1 };

}  // namespace ssd
