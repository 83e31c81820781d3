// Host-side launchers of every kernel (internal).  Each enqueues on `st` and returns a hydra_status.
#pragma once
#include "common.cuh"

namespace hydra {

// ---- GEMM: partial sums of x[m][k] * w[n][k] (see SplitDesc for where they land)
// tcgen05 path (bfloat16 operands).  x_rows_alloc = rows the x buffer really holds (>= m); rows of the last
// tile beyond m are computed and dropped.  part needs gemm_tc_plan(...)'s max_slots * m * n floats.
// x holds x_planes (1 or 2) planes of x_rows_alloc rows each: plane 0 = bf16(v), plane 1 = bf16(v - plane 0).  The m rows begin at row x_row0
// of a plane; x itself is the buffer's beginning, so that no row behind its end is ever described to the hardware.
// w_const: no kernel in flight writes w (the weights of a context); its first tiles are then read ahead of the preceding kernel's completion.
// dbg (tests of the bounded waits only): a shorter poll limit and one weight-tile request that CTA 0 leaves out.
struct GemmDebug { uint32_t wait_limit; int skip_unit; };
struct GemmArrivals { unsigned long long* count; unsigned long long ticket; };
hydra_status gemm_tc(const bf16* x, int x_rows_alloc, int x_planes, const bf16* w, float* part, int m, int n, int k,
                     SplitDesc* sd_out, bool w_const, int* status, int* diag /*int[8] or null*/, const GemmDebug* dbg /*null: defaults*/, cudaStream_t st,
                     size_t part_cap = 0 /*floats in part; 0: as many as the plan asks for*/,
                     float* out = nullptr /*[m][n]: the sums themselves*/, const GemmArrivals* arrivals = nullptr /*with out: for one-launch calls*/, int x_row0 = 0);
// Stand-alone calls of up to GEMM_ONE_LAUNCH_WEIGHTS weights and 16 rows add their partial sums in the GEMM's own launch (gemm_tc.cu has the
// figures).  A counter per tile (128 columns, at least 64 k) says how many CTAs have stored it: the call's ticket in the upper 48 bits,
// the count below.  Tickets rise from call to call, so whatever an earlier call left in a counter - one that timed out, or that another call
// overlapped - counts for nothing in a later one.
constexpr long long GEMM_ONE_LAUNCH_WEIGHTS = 6 * 1000 * 1000;
constexpr size_t GEMM_ONE_LAUNCH_TILES = GEMM_ONE_LAUNCH_WEIGHTS / (128 * 64);
// grid: CTAs.  part_cap (floats, 0: no limit): fewer CTAs, hence fewer slots, where the partial sums would not fit otherwise.
SplitDesc gemm_tc_plan(int m, int n, int k, int* grid, int* max_slots, size_t part_cap = 0);
bool gemm_tc_available();                 // driver entry point for tensor-map encoding found
// SIMT path (float or bfloat16 operands), single slot.  w_const: no kernel in flight writes w (the weights of a context), so it is
// read ahead of the preceding kernel's completion.
hydra_status gemm_simt(const void* x, const void* w, float* out, int m, int n, int k, int dtype, bool w_const, cudaStream_t st);
// out[m][n] = sum of the slots of part
hydra_status reduce_splits(const float* part, SplitDesc sd, float* out, int m, int n, cudaStream_t st);

// ---- element-wise / row-wise stages of a decoder layer (dtype: 0 float, 1 bfloat16 for the "act" outputs)
// x_out = (res ? res : 0) + sum_s part[s]; if gain: xn = rmsnorm(x_out)*gain (act dtype, optional) and hn = the same in
// float (optional).  part may be null.  x_out may alias res.
hydra_status residual_rmsnorm(const float* res, const float* part, SplitDesc sd, float* x_out,
                              const void* gain, void* xn, size_t xn_ps, float* hn, int rows, int d, float eps, int dtype,
                              cudaStream_t st);
// The first kernel of a forward call: table[r][j] = (cos, sin) of (pos0[b]+depth[i]) * theta^(-2j/head_dim), evaluated in double, and with tok x[r] = embed[tok[r]]
hydra_status forward_start(RowSet rs, float2* table, int head_dim, float theta, const void* embed, const int* tok, float* x, int d, int vocab, int dtype, int* status,
                           cudaStream_t st);
// bfloat16 path: q ([rows][H][hd], rotated) and the K/V cache rows (rotated K) from the QKV partial sums;
// float16 with a lo plane (f16(v - f16(v))) q_ps / kv_ps elements after the hi plane (0: hi only).  kv_only: the projection has the
// 2 d columns of K and V, q is not written.
hydra_status qkv_rope_store(const float* part, SplitDesc sd, const float2* table, void* q, size_t q_ps, void* kcache, void* vcache,
                            size_t kv_ps, RowSet rs, int n_heads, int head_dim, int max_seq, bool kv_only, int* status, cudaStream_t st);
// Float model path: SIMT kernel + combine kernel, partial rows of ATT_CHUNK_ROWS-row chunks in `scratch`
// (attention_scratch_bytes).  q, caches and out are float.
constexpr int ATT_CHUNK_ROWS = 128;
size_t attention_scratch_bytes(int batch, int tc, int n_heads, int head_dim, int max_seq);
hydra_status tree_attention_f32(const float* q, const float* kcache, const float* vcache, RowSet rs, float* out, void* scratch,
                                int n_heads, int head_dim, int max_seq, int len_upper, cudaStream_t st);
// bfloat16 model path: tensor-core kernel (attention_tc.cu).  q [planes][q_rows][H*hd] and the caches
// [planes][cache_batch][H][max_seq][hd] are float16 in 1 or 2 planes (hi = f16(v), lo = f16(v - hi)); out is bfloat16
// [rows][H*hd] in two planes out_ps elements apart (0: hi only).  rs.mask == null selects a causal chunk (row i sees
// the committed slots and new slots 0..i) of up to 128 rows; with a mask, up to 64 rows.
// A packed row set runs one CTA column per attention block of at most ATT_BLOCK_ROWS rows.
// stable_lengths: rs.pos0 / rs.n_rows and every cache row below pos0 were written by kernels that had COMPLETED before the
// kernel preceding this one in the stream started (true inside a forward call of the library, whose first kernel holds
// its successors back until everything earlier has completed); the kernel then requests committed cache tiles before it
// waits for its predecessor.
hydra_status tree_attention_tc(const __half* q, int q_rows, const __half* kc, const __half* vc, int cache_batch, int planes, RowSet rs,
                               bf16* out, size_t out_ps, int n_heads, int head_dim, int max_seq, int len_upper, int* status,
                               bool stable_lengths, cudaStream_t st);
constexpr int ATT_BLOCK_ROWS = 128;
// The same for one or two rows a sequence, without tensor cores (attention_rows.cu).
hydra_status tree_attention_rows(const __half* q, int q_rows, const __half* kc, const __half* vc, int cache_batch, int planes, RowSet rs, bf16* out, size_t out_ps, int n_heads,
                                 int head_dim, int max_seq, int len_upper, bool stable_lengths, cudaStream_t st);
hydra_status silu_mul(const float* part, SplitDesc sd, void* act, size_t act_ps, int rows, int f, cudaStream_t st);
// amax[r] = argmax_v of the summed partial logits (lowest id among equal maxima); the sums go to logits_out if given
// scratch: topk_scratch_bytes(rows_cap, vocab) bytes of candidate storage
size_t topk_scratch_bytes(int rows, int vocab);
hydra_status argmax_rows(const float* part, SplitDesc sd, float* logits_out, int* amax, void* scratch, int rows_cap, int rows,
                         int vocab, cudaStream_t st);

// ---- draft heads
struct LevelDesc {           // one tree level d (1-based): the parents that have children
  int d, n_parents;
  const int* parents;        // device [n_parents] row ids
};
// z[b*P+j] = [hprime[b] ; E[tok[b][path(parent j)]]] in act dtype (lv.d path tokens; lv.d = 0: the hidden state alone);
// with write_root also tree_tok[b][0] = root_tok[b].
hydra_status head_gather(const float* hprime, const void* embed, const int* root_tok, int* tree_tok, const int* path_tab,
                         LevelDesc lv, int write_root, void* z, size_t z_ps, int batch, int T, int kp1, int d_model, int vocab,
                         int* status, cudaStream_t st);
// y_out = res + silu(sum_s part[s] + bias); res row = hprime[b] when res_is_hprime else y row.  yb = act-dtype copy.
hydra_status head_act(const float* res, int res_is_hprime, int rows_per_b, const float* part, SplitDesc sd,
                      const void* bias, float* y_out, void* yb, size_t yb_ps, int rows, int d, cudaStream_t st);
// Children of a level in two steps.  The max_children best tokens of every logits row, descending (ties: lower id first); the logits are the
// summed partials, also written to `logits` [rows][vocab].  Then the children of parent j of sequence b = the first n_child of row b*P+j's; with depth, lv has
// the parents of all levels (sequentially independent heads, one row per sequence and head), and those at depth t take theirs from row (top - t)*batch + b.
hydra_status topk_candidates(const float* part, SplitDesc sd, float* logits, int max_children, void* scratch, int rows_cap, int rows, int vocab,
                             cudaStream_t st);
hydra_status topk_merge(LevelDesc lv, int max_children, const int* first_child, const int* n_child, int* tree_tok, void* scratch, int rows_cap, int cand_rows,
                        int batch, int T, int vocab, const int* depth, int top, cudaStream_t st);

// Both, for a level whose rows are its own.
hydra_status topk_children(const float* part, SplitDesc sd, float* logits, LevelDesc lv, int max_children, const int* first_child, const int* n_child,
                           int* tree_tok, void* scratch, int rows_cap, int batch, int T, int vocab, cudaStream_t st);

// ---- float path: products with what follows them (float_path.cu).  w rows, x and gain on four elements; sums in one slot
// out[m][n] = x[m][k] w[n][k]^T.  w_const as in gemm_simt
hydra_status f32_gemm(const float* x, const float* w, float* out, int m, int n, int k, bool w_const, cudaStream_t st);
// the same of rmsnorm(x)*gain, whose rows also go to hn
hydra_status f32_normed_gemm(const float* x, const float* gain, const float* w, float* out, float* hn, int m, int n, int k, float eps, cudaStream_t st);
// out[m][n] = res[m][n] + x[m][k] w[n][k]^T; out may be res
hydra_status f32_add(const float* x, const float* w, const float* res, float* out, int m, int n, int k, cudaStream_t st);
// act[m][f] = SiLU(gate) * up of rmsnorm(x)*gain, w [2 f][d]: gate rows, then up rows
hydra_status f32_glu(const float* x, const float* gain, const float* w, float* act, int m, int f, int d, float eps, cudaStream_t st);
// qkv_rope_store of the projection of rmsnorm(x)*gain; w [3 d][d], or the [2 d][d] of K and V (kv_only)
hydra_status f32_qkv(const float* x, const float* gain, const float* w, const float2* table, float* q, float* kc, float* vc, RowSet rs, int n_heads, int head_dim, int max_seq,
                     bool kv_only, float eps, int* status, cudaStream_t st);
// first layer of a head: y = h' + SiLU(W [h' ; E of lv.d path tokens] + bias), rows (sequence, parent); write_root as in head_gather.  h' of sequence b is row
// n[b] - 1 of its tc rows (n null: the only one) and goes to copy[b] as well if that is given (one parent then)
struct LastRows { const float* rows; const int* n; int tc; float* copy; };
hydra_status f32_head_first(const LastRows& h, const float* embed, const int* root_tok, int* tree_tok, const int* path_tab, LevelDesc lv, int write_root,
                            const float* w, const float* bias, float* y, int batch, int T, int kp1, int d_model, int vocab, int* status, cudaStream_t st);
// a further layer: y = y_in + SiLU(W y_in + bias); y is another buffer than y_in
hydra_status f32_head_next(const float* y_in, const float* w, const float* bias, float* y, int m, int d, cudaStream_t st);

// ---- acceptance + compaction (one kernel)
struct AcceptArgs {
  const int* tree_tok; const int* amax;
  const int* parent; const int* depth; const uint64_t* anc;
  int T, K, batch, n_layers, n_heads, head_dim, max_seq, max_batch, d_model, esize, kv_planes;
  void* kv_base; const float* h_tree; int h_tree_stride;   // h_tree row = b*h_tree_stride + i
  float* h_new; int* n_new; int* len; int* root_tok;
  int* n_acc; int* path; int* out_tok; unsigned int* done_counter; int* status;
  // acceptance criterion: 0 greedy (token == argmax at the parent); 1 typical (probability of the token under the
  // temperature-tau distribution at the parent > min(eps, alpha * exp(-entropy)))
  int mode; float tau, eps, alpha;
  const float* logits;       // [batch*T][vocab] of the last verification (typical mode)
  const float4* row_stats;   // [batch*T] (max logit, sum exp((l - max)/tau), sum exp(.) (l - max)/tau, 0) (typical mode)
  int vocab;
  const float* u;            // [batch] uniform numbers for the token after the accepted path, or null (= its argmax)
  unsigned long long* pass_bits;   // [batch] out: bit i = candidate row i passed the criterion at its parent
  int* bonus_tmp;            // [batch] scratch: the sampled token, handed from CTA 0 of a sequence to the CTA that publishes the state
};
// row_stats[r] for every logits row (typical acceptance)
hydra_status softmax_row_stats(const float* logits, float4* row_stats, int rows, int vocab, float tau, cudaStream_t st);
hydra_status accept_compact(const AcceptArgs& a, cudaStream_t st);
// the acceptance node of a captured step, and new arguments for it in an instantiated graph
cudaError_t accept_graph_node(cudaGraph_t graph, cudaGraphNode_t* node);
cudaError_t accept_graph_update(cudaGraphExec_t exec, cudaGraphNode_t node, const AcceptArgs& a);

// Whether a stream is being captured, from what cudaStreamIsCapturing answered.  The default stream cannot be used while another one captures: that counts as
// captured.  Any other error is reported as it is.  Either way the runtime does not hand it to the next launch's check.
inline hydra_status capture_answer(cudaError_t asked, cudaStreamCaptureStatus s, bool* captured) {
  *captured = s != cudaStreamCaptureStatusNone;
  if (asked == cudaSuccess) return HYDRA_OK;
  cudaGetLastError();
  if (asked == cudaErrorStreamCaptureImplicit) { *captured = true; return HYDRA_OK; }
  set_last_error("cudaStreamIsCapturing", asked);
  return HYDRA_ERR_CUDA;
}

// ---- small state kernels
// prompt lengths and offsets of a batch, as kernel arguments: no copy from host memory, which would have to outlive the call
constexpr int MAX_BATCH = 64;
struct PromptOffsets { int off[MAX_BATCH + 1]; };
hydra_status set_prompts(const PromptOffsets& p, int batch, int* prompt_len, int* offsets, cudaStream_t st);
hydra_status set_chunk(const int* prompt_len, int chunk, int tc, int* pos0, int* n_rows, int batch, cudaStream_t st);
hydra_status gather_chunk_tokens(const int* tokens, const int* offsets, int chunk, int tc, int* tok_out, int batch,
                                 cudaStream_t st);
// for sequences whose last prompt row lies in this chunk: h_new[b][0] = h[b*tc + i], n_new = 1, len = prompt_len
hydra_status capture_last(const float* h, const int* prompt_len, int chunk, int tc, float* h_new, int kp1, int* n_new,
                          int* len, int batch, int d, cudaStream_t st);
// packed prompts (bfloat16 path): row_at[g] = (sequence, slot) of token g of the concatenated prompts
hydra_status pack_rows(const int* offsets, int batch, int2* row_at, int base, int total, cudaStream_t st);
// capture_last for a packed pass over tokens g0 .. g0+rows-1
hydra_status capture_last_packed(const float* h, const int* offsets, int g0, int rows, float* h_new, int kp1, int* n_new, int* len,
                                 int batch, int d, cudaStream_t st);
// pos0[b] = len[b] - n_new[b]; n_rows[b] = n_new[b]
hydra_status prefix_rowset(const int* len, const int* n_new, int* pos0, int* n_rows, int batch, cudaStream_t st);
// hprime[b] = x[b*tc + n_rows[b]-1]
hydra_status pick_last_row(const float* x, const int* n_rows, int tc, float* hprime, int batch, int d, cudaStream_t st);
hydra_status apply_plant(int* tree_tok, const int* plant, int count, cudaStream_t st);
// dst = src converted to the operand type
hydra_status cast_rows(const float* src, void* dst, size_t dst_ps, size_t count, int dtype, cudaStream_t st);
hydra_status copy_i32(int* dst, const int* src, int count, cudaStream_t st);

}  // namespace hydra
