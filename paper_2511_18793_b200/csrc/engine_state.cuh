// Device-resident state of one decode call and the launchers of the beam-search kernels that work on it.
//
// Indexing convention: a "level n" beam has n codes (n = 0 is the empty beam).  Arrays named tb_* hold the true
// beam sets B_n of the primary model for n = 0..L; dw_* hold the draft head's working beam sets.
#pragma once

#include "common.cuh"

namespace nz {

struct EngineState {
  int Bmax, Kmax, L, d, Hkv, hd;
  LevelInfo li;
  HashSetView hs;
  PrefixMapView pm;
  int* status;
  // draft-head variants (the ablations of Section 4.3); defaults 1, 1, 0 = Eq. 2 and Eq. 3 as printed
  int draft_use_h, draft_use_s, draft_additive;

  // true beams, [L+1][Bmax][Kmax]([L])
  int* tb_codes; float* tb_score; int* tb_parent; int* tb_count;   // tb_count: [L+1][Bmax]
  int* tb_anc;      // [L+1][Bmax][Kmax][L]: slot (in the draft-KV slab of level i+1) of the ancestor with i+1 codes
  int* tb_self;     // [L+1][Bmax][Kmax]: slot of the beam's own KV in the slab of its level
  int* tb_src;      // [L+1][Bmax][Kmax]: token index whose hidden state predicts the beam's next code

  int* row_m;       // [Bmax] levels settled (L = row finished)
  int* row_cur;     // [Bmax] level whose beams have logits in the current pass, -1 = row stopped this round
  int* row_P;       // [Bmax] context length of the row (BOS + history tokens)
  int* row_m_start; // [Bmax] levels the row had settled when the current round began
  int* draft_rows;  // [1] rows of the draft head's products in the coming round: batch * Kmax, or 0 when no request drafts
  int* row_spec;    // [Bmax] 1: the draft head drafts for the row in the next round (always 1 unless the adaptive policy is on)

  // The round's draft tree, [L+1][Bmax][Kmax]([L]): level l holds the drafted nodes with l codes (the draft head's beam
  // set of that level, or the distinct l-prefixes of caller-supplied tuples); dw_parent = slot of the node's parent in
  // level l - 1.  The drafted tuples of the round are level L.
  int* dw_codes; float* dw_score; int* dw_parent; int* dw_count;
  int* d_m;         // [Bmax] level the row's drafting started from this round (L = the draft head takes no part)
  int* d_beam;      // [L+1][Bmax][Kmax] for a node in this round's pass: rank of the true beam of B_m it descends from
                    //                   (-1: the node is dead -- its first m codes are no beam, or it has no parent)
  float* state_lv;  // [L+1][Bmax][Kmax][d] draft-head context states s_l (l = 2..L used; s_1 = h_0)

  // verify-pass token list
  int* node_index;  // [Bmax][L][Kmax] token index of node (level n = 1..L-1 stored at n, slot), -1 if absent
  int* tok_row; int* tok_pos; int* tok_id; int* tok_ctx_len; long long* tok_kv_dst; long long* tok_ext;  // tok_ext [Mv][L]
  int* row_tok_count;   // [Bmax]
  int* row_tok_start;   // [Bmax] first token of the request in the list
  int* pf_row_start; int* pf_row_count;   // [Bmax] the same for a prefill chunk (indexed by row within the chunk)
  int4* req_info; int4* pf_req_info;      // [Bmax] {first token, token count, cache row, context length or -1 = causal}:
                                          //        all the attention kernel needs to know about a request, in one load
  int* n_tokens;        // [1] tokens of the verify pass
  int* pf_n_tokens;     // [1] tokens of the prefill chunk

  const float* h_f32;   // [Bmax][L+1][d]
};

inline __host__ __device__ long long lvl_bk(const EngineState& e, int n, int b, int k) {
  return ((long long)n * e.Bmax + b) * e.Kmax + k;
}

#ifdef __CUDACC__
// Where slot k of request b gets its state s_{l+1} from (Eq. 3's step from level l): the slot of the state s_l and the code, -1 = none.
//   requests still teacher-forcing (d_m >= l): beam k of the start set, its own state, its l-th code;
//   requests drafting (d_m < l): survivor k of level l, its parent's state, the code just chosen.
// What a drafting request asks for is asked for at once (one after the other these were four round trips to the L2).
struct DraftSource { int parent, code; };
__device__ __forceinline__ DraftSource draft_source(const EngineState& e, int b, int k, int l) {
  const int dm = e.d_m[b], m = e.row_m[b];
  const long long s_l = lvl_bk(e, l, b, k);
  int count = e.dw_count[l * e.Bmax + b], parent = e.dw_parent[s_l], code = e.dw_codes[s_l * e.L + (l - 1)];
  if (dm >= l) {
    const int src = min(dm, e.L);
    count = e.dw_count[src * e.Bmax + b]; parent = k; code = e.dw_codes[lvl_bk(e, src, b, k) * e.L + (l - 1)];
  }
  const bool live = (dm < e.L || m < e.L) && k < count;
  return DraftSource{live ? parent : -1, live ? code : -1};
}
#endif

struct SelectArgs {
  const float* logits; long long row_stride; int col_off;
  const int* src_row; int src_mul;      // logits row of beam r of request b: src_row ? src_row[b*in_stride+r] : b*src_mul+r
  const int* in_codes; const float* in_score; const int* in_count; int in_stride;
  int n;                                // codes the input beams have; the level's codebook is T[n]
  int T, K, per_beam, filter;
  const int* gate; int gate_mode, gate_value;   // 0: none, 1: run iff gate[b] == value, 2: run iff gate[b] < value
  const float* logit_bias; long long bias_stride;   // optional: logits of request b get logit_bias[b * bias_stride + t] added
  int* out_codes; int* out_token; float* out_score; int* out_parent; int* out_count; int out_stride;
  int tuple_len;                        // row length of in_codes / out_codes (L)
  int batch;
  LevelInfo li; HashSetView hs;
  PrefixMapView pm;
  int final_mask_from_map;              // 1: the last-level mask of a beam (all T_L extensions) reads the prefix map; 0: hash probes
  int prefix_filter;                    // 1: this is an earlier level and candidates that begin no valid ID are dropped
  const int* status; int* host_status;  // optional: the status words are copied to pinned host memory
};
void launch_select(const SelectArgs& a, cudaStream_t st);
// What closes a round, behind its last selection (host == null: not this one): the trace's outputs and, in pinned host memory, the status
// words (host) and each request's counters (rows).
struct RoundEnd { int* host; int4* rows; int round, adaptive, draft_next; nezha_trace tr; };
// launch_select of level a.n (gated on row_cur == a.n) followed, in the same launch, by the accept / roll-back step of that level, the
// same for the levels up to (not including) `last` as long as the request's beams are nodes of the pass and, where re.host is
// given, the end of the round.  Levels behind the first: logits next to each other, tables tb_* of the next level.
void launch_select_advance(const SelectArgs& a, const EngineState& e, int last, int K, int* out_codes, float* out_score,
                           int* out_count, const RoundEnd& re, cudaStream_t st);
// launch_select followed, in the same launch, by launch_draft_step of level l (same arguments as there)
void launch_select_step(const SelectArgs& a, const EngineState& e, int l, const float* G, int per_req, long long g_stride, int t_cols,
                        const float* U, const float* bias, void* s_act, cudaStream_t st);
// launch_select and, beside it in the same launch, launch_build_nodes
void launch_select_nodes(const SelectArgs& a, const EngineState& e, cudaStream_t st);
size_t select_smem_bytes(int in_stride, int K);
cudaError_t select_configure(int max_beam);

// out_* and every pointer of tr may be null
void launch_decode_begin(const EngineState& e, int batch, int K, int from_scratch, int* out_codes, float* out_scores, int* out_count,
                         const nezha_trace& tr, cudaStream_t st);
void launch_draft_set(const EngineState& e, int batch, int K, const int* drafts, const int* n_draft, cudaStream_t st);
// the whole tree given by the caller: tree_codes [L][batch][K][L], tree_count [L][batch]
void launch_draft_tree_set(const EngineState& e, int batch, int K, const int* tree_codes, const int* tree_count, cudaStream_t st);
void launch_draft_x(const EngineState& e, int batch, int l, void* x, bool bf16, cudaStream_t st);
void launch_trans_gather(const EngineState& e, int batch, int l, const void* embed, void* A, bool bf16,
                         cudaStream_t st);
void launch_trans_add(const EngineState& e, int batch, int l, const void* embed, bool bf16, cudaStream_t st);
// The draft head with its two per-level products merged (see DraftFast in api.cu)
void launch_draft_state_init(const EngineState& e, int batch, void* s_act, cudaStream_t st);
void launch_draft_step(const EngineState& e, int batch, int l, const float* G, int per_req, long long g_stride, int t_cols, const float* U,
                       const float* bias, void* s_act, cudaStream_t st);
// fp32: launch_draft_x, or launch_trans_gather (`state`), with the product behind it in one launch
bool draft_gemm_rows_applies(int M, int N, const EngineState& e, const void* W);
void launch_draft_gemm_rows(const GemmArgs& a, const EngineState& e, int l, const void* embed, bool state, cudaStream_t st);
void launch_copy_logits_bias(const float* src, long long row_stride, int row_mul, int batch, int n_beams, int T,
                             const float* bias, long long bias_stride, float* dst, cudaStream_t st);
void launch_build_nodes(const EngineState& e, int batch, cudaStream_t st);
void launch_nodes_from_prefixes(const EngineState& e, int batch, int n_beams, int level, const int* prefixes,
                                cudaStream_t st);
void launch_copy_logits(const float* src, long long row_stride, int col_off, const int* row_index, int row_mul,
                        int beam_mul, int batch, int n_beams, int idx_stride, int T, float* dst, cudaStream_t st);
void launch_fill_i32(int* p, long long n, int v, cudaStream_t st);
void launch_trace_beams(const EngineState& e, int batch, int K, const nezha_trace& tr, cudaStream_t st);

}  // namespace nz
