// Internal launcher interface between the step scheduler and the kernels.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/depcap.h"

namespace dc {

// reason of the last failed call that had no context (what dc_last_error(NULL) returns)
void set_thread_error(const char* msg);

// Per-step sequence description, passed by value to kernels (baked into a captured graph).
struct SeqMeta {
  int ctx_len[DC_MAX_BATCH];
  int last_len[DC_MAX_BATCH];
  int win_len[DC_MAX_BATCH];
  int remain[DC_MAX_BATCH];
  int have_prev[DC_MAX_BATCH];
  int pos0[DC_MAX_BATCH];   // absolute position of active row 0 (ctx_len unless a prefill says otherwise)
  int batch;     // B
  int nv;        // variants in the pass: 1 (curr) or 2 (curr, prev)
  int R_cap;     // the most active rows of a sequence, rounded up to 16
  // active rows [last ; window ; pad] of a sequence, rounded up to 16 each (the dense chain rotates 16 rows in
  // a step), lie behind those of the one before: a ragged batch has no rows that only fill it up to its longest
  // sequence (eight denoising steps of 8..24 rows are 192 rows instead of 256: 5925 -> 5303 us; four prompts
  // of 450..600 tokens 33.4 -> 29.1 ms).
  int rows;                     // rows of one variant
  int row0[DC_MAX_BATCH];       // first row of each sequence in its variant
  int W_cap;     // window rows per sequence, multiple of 16
  int G;         // LM-head group: positions per group (<= 128)
  int npos_pad;  // B * W_cap rounded up to a multiple of G
};

// active row index of (variant v, sequence b, row r)
__host__ __device__ inline int act_row(const SeqMeta& m, int v, int b, int r) {
  return v * m.rows + m.row0[b] + r;
}
// sequence of row br of a variant
__host__ __device__ inline int act_seq(const SeqMeta& m, int br) {
  int b = 0;
  while (b + 1 < m.batch && br >= m.row0[b + 1]) ++b;
  return b;
}
// LM-head row of (variant v, flattened position p = b * W_cap + k): groups of G positions,
// inside a group the curr rows come first, then the prev rows.
__host__ __device__ inline int lm_row(const SeqMeta& m, int v, int p) {
  return (p / m.G) * (m.nv * m.G) + v * m.G + (p % m.G);
}

struct Hyper {
  float lambda;
  int L_min, L_max;
  float tau_low, tau_high, gamma;
  int smooth_radius, norm_mode, boundary_mode, cap_mode;
};

// ---- CUDA-core kernels (any shape, fp32 or bf16 storage) -------------------------------------
// start of a step: x[row] = E[token], status[batch], RoPE table; clears words[n_words]
template <typename T>
void launch_step_begin(const T* embed, const int32_t* last_ids, const int32_t* win_ids, int max_last, int max_window,
                       int mask_id, int vocab, int d, const SeqMeta& m, float* x, int32_t* status, int head_dim,
                       float theta, float* cos_sin, unsigned int* words, int n_words, cudaStream_t s);

// x += sum of nsplit partials (if part != null), then out = T(rmsnorm(x) * g).  rows of x: M.
template <typename T>
void launch_rmsnorm(float* x, const float* part, int nsplit, size_t part_stride, const T* g,
                    float eps, int M, int d, T* out, cudaStream_t s);

// LM-head input rows (k_lm_rows): the final norm of the window's rows, and what may stand in for them
struct PrevLen { int n[DC_MAX_BATCH]; };
template <typename T>
struct LmRowsIo {
  const T* h_in = nullptr;       // [B][2][max_window][d]: replaces every row
  const T* h_prev_in = nullptr;  // [B][max_window][d]: prev row k of sequence b for k < prev.n[b]
  T* h_out = nullptr;            // [B][max_window][d]: gets the curr rows
  int max_window = 0;
  PrevLen prev{};
};
// x holds nv_x variants; with nv_x < m.nv the prev rows are carried in.  Pad rows are zeroed.
template <typename T>
void launch_lm_rows(const float* x, const float* part, int nsplit, size_t part_stride, const T* g, float eps, int d,
                    const SeqMeta& m, int nv_x, const LmRowsIo<T>& io, T* h, cudaStream_t s);

// One CUDA-core GEMM over A [M, K] with the epilogue of its place in a layer.  w0 .. w2: weight
// matrices [rows, K] (QKV: q, k, v;  SWIGLU: gate, up;  otherwise w0 [N, K]).
enum { EPI_STORE_F32 = 0,  // C = acc                                             (fp32, row pitch ldc)
       EPI_ADD_F32 = 1,    // C += acc
       EPI_SWIGLU = 2,     // act [M, N] = silu(gate) * up
       EPI_QKV = 3 };      // q, k: + bias, rotated;  v: + bias; and into the cache (head_dim % 32 == 0)
template <typename T>
struct SimtGemm {
  const T* A = nullptr;
  const T *w0 = nullptr, *w1 = nullptr, *w2 = nullptr;
  int M = 0, N = 0, K = 0, ldc = 0;
  int vec = 0;              // set by the launcher: rows start on 16-byte boundaries
  float* C = nullptr;
  T* act = nullptr;
  // QKV
  int nq = 0, nkv = 0, hd = 0, max_ctx = 0;
  const float* cos_sin = nullptr;
  const T *bq = nullptr, *bk = nullptr, *bv = nullptr;   // projection biases or null
  T *q = nullptr, *k = nullptr, *v = nullptr;            // [M, heads * hd]
  T *k_cache = nullptr, *v_cache = nullptr;              // one layer's context cache to append the last block's rows to, or null
  SeqMeta m{};
};
template <typename T>
void launch_gemm_simt(const SimtGemm<T>& g, int epi, cudaStream_t s);

// the QKV epilogue over projections in `tmp` [M, (nq + 2 nkv) * hd], for any head_dim
template <typename T>
void launch_rope_store(const float* tmp, const SimtGemm<T>& g, cudaStream_t s);

// k_cache [.. max_ctx][hd], v_cache [.. hd][max_ctx] of one layer: [max_batch][nkv][...]
template <typename T>
void launch_attn_simt(const T* q, const T* k, const T* v, const T* k_cache, const T* v_cache,
                      int max_ctx, const SeqMeta& m, int nq, int nkv, int hd, T* o,
                      cudaStream_t s);

// once per context: shared-memory opt-in of the CUDA-core kernels on the current device; false when the attention of
// this head_dim (0: none) does not fit
bool simt_init(bool bf16, int head_dim);

struct SignalOut {
  int32_t* pred_id;
  float *conf, *entropy, *influence, *lse;
  int max_window;
};
// logits [M_lm, V] fp32 in LM-head row order -> per-position signals (into ws arrays, always
// non-null, laid out [B][W_cap]) and optionally the caller's arrays.
struct SimtSignals {
  const float* logits;
  int V, mask_id, forbid;
  int32_t* ws_pred;
  float *ws_conf, *ws_ent, *ws_infl, *ws_lse;
  SignalOut out;
  int32_t* status;
};
void launch_signals_from_logits(const SimtSignals& sg, const SeqMeta& m, cudaStream_t s);

template <typename T>
void launch_xlogp(const T* h, const T* lm_head, const int32_t* ws_pred, const float* ws_lse,
                  int d, int V, const SeqMeta& m, int max_window, float* xlogp, cudaStream_t s);

// ---- decision kernels --------------------------------------------------------------------------
// per-sequence lengths in device memory (all null: the lengths inside SeqMeta are used)
struct DevLens {
  const int32_t* win_len = nullptr;
  const int32_t* remain = nullptr;
  const int32_t* have_prev = nullptr;
};
// influence / entropy rows have stride ld, outputs stride max_window (and may be null but block_len);
// vec: every row starts on a 16-byte boundary
struct BoundaryIo {
  int ld, max_window, vec;
  float *score, *cum_i, *cum_s;
  int32_t* block_len;
};
inline BoundaryIo make_boundary_io(const float* influence, const float* entropy, int ld, int max_window, float* score,
                                   float* cum_i, float* cum_s, int32_t* block_len) {
  auto aligned = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  const int vec = ld % 4 == 0 && max_window % 4 == 0 && aligned(influence) && aligned(entropy) && aligned(score) &&
                  aligned(cum_i) && aligned(cum_s);
  return BoundaryIo{ld, max_window, vec, score, cum_i, cum_s, block_len};
}
void launch_boundary(const float* influence, const float* entropy, int ld, const SeqMeta& m,
                     const Hyper& hp, int max_window, float* score, float* cum_i, float* cum_s,
                     int32_t* block_len, cudaStream_t s);

// the same kernel over `batch` sequences (any number) whose lengths are arrays in device memory
void launch_boundary_dev(const float* influence, const float* entropy, int ld, int batch, const DevLens& dl,
                         const Hyper& hp, int max_window, float* score, float* cum_i, float* cum_s,
                         int32_t* block_len, cudaStream_t s);
void launch_select_dev(const float* conf, const int32_t* win_ids, const float* xlogp,
                       const int32_t* block_len, int batch, const DevLens& dl, const Hyper& hp, int mask_id,
                       int max_window, uint8_t* sel_mask, int32_t* sel_idx, int32_t* sel_count,
                       cudaStream_t s);

void launch_select(const float* conf, const int32_t* win_ids, const float* xlogp,
                   const int32_t* block_len, const SeqMeta& m, const Hyper& hp, int mask_id,
                   int max_window, uint8_t* sel_mask, int32_t* sel_idx, int32_t* sel_count,
                   cudaStream_t s);

// Eq. (2): win_ids[i] <- pred_id[i] where selected and still masked, inside [0, block_len);
// remaining[b] = masked positions left in the block (may be null)
void launch_commit(int32_t* win_ids, const int32_t* pred_id, const uint8_t* sel_mask,
                   const int32_t* block_len, const SeqMeta& m, int mask_id, int max_window,
                   int32_t* remaining, cudaStream_t s);

// CAP-Decoding and the commit in one launch, for the decoding loop: sequences with keep.n[b] >= 0 are inside a
// block of that length (block_len[b] is not read); win_ids is updated as by launch_commit, and the host's
// copies (pinned memory: block length, masked positions left, status, window ids) are written
struct SelectCommit {
  int32_t* win_ids = nullptr;         // null: select only
  const int32_t *pred_id = nullptr, *status = nullptr;
  PrevLen keep{};
  int32_t *host_blk = nullptr, *host_left = nullptr, *host_status = nullptr, *host_ids = nullptr;
};
void launch_select_commit(const float* conf, const float* xlogp, const int32_t* block_len, const SeqMeta& m,
                          const Hyper& hp, int mask_id, int max_window, const SelectCommit& cm, cudaStream_t s);

}  // namespace dc
