// Host interface of the fused CUDA-core step (simt_step.cu).
#pragma once
#include "kernels.h"

namespace dc {

template <typename T>
struct SimtLayer {
  const T *wq, *wk, *wv, *wo, *wg, *wu, *wd, *n1, *n2, *bq, *bk, *bv;   // biases null without them
};

template <typename T>
struct SimtStep {
  const SimtLayer<T>* layers;   // device
  int n_layers, kv_only, export_kv;
  SeqMeta m, ml;                // of the stack, and what the LM-head stage sees
  int d, F, nq, nkv, hd, V, max_ctx, max_window;
  size_t cache_layer;           // elements of one layer's cache
  float eps;
  float* x;
  T *q, *k, *v, *o, *act, *h;
  const float* cos_sin;
  T *k_cache, *v_cache;         // whole caches
  const T *final_norm, *lm_head;
  LmRowsIo<T> io;
  float* logits;
  SimtSignals sig;
  float* xlogp;                 // null: not wanted
  BoundaryIo bnd;               // block_len null: no boundary rule
  Hyper hp;
  unsigned int* bar;            // arrivals, and a word that a CTA which gave up sets; zero at the start
  int kt, group_smem;           // set by the launcher
  int stall;                    // test hook: one CTA leaves at once, so that the others wait for it in vain
};

// What the fused step needs to know about a context; grid == 0: the shape or the device does not take it
struct SimtFuse { int grid = 0, kt = 0, group_smem = 0; };
// Tiles of 16 x 16 of the largest GEMM.  d 256, MLP 1024, vocab 4096, one launch against separate ones: 107
// against 153 us at 1024 tiles, 168 / 203 at 2048, 263 / 248 at 4096, 331 / 266 at 6144.
constexpr int kFuseMaxTiles = 148 * 18;

template <typename T>
bool simt_step_init(SimtFuse* f, int d, int F, int nq, int nkv, int hd, int vocab, int max_ctx);   // false: a CUDA call failed
template <typename T>
bool simt_step_ok(const SimtFuse& f, const SimtStep<T>& p);   // this step's sizes are what it is for
template <typename T>
int launch_simt_step(const SimtFuse& f, SimtStep<T> p, cudaStream_t s);   // cudaError_t
int simt_set_wait_limit_us(long long us, cudaStream_t s);

}  // namespace dc
