// Decision kernels: the DepGA-Block boundary scan (Section 4.2, cumulative form Section 4.4)
// and CAP-Decoding (Section 4.3, Algorithm 1).  One warp per sequence.
//
// Every floating-point step that decides an integer is written with explicit round-to-nearest
// intrinsics (no contraction into FMA) and a fixed operation order, so the decisions are a
// function of the input bits alone; running sums use 2^40 fixed point, which is order-free.
#include <math.h>

#include <type_traits>

#include "decisions.cuh"
#include "pdl.cuh"

namespace dc {

constexpr int kThreads = 256;         // one thread per window position (k_commit)

template <int NQ>
__global__ void __launch_bounds__(32 * kSeqWarps) k_boundary(const float* influence, const float* entropy, int batch,
                                                             const __grid_constant__ SeqMeta m, DevLens dl, Hyper hp,
                                                             BoundaryIo io) {
  __shared__ float sI[kSeqWarps][33 * NQ], sH[kSeqWarps][33 * NQ];
  pdl_trigger();
  pdl_wait();
  const int w = threadIdx.x >> 5, b = blockIdx.x * (blockDim.x >> 5) + w;
  if (b < batch) boundary_seq<NQ>(influence, entropy, b, m, dl, hp, io, sI[w], sH[w]);
}

// f(NQ as a constant): positions per lane for a window of max_window, warps per CTA for a batch
template <typename F>
static void decide_launch(int batch, int max_window, F&& f) {
  const int warps = batch > kSpread ? kSeqWarps : 1;
  const dim3 grid((batch + warps - 1) / warps);
  if (max_window <= 64) f(std::integral_constant<int, 2>{}, grid, 32 * warps);
  else if (max_window <= 128) f(std::integral_constant<int, 4>{}, grid, 32 * warps);
  else f(std::integral_constant<int, kMaxW / 32>{}, grid, 32 * warps);
}

static void boundary(const float* influence, const float* entropy, int ld, int batch, const SeqMeta& m,
                     const DevLens& dl, const Hyper& hp, int max_window, float* score, float* cum_i, float* cum_s,
                     int32_t* block_len, cudaStream_t s) {
  const BoundaryIo io = make_boundary_io(influence, entropy, ld, max_window, score, cum_i, cum_s, block_len);
  decide_launch(batch, max_window, [&](auto nq, dim3 grid, int threads) {
    launch_chained(k_boundary<decltype(nq)::value>, grid, threads, 0, s, influence, entropy, batch, m, dl, hp, io);
  });
}

void launch_boundary(const float* influence, const float* entropy, int ld, const SeqMeta& m,
                     const Hyper& hp, int max_window, float* score, float* cum_i, float* cum_s,
                     int32_t* block_len, cudaStream_t s) {
  boundary(influence, entropy, ld, m.batch, m, DevLens{}, hp, max_window, score, cum_i, cum_s, block_len, s);
}

void launch_boundary_dev(const float* influence, const float* entropy, int ld, int batch, const DevLens& dl,
                         const Hyper& hp, int max_window, float* score, float* cum_i, float* cum_s,
                         int32_t* block_len, cudaStream_t s) {
  boundary(influence, entropy, ld, batch, SeqMeta{}, dl, hp, max_window, score, cum_i, cum_s, block_len, s);
}

// ---- CAP-Decoding ------------------------------------------------------------------------------
// Algorithm 1 with the conflicts evaluated where they decide something: only a member of S removes
// candidates, so D_ij is read for i in S and j still alive - a row and a column of xlogp per selected
// position, never the matrix of the whole pool (Eq. 6: conflict iff xlogp[i,j] + xlogp[j,i] > gamma).
// Position 32 q + lane belongs to the lane; a set of candidates is the array of their sort keys, 0 where
// a position is not in it.  The kernel is bound by instruction issue and by the latency of those
// rows and columns, so the code is kept to few instructions and five CTAs of eight warps per SM.
// (Loading the conflicts of the last 16 candidates at once instead of a round per selected position
// was slower: 63 against 40 us, most of its loads were for pairs that never meet; prefetching the
// pool's rows into L2 changed nothing at 8192 x 128 and cost 8 us at 1000 x 256.)

// float -> unsigned with the same order (confidences may be any finite float); never 0
__device__ __forceinline__ unsigned order_key(float c) {
  const unsigned u = __float_as_uint(__fadd_rn(c, 0.f));   // (-0 and 0 are the same confidence)
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// removes from `key` what conflicts with one of the positions a[0..NA)
template <int NQ, int NA>
__device__ __forceinline__ void drop_conflicts(const float* __restrict__ xb, unsigned ld, int L, const int (&a)[NA],
                                               unsigned (&key)[NQ], float gamma) {
  constexpr int G = NQ < 2 ? NQ : 2;   // 64 positions per round of loads: shorter blocks skip the rest
  const unsigned lane = threadIdx.x & 31;
#pragma unroll
  for (int q0 = 0; q0 < NQ; q0 += G) {
    if (q0 > 0 && 32 * q0 >= L) break;
    float row[NA][G], col[NA][G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const bool want = key[q0 + g] != 0u;
      const unsigned j = 32 * (q0 + g) + lane;
#pragma unroll
      for (int t = 0; t < NA; ++t) {
        row[t][g] = want ? xb[(unsigned)a[t] * ld + j] : 0.f;
        col[t][g] = want ? xb[j * ld + (unsigned)a[t]] : 0.f;
      }
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
      float d = -INFINITY;
#pragma unroll
      for (int t = 0; t < NA; ++t) d = fmaxf(d, __fadd_rn(row[t][g], col[t][g]));
      if (d > gamma) key[q0 + g] = 0u;
    }
  }
}

// the position first in (confidence descending, position ascending) order, -1 if there is none
template <int NQ>
__device__ __forceinline__ int first_of(const unsigned (&key)[NQ]) {
  unsigned best = key[0];
#pragma unroll
  for (int q = 1; q < NQ; ++q) best = max(best, key[q]);
  const unsigned top = __reduce_max_sync(kAll, best);
  if (top == 0u) return -1;
  unsigned pos = 0x7fffffffu;
#pragma unroll
  for (int q = NQ - 1; q >= 0; --q)
    if (key[q] == top) pos = 32 * q + (threadIdx.x & 31);
  return (int)__reduce_min_sync(kAll, pos);
}

// Greedy pass over the candidates in confidence order: take a position, drop what conflicts with it.
template <int NQ>
__device__ __forceinline__ unsigned greedy(const float* __restrict__ xb, unsigned ld, int L, unsigned (&key)[NQ], float gamma) {
  unsigned sel = 0u;   // bit q: position 32 q + lane
  while (true) {
    const int a[1] = {first_of<NQ>(key)};
    if (a[0] < 0) return sel;
    const bool mine = (int)(threadIdx.x & 31) == (a[0] & 31);
#pragma unroll
    for (int q = 0; q < NQ; ++q)
      if (mine && q == (a[0] >> 5)) { key[q] = 0u; sel |= 1u << q; }
    drop_conflicts<NQ, 1>(xb, ld, L, a, key, gamma);
  }
}

template <int NQ>
__global__ void __launch_bounds__(32 * kSeqWarps, 5) k_select(
    const float* __restrict__ conf, const int32_t* win_ids,
    const float* __restrict__ xlogp, const int32_t* __restrict__ block_len, int batch,
    const __grid_constant__ SeqMeta m, DevLens dl, Hyper hp, int mask_id, int max_window,
    uint8_t* __restrict__ sel_mask, int32_t* __restrict__ sel_idx, int32_t* __restrict__ sel_count,
    const __grid_constant__ SelectCommit cm) {
  constexpr int NA = 4;
  __shared__ __align__(16) int members[kSeqWarps][32 * NQ + NA];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int b = blockIdx.x * (blockDim.x >> 5) + w;
  pdl_wait();
  if (b >= batch) return;
  const int W = len_of(dl.win_len, m.win_len, b);
  const int kept = cm.win_ids != nullptr ? cm.keep.n[b] : -1;   // the length of a block that a generation is in the middle of
  const int blk = kept >= 0 ? kept : block_len[b];
  const int L = min(max(blk, 0), W);
  const size_t o = (size_t)b * max_window;
  const float* xb = xlogp + o * max_window;
  unsigned key[NQ];                           // M^t ∩ B^t
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int k = 32 * q + lane;
    key[q] = 0u;
    if (k < L) {
      const float c = conf[o + k];
      if (win_ids[o + k] == mask_id) key[q] = c == c ? order_key(c) : 1u;   // NaN: below every threshold
    }
  }
  auto bar = [](float tau) { return tau == tau ? order_key(tau) : kAll; };   // (nothing reaches a NaN)
  const unsigned k_low = bar(hp.tau_low), k_high = max(k_low, bar(hp.tau_high));
  unsigned cand[NQ];
  unsigned sel = 0u;
  if (hp.cap_mode == DC_CAP_STRICT) {         // phase 1, greedily with conflict checks
#pragma unroll
    for (int q = 0; q < NQ; ++q) cand[q] = key[q] >= k_high ? key[q] : 0u;
    sel = greedy<NQ>(xb, max_window, L, cand, hp.gamma);
  } else {                                    // phase 1 as printed: every c_i >= tau_high enters S
#pragma unroll
    for (int q = 0; q < NQ; ++q) sel |= (key[q] >= k_high ? 1u : 0u) << q;
  }
  // the pool of Eq. (5) without S and without what conflicts with a member of S, four members at a time
  int n = 0;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const bool on = (sel >> q) & 1u;
    const unsigned word = __ballot_sync(kAll, on);
    if (on) members[w][n + __popc(word & ((1u << lane) - 1u))] = 32 * q + lane;
    n += __popc(word);
    cand[q] = (!on && key[q] >= k_low) ? key[q] : 0u;
  }
  __syncwarp();
  if (n > 0 && lane < NA) members[w][n + lane] = members[w][n - 1];   // the last group is filled with the last member
  __syncwarp();
  for (int t = 0; t < n; t += NA) {
    const int4 g = *reinterpret_cast<const int4*>(&members[w][t]);
    const int a[NA] = {g.x, g.y, g.z, g.w};
    drop_conflicts<NQ, NA>(xb, max_window, L, a, cand, hp.gamma);
  }
  // phase 2: greedy completion in descending confidence
  sel |= greedy<NQ>(xb, max_window, L, cand, hp.gamma);
  // fallback: the most confident masked position of the block
  if (!__any_sync(kAll, sel != 0u)) {
    const int a = first_of<NQ>(key);
    if (a >= 0 && lane == (a & 31)) sel = 1u << (a >> 5);
  }
  // outputs: mask, ascending index list, count
  int total = 0;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int k = 32 * q + lane;
    const bool on = (sel >> q) & 1u;
    const unsigned word = __ballot_sync(kAll, on);
    if (sel_mask && k < W) sel_mask[o + k] = on ? 1 : 0;
    if (sel_idx && on) sel_idx[o + total + __popc(word & ((1u << lane) - 1u))] = k;
    total += __popc(word);
  }
  if (lane == 0 && sel_count) sel_count[b] = total;
  if (cm.win_ids == nullptr) return;
  // Eq. (2) and what the host loop of a generation reads, straight into its pinned buffer
  int left = 0;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int k = 32 * q + lane;
    left += __popc(__ballot_sync(kAll, key[q] != 0u && !((sel >> q) & 1u)));
    if (k < W) {
      int id = win_ids[o + k];
      if ((sel >> q) & 1u) { id = cm.pred_id[o + k]; cm.win_ids[o + k] = id; }
      cm.host_ids[o + k] = id;
    }
  }
  if (lane == 0) { cm.host_blk[b] = blk; cm.host_left[b] = left; cm.host_status[b] = cm.status[b]; }
}

static void select(const float* conf, const int32_t* win_ids, const float* xlogp, const int32_t* block_len, int batch,
                   const SeqMeta& m, const DevLens& dl, const Hyper& hp, int mask_id, int max_window,
                   uint8_t* sel_mask, int32_t* sel_idx, int32_t* sel_count, cudaStream_t s,
                   const SelectCommit& cm = SelectCommit{}) {
  decide_launch(batch, max_window, [&](auto nq, dim3 grid, int threads) {
    launch_chained(k_select<decltype(nq)::value>, grid, threads, 0, s, conf, win_ids, xlogp, block_len, batch, m, dl, hp,
                   mask_id, max_window, sel_mask, sel_idx, sel_count, cm);
  });
}

void launch_select(const float* conf, const int32_t* win_ids, const float* xlogp,
                   const int32_t* block_len, const SeqMeta& m, const Hyper& hp, int mask_id,
                   int max_window, uint8_t* sel_mask, int32_t* sel_idx, int32_t* sel_count,
                   cudaStream_t s) {
  select(conf, win_ids, xlogp, block_len, m.batch, m, DevLens{}, hp, mask_id, max_window, sel_mask, sel_idx, sel_count, s);
}

void launch_select_dev(const float* conf, const int32_t* win_ids, const float* xlogp,
                       const int32_t* block_len, int batch, const DevLens& dl, const Hyper& hp, int mask_id,
                       int max_window, uint8_t* sel_mask, int32_t* sel_idx, int32_t* sel_count,
                       cudaStream_t s) {
  select(conf, win_ids, xlogp, block_len, batch, SeqMeta{}, dl, hp, mask_id, max_window, sel_mask, sel_idx, sel_count, s);
}

// ---- commit (Eq. 2): y_i <- yhat_i for the selected positions; masked positions left in the block --
__global__ void __launch_bounds__(kThreads) k_commit(int32_t* __restrict__ win_ids,
                                                    const int32_t* __restrict__ pred_id,
                                                    const uint8_t* __restrict__ sel_mask,
                                                    const int32_t* __restrict__ block_len, SeqMeta m,
                                                    int mask_id, int max_window,
                                                    int32_t* __restrict__ remaining) {
  __shared__ int red[kThreads / 32];
  const int b = blockIdx.x, i = threadIdx.x;
  const int W = m.win_len[b];
  const int L = min(max(block_len[b], 0), W);
  int left = 0;
  if (i < W) {
    const size_t o = (size_t)b * max_window + i;
    int id = win_ids[o];
    if (i < L && id == mask_id && sel_mask[o]) { id = pred_id[o]; win_ids[o] = id; }
    left = (i < L && id == mask_id) ? 1 : 0;
  }
  for (int o = 16; o > 0; o >>= 1) left += __shfl_xor_sync(0xffffffffu, left, o);
  if ((i & 31) == 0) red[i >> 5] = left;
  __syncthreads();
  if (i == 0 && remaining) {
    int t = 0;
    for (int w = 0; w < kThreads / 32; ++w) t += red[w];
    remaining[b] = t;
  }
}

void launch_select_commit(const float* conf, const float* xlogp, const int32_t* block_len, const SeqMeta& m,
                          const Hyper& hp, int mask_id, int max_window, const SelectCommit& cm, cudaStream_t s) {
  select(conf, cm.win_ids, xlogp, block_len, m.batch, m, DevLens{}, hp, mask_id, max_window, nullptr, nullptr, nullptr, s, cm);
}

void launch_commit(int32_t* win_ids, const int32_t* pred_id, const uint8_t* sel_mask,
                   const int32_t* block_len, const SeqMeta& m, int mask_id, int max_window,
                   int32_t* remaining, cudaStream_t s) {
  k_commit<<<m.batch, kThreads, 0, s>>>(win_ids, pred_id, sel_mask, block_len, m, mask_id, max_window,
                                        remaining);
}

}  // namespace dc
