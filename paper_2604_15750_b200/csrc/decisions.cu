// Decision kernels: the DepGA-Block boundary scan (Section 4.2, cumulative form Section 4.4)
// and CAP-Decoding (Section 4.3, Algorithm 1).  One warp per sequence.
//
// Every floating-point step that decides an integer is written with explicit round-to-nearest
// intrinsics (no contraction into FMA) and a fixed operation order, so the decisions are a
// function of the input bits alone; running sums use 2^40 fixed point, which is order-free.
#include <math.h>

#include <type_traits>

#include "kernels.h"

namespace dc {

constexpr int kMaxW = DC_MAX_WINDOW;  // 256
constexpr int kThreads = 256;         // one thread per window position (k_commit)
constexpr float kFxScale = 1099511627776.f;           // 2^40
constexpr unsigned kAll = 0xffffffffu;

// 2^40 fixed point.  Scaling by a power of two is exact, so one conversion rounds (to nearest) either
// way; a sum of 2^53 or more goes through a double first, as it always did, and may round twice.
__device__ __forceinline__ long long to_fixed(float v) { return __float2ll_rn(__fmul_rn(v, kFxScale)); }
__device__ __forceinline__ float from_fixed(long long v) {
  if (v > -(1ll << 53) && v < (1ll << 53)) return __fmul_rn(__ll2float_rn(v), 1.f / kFxScale);
  return __double2float_rn(__ll2double_rn(v) * (1.0 / 1099511627776.0));
}

// Both decisions are a few hundred dependent operations per sequence, so a sequence is one warp with
// NQ positions per lane, every reduction and scan is a shuffle, and nothing waits on a block-wide
// barrier.  A call over many sequences is
// then bound by its memory traffic: all 8192 sequences of a large call are resident at once and
// their load latencies overlap (8192 x 128: k_boundary 26 -> 13 us, k_select 222 -> 39 us against
// one block with a thread per position).  With few sequences - a step - every warp is a CTA of its
// own, so that they spread over the SMs.
constexpr int kSeqWarps = 8;          // sequences per CTA of a call with more sequences than kSpread
constexpr int kSpread = 4 * 148;

// NQ consecutive values of a row from position k0 on; positions >= n are 0 / not written
template <int NQ>
__device__ __forceinline__ void load_run(const float* __restrict__ row, int k0, int n, int vec, float (&v)[NQ]) {
  constexpr int V = NQ >= 4 ? 4 : 2;
#pragma unroll
  for (int q = 0; q < NQ; q += V) {
    if (vec && k0 + q + V <= n) {
      if (V == 4) {
        const float4 t = *reinterpret_cast<const float4*>(row + k0 + q);
        v[q] = t.x; v[q + 1] = t.y; v[q + V / 2] = t.z; v[q + V - 1] = t.w;
      } else {
        const float2 t = *reinterpret_cast<const float2*>(row + k0 + q);
        v[q] = t.x; v[q + 1] = t.y;
      }
    } else {
#pragma unroll
      for (int u = 0; u < V; ++u) v[q + u] = k0 + q + u < n ? row[k0 + q + u] : 0.f;
    }
  }
}
template <int NQ>
__device__ __forceinline__ void store_run(float* __restrict__ row, int k0, int n, int vec, const float (&v)[NQ]) {
  constexpr int V = NQ >= 4 ? 4 : 2;
#pragma unroll
  for (int q = 0; q < NQ; q += V) {
    if (vec && k0 + q + V <= n) {
      if (V == 4) *reinterpret_cast<float4*>(row + k0 + q) = make_float4(v[q], v[q + 1], v[q + V / 2], v[q + V - 1]);
      else *reinterpret_cast<float2*>(row + k0 + q) = make_float2(v[q], v[q + 1]);
    } else {
#pragma unroll
      for (int u = 0; u < V; ++u)
        if (k0 + q + u < n) row[k0 + q + u] = v[q + u];
    }
  }
}
__device__ __forceinline__ float warp_max(float v) {   // exact, order-free
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kAll, v, o));
  return v;
}
// inclusive prefix sum over the lanes
__device__ __forceinline__ long long warp_scan(long long v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long t = __shfl_up_sync(kAll, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

__device__ __forceinline__ float normalise(float x, float hi, float lo, int mode) {
  if (mode == DC_NORM_NONE) return x;
  if (mode == DC_NORM_MAX) return __fdiv_rn(x, fmaxf(hi, 1e-8f));
  return __fdiv_rn(__fsub_rn(x, lo), fmaxf(__fsub_rn(hi, lo), 1e-8f));
}

// Lengths of the sequences of a call: by value inside SeqMeta (a step: at most DC_MAX_BATCH
// sequences), or - when the pointers are set - arrays in device memory, for calls over any number
// of sequences.
__device__ __forceinline__ int len_of(const int32_t* dev, const int* by_value, int b) {
  return dev != nullptr ? dev[b] : by_value[b];
}

template <int NQ>
__global__ void __launch_bounds__(32 * kSeqWarps) k_boundary(
    const float* __restrict__ influence, const float* __restrict__ entropy, int ld, int batch,
    const __grid_constant__ SeqMeta m, DevLens dl, Hyper hp, int max_window, float* __restrict__ score,
    float* __restrict__ cum_i, float* __restrict__ cum_s, int32_t* __restrict__ block_len, int vec) {
  __shared__ float sI[kSeqWarps][33 * NQ], sH[kSeqWarps][33 * NQ];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x * (blockDim.x >> 5) + w;
  if (b >= batch) return;
  const int Lw = max(0, min(min(hp.L_max, len_of(dl.remain, m.remain, b)), len_of(dl.win_len, m.win_len, b)));
  const size_t o = (size_t)b * max_window;
  if (!len_of(dl.have_prev, m.have_prev, b)) {  // cold start: the first block uses L_min
    for (int k = lane; k < Lw; k += 32) {
      if (score) score[o + k] = 0.f;
      if (cum_i) cum_i[o + k] = 0.f;
      if (cum_s) cum_s[o + k] = 0.f;
    }
    if (lane == 0) block_len[b] = min(hp.L_min, Lw);
    return;
  }
  // lane l holds the NQ consecutive positions NQ l ..: 16-byte accesses where the rows allow it, and
  // one scan over the lanes' totals instead of NQ scans (the kernel is bound by instruction issue)
  const int k0 = NQ * lane;
  float rawI[NQ], Is[NQ], Hs[NQ];
  load_run<NQ>(influence + (size_t)b * ld, k0, Lw, vec, rawI);
  load_run<NQ>(entropy + (size_t)b * ld, k0, Lw, vec, Hs);
  // centred moving average over the in-range taps, added left to right
  if (hp.smooth_radius == 1) {   // the default: the neighbours are in this lane or the next ones
    const float lI = __shfl_up_sync(kAll, rawI[NQ - 1], 1), rI = __shfl_down_sync(kAll, rawI[0], 1);
    const float lH = __shfl_up_sync(kAll, Hs[NQ - 1], 1), rH = __shfl_down_sync(kAll, Hs[0], 1);
    float hPrev = lH;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int k = k0 + q;
      const bool l = k > 0, r = k + 1 < Lw;
      const float iL = q ? rawI[q ? q - 1 : 0] : lI, iR = q + 1 < NQ ? rawI[q + 1 < NQ ? q + 1 : q] : rI;
      const float hR = q + 1 < NQ ? Hs[q + 1 < NQ ? q + 1 : q] : rH;
      float aI = l ? __fadd_rn(iL, rawI[q]) : rawI[q], aH = l ? __fadd_rn(hPrev, Hs[q]) : Hs[q];
      if (r) { aI = __fadd_rn(aI, iR); aH = __fadd_rn(aH, hR); }
      hPrev = Hs[q];
      const float n = (float)(1 + (l ? 1 : 0) + (r ? 1 : 0));
      Is[q] = k < Lw ? __fdiv_rn(aI, n) : 0.f;
      Hs[q] = k < Lw ? __fdiv_rn(aH, n) : 0.f;
    }
  } else {
    // (one word of padding per 32: lanes read at a stride of NQ words)
    auto at = [](int k) { return k + (k >> 5); };
#pragma unroll
    for (int q = 0; q < NQ; ++q) { sI[w][at(k0 + q)] = rawI[q]; sH[w][at(k0 + q)] = Hs[q]; }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int k = k0 + q;
      Is[q] = 0.f; Hs[q] = 0.f;
      if (k < Lw) {
        const int lo = max(0, k - hp.smooth_radius), hi = min(Lw - 1, k + hp.smooth_radius);
        float aI = sI[w][at(lo)], aH = sH[w][at(lo)];
        for (int j = lo + 1; j <= hi; ++j) { aI = __fadd_rn(aI, sI[w][at(j)]); aH = __fadd_rn(aH, sH[w][at(j)]); }
        const float n = (float)(hi - lo + 1);
        Is[q] = __fdiv_rn(aI, n); Hs[q] = __fdiv_rn(aH, n);
      }
    }
  }
  float hiI = -INFINITY, hiH = -INFINITY, nlI = -INFINITY, nlH = -INFINITY;   // maxima, and of the negated values
#pragma unroll
  for (int q = 0; q < NQ; ++q)
    if (k0 + q < Lw) {
      hiI = fmaxf(hiI, Is[q]); hiH = fmaxf(hiH, Hs[q]);
      nlI = fmaxf(nlI, -Is[q]); nlH = fmaxf(nlH, -Hs[q]);
    }
  if (hp.norm_mode != DC_NORM_NONE) {
    hiI = warp_max(hiI); hiH = warp_max(hiH);
    if (hp.norm_mode == DC_NORM_MINMAX) { nlI = -warp_max(nlI); nlH = -warp_max(nlH); }
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      Is[q] = normalise(Is[q], hiI, nlI, hp.norm_mode);
      Hs[q] = normalise(Hs[q], hiH, nlH, hp.norm_mode);
    }
  }
  float S[NQ];
  long long accS[NQ], accI[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const bool in = k0 + q < Lw;
    S[q] = in ? __fsub_rn(Is[q], __fmul_rn(hp.lambda, Hs[q])) : 0.f;
    const long long fS = in ? to_fixed(S[q]) : 0, fI = in ? to_fixed(rawI[q]) : 0;
    accS[q] = (q ? accS[q ? q - 1 : 0] : 0) + fS;
    accI[q] = (q ? accI[q ? q - 1 : 0] : 0) + fI;
  }
  const long long baseS = warp_scan(accS[NQ - 1]) - accS[NQ - 1], baseI = warp_scan(accI[NQ - 1]) - accI[NQ - 1];
  int first = Lw;
  float ci[NQ], cs[NQ];
#pragma unroll
  for (int q = NQ - 1; q >= 0; --q) {
    const long long tS = baseS + accS[q], tI = baseI + accI[q];
    if (k0 + q < Lw && ((hp.boundary_mode == DC_BOUNDARY_CUMULATIVE) ? (tS < 0) : (S[q] < 0.f))) first = k0 + q;
    ci[q] = from_fixed(tI);
    cs[q] = from_fixed(tS);
  }
  const int kstar = __reduce_min_sync(kAll, first);
  if (score) store_run<NQ>(score + o, k0, Lw, vec, S);
  if (cum_i) store_run<NQ>(cum_i + o, k0, Lw, vec, ci);
  if (cum_s) store_run<NQ>(cum_s + o, k0, Lw, vec, cs);
  if (lane == 0) block_len[b] = min(max(kstar, hp.L_min), Lw);
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
  auto aligned = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  const int vec = ld % 4 == 0 && max_window % 4 == 0 && aligned(influence) && aligned(entropy) && aligned(score) &&
                  aligned(cum_i) && aligned(cum_s);
  decide_launch(batch, max_window, [&](auto nq, dim3 grid, int threads) {
    k_boundary<decltype(nq)::value><<<grid, threads, 0, s>>>(influence, entropy, ld, batch, m, dl, hp, max_window, score,
                                                             cum_i, cum_s, block_len, vec);
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
    const float* __restrict__ conf, const int32_t* __restrict__ win_ids,
    const float* __restrict__ xlogp, const int32_t* __restrict__ block_len, int batch,
    const __grid_constant__ SeqMeta m, DevLens dl, Hyper hp, int mask_id, int max_window,
    uint8_t* __restrict__ sel_mask, int32_t* __restrict__ sel_idx, int32_t* __restrict__ sel_count) {
  constexpr int NA = 4;
  __shared__ __align__(16) int members[kSeqWarps][32 * NQ + NA];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int b = blockIdx.x * (blockDim.x >> 5) + w;
  if (b >= batch) return;
  const int W = len_of(dl.win_len, m.win_len, b);
  const int L = min(max(block_len[b], 0), W);
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
  const unsigned k_low = order_key(hp.tau_low), k_high = order_key(fmaxf(hp.tau_low, hp.tau_high));
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
}

static void select(const float* conf, const int32_t* win_ids, const float* xlogp, const int32_t* block_len, int batch,
                   const SeqMeta& m, const DevLens& dl, const Hyper& hp, int mask_id, int max_window,
                   uint8_t* sel_mask, int32_t* sel_idx, int32_t* sel_count, cudaStream_t s) {
  decide_launch(batch, max_window, [&](auto nq, dim3 grid, int threads) {
    k_select<decltype(nq)::value><<<grid, threads, 0, s>>>(conf, win_ids, xlogp, block_len, batch, m, dl, hp, mask_id,
                                                           max_window, sel_mask, sel_idx, sel_count);
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

__global__ void k_keep_block_len(int32_t* block_len, const PrevLen keep, int batch) {
  const int b = threadIdx.x;
  if (b < batch && keep.n[b] >= 0) block_len[b] = keep.n[b];
}

void launch_keep_block_len(int32_t* block_len, const PrevLen& keep, int batch, cudaStream_t s) {
  k_keep_block_len<<<1, DC_MAX_BATCH, 0, s>>>(block_len, keep, batch);
}

void launch_commit(int32_t* win_ids, const int32_t* pred_id, const uint8_t* sel_mask,
                   const int32_t* block_len, const SeqMeta& m, int mask_id, int max_window,
                   int32_t* remaining, cudaStream_t s) {
  k_commit<<<m.batch, kThreads, 0, s>>>(win_ids, pred_id, sel_mask, block_len, m, mask_id, max_window,
                                        remaining);
}

}  // namespace dc
