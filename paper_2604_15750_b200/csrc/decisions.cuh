// Device side of the boundary rule, shared by the decision kernels and the fused CUDA-core step.
#pragma once
#include <math.h>

#include "kernels.h"

namespace dc {

constexpr int kMaxW = DC_MAX_WINDOW;  // 256
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
// barrier (8192 x 128: k_boundary 26 -> 13 us, k_select 222 -> 37 us against one block with a thread per
// position).  What bounds a call over many sequences is instruction issue and latency: 63 registers a
// thread let 32 warps of k_boundary on an SM, 48 let 40 of k_select, so 8192 sequences are 1.7 and 1.4 rounds; 63% and
// 52% of the issue slots are used, 6% and 24% of the DRAM throughput.  With few sequences - a step - every warp is a
// CTA of its own, so that they spread over the SMs.
constexpr int kSeqWarps = 8;          // sequences per CTA of a call with more sequences than kSpread
constexpr int kSpread = 4 * 148;

// NQ consecutive values of a row from position k0 on; positions >= n are 0 / not written.  SAME: the row may have been
// written earlier in this launch, by another CTA: it is read past L1, and never as constant data
template <int NQ, bool SAME>
__device__ __forceinline__ void load_run(const float* row, int k0, int n, int vec, float (&v)[NQ]) {
  constexpr int V = NQ >= 4 ? 4 : 2;
  auto get = [](const auto* p) { return SAME ? __ldcg(p) : *p; };
#pragma unroll
  for (int q = 0; q < NQ; q += V) {
    if (vec && k0 + q + V <= n) {
      if (V == 4) {
        const float4 t = get(reinterpret_cast<const float4*>(row + k0 + q));
        v[q] = t.x; v[q + 1] = t.y; v[q + V / 2] = t.z; v[q + V - 1] = t.w;
      } else {
        const float2 t = get(reinterpret_cast<const float2*>(row + k0 + q));
        v[q] = t.x; v[q + 1] = t.y;
      }
    } else {
#pragma unroll
      for (int u = 0; u < V; ++u) v[q + u] = k0 + q + u < n ? get(row + k0 + q + u) : 0.f;
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
__device__ __forceinline__ float lanes_max(float v) {   // exact, order-free
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kAll, v, o));
  return v;
}
// inclusive prefix sum over the lanes
__device__ __forceinline__ long long lanes_scan(long long v) {
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

// What the warps of a sequence tell one another (TW of them).
template <int TW>
struct BoundaryTeam { float top[4][TW]; long long sum[2][TW]; int first[TW]; };

// The boundary rule for sequence b, by TW warps that are a CTA of their own, or one warp; sI, sH: 33 * NQ * TW floats of
// shared memory each.  SAME: see load_run.
template <int NQ, int TW = 1, bool SAME = false>
__device__ __forceinline__ void boundary_seq(const float* influence, const float* entropy, int b, const SeqMeta& m,
                                             const DevLens& dl, const Hyper& hp, const BoundaryIo& io, float* sI, float* sH,
                                             BoundaryTeam<TW>* team = nullptr) {
  const int lane = threadIdx.x & (32 * TW - 1), ld = io.ld, max_window = io.max_window, vec = io.vec;
  const int warp = TW > 1 ? lane >> 5 : 0;
  auto sync = [] { if (TW > 1) __syncthreads(); else __syncwarp(); };
  float *score = io.score, *cum_i = io.cum_i, *cum_s = io.cum_s;
  int32_t* block_len = io.block_len;
  const int Lw = max(0, min(min(hp.L_max, len_of(dl.remain, m.remain, b)), len_of(dl.win_len, m.win_len, b)));
  const size_t o = (size_t)b * max_window;
  if (!len_of(dl.have_prev, m.have_prev, b)) {  // cold start: the first block uses L_min
    for (int k = lane; k < Lw; k += 32 * TW) {
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
  load_run<NQ, SAME>(influence + (size_t)b * ld, k0, Lw, vec, rawI);
  load_run<NQ, SAME>(entropy + (size_t)b * ld, k0, Lw, vec, Hs);
  // centred moving average over the in-range taps, added left to right
  if (TW == 1 && hp.smooth_radius == 1) {   // the default: the neighbours are in this lane or the next ones
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
    for (int q = 0; q < NQ; ++q) { sI[at(k0 + q)] = rawI[q]; sH[at(k0 + q)] = Hs[q]; }
    sync();
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int k = k0 + q;
      Is[q] = 0.f; Hs[q] = 0.f;
      if (k < Lw) {
        const int lo = max(0, k - hp.smooth_radius), hi = min(Lw - 1, k + hp.smooth_radius);
        float aI = sI[at(lo)], aH = sH[at(lo)];
        for (int j = lo + 1; j <= hi; ++j) { aI = __fadd_rn(aI, sI[at(j)]); aH = __fadd_rn(aH, sH[at(j)]); }
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
    hiI = lanes_max(hiI); hiH = lanes_max(hiH);
    if (hp.norm_mode == DC_NORM_MINMAX) { nlI = lanes_max(nlI); nlH = lanes_max(nlH); }
    if (TW > 1) {
      if ((lane & 31) == 0) { team->top[0][warp] = hiI; team->top[1][warp] = hiH; team->top[2][warp] = nlI; team->top[3][warp] = nlH; }
      sync();
#pragma unroll
      for (int i = 0; i < TW; ++i) {
        hiI = fmaxf(hiI, team->top[0][i]); hiH = fmaxf(hiH, team->top[1][i]);
        nlI = fmaxf(nlI, team->top[2][i]); nlH = fmaxf(nlH, team->top[3][i]);
      }
    }
    nlI = -nlI; nlH = -nlH;
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
  long long baseS = lanes_scan(accS[NQ - 1]), baseI = lanes_scan(accI[NQ - 1]);
  if (TW > 1) {
    if ((lane & 31) == 31) { team->sum[0][warp] = baseS; team->sum[1][warp] = baseI; }
    sync();
#pragma unroll
    for (int i = 0; i + 1 < TW; ++i)
      if (i < warp) { baseS += team->sum[0][i]; baseI += team->sum[1][i]; }
  }
  baseS -= accS[NQ - 1]; baseI -= accI[NQ - 1];
  int first = Lw;
  float ci[NQ], cs[NQ];
#pragma unroll
  for (int q = NQ - 1; q >= 0; --q) {
    const long long tS = baseS + accS[q], tI = baseI + accI[q];
    if (k0 + q < Lw && ((hp.boundary_mode == DC_BOUNDARY_CUMULATIVE) ? (tS < 0) : (S[q] < 0.f))) first = k0 + q;
    ci[q] = from_fixed(tI);
    cs[q] = from_fixed(tS);
  }
  int kstar = __reduce_min_sync(kAll, first);
  if (TW > 1) {
    if ((lane & 31) == 0) team->first[warp] = kstar;
    sync();
#pragma unroll
    for (int i = 0; i < TW; ++i) kstar = min(kstar, team->first[i]);
  }
  if (score) store_run<NQ>(score + o, k0, Lw, vec, S);
  if (cum_i) store_run<NQ>(cum_i + o, k0, Lw, vec, ci);
  if (cum_s) store_run<NQ>(cum_s + o, k0, Lw, vec, cs);
  if (lane == 0) block_len[b] = min(max(kstar, hp.L_min), Lw);
}

}  // namespace dc
