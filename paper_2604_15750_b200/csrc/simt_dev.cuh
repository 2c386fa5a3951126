// Device helpers shared by the CUDA-core kernels: element conversion, vector access, asynchronous
// copies, packed FMAs, the QKV epilogue and the per-position signals.
#pragma once
#include <math.h>

#include "kernels.h"

namespace dc {

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) {
  return __bfloat162float(v);
}
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// ---- 4-element vector loads / stores ------------------------------------------------------------
template <typename T> __device__ __forceinline__ void store4(T* dst, const float (&v)[4]);
template <> __device__ __forceinline__ void store4<float>(float* dst, const float (&v)[4]) {
  *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
}
template <> __device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16* dst,
                                                                   const float (&v)[4]) {
  __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
  *reinterpret_cast<uint2*>(dst) =
      make_uint2(*reinterpret_cast<uint32_t*>(&a), *reinterpret_cast<uint32_t*>(&b));
}
template <typename T> __device__ __forceinline__ void load4(const T* src, float (&v)[4]);
template <> __device__ __forceinline__ void load4<float>(const float* src, float (&v)[4]) {
  const float4 t = *reinterpret_cast<const float4*>(src);
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
template <> __device__ __forceinline__ void load4<__nv_bfloat16>(const __nv_bfloat16* src,
                                                                  float (&v)[4]) {
  const uint2 t = *reinterpret_cast<const uint2*>(src);
  const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&t.x);
  const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(&t.y);
  v[0] = __low2float(a); v[1] = __high2float(a); v[2] = __low2float(b); v[3] = __high2float(b);
}

template <typename T> struct GemmIo {
  static constexpr int kPiece = 16 / (int)sizeof(T);   // elements of a 16-byte copy
  static constexpr int kPad = kPiece;                  // row padding: no bank conflicts between 8 rows
};
__device__ __forceinline__ void cp_async16(void* dst, const void* src, int bytes) {   // the rest of the 16 bytes is zeroed
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
               ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack2(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void fma2(f2& d, f2 a, f2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ float sum2(f2 v) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
  return lo + hi;
}

// One rotated pair (features e and e + head_dim / 2 of a head) of activation row m: bias, rotation,
// store, and the copy into the context cache when the row belongs to an exported last block.
template <typename T, typename G>
__device__ __forceinline__ void simt_store_qkv(const G& g, int m, int head, int e, float y1, float y2) {
  const int hd = g.hd, half = hd >> 1;
  const int rv = g.m.rows, br = m % rv;   // (b, r): the RoPE table is shared by both variants
  if (g.bq != nullptr) {   // projection bias, before the rotation
    const T* bb = head < g.nq ? g.bq + head * hd : head < g.nq + g.nkv ? g.bk + (head - g.nq) * hd
                                                                       : g.bv + (head - g.nq - g.nkv) * hd;
    y1 += to_f<T>(bb[e]); y2 += to_f<T>(bb[half + e]);
  }
  const bool is_v = head >= g.nq + g.nkv;
  if (!is_v) {
    const float c = g.cos_sin[(size_t)br * hd + e], sn = g.cos_sin[(size_t)br * hd + half + e];
    const float t = y1 * c - y2 * sn;
    y2 = y2 * c + y1 * sn;
    y1 = t;
  }
  const T o1 = from_f<T>(y1), o2 = from_f<T>(y2);
  if (head < g.nq) {
    T* dst = g.q + (size_t)m * g.nq * hd + head * hd + e;
    dst[0] = o1; dst[half] = o2;
    return;
  }
  const int hk = is_v ? head - g.nq - g.nkv : head - g.nq;
  T* dst = (is_v ? g.v : g.k) + (size_t)m * g.nkv * hd + hk * hd + e;
  dst[0] = o1; dst[half] = o2;
  if (g.k_cache != nullptr && m < rv) {
    const int b = act_seq(g.m, br), r = br - g.m.row0[b];
    if (r < g.m.last_len[b]) {
      const size_t kv = (size_t)b * g.nkv + hk;
      const int key = g.m.ctx_len[b] + r;
      if (is_v) {
        g.v_cache[(kv * hd + e) * g.max_ctx + key] = o1;
        g.v_cache[(kv * hd + half + e) * g.max_ctx + key] = o2;
      } else {
        g.k_cache[(kv * g.max_ctx + key) * hd + e] = o1;
        g.k_cache[(kv * g.max_ctx + key) * hd + half + e] = o2;
      }
    }
  }
}


// ---- per-position signals from full logits ---------------------------------------------------------
// c = max_v p(v), yhat = argmax (lowest id on ties), H = lse - sum p z,
// I = sum p [(z - lse) - (z' - lse')] clamped at 0 (Eq. 3).  NT threads work on one window position.
// One pass: every thread keeps its own reference points and scales its sums when they move.
template <int NT> struct SignalsShared { float red[4][NT / 32], m[NT / 32], m2[NT / 32]; int i[NT / 32]; };
template <int NT, typename Sync>
__device__ __forceinline__ void signals_pos(const SimtSignals& sg, const SeqMeta& m, int p, int t, SignalsShared<NT>& sh,
                                            Sync&& sync) {
  const int b = p / m.W_cap, k = p % m.W_cap, V = sg.V;
  if (b >= m.batch || k >= m.win_len[b]) return;   // uniform over the NT threads
  const bool prev = (m.nv == 2);
  const float* z = sg.logits + (size_t)lm_row(m, 0, p) * V;
  const float* z2 = prev ? sg.logits + (size_t)lm_row(m, 1, p) * V : nullptr;
  const int skip = sg.forbid ? sg.mask_id : -1;
  float mx = -INFINITY, mx2 = -INFINITY;
  int am = 0x7fffffff;
  float sum[4] = {0.f, 0.f, 0.f, 0.f};   // S, A, D, S'
  auto four = [&](int v, const float (&a)[4], const float (&a2)[4], int n) {
    float top = -INFINITY, top2 = -INFINITY;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i < n && v + i != skip) {
        if (a[i] > fmaxf(mx, top)) am = v + i;     // ascending ids: the first maximum is kept
        top = fmaxf(top, a[i]);
        top2 = fmaxf(top2, a2[i]);
      }
    if (top > mx) {
      const float c = expf(mx - top);
      sum[0] *= c; sum[1] *= c; sum[2] *= c;
      mx = top;
    }
    if (prev && top2 > mx2) { sum[3] *= expf(mx2 - top2); mx2 = top2; }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i < n && v + i != skip) {
        const float e = a[i] == -INFINITY ? 0.f : expf(a[i] - mx);   // (the reference point may still be -inf)
        sum[0] += e;
        if (e > 0.f) {
          sum[1] = fmaf(e, a[i], sum[1]);
          if (prev) sum[2] = fmaf(e, a[i] - a2[i], sum[2]);
        }
        if (prev && a2[i] != -INFINITY) sum[3] += expf(a2[i] - mx2);
      }
  };
  // four logits at a time where the rows are 16-byte aligned
  if (V % 4 == 0) {
    float4 na = make_float4(0.f, 0.f, 0.f, 0.f), nq = na;
    auto fetch = [&](int v) {
      if (v >= V) return;
      na = __ldcg(reinterpret_cast<const float4*>(z + v));
      if (prev) nq = __ldcg(reinterpret_cast<const float4*>(z2 + v));
    };
    fetch(t * 4);
#pragma unroll 1
    for (int v = t * 4; v < V; v += NT * 4) {
      const float4 a = na, q = nq;
      fetch(v + NT * 4);
      const float av[4] = {a.x, a.y, a.z, a.w}, qv[4] = {q.x, q.y, q.z, q.w};
      four(v, av, qv, 4);
    }
  } else {
    for (int v = t; v < V; v += NT) {
      const float av[4] = {__ldcg(z + v)}, qv[4] = {prev ? __ldcg(z2 + v) : 0.f};
      four(v, av, qv, 1);
    }
  }
  const float own = mx, own2 = mx2;
  // reduce (max, lowest index) across the threads
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float om = __shfl_xor_sync(0xffffffffu, mx, o);
    const int oi = __shfl_xor_sync(0xffffffffu, am, o);
    if (om > mx || (om == mx && oi < am)) { mx = om; am = oi; }
    mx2 = fmaxf(mx2, __shfl_xor_sync(0xffffffffu, mx2, o));
  }
  const int w = t >> 5, l = t & 31;
  if (l == 0) { sh.m[w] = mx; sh.i[w] = am; sh.m2[w] = mx2; }
  sync();
  mx = sh.m[0]; am = sh.i[0]; mx2 = sh.m2[0];
  for (int i = 1; i < NT / 32; ++i) {
    if (sh.m[i] > mx || (sh.m[i] == mx && sh.i[i] < am)) { mx = sh.m[i]; am = sh.i[i]; }
    mx2 = fmaxf(mx2, sh.m2[i]);
  }
  const float c = own > -INFINITY ? expf(own - mx) : 0.f, c2 = own2 > -INFINITY ? expf(own2 - mx2) : 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    sum[i] = warp_sum(sum[i] * (i < 3 ? c : c2));
    if (l == 0) sh.red[i][w] = sum[i];
  }
  sync();
  if (t == 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      sum[i] = 0.f;
      for (int j = 0; j < NT / 32; ++j) sum[i] += sh.red[i][j];
    }
    // (no logit above -inf: not a sum of 0, whose 1 / S would be the highest confidence of all)
    const float S = mx > -INFINITY ? sum[0] : __int_as_float(0x7fffffff);
    const float lse = mx + logf(S);
    const float conf = 1.f / S;
    const float ent = lse - sum[1] / S;
    float infl = 0.f;
    if (prev && m.have_prev[b]) {
      const float lse2 = mx2 + logf(sum[3]);
      infl = fmaxf(sum[2] / S - lse + lse2, 0.f);
    }
    // no finite admissible logit (a NaN / inf hidden row): the argmax sentinel must not reach
    // the kernels that index the vocabulary matrix with the id
    if (am < 0 || am >= V || !isfinite(lse)) {
      am = sg.mask_id;
      if (sg.status) atomicMax(sg.status + b, (int)DC_ERR_NUMERIC);
    }
    const int wi = b * m.W_cap + k;
    sg.ws_pred[wi] = am; sg.ws_conf[wi] = conf; sg.ws_ent[wi] = ent; sg.ws_infl[wi] = infl; sg.ws_lse[wi] = lse;
    const SignalOut& out = sg.out;
    const int oi = b * out.max_window + k;
    if (out.pred_id) out.pred_id[oi] = am;
    if (out.conf) out.conf[oi] = conf;
    if (out.entropy) out.entropy[oi] = ent;
    if (out.influence) out.influence[oi] = infl;
    if (out.lse) out.lse[oi] = lse;
  }
}

}  // namespace dc
